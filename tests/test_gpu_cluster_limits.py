"""The cluster builder at the limits of what its records hold: image indices
of a byte, and sort keys of 32 bits."""
import numpy as np
import pytest

from paper_1803_07491_gb300 import inputs as I
from conftest import oracle_model

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bop():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_07491_gb300 import build, bop as b
    build.build()
    return b


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("reach", [15, 16])
def test_chain_of_images(bop, axis, reach):
    """One atom that sees `reach` images on either side along one axis: eight
    hops reach image 8 reach, which is 120, or 128 and refused."""
    length = np.full(3, 40.0)
    length[axis] = I.MODEL_S.rc / (reach + 0.5)
    pbc = [int(a == axis) for a in range(3)]
    ctx = bop.Context(I.MODEL_S, I.RunParams(n_e=0.7, n_mom=17), "fp64")
    args = (np.array([[0.1, 0.1, 0.1]]), np.diag(length), pbc)
    if 8 * reach <= 127:
        assert ctx.build(*args)["max_cluster"] == 16 * reach + 1
    else:
        with pytest.raises(bop.BopError) as e:
            ctx.build(*args)
        assert e.value.status == bop.BOP_ERR_OVERFLOW
        ok = ctx.build(args[0], np.diag(length * np.where(np.array(pbc) == 1, 16.5 / 15.5, 1.0)), pbc)
        assert ok["max_cluster"] == 241
    ctx.close()
