"""The structure build's batched small jobs (counters zeroed, prefix sums and
host reads in one launch each) at the sizes where they change hands: prefix
sums of one block end at 8,192 elements."""
import numpy as np
import pytest

from paper_1803_07491_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bop():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_07491_gb300 import build, bop as b
    build.build()
    return b


@pytest.mark.parametrize("cells", [(1, 1, 1), (16, 16, 15), (16, 16, 16), (17, 16, 16)])
def test_build_at_the_prefix_sum_limits(bop, cells):
    """2, 7,680, 8,192 (8,193 sums) and 8,704 atoms, built twice in one context with
    a smaller structure between: a perfect bcc crystal has 14 neighbours in
    two shells and clusters of 15 sites at one hop, whatever its size."""
    run = I.RunParams(n_e=0.7, n_mom=3)
    ctx = bop.Context(I.MODEL_S, run, "fp64")
    for c in (cells, (3, 3, 3), cells):
        pos, cell = I.bcc_cell(*c)
        n = len(pos)
        st = ctx.build(pos, cell, (1, 1, 1))
        assert st["n_edges"] == 14 * n and st["n_bonds"] == 7 * n and st["n_sites"] == 15 * n
        assert st["max_cluster"] == 15 and st["moment_products"] == 14 * n
        row, col, img = bop.bop_get_neighbors(ctx.h)
        assert np.array_equal(row.cpu().numpy(), 14 * np.arange(n + 1))
        mu = bop.bop_moments(ctx.h, 1, n, 1, 3).cpu().numpy()
        assert np.all(np.abs(mu - mu[:, :1]) < 1e-12 * np.abs(mu).max())
    ctx.close()
