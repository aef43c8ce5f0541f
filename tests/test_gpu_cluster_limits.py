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


@pytest.mark.parametrize("nx", [365, 366])
def test_sort_keys_below_and_above_the_codes(bop, ob, nx):
    """A slab one bcc cell thick: 63 image codes per atom, several images of an
    atom in a level, and 265,720 / 266,448 atoms around the 266,305 whose codes
    fit 32 bits.  Clusters of scattered centres against the oracle's (on a patch
    of the slab around the centre), and two moments, which count neighbours."""
    pos, cell = I.bcc_cell(nx, 364, 1)
    rng = np.random.default_rng(9)
    pos = I.jittered(pos, cell, (1, 1, 1), 0.03, rng)
    n = len(pos)
    ctx = bop.Context(I.MODEL_S, I.RunParams(n_e=0.7, n_mom=5), "fp64")
    ctx.build(pos, cell, (1, 1, 1))
    m = oracle_model(I.MODEL_S)
    box = np.diag(cell)
    for a in (0, 1, n // 2, n - 1, *rng.integers(0, n, 4)):
        # the patch: atoms within 11 Angstrom along x and y (two hops reach 7.2), in their order
        d = pos[:, :2] - pos[a, :2]
        wrap = np.round(d / box[:2])
        near = np.flatnonzero(np.all(np.abs(d - wrap * box[:2]) < 11.0, axis=1))
        shift = np.concatenate([-wrap[near], np.zeros((len(near), 1))], 1).astype(int)
        p = pos[near] + shift * box
        lo = np.array([*(pos[a, :2] - 12.0), 0.0])
        pcell = np.diag([24.0, 24.0, box[2]])
        nbr = ob.neighbors(p - lo, pcell, (0, 0, 1), m.rc)
        ra, ri, rl = ob.cluster(int(np.flatnonzero(near == a)[0]), 2, nbr)
        # back to the atoms and images of the whole slab, in canonical order
        ga, gi = near[ra], ri + shift[ra] - shift[near == a]
        key = np.lexsort((gi[:, 2], gi[:, 1], gi[:, 0], ga, np.searchsorted(rl, np.arange(len(ra)), side="right")))
        sa, si, lev = bop.bop_get_cluster(ctx.h, int(a), 2, len(ra))
        assert np.array_equal(lev.cpu().numpy(), rl)
        assert np.array_equal(sa.cpu().numpy(), ga[key])
        assert np.array_equal(si.cpu().numpy(), gi[key])
    mu = bop.bop_moments(ctx.h, 1, n, 1, 5).cpu().numpy()[0, :, 0]
    atoms, dist, blocks = bop.bop_get_bonds(ctx.h, 1)
    i, j = atoms.cpu().numpy().T.astype(int)
    h2 = blocks.cpu().numpy().ravel() ** 2
    ref = np.bincount(i, h2, n) + np.bincount(j, h2, n)
    assert np.max(np.abs(mu[:, 2] - ref)) < 1e-10 * ref.max()
    ctx.close()
