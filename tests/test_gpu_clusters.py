"""GPU clusters (the linked-cell table builder and the general one it hands
over to) against the oracle: sites and levels bit for bit, and the FP64
moments, which walk the adjacency, to 1e-10 relative.  The structures sit at
the builder's edges: cells smaller than the cutoff (many images of one atom),
free boundaries, triclinic cells, rows of 16 / 17 / 32 / 33 neighbours, one
hop and eight hops, clusters that outgrow a capacity tier, the path cut, and
a crowded linked cell."""
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


def _shell(n, radius, seed):
    """A centre with n atoms on a sphere (free boundaries): its row has n entries."""
    k = np.arange(n) + 0.5
    ph, z = np.pi * (1 + 5 ** 0.5) * k, 1 - 2 * k / n
    s = np.sqrt(1 - z * z)
    p = radius * np.stack([s * np.cos(ph), s * np.sin(ph), z], 1)
    rng = np.random.default_rng(seed)
    return np.concatenate([np.zeros((1, 3)), p + rng.normal(0, 0.02, p.shape)]) + 15.0, np.eye(3) * 30.0, (0, 0, 0)


def _triclinic(seed):
    pos, cell = I.bcc_cell(3, 4, 5)
    F = np.array([[1.0, 0.25, -0.1], [0.0, 0.97, 0.3], [0.05, 0.0, 1.02]])
    return I.jittered(pos @ F, cell @ F, (1, 1, 1), 0.05, np.random.default_rng(seed)), cell @ F, (1, 1, 1)


def _structure(name):
    if name.startswith("shell"):
        return _shell(int(name[5:]), 3.3, 3)
    if name == "one":  # one atom, cell smaller than the cutoff
        return np.array([[0.3, 0.2, 0.1]]), np.eye(3) * 2.6, (1, 1, 1)
    if name == "thin":  # two cells along x, one along y, free along z
        p, c = I.bcc_jittered(3, 1, 4, 0.05, 5)
        c = c.copy()
        c[2, 2] += 9.0
        return p, c, (1, 1, 0)
    if name == "triclinic":
        return _triclinic(6)
    if name == "crowded":  # a dense clump in a large cell: many atoms in one linked cell
        rng = np.random.default_rng(8)
        g = np.stack(np.meshgrid(*[np.arange(3)] * 3, indexing="ij"), -1).reshape(-1, 3) * 1.9
        return g + rng.normal(0, 0.05, g.shape) + 1.0, np.eye(3) * 40.0, (1, 1, 1)
    n = {"bcc2": (2, 2, 2), "bcc5": (5, 4, 6), "bcc9": (9, 9, 9)}[name]
    return (*I.bcc_jittered(*n, 0.05, 4), (1, 1, 1))


@pytest.mark.parametrize("name,n_mom,r_path", [
    ("one", 9, 0.0), ("one", 17, 0.0), ("thin", 9, 0.0), ("triclinic", 9, 0.0), ("triclinic", 13, 0.0),
    ("shell16", 5, 0.0), ("shell17", 5, 0.0), ("shell32", 5, 0.0), ("shell33", 5, 0.0), ("crowded", 9, 0.0),
    ("bcc2", 3, 0.0), ("bcc2", 17, 0.0), ("bcc5", 11, 0.0), ("bcc5", 13, 5.5), ("bcc9", 7, 0.0), ("bcc9", 7, 4.5)])
def test_clusters_and_moments_match_oracle(bop, ob, name, n_mom, r_path):
    pos, cell, pbc = _structure(name)
    run = I.RunParams(n_e=0.7, n_mom=n_mom, r_path=r_path)
    m = oracle_model(I.MODEL_S)
    nbr = ob.neighbors(pos, cell, pbc, m.rc).with_path_radius(pos, cell, r_path)
    K = (n_mom - 1) // 2
    ctx = bop.Context(I.MODEL_S, run, "fp64")
    for _ in range(2):  # the second build starts at the capacity tier the first one found
        st = ctx.build(pos, cell, pbc)
        sites = 0
        for a in range(0, len(pos), max(1, len(pos) // 40)):
            ra, ri, rl = ob.cluster(a, K, nbr)
            sa, si, lev = bop.bop_get_cluster(ctx.h, a, K, len(ra))
            assert np.array_equal(lev.cpu().numpy(), rl)
            assert np.array_equal(sa.cpu().numpy(), ra)
            assert np.array_equal(si.cpu().numpy(), ri)
            sites = max(sites, len(ra))
        assert st["max_cluster"] >= sites
        mu = bop.bop_moments(ctx.h, 1, len(pos), 1, n_mom).cpu().numpy()[0]
        ref = ob.moments(nbr, ob.blocks(m, pos, cell, nbr), np.zeros((len(pos), 1)), n_mom)
        assert np.max(np.abs(mu - ref) / np.maximum(1.0, np.abs(ref).max(axis=(0, 1)))) < 1e-10
    ctx.close()
