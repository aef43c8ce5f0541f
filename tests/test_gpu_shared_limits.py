"""First calls of a process whose kernels take just under 48 KB of dynamic
shared memory: with the static arrays that is more than a launch may use
without asking.  Each structure runs in a process of its own (what one call
has been allowed, later ones of the process keep); moments against the
oracle, 1e-9 relative (FP64)."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1803_07491_gb300 import inputs as I
from conftest import oracle_model, oracle_settings

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MODELS = {"s": I.MODEL_S, "d": I.MODEL_D, "sd": I.MODEL_SD}


def workload(name):
    """Structures whose largest cluster gives 48,524, 49,020, 49,120 and 48,784 bytes."""
    model, n_mom, cells, sigma, seed, nc = {
        "d": ("d", 7, (2, 2, 2), 0.2, 22, False), "s": ("s", 9, (2, 2, 2), 0.2, 45, False),
        "sd_noncollinear": ("sd", 7, (3, 3, 3), 0.03, 11, True),
        "d_noncollinear": ("d", 7, (2, 2, 2), 0.2, 18, True)}[name]
    pos, cell = I.bcc_jittered(*cells, sigma, seed)
    w = I.with_run(I.Workload(name, pos, cell, (1, 1, 1), MODELS[model], I.RunParams(n_e={"s": 0.7, "d": 6.8, "sd": 8.0}[model])),
                   n_mom=n_mom)
    return I.with_run(w, n_spin=2, stoner_I=0.8, noncollinear=True) if nc else w


def directions(w):
    return I.random_directions(w.n_atoms, 3), np.full(w.n_atoms, 0.5)


CHILD = """
import sys
import numpy as np, torch
sys.path[:0] = [{root!r}, {tests!r}]
from paper_1803_07491_gb300 import bop
from test_gpu_shared_limits import workload, directions
w = workload({name!r})
ctx = bop.Context(w.model, w.run, "fp64")
ctx.build(w.pos, w.cell, w.pbc)
m = None
if w.run.noncollinear:
    s, m = directions(w)
    ctx.set_spin_directions(s)
    m = torch.as_tensor(m, dtype=torch.float64, device="cuda")
ctx.energy(m=m)
np.save({out!r}, bop.bop_get_orbital_state(ctx.h, w.run.n_spin * w.n_atoms * w.model.norb, w.run.n_mom)["mu"].cpu().numpy())
"""


@pytest.mark.parametrize("name", ["d", "s", "sd_noncollinear", "d_noncollinear"])
def test_first_call_just_under_48_kilobytes(ob, tmp_path, name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_07491_gb300 import build
    build.build()
    out = str(tmp_path / "mu.npy")
    code = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"), name=name, out=out)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    w = workload(name)
    kw = {}
    if w.run.noncollinear:
        kw["spin_dir"], kw["m_init"] = directions(w)
    ref = ob.evaluate(oracle_model(w.model), oracle_settings(w.run), w.pos, w.cell, w.pbc,
                      want_forces=False, **kw)
    mu = np.load(out)
    ref = np.asarray(ref["mu"]).reshape(mu.shape)
    assert np.max(np.abs(mu - ref) / np.maximum(1.0, np.abs(ref))) < 1e-9
