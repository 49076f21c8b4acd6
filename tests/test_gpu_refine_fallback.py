"""Where the mixed form's BiCGStab corrections hand a system to restarted FOM, and where they stop.

The library's log (SGN_DEBUG) says how many systems went where; launch shapes are fixed (SGN_NO_TUNE), so
that the same numbers come out on every run."""
import json
import os
import re
import subprocess
import sys

import numpy as np
import pytest

import oracle as O
import seeded_inputs as si

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SCRIPT = """
import json, sys
import numpy as np, torch
import paper_0910_2927_gb300 as pkg, seeded_inputs as si
a = json.loads(sys.argv[1])
dims = tuple(a["dims"])
U = torch.from_numpy(si.random_su3_links(dims, a["spread"], 91)).cuda()
b = torch.from_numpy(si.gaussian_block(dims, a["nrhs"], 92)).cuda()
with pkg.SignContext(dims, mu=a["mu"], antiperiodic=(0, 0, 0, a["ap"])) as ctx:
    ctx.set_kernel_mass(a["mass"])
    ctx.load_gauge(U)
    ctx.set_rational(*pkg.kenney_laub(a["s"], a["c"]))
    ctx.set_restart(k=a["k"], tol=a["tol"], max_cycles=a["max_cycles"])
    ctx.set_precision(pkg.PREC_MIXED, 1e-8, 0)
    x, rep = ctx.apply(b)
np.save(a["out"], x.cpu().numpy())
print(json.dumps({k: rep[k] for k in ("status", "refine_rounds", "err_est")}))
"""
ROUND = re.compile(r"round (\d+): .* (\d+) of (\d+) systems above tol, (\d+) stuck")


def _solve(tmp_path, dims, nrhs=2, mu=0.0, mass=-1.6, ap=1, spread=0.7, s=20, c=1.0, k=40, tol=1e-8, max_cycles=400):
    a = dict(dims=dims, nrhs=nrhs, mu=mu, mass=mass, ap=ap, spread=spread, s=s, c=c, k=k, tol=tol,
             max_cycles=max_cycles, out=str(tmp_path / "x.npy"))
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, SGN_DEBUG="1", SGN_NO_TUNE="1", PYTHONPATH=root)
    p = subprocess.run([sys.executable, "-c", SCRIPT, json.dumps(a)], env=env, cwd=root, capture_output=True, text=True,
                       timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    return json.loads(p.stdout.strip().splitlines()[-1]), p.stderr, np.load(a["out"])


@pytest.mark.parametrize("mu", [0.0, 0.3])
def test_rounds_end_where_nothing_is_gained(tmp_path, mu):
    """Tolerances whose aims (a fraction of the tolerance) lie below what the residuals resolve: one round
    that gains nothing ends the refinement once every system is below the tolerance."""
    rep, _, _ = _solve(tmp_path, (4, 3, 5, 4), mu=mu, c=1.0 / np.sqrt(0.2 * 8.0), tol=3e-14)
    assert rep["status"] == 0 and rep["refine_rounds"] <= 4


def test_columns_without_gain_go_to_fom(tmp_path):
    """An operator with |lambda| = 0.0015 and shifts down to 5e-7: BiCGStab columns whose recursive residual
    converges and whose true one does not are solved by FOM in the next round."""
    seen = 0
    for s, low in ((20, 1e-4), (32, 3e-4), (32, 1e-4)):
        rep, log, _ = _solve(tmp_path, (4, 3, 4, 3), mass=-0.006666691938058431, ap=0, spread=0.05, s=s,
                             c=1.0 / np.sqrt(low * 7.1))
        assert rep["status"] == 0 and rep["err_est"] <= 1e-8
        stuck = 0
        for part in re.split(r"(?=\[sgn mixed\] round)", log):
            m = ROUND.search(part)
            if not m:
                continue
            if int(m[4]) > stuck:  # newly stuck: this round has a FOM batch
                seen += int(m[4]) - stuck
                assert ", FOM)" in part
            stuck = int(m[4])
    assert seen > 0


@pytest.mark.parametrize("max_cycles", [2, 3])
def test_iteration_cap_reached_by_some_columns(tmp_path, max_cycles):
    """BiCGStab's cap (16 max_cycles / 2 iterations) is reached by the small shifts only: their columns are
    left out of the batch's update and solved by FOM, the others are corrected; x meets the bound of
    test_gpu_refine.py."""
    dims, tol = (3, 4, 2, 4), 1e-9
    sigma, omega = O.kenney_laub(12, 0.5)
    rep, log, x = _solve(tmp_path, dims, nrhs=3, mu=0.2, spread=0.6, s=12, c=0.5, k=20, tol=tol,
                         max_cycles=max_cycles)
    split = [(int(n), int(f)) for n, f in re.findall(r"\((\d+) systems\): \d+ iterations, (\d+) to FOM", log)]
    assert any(0 < f < n for n, f in split), split
    assert rep["status"] == 0 and rep["err_est"] <= tol
    U = si.random_su3_links(dims, 0.6, 91)
    b = si.gaussian_block(dims, 3, 92)
    A = O.dense_hw(dims, U, 0.2)
    for r in range(3):
        ref = O.deflated_target(A, b[r], sigma, omega)
        assert np.linalg.norm(x[r] - ref) < 1e-7 * np.linalg.norm(ref)
