"""The residuals that the mixed form reports are the true ones, on an operator whose smallest eigenvalue
(|lambda| = 0.003 at norm 7.1) makes the corrections large against the residuals they remove.

Bound: the report may differ from the residuals formed here in FP64 by the accuracy of the float-float
stencil, 1e-13 of a result's largest entry per application (test_gpu_stencil.py), and 1e-3 of itself."""
import numpy as np
import pytest

import oracle as O
import seeded_inputs as si

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIMS, MASS, PERIODIC = (4, 3, 4, 3), -0.02660769534298367, (0, 0, 0, 0)


@pytest.mark.parametrize("links,tol,k_refine", [(0, 1e-8, 0), (0, 1e-10, 0), (0, 1e-10, 16), (0, 1e-11, 0),
                                                (0, 1e-11, 16), (2, 1e-8, 0), (2, 1e-8, 16)])
def test_reported_residual_is_true(links, tol, k_refine):
    import paper_0910_2927_gb300 as pkg
    U = si.random_su3_links(DIMS, 0.1, 91)
    b = si.gaussian_block(DIMS, 2, 92)
    sigma, omega = pkg.kenney_laub(20, 1.0 / np.sqrt(0.003 * 7.1))
    with pkg.SignContext(DIMS, mu=0.0, antiperiodic=PERIODIC) as ctx:
        ctx.set_kernel_mass(MASS)
        ctx.load_gauge(torch.from_numpy(U).cuda())
        ctx.set_rational(sigma, omega)
        ctx.set_restart(k=40, tol=tol, max_cycles=400)
        ctx.set_precision(pkg.PREC_MIXED, 1e-8, links)
        ctx.set_refinement(k_refine, 0)
        _, xs, rep = ctx.apply(torch.from_numpy(b).cuda(), shifts=True)
    A = O.dense_hw(DIMS, U, 0.0, MASS, PERIODIC)
    bt = b @ A.T
    norm = np.linalg.norm(bt, axis=1)
    worst = noise = 0.0
    for s, x in zip(sigma, xs.cpu().numpy()):
        ax = x @ A.T
        aax = ax @ A.T
        worst = max(worst, np.max(np.linalg.norm(bt - aax + s * x, axis=1) / norm))
        entry = np.sqrt(x.shape[1]) * (np.abs(aax).max(1) + 7.2 * np.abs(ax).max(1))
        noise = max(noise, np.max(1e-13 * entry / norm))
    assert abs(rep["err_est"] - worst) < 1e-3 * worst + noise
    assert rep["status"] == (0 if rep["err_est"] <= tol else 3)
