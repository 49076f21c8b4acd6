"""Refinement of the mixed form by BiCGStab (bicgstab.cu) and by restarted FOM: both bring every shifted
system below the tolerance, on field counts and lattices that leave the kernels' tiles ragged, in
batches smaller than the systems to correct, and for columns that are zero.

Bound on x: the shifted systems' residuals are below tol ||b~||, which leaves at most
sum_i |omega_i| tol ||b~|| / |A^2 - sigma_i| in x; on these lattices (|lambda| > 0.1 after deflation or
without) that is below 1e-7 ||x|| at tol 1e-10 by two orders of magnitude."""
import numpy as np
import pytest

import oracle as O
import seeded_inputs as si

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((3, 2, 5, 3), 3), ((3, 4, 2, 4), 13)])
@pytest.mark.parametrize("k_refine,batch,links", [(0, 0, 0), (0, 7, 0), (0, 0, 1), (0, 0, 2), (12, 0, 0)])
def test_refinement_meets_tolerance(dims, nrhs, k_refine, batch, links):
    import paper_0910_2927_gb300 as pkg
    mu = 0.2
    U = si.random_su3_links(dims, 0.6, 71)
    sigma, omega = pkg.kenney_laub(12, 0.5)
    b = si.gaussian_block(dims, nrhs, 72)
    if nrhs > 1:
        b[1] = 0.0  # a zero column converges at once
    with pkg.SignContext(dims, mu=mu) as ctx:
        ctx.load_gauge(torch.from_numpy(U).cuda())
        ctx.set_rational(sigma, omega)
        ctx.set_restart(k=20, tol=1e-10, max_cycles=2000)
        ctx.set_precision(pkg.PREC_MIXED, 1e-8, links)
        ctx.set_refinement(k_refine, batch)
        bd = torch.from_numpy(b).cuda()
        x, rep = ctx.apply(bd)
        x2, _ = ctx.apply(bd)
    assert rep["status"] == 0 and rep["err_est"] <= 1e-10
    assert torch.equal(x, x2)
    x = x.cpu().numpy()
    A = O.dense_hw(dims, U, mu)
    for r in {0, nrhs - 1}:
        ref = O.deflated_target(A, b[r], sigma, omega)
        assert np.linalg.norm(x[r] - ref) < 1e-7 * np.linalg.norm(ref)
    if nrhs > 1:
        assert not np.any(x[1])
