"""The mixed form does not depend on the size of the right-hand side: a power of two times b gives the
same power of two times x, bit for bit (every norm is scaled exactly, and nothing that a result depends
on leaves the range of its type), by the default corrections and by restarted FOM."""
import numpy as np
import pytest

import seeded_inputs as si

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims,nrhs,mu", [((4, 3, 5, 4), 2, 0.3), ((6, 6, 6, 6), 1, 0.0)])
@pytest.mark.parametrize("k_refine", [0, 16])
def test_scaled_right_hand_side(dims, nrhs, mu, k_refine):
    import paper_0910_2927_gb300 as pkg
    U = si.random_su3_links(dims, 0.7, 95)
    b = torch.from_numpy(si.gaussian_block(dims, nrhs, 96)).cuda()
    with pkg.SignContext(dims, mu=mu) as ctx:
        ctx.load_gauge(torch.from_numpy(U).cuda())
        ctx.set_rational(*pkg.kenney_laub(20, 1.0 / np.sqrt(0.2 * 8.1)))
        ctx.set_restart(k=40, tol=1e-10, max_cycles=500)
        ctx.set_precision(pkg.PREC_MIXED, 1e-8, 0)
        ctx.set_refinement(k_refine, 0)
        x, rep = ctx.apply(b)
        assert rep["status"] == 0
        for e in (-46, -33, -20, 40):
            y, r = ctx.apply(b * 2.0 ** e)
            assert r["status"] == 0
            assert (r["cycles"], r["refine_rounds"], r["refine_cycles"]) == (rep["cycles"], rep["refine_rounds"],
                                                                             rep["refine_cycles"])
            assert torch.equal(y, x * 2.0 ** e)
