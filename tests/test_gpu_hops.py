"""The stencil with a lane per hop (hops.cuh): FP64 with a row of the link per warp and with whole links,
in one-warp and four-warp CTAs, FP32 with every link storage as a fixed launch shape; natural and packed
fields, both directions, site counts that leave the last tile ragged; and the float-float stencil on
packed fields, which equals the natural-order result.

Bounds: those of the other stencil kernels (test_gpu_stencil.py)."""
import numpy as np
import pytest

import oracle as O
import seeded_inputs as si

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _ctx(dims, U, mu, ap):
    import paper_0910_2927_gb300 as pkg
    ctx = pkg.SignContext(dims, mu=mu, antiperiodic=ap)
    ctx.load_gauge(torch.from_numpy(U).cuda())
    return ctx


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((3, 5, 3, 7), 1), ((3, 5, 3, 7), 5), ((7, 5, 9, 6), 1),
                                       ((7, 5, 9, 6), 6)])
@pytest.mark.parametrize("mu,ap", [(0.3, (0, 0, 0, 1)), (-0.9, (1, 0, 1, 0)), (60.0, (0, 1, 0, 1))])
@pytest.mark.parametrize("float_float", [False, True])
def test_fp64_lane_per_hop(dims, nrhs, mu, ap, float_float):
    U = si.random_su3_links(dims, 0.7, 81)
    b = si.gaussian_block(dims, nrhs, 82)
    if float_float and mu > 1.0:
        pytest.skip("e^60 leaves the float-float stencil's FP32 range")
    with _ctx(dims, U, mu, ap) as ctx:
        bd = torch.from_numpy(b).cuda()
        for adj in (False, True):
            out = ctx.hw(bd, adjoint=adj, float_float=float_float)
            pk = ctx.unpack(ctx.hw(ctx.pack(bd), adjoint=adj, packed=True, float_float=float_float))
            assert torch.equal(out, pk)
            for r in {0, nrhs - 1}:
                ref = O.hw(dims, U, b[r], -mu if adj else mu, -1.6, ap)
                np.testing.assert_allclose(out[r].cpu().numpy(), ref, rtol=0, atol=1e-13 * np.abs(ref).max())


@pytest.mark.parametrize("links,tol", [(0, 2e-6), (1, 2e-2), (2, 3e-3)])
@pytest.mark.parametrize("shape", ["32,1,1,5", "32,3,1,5"])
@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((3, 5, 3, 7), 5), ((7, 5, 9, 6), 3)])
def test_fp32_lane_per_hop(dims, nrhs, shape, links, tol, monkeypatch):
    import paper_0910_2927_gb300 as pkg
    monkeypatch.setenv("SGN_STENCIL_SHAPE", shape)
    mu, ap = 0.4, (0, 1, 0, 1)
    U = si.random_su3_links(dims, 0.7, 83)
    b = si.gaussian_block(dims, nrhs, 84)
    with _ctx(dims, U, mu, ap) as ctx:
        ctx.set_precision(pkg.PREC_MIXED, 1e-8, links)
        bd = torch.from_numpy(b.astype(np.complex64)).cuda()
        for adj in (False, True):
            out = ctx.hw(bd, precision=pkg.PREC_MIXED, adjoint=adj)
            pk = ctx.hw(ctx.pack(bd, pkg.PREC_MIXED), precision=pkg.PREC_MIXED, adjoint=adj, packed=True)
            assert torch.equal(out, ctx.unpack(pk, pkg.PREC_MIXED))
            for r in {0, nrhs - 1}:
                ref = O.hw(dims, U, b[r], -mu if adj else mu, -1.6, ap)
                assert np.linalg.norm(out[r].cpu().numpy() - ref) / np.linalg.norm(ref) < tol


def test_unaligned_natural_fields():
    """complex64 fields that start 8 bytes off a 16-byte boundary give the aligned fields' result."""
    import paper_0910_2927_gb300 as pkg
    dims = (3, 4, 5, 2)
    U = si.random_su3_links(dims, 0.7, 85)
    b = torch.from_numpy(si.gaussian_block(dims, 3, 86).astype(np.complex64)).cuda()
    with _ctx(dims, U, 0.3, (0, 0, 0, 1)) as ctx:
        want = ctx.hw(b, precision=pkg.PREC_MIXED)
        store = torch.empty(b.numel() + 1, dtype=torch.complex64, device="cuda")
        off = store[1:].view_as(b)
        off.copy_(b)
        assert off.data_ptr() % 16 == 8
        assert torch.equal(ctx.hw(off, precision=pkg.PREC_MIXED), want)
