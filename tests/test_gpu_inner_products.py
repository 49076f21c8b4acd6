"""The FP64 inner-product kernel at the edges of its splits: fewer elements than a CTA, ragged tails,
one to eight elements per thread, and basis sizes around the groups of 16 vectors.

Bound: a sum passes through at most about 100 roundings (16 multiply-adds per thread, the adds over
lanes, warps and CTAs), each of them 2^-53 of the sum of the products' moduli, which Cauchy-Schwarz
bounds by |v||w|; complex parts take two products each."""
import numpy as np
import pytest

import seeded_inputs as si

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((2, 2, 2, 2), 40), ((5, 2, 3, 7), 3), ((9, 8, 7, 10), 1),
                                       ((9, 8, 7, 10), 12)])
@pytest.mark.parametrize("J", [1, 15, 16, 17, 33, 64])
def test_inner_products_edges(dims, nrhs, J):
    import paper_0910_2927_gb300 as pkg
    V = si.gaussian_block(dims, J, 61)
    w = si.gaussian_block(dims, nrhs, 62)
    with pkg.SignContext(dims, mu=0.3) as ctx:
        got = ctx.inner_products(torch.from_numpy(V).cuda(), torch.from_numpy(w).cuda())
    ref = w @ V.conj().T
    scale = np.linalg.norm(w, axis=1)[:, None] * np.linalg.norm(V, axis=1)[None]
    assert np.max(np.abs(got - ref) / scale) < 4e-14
