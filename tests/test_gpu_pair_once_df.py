"""The double-float and FP32 sums that take each pair of nodes once, against the
FP64 operator.

Sizes about their rule (a block pair has 256 x 256 nodes) and beyond: one node past
a block, one node short of one, an odd number of blocks; real and complex A, one
part of z and both (f_B reads Im z, f_C Re z, the adjoint both).  A double-float
operation is exact to about 2^-46 and (2/n) sum_j |w_j/d| is below 50 here:
50 x 2^-46 = 7e-13, taken as 1e-11 of the largest value.  In FP32 the two nearest
neighbours decide: offsets below 0.5 rounded to 3e-8 against distances above 2.5e-4
give (2/n)|w/d| <= 2 an error of 1.2e-4 relative each, taken as 3e-4 of the largest
value (about 4 for normal x).
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1308_5351_gb300 import domains as Dm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1308_5351_gb300 import build, gnk
    build.build()
    gnk.load()
    return gnk


@pytest.mark.parametrize("n", [366, 622, 1792, 1794, 2306])
@pytest.mark.parametrize("turned", [False, True])
def test_pairs_once(G, n, turned):
    rng = np.random.default_rng(n)
    ell = Dm.random_ellipses(rng, 7, 2.0)
    theta = [math.pi / 2, 0, 0.4, math.pi / 2, 1.0, 0, 0.3] if turned else None
    d = Dm.build_domain(ell, n, bounded=False, theta=theta)
    x = torch.as_tensor(rng.normal(size=d.N), device="cuda")
    with G.Boundary.from_domain(d, adjoint=True, device="cuda", precision=G.GNK_PREC_FP64) as b:
        for f in (b.apply_IminusN, b.apply_M, b.apply_adjoint):
            want = f(x, G.GNK_PREC_FP64)
            for prec, tol in ((G.GNK_PREC_DF32, 1e-11), (G.GNK_PREC_FP32, 3e-4)):
                got = f(x, prec)
                assert float((got - want).abs().max()) <= tol * float(want.abs().max())


@pytest.mark.parametrize("name", ["GNK_PREC_FP64", "GNK_PREC_DF32", "GNK_PREC_FP32"])
def test_captured_product_keeps_its_workspace(G, name):
    """A product captured into a graph, replayed after a call with two right-hand
    sides made the pool's workspace grow: the same operator, other inputs."""
    prec = getattr(G, name)
    d = Dm.build_domain(Dm.random_ellipses(np.random.default_rng(3), 7, 2.0), 1792, bounded=False)
    x = torch.zeros(d.N, dtype=torch.float64, device="cuda")
    y = torch.empty_like(x)
    new = torch.as_tensor(np.random.default_rng(4).normal(size=d.N), device="cuda")
    with G.Boundary.from_domain(d, adjoint=True, device="cuda", precision=G.GNK_PREC_FP64) as b:
        b.apply_IminusN(x, prec, out=y)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            b.apply_IminusN(x, prec, out=y)
        gam = torch.as_tensor(Dm.gamma_log(d, d.holes[0]), device="cuda")
        b.fbie(gam, precision=G.GNK_PREC_FP64, tol=1e-10)
        x.copy_(new)
        g.replay()
        torch.cuda.synchronize()
        want = b.apply_IminusN(new, G.GNK_PREC_FP64)
        tol = 3e-4 if name == "GNK_PREC_FP32" else 1e-11
        assert float((y - want).abs().max()) <= tol * float(want.abs().max())
