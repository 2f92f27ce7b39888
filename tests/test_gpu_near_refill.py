"""A near-field item with more sources than the kernel gathers at once.

Six tiny circles close together lie in one leaf: its items have 3,072 sources, four
gathers of at most 960, and there are items enough (565) that none is split into
shares.  The FMM's operators are within 1e-12 of (2/n) sum |A q x / d| <= 16 for
|x| <= 1 of the direct FP64 ones, taken as 1e-10; a solve to 1e-12, whose operator
reads its near field from the cache of the weights A x, leaves a residual of the
direct operator below that too.  Then a product on one stream and a solve on another,
ordered by events, give what they give on one.
"""
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


def _domain(turned):
    ell = Dm.random_ellipses(np.random.default_rng(2), 24, 2.6)
    tiny = [Dm.Circle(5.2 + 0.3j + 0.012 * (k % 3) + 0.012j * (k // 3), 0.004, ccw=False) for k in range(6)]
    return Dm.build_domain(ell + tiny, 512, bounded=False, theta=[0.1 * k for k in range(30)] if turned else None)


@pytest.mark.parametrize("turned", [False, True], ids=["real_A", "complex_A"])
def test_items_of_many_sources(G, turned):
    d = _domain(turned)
    x = torch.as_tensor(np.random.default_rng(5).uniform(-1, 1, d.N), device="cuda")
    gam = torch.as_tensor(Dm.gamma_log(d, d.holes[0]), device="cuda")
    fmm, fp64 = G.GNK_PREC_FMM, G.GNK_PREC_FP64
    with G.Boundary.from_domain(d, adjoint=True, device="cuda", precision=fmm) as b:
        for f in (b.apply_IminusN, b.apply_M):
            assert float((f(x, fmm) - f(x, fp64)).abs().max()) <= 1e-10
        phi, res = b.solve_adjoint_ie(gam, precision=fmm, tol=1e-12)
        assert res.status == 0
        assert float((b.apply_adjoint(phi, fp64) - gam).norm()) <= 1e-10 * float(gam.norm())


def test_product_and_solve_on_two_streams(G):
    d = _domain(True)
    x = torch.as_tensor(np.random.default_rng(5).uniform(-1, 1, d.N), device="cuda")
    gam = torch.as_tensor(Dm.gamma_log(d, d.holes[0]), device="cuda")
    fmm = G.GNK_PREC_FMM
    got = []
    for two in (False, True):
        s0 = torch.cuda.Stream()
        s1 = torch.cuda.Stream() if two else s0
        torch.cuda.synchronize()
        with G.Boundary.from_domain(d, adjoint=True, device="cuda", precision=fmm) as b:
            torch.cuda.synchronize()
            y = torch.empty_like(x)
            phi = torch.empty_like(x)
            z = torch.empty_like(x)
            G.gnk_apply_IminusN(b.handle, x, y, fmm, s0)
            s1.wait_stream(s0)
            G.gnk_solve_adjoint_ie(b.handle, gam, phi, G.options(precision=fmm, tol=1e-12), s1)
            s0.wait_stream(s1)
            G.gnk_apply_M(b.handle, phi, z, fmm, s0)
            torch.cuda.synchronize()
        got.append((y, phi, z))
    for a, c in zip(*got):
        assert torch.equal(a, c)  # sums in a fixed order
