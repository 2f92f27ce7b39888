"""gnk_fbie_backward on an FMM handle with and without GNK_BUILD_DIFF.

Graded corners at n = 2048 (the header's bound): dL/d eta of the two handles differs
by less than 1e-7 of its norm, and each is as far from the dense oracle's as the
solves' tolerance leaves it, so neither is farther than the other by more than that.
Smooth boundaries: dL/d eta takes the sums of w/d^2, whose far field is the
derivative of the expansions; P = 32 times the FMM's 2e-12 of sum |w/d| is 6.4e-11,
taken as 1e-10 of the norm, for either handle.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import gnk_dense as O
from paper_1308_5351_gb300 import domains as Dm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1308_5351_gb300 import build, gnk
    build.build()
    gnk.load()
    return gnk


def _gradients(G, d, gam, cm, ch):
    """dL/d eta without and with the flag."""
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    out = []
    for flag in (0, G.GNK_BUILD_DIFF):
        with G.Boundary.from_domain(d, adjoint=False, device="cuda", precision=G.GNK_PREC_FMM | flag) as b:
            mu, h, hk, res = b.fbie(dev(gam), tol=1e-12, precision=G.GNK_PREC_FMM)
            g = [torch.empty(d.N, dtype=torch.complex128, device="cuda") for _ in range(3)]
            back = G.gnk_fbie_backward(b.handle, mu, dev(gam), dev(cm), dev(ch), g[0], g[1], g[2],
                                       torch.empty_like(mu), G.options(tol=1e-12, precision=G.GNK_PREC_FMM))
            assert res.status == 0 and back.status == 0
        out.append(g[0].cpu().numpy())
    return out


def test_graded_corners(G):
    d = Dm.build_domain([Dm.Circle(0j, 1.6, ccw=True), Dm.square(0.3 + 0.1j, 0.5, ccw=False)], 2048, bounded=True,
                        alpha=-1.2 + 0.3j)
    gam = Dm.manufactured(d, Dm.f_bounded_ex1)[0]
    rng = np.random.default_rng(5)
    cm, ch = rng.normal(size=d.N), rng.normal(size=d.N)
    ref = O.fbie_gradient(d.et, d.etp, d.A, d.n, gam, cm, ch)[0]
    plain, diff = _gradients(G, d, gam, cm, ch)
    norm = np.linalg.norm
    assert norm(plain - diff) <= 1e-7 * norm(ref)
    assert norm(plain - ref) <= norm(diff - ref) + 1e-7 * norm(ref)


def test_smooth_boundaries(G):
    d = Dm.build_domain(Dm.random_ellipses(np.random.default_rng(3), 16, 2.5), 512, bounded=False)
    gam = Dm.gamma_log(d, d.holes[0])
    rng = np.random.default_rng(5)
    cm, ch = rng.normal(size=d.N), rng.normal(size=d.N)
    ref = O.fbie_gradient(d.et, d.etp, d.A, d.n, gam, cm, ch)[0]
    for got in _gradients(G, d, gam, cm, ch):
        assert np.linalg.norm(got - ref) <= 1e-10 * np.linalg.norm(ref)
