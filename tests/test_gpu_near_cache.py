"""The FMM's cached near fields: the operators that read them against the dense
oracle, at the shapes where the caches can go wrong.

Domains: real and complex A (one part of A z or Im(q z) of a complex factor),
graded corners (q = 0 at a node), odd m+1, leaves with odd source counts (the
padding of a source pair), more than one chunk of 32 source pairs, a single
leaf's worth of nodes.  The products without a solve (no cache for the weights
A x) and the solves (with it) must agree with the oracle to the solve bounds of
test_gpu_parity (1e-10) and each other's equation: the residual of the cached
solve, formed by the direct FP64 operator, is within 1e-11 of the right-hand side
(tol 1e-12, FMM error 1e-12 S_i, condition below 100).
"""
import math

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


def _domains():
    rng = np.random.default_rng(21)
    ell = Dm.random_ellipses(rng, 7, 2.0)
    return {
        "disk_n34": Dm.disk(34),
        "ellipses7_n150": Dm.build_domain(ell, 150, bounded=False),
        "ellipses7_theta_n302": Dm.build_domain(ell, 302, bounded=False,
                                                theta=[math.pi / 2, 0, 0.4, math.pi / 2, 1.0, 0, 0.3]),
        "circles3_n256": Dm.three_circles(256),
        "square_n512": Dm.build_domain([Dm.Circle(0j, 1.6, ccw=True), Dm.square(0.3 + 0.1j, 0.5, ccw=False)], 512,
                                       bounded=True, alpha=-1.2 + 0.3j),
    }


DOMS = _domains()


@pytest.mark.parametrize("name", list(DOMS))
def test_cached_near_fields(G, name):
    d = DOMS[name]
    rng = np.random.default_rng(4)
    x = rng.normal(size=d.N)
    gam = Dm.gamma_log(d, d.holes[0]) if d.m1 > 1 else np.cos(Dm.nodes(d.n))
    K, M = O.matrix_IminusN(d.et, d.etp, d.A, d.n), O.matrix_M(d.et, d.etp, d.A, d.n)
    Ad = O.matrix_adjoint(d.et, d.etp, d.etpp, d.A, d.Ap, d.n, d.c)
    fmm = G.GNK_PREC_FMM
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    with G.Boundary.from_domain(d, adjoint=True, device="cuda", precision=fmm) as b:
        before = b.apply_adjoint(dev(x), fmm).cpu().numpy()
        phi, r1 = b.solve_adjoint_ie(dev(gam), precision=fmm, tol=1e-12)
        after = b.apply_adjoint(dev(x), fmm).cpu().numpy()
        y, m = b.apply_IminusN(dev(x), fmm).cpu().numpy(), b.apply_M(dev(x), fmm).cpu().numpy()
        lam = torch.empty_like(phi)
        r2 = G.gnk_solve_ie_transpose(b.handle, dev(x), lam, G.options(precision=fmm, tol=1e-12))
    assert r1.status == 0 and r2.status == 0
    bound = lambda A, v: 1e-11 * (np.abs(A) @ np.abs(v)).max()
    for got, A in ((before, Ad), (after, Ad), (y, K), (m, M)):
        assert np.abs(got - A @ x).max() <= bound(A, x)
    phi, lam = phi.cpu().numpy(), lam.cpu().numpy()
    assert np.linalg.norm(Ad @ phi - gam) <= 1e-11 * np.linalg.norm(gam)
    assert np.linalg.norm(K.T @ lam - x) <= 1e-11 * np.linalg.norm(x)


def test_diff_handle_keeps_its_arithmetic(G):
    """GNK_BUILD_DIFF: the transposed solve forms its near field directly, and its
    result agrees with that of the cache to the solves' tolerance."""
    d = DOMS["ellipses7_n150"]
    x = np.random.default_rng(5).normal(size=d.N)
    out = []
    for flag in (0, G.GNK_BUILD_DIFF):
        with G.Boundary.from_domain(d, adjoint=False, device="cuda", precision=G.GNK_PREC_FMM | flag) as b:
            lam = torch.empty(d.N, dtype=torch.float64, device="cuda")
            G.gnk_solve_ie_transpose(b.handle, torch.as_tensor(x, device="cuda"), lam,
                                     G.options(precision=G.GNK_PREC_FMM, tol=1e-12))
            out.append(lam.cpu().numpy())
    assert np.abs(out[0] - out[1]).max() <= 1e-10 * np.abs(out[1]).max()


@pytest.mark.parametrize("name", list(DOMS))
def test_inverse_cache_changes_no_bit(G, name):
    """GNK_BUILD_DIFF: the same product before a solve (1/d formed in the kernel)
    and after one (1/d read from the cache that the solve formed)."""
    d = DOMS[name]
    rng = np.random.default_rng(6)
    x = torch.as_tensor(rng.normal(size=d.N), device="cuda")
    gam = torch.as_tensor(Dm.gamma_log(d, d.holes[0]) if d.m1 > 1 else np.cos(Dm.nodes(d.n)), device="cuda")
    fmm = G.GNK_PREC_FMM
    with G.Boundary.from_domain(d, adjoint=True, device="cuda", precision=fmm | G.GNK_BUILD_DIFF) as b:
        before = b.apply_adjoint(x, fmm).cpu().numpy()
        b.solve_adjoint_ie(gam, precision=fmm, tol=1e-12)
        after = b.apply_adjoint(x, fmm).cpu().numpy()
    assert np.array_equal(before, after)


@pytest.mark.parametrize("n", [24, 34, 66, 70, 78, 94, 130])
def test_folded_items(G, n):
    """The directly summed near field (weights of the caller's) with last items of 1
    to 32 targets: within the FMM's bound, 1e-11 of sum |w/d|, of the dense sum."""
    d = Dm.build_domain(Dm.random_ellipses(np.random.default_rng(n), 5, 2.0), n, bounded=False)
    rng = np.random.default_rng(n)
    w = rng.normal(size=d.N) + 1j * rng.normal(size=d.N)
    diff = d.et[:, None] - d.et[None, :]
    np.fill_diagonal(diff, np.inf)
    with G.Boundary.from_domain(d, adjoint=False, device="cuda", precision=G.GNK_PREC_FMM) as b:
        z = b.cauchy_sum(torch.as_tensor(w, device="cuda"), precision=G.GNK_PREC_FMM).cpu().numpy()
    assert np.abs(z - (w[None, :] / diff).sum(1)).max() <= 1e-11 * (np.abs(w)[None, :] / np.abs(diff)).sum(1).max()


@pytest.mark.parametrize("grid,n", [(20, 80), (20, 100), (22, 64)])
def test_domains_that_fill_the_plane(G, grid, n):
    """Trees whose leaf level is chosen against its parent's mean (28 to 44 nodes per
    leaf, 120 to 160 one level up): the FMM's operator against the double-float direct
    sums, both within 1e-12 of (2/n) sum |A q x/d| <= 100, so within 1e-10 of |x| <= 1."""
    d = Dm.close_curves(seed=5, n=n, grid=grid, squares=1)
    x = torch.as_tensor(np.random.default_rng(n).uniform(-1, 1, d.N), device="cuda")
    with G.Boundary.from_domain(d, adjoint=False, device="cuda", precision=G.GNK_PREC_FMM) as b:
        y, z = b.apply_IminusN(x, G.GNK_PREC_FMM), b.apply_IminusN(x, G.GNK_PREC_DF32)
    assert float((y - z).abs().max()) <= 2e-10
