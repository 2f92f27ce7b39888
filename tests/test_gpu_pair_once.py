"""The FP64 Cauchy sums that take each pair of nodes once, at the sizes where
their node blocks can go wrong: one node block, a node more or less than whole
blocks, odd and even block counts, every block shape, the largest count.

Sampled rows (the first and last nodes, the nodes at block edges, random ones)
against the oracle, with test_gpu_parity's bounds: |z - z_ref|_i <=
(64 + N) u S_i, S_i = sum_j |w_j / (eta_i - eta_j)|, u = 2^-53; operators the
same on |A||x| with a factor 4.  Real A (one part of the sum) and complex A
(both), and the two-right-hand-side sums of a handle with eta''.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import gnk_dense as O
from paper_1308_5351_gb300 import domains as Dm

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53
# (m1, n): N = 4, 32, 34 | 62, 66 | 768, 1022, 1026 | 4094, 4098 | 8190, 8198 | 16386 | 33280
SIZES = [(1, 4), (1, 32), (1, 34), (1, 62), (3, 22), (3, 256), (7, 146), (1, 1026), (23, 178), (3, 1366), (5, 1638),
         (1, 8198), (2, 8193 - 1), (1, 16386), (65, 512)]


@pytest.fixture(scope="module")
def G():
    from paper_1308_5351_gb300 import build, gnk
    build.build()
    gnk.load()
    return gnk


def _domain(m1, n, theta):
    k = math.ceil(math.sqrt(m1))
    curves = [Dm.Ellipse(complex(i % k, i // k), 0.4, 0.3, 0.2 * i) for i in range(m1)]
    th = None if theta is None else [theta if i % 2 else math.pi / 2 for i in range(m1)]
    return Dm.build_domain(curves, n, bounded=False, theta=th)


def _rows(N, rng):
    edge = [0, 1, N - 1, N - 2] + [e + o for e in (32, 64, 128, 256, 512, N // 2) for o in (-1, 0)]
    r = set(int(e) for e in edge if 0 <= e < N) | set(int(e) for e in rng.integers(0, N, 12))
    return np.array(sorted(r))


@pytest.mark.parametrize("m1,n", SIZES)
@pytest.mark.parametrize("theta", [None, 0.7], ids=["real_A", "complex_A"])
def test_pairs_once(G, m1, n, theta):
    d = _domain(m1, n, theta)
    rng = np.random.default_rng([m1, n])
    w = rng.normal(size=d.N) + 1j * rng.normal(size=d.N)
    x = rng.normal(size=d.N)
    rows = _rows(d.N, rng)
    dist = np.abs(d.et[rows][:, None] - d.et[None, :])
    dist[np.arange(rows.size), rows] = np.inf
    with G.Boundary.from_domain(d, adjoint=True, device="cuda") as b:
        z = b.cauchy_sum(torch.as_tensor(w, device="cuda")).cpu().numpy()
        xd = torch.as_tensor(x, device="cuda")
        got = [f(xd).cpu().numpy() for f in (b.apply_IminusN, b.apply_M, b.apply_adjoint)]
    S = (np.abs(w)[None, :] / dist).sum(1)
    assert np.all(np.abs(z[rows] - O.cauchy_rows(d.et, w, rows)) <= (64 + d.N) * U64 * S)
    refs = [O.rows_IminusN(d.et, d.etp, d.A, d.n, x, rows), O.rows_M(d.et, d.etp, d.A, d.n, x, rows),
            O.rows_adjoint(d.et, d.etp, d.etpp, d.A, d.Ap, d.n, d.c, x, rows)]
    # |A||x| of the kernel sums (both orders) and of the circulant's rows
    q = np.abs(d.etp / d.A)
    K = np.maximum(np.abs(d.A)[rows][:, None] * q[None, :], q[rows][:, None] * np.abs(d.A)[None, :]) / dist * (2 / d.n)
    s1, sx = K.sum(1), K @ np.abs(x)
    lx = np.abs(O.circulant_L(d.n)[0]).sum() * np.abs(x).max()
    tol = 4 * (64 + d.N) * U64 * (sx + (2 + s1) * np.abs(x[rows]) + lx + np.abs(x).max())
    for y, ref in zip(got, refs):
        assert np.all(np.abs(y[rows] - ref) <= tol)


@pytest.mark.parametrize("m1,n", [(1, 768), (1, 4096), (1, 4098)], ids=["fp64_sequence", "split_fast", "blocks_fast"])
@pytest.mark.parametrize("scale", ["ones", "wide", "huge", "tiny", "axis"])
def test_one_over_d(G, m1, n, scale):
    """One unit weight: z_i = 1 / (eta_i - eta_j) within 2^-51 of its modulus (2 ulp
    of the larger part), for distances over many powers of two, equal
    coordinates, and ranges that leave the three-float form."""
    rng = np.random.default_rng([n, len(scale)])
    e = rng.uniform(-1, 1, n) + 1j * rng.uniform(-1, 1, n)
    if scale == "wide":
        e = e * 2.0 ** rng.integers(-60, 60, n)
    elif scale == "huge":
        e = e * 2.0 ** 120
    elif scale == "tiny":
        e = e * 2.0 ** -120
    elif scale == "axis":  # a grid: every second difference has an exactly zero part
        k = np.arange(n)
        e = (k % 64) * 0.37 + 1j * (k // 64) * 2.0 ** -20
    one = np.ones(n, dtype=np.complex128)
    with G.Boundary(m1, n, e, one, one, None, None, False) as b:
        for j in (0, n // 2 + 1, n - 1):
            w = torch.zeros(n, dtype=torch.complex128, device="cuda")
            w[j] = 1.0
            z = b.cauchy_sum(w).cpu().numpy()
            d = e - e[j]  # rounded as on the GPU
            i = np.arange(n) != j
            x, y = d.real[i].astype(np.longdouble), d.imag[i].astype(np.longdouble)
            r2 = x * x + y * y
            err = np.hypot((z.real[i] - x / r2), (z.imag[i] + y / r2))
            assert np.all(err <= 2.0 ** -51 / np.sqrt(r2)), float((err * np.sqrt(r2)).max())
            assert z[j] == 0
