"""The batched pair kernels at the sizes where they can go wrong: group sizes of
every remainder (1 to 9 right-hand sides), domains smaller than a target tile, a
node more or less than a source tile, real and complex A.

Products against the dense oracle with test_gpu_parity's bounds on |A||x|
(FP32: 8 (64 + N) u32; double-float: (64 + N) 2^-45 plus the tile-offset term,
the largest node-to-reference distance over the smallest node distance), and the
solves against its LU solutions (1e-9: the systems stop at 1e-12).
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


def _domains(theta):
    rng = np.random.default_rng(17)
    out = []
    for m1, n, nrhs in ((1, 8, 1), (2, 32, 2), (3, 22, 3), (2, 128, 5), (3, 86, 4), (5, 52, 6), (7, 128, 9), (8, 66, 8)):
        th = None if theta is None else [theta if k % 2 else math.pi / 2 for k in range(m1)]
        out.append((Dm.build_domain(Dm.random_ellipses(rng, m1, 0.6 * m1 + 0.5), n, bounded=False, theta=th), nrhs))
    return out


@pytest.mark.parametrize("theta", [None, 0.6], ids=["real_A", "complex_A"])
@pytest.mark.parametrize("variant", range(1, 8))
def test_groups(G, theta, variant):
    doms = _domains(theta)
    rng = np.random.default_rng(variant)
    gam = [np.stack([Dm.gamma_log(d, d.holes[r % d.m1]) + 0.1 * r for r in range(k)]) for d, k in doms]
    x = [rng.normal(size=(k, d.N)) for d, k in doms]
    dev = lambda v: torch.as_tensor(np.concatenate([a.reshape(-1) for a in v]), device="cuda")
    with G.Batch([d for d, _ in doms], [k for _, k in doms], autotune=False, device="cuda") as b:
        mu, h, hk, res, rel = b.fbie(dev(gam), tol=1e-12, tile_variant=variant)
        y32 = b.apply_IminusN(dev(x), G.GNK_PREC_FP32).cpu().numpy()
        ydf = b.apply_IminusN(dev(x), G.GNK_PREC_DF32).cpu().numpy()
    assert res.status == 0
    mu, h = mu.cpu().numpy(), h.cpu().numpy()
    at = 0
    for (d, k), g, v in zip(doms, gam, x):
        K = O.matrix_IminusN(d.et, d.etp, d.A, d.n)
        dist = np.abs(d.et[:, None] - d.et[None, :]) + np.diag(np.full(d.N, np.inf))
        span = max(np.abs(d.et[j:j + 256] - d.et[j:j + 256][len(d.et[j:j + 256]) // 2]).max() for j in range(0, d.N, 256))
        S = np.abs(K) + np.diag(np.abs(K - np.diag(np.diag(K))).sum(1))
        for r in range(k):
            ref = K @ v[r]
            sx = (S * np.maximum(1.0, (span / dist.min(1)) * 2.0 ** -3)[:, None]) @ np.abs(v[r])
            sl = slice(at + r * d.N, at + (r + 1) * d.N)
            assert np.all(np.abs(y32[sl] - ref) <= 8 * (64 + d.N) * 2.0 ** -24 * 4 * sx)
            assert np.all(np.abs(ydf[sl] - ref) <= (64 + d.N) * 2.0 ** -45 * 4 * sx)
            mo, ho, _ = O.fbie(d.et, d.etp, d.A, d.n, g[r])
            assert np.abs(mu[sl] - mo).max() <= 1e-9 * np.abs(mo).max()
            assert np.abs(h[sl] - ho).max() <= 1e-9 * max(1.0, np.abs(ho).max())
        at += k * d.N
