"""The tensor-core M2L against the double-float one (the handles built for
differentiation keep it) and against direct sums.

Weights: random, with zero sums per curve (leading coefficients that cancel),
zero on most curves (columns of zeros), and scaled by 2^-60 and 2^60 (the digits
are taken below a power of two per pair).  Bounds: both forms within
test_fmm's 1e-12 S_i of the direct sum, and their difference within 2^-44 of
the largest S_i (each rounds below 2^-46 of the sums it adds)."""
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


@pytest.mark.parametrize("kind", ["random", "zero_sum", "sparse", "tiny", "huge", "zero"])
def test_m2l_forms_agree(G, kind):
    rng = np.random.default_rng(3)
    d = Dm.build_domain(Dm.random_ellipses(rng, 13, 2.5), 300, bounded=False)
    w = rng.normal(size=d.N) + 1j * rng.normal(size=d.N)
    if kind == "zero_sum":
        w = (w.reshape(d.m1, d.n) - w.reshape(d.m1, d.n).mean(1, keepdims=True)).reshape(-1)
    elif kind == "sparse":
        w[d.n:] = 0.0
    elif kind in ("tiny", "huge"):
        w *= 2.0 ** (-60 if kind == "tiny" else 60)
    elif kind == "zero":
        w[:] = 0.0
    z = []
    for flag in (0, G.GNK_BUILD_DIFF):
        with G.Boundary.from_domain(d, adjoint=False, device="cuda", precision=G.GNK_PREC_FMM | flag) as b:
            z.append(b.cauchy_sum(torch.as_tensor(w, device="cuda"), precision=G.GNK_PREC_FMM).cpu().numpy())
    E = O.cauchy_matrix(d.et)
    S, ref = np.abs(E) @ np.abs(w), E @ w
    for v in z:
        assert np.all(np.abs(v - ref) <= 1e-12 * S)
    assert np.abs(z[0] - z[1]).max() <= 2.0 ** -44 * S.max()
