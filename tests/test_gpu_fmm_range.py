"""FMM sums with the translations on the tensor cores scale with their weights:
multiplying by a power of two changes no other bit, up to the largest exponent that
single precision holds (2^127, where the scale of the digits has to have room) and down
to 2^-60."""
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


@pytest.mark.parametrize("power", [127, 126, 60, -60])
def test_weights_times_a_power_of_two(G, power):
    d = Dm.build_domain(Dm.random_ellipses(np.random.default_rng(3), 16, 2.5), 512, bounded=False)
    one = torch.ones(d.N, dtype=torch.complex128, device="cuda")
    et = torch.as_tensor(d.et * 1024.0, device="cuda")  # nodes 1 and more apart: |z| below the weight
    with G.Boundary(d.m1, d.n, et, one, one, None, None, False, precision=G.GNK_PREC_FMM) as b:
        for j in (0, 4000, d.N - 1):
            w = torch.zeros(d.N, dtype=torch.complex128, device="cuda")
            w[j] = 1.0 + 0.5j
            z = b.cauchy_sum(w, G.GNK_PREC_FMM)
            s = b.cauchy_sum(w * 2.0 ** power, G.GNK_PREC_FMM)
            assert bool(torch.isfinite(torch.view_as_real(s)).all())
            assert torch.equal(s, z * 2.0 ** power)
