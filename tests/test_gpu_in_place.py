"""Products whose result lies over their input give what they give into another array.

Every block of a small FP64 sum (up to 4,096 nodes) reads all inputs, and the blocks
that finish first write results; the larger sums and the other precisions write theirs
in a launch of its own.  The same operations in the same order: equal bits.
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


@pytest.mark.parametrize("n", [34, 256, 1364, 2050])  # N = 102, 768, 4,092, 6,150
@pytest.mark.parametrize("name", ["GNK_PREC_FP64", "GNK_PREC_DF32", "GNK_PREC_FP32", "GNK_PREC_FMM"])
def test_result_over_the_input(G, n, name):
    prec = getattr(G, name)
    d = Dm.three_circles(n)
    rng = np.random.default_rng(n)
    x = torch.as_tensor(rng.normal(size=d.N), device="cuda")
    g = torch.as_tensor(rng.normal(size=d.N), device="cuda")
    w = torch.complex(x, g)
    with G.Boundary.from_domain(d, adjoint=True, device="cuda",
                                precision=prec if name == "GNK_PREC_FMM" else G.GNK_PREC_FP64) as b:
        for f, v in ((b.apply_IminusN, x), (b.apply_M, x), (b.apply_adjoint, x), (b.cauchy_sum, w)):
            want = f(v, prec)
            for _ in range(5):
                y = v.clone()
                f(y, prec, out=y)
                assert torch.equal(y, want)
        h = torch.empty_like(x)
        G.gnk_compute_h(b.handle, x, g, h, None)
        for k in range(2):
            y = (x, g)[k].clone()
            G.gnk_compute_h(b.handle, *((y, g) if k == 0 else (x, y)), y, None)
            assert torch.equal(y, h)
