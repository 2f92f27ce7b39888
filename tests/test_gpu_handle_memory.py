"""What kept handles hold after direct sums.

A direct sum that takes each pair once needs partial sums of node blocks x N, 38 to
150 MB here by precision and right-hand sides.  They belong to the product, not to
the handle: as in test_gpu_memory, after the first two handles' products the pool
serves those of six more from memory it keeps (to 64 MB).
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


def test_kept_handles_do_not_hold_the_partial_sums(G):
    d = Dm.build_domain(Dm.random_ellipses(np.random.default_rng(3), 24, 3.0), 1024, bounded=False)
    x = torch.as_tensor(np.random.default_rng(4).normal(size=d.N), device="cuda")
    precs = (G.GNK_PREC_FP64, G.GNK_PREC_DF32, G.GNK_PREC_FP32)
    y = [torch.empty_like(x) for _ in precs]
    first = [torch.empty_like(x) for _ in precs]
    kept = [G.Boundary.from_domain(d, adjoint=True, device="cuda", precision=G.GNK_PREC_FP64 | G.GNK_BUILD_DEFER)
            for _ in range(8)]
    free = []
    try:
        for k, b in enumerate(kept):
            for p, out in zip(precs, first if k == 0 else y):
                b.apply_IminusN(x, p, out=out)
            torch.cuda.synchronize()
            free.append(torch.cuda.mem_get_info()[0])
            if k:  # sums in a block that other handles have used
                assert all(torch.equal(a, c) for a, c in zip(y, first))
        assert max(free[2:]) - min(free[2:]) <= 64 << 20, [f >> 20 for f in free]
    finally:
        for b in kept:
            b.close()
