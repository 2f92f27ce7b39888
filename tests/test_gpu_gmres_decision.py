"""Where a cycle leaves the residual on the tolerance, the host and the kernels take
one decision.

A solve is run for one cycle, then again with the tolerance one unit in the last
place below the residual that this cycle reached: the second run is not converged
there and has to go on to a smaller residual.  (With tol * ||b|| rounded on one
side and ||r|| / ||b|| on the other, about one in ten of these solves took its
residual for converged on the device alone, and every later cycle did nothing.)
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


@pytest.mark.parametrize("name", ["GNK_PREC_FP64", "GNK_PREC_FMM"])
def test_tolerance_at_the_residual_of_a_cycle(G, name):
    prec = getattr(G, name)
    d = Dm.three_circles(64)
    rng = np.random.default_rng(8)
    x = torch.empty(d.N, dtype=torch.float64, device="cuda")
    with G.Boundary.from_domain(d, adjoint=False, device="cuda",
                                precision=prec if name == "GNK_PREC_FMM" else G.GNK_PREC_FP64) as b:
        for _ in range(64):
            rhs = torch.as_tensor(rng.normal(size=d.N), device="cuda")
            one = G.gnk_solve_ie_transpose(b.handle, rhs, x, G.options(precision=prec, tol=1e-14, restart=4, maxit=1))
            tol = float(np.nextafter(one.relres, 0.0))
            assert one.status == G.GNK_ENOTCONV and tol > 1e-6
            two = G.gnk_solve_ie_transpose(b.handle, rhs, x, G.options(precision=prec, tol=tol, restart=4, maxit=50))
            assert two.status == G.GNK_OK and two.relres <= tol and two.cycles == 2
