"""1D Euler in FP64 where the flow is uniform and supersonic: every face flux is the
physical flux, and so is every point's flux of the quadrature, by the same operations.
What is left of the first moments' right-hand side is the rounding of the weighted sum."""
import numpy as np
import pytest

from paper_2201_12193_gb300 import hweno

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused", [True, False])
def test_uniform_flow_leaves_the_sums_rounding(fused):
    import torch
    n, w = 4000, 12                          # blocks of w equal cells; the middle ones see nothing else
    g = np.random.default_rng(12)
    rho, c = np.exp(g.uniform(-3, 3, n)), np.exp(g.uniform(-1, 1, n))
    u = g.uniform(1.2, 6.0, n) * c * np.where(g.random(n) < 0.5, -1, 1)
    p = rho * c * c / 1.4
    q = np.stack([rho, rho * u, p / 0.4 + 0.5 * rho * u * u])
    m = np.zeros((3, 2, 1, n * w))
    m[:, 0, 0] = np.repeat(q, w, axis=1)
    s = hweno.Solver(1, n * w, x1=float(n * w), indicator="none", bc=("transmissive",) * 4)
    s.set_fused(fused)
    U = torch.from_numpy(m).cuda()
    L, Um = torch.empty_like(U), torch.empty_like(U)
    s.rhs(U, Um, L, torch.empty((1, n * w), dtype=torch.uint8, device="cuda"))
    torch.cuda.synchronize()
    got = np.abs(L.cpu().numpy()[:, 1, 0].reshape(3, n, w)[:, :, 5:7])
    flux = np.abs(np.stack([rho * u, rho * u * u + p, u * (q[2] + p)]))[:, :, None]
    # 1/12, 1/2, 11/12 and 1 of the flux, each rounded at 2^-53 of itself, the weights
    # rounded at 2^-54 in all, and the last product (dx = 1)
    assert (got <= 2.0 ** -53 * (2.5 + 0.5 + 0.01) * flux).all(), (got / flux).max() * 2.0 ** 53
