"""The FP64 step's own error, against the same method in extended precision (numpy's longdouble: 64 bits of
mantissa on x86, 113 on Arm)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_05009_gb300 import binding as B  # noqa: E402
from paper_2211_05009_gb300.cavity import Cavity  # noqa: E402

L = np.longdouble
CX, CY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = [L(4) / 9] + [L(1) / 9] * 4 + [L(1) / 36] * 4


def moments(g):
    drho = g.sum(0)
    rho = 1 + drho
    return drho, rho, sum(c * g[j] for j, c in enumerate(CX)) / rho, sum(c * g[j] for j, c in enumerate(CY)) / rho


def equilibrium(drho, rho, ux, uy):
    """Deviations f^eq_j - w_j."""
    sq = L(3) / 2 * (ux * ux + uy * uy)
    return np.stack([w * (drho + rho * (3 * (a * ux + b * uy) + L(9) / 2 * (a * ux + b * uy) ** 2 - sq))
                     for a, b, w in zip(CX, CY, W)])


def velocity(nx, ny, tau, U, steps):
    zero, wall_u = np.zeros((ny, nx), dtype=L), np.zeros((ny, nx), dtype=L)
    wall_u[-1, 1:-1] = L(U)
    ring = np.ones((ny, nx), dtype=bool)
    ring[1:-1, 1:-1] = False
    y, x = np.mgrid[0:ny, 0:nx]
    yc, xc = np.clip(y, 1, ny - 2), np.clip(x, 1, nx - 2)
    omega = 1 / L(tau)
    g = equilibrium(zero, zero + 1, wall_u, zero)
    for _ in range(steps):
        p = np.stack([g[j][yc - CY[j], xc - CX[j]] for j in range(9)])
        drho, rho, ux, uy = moments(p)
        e = equilibrium(drho, rho, ux, uy)
        g = np.where(ring, equilibrium(drho, rho, wall_u, zero) + (1 - omega) * (p - e), p + omega * (e - p))
    return moments(g)[2:]


@pytest.mark.parametrize("re", [400.0, 100.0, 30.0])  # tau 0.53, 0.62, 0.9
def test_velocity_error_has_no_drift(re):
    """Constants that leave out one unit in the last place of the momentum, 1.1e-16, every step would be
    off by up to 250 x 1.1e-16 = 3e-14; roundings without a direction stay below a few of them, 2e-15."""
    nx, ny, U, steps = 40, 32, 0.1, 250
    tau = 3.0 * U * nx / re + 0.5  # as a batch forms it
    want = velocity(nx, ny, tau, U, steps)
    with Cavity(nx, ny, tau=tau, U=U, dtype="f64") as cav:
        cav.step(steps)
        single = [f.cpu().numpy() for f in cav.moments()]
    b = B.lbm_batch_create([nx, 5], [ny, 4], [re, 10.0], [U, U], "f64")
    try:
        B.lbm_batch_step(b, steps)
        batch = [torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(3)]
        B.lbm_batch_moments(b, 0, *batch)
    finally:
        B.lbm_batch_destroy(b)
    for got in (single, [f.cpu().numpy() for f in batch]):
        for f, w in zip(got[1:], want):
            error = np.linalg.norm((f - w).astype(float)) / np.linalg.norm(w.astype(float))
            print(f"tau {tau}: {error:.2e}")
            assert error < 2e-15
