"""One adjoint step against extended precision, cell by cell: the fixed-point
form (its scale is the cell's own largest adjoint) and the FP64 form that
takes the cells outside its range; and the objective's fields over several
batches of levels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
LD = np.longdouble
T = [LD(4) / 9] + [LD(1) / 9] * 4 + [LD(1) / 36] * 4


def _exact(f, lam, tau, alpha, F0, kf):
    """lam_out, dJ/dtau, dJ/dF0 of f -> f - om (f - feq(rho, j)) +
    feq(rho, m') - feq(rho, j) followed by streaming, m' = (1 - alpha) j + F."""
    ny, nx = f.shape[1:]
    f, om, al = f.astype(LD), LD(1.0 / tau), LD(alpha)
    sx = np.sin(2 * np.pi * kf * np.arange(ny) / ny).astype(LD)[:, None] + np.zeros((1, nx), LD)
    sy = np.sin(2 * np.pi * kf * np.arange(nx) / nx).astype(LD)[None, :] + np.zeros((ny, 1), LD)
    mu = np.stack([np.roll(lam[l].astype(LD), (-CY[l], -CX[l]), (0, 1)) for l in range(9)])
    rho = f.sum(0)
    jx, jy = sum(CX[l] * f[l] for l in range(9)), sum(CY[l] * f[l] for l in range(9))

    def contract(mx, my):
        r = bx = by = e = 0
        for l in range(9):
            cm = CX[l] * mx + CY[l] * my
            q = LD(4.5) * cm * cm - LD(1.5) * (mx * mx + my * my)
            r = r + T[l] * mu[l] * (1 - q / rho ** 2)
            e = e + T[l] * mu[l] * (rho + 3 * cm + q / rho)
            bx = bx + T[l] * mu[l] * (3 * CX[l] + (9 * cm * CX[l] - 3 * mx) / rho)
            by = by + T[l] * mu[l] * (3 * CY[l] + (9 * cm * CY[l] - 3 * my) / rho)
        return r, bx, by, e

    ra, xa, ya, ea = contract(jx, jy)
    rb, xb, yb, _ = contract((1 - al) * jx + LD(F0) * sx, (1 - al) * jy + LD(F0) * sy)
    R, X, Y = (om - 1) * ra + rb, (om - 1) * xa + (1 - al) * xb, (om - 1) * ya + (1 - al) * yb
    out = np.stack([(1 - om) * mu[l] + R + CX[l] * X + CY[l] * Y for l in range(9)])
    dtau = (om * om * ((mu * f).sum(0) - ea)).sum()
    return out, dtau, (xb * sx + yb * sy).sum(), np.abs(mu).max(0), rho


@pytest.mark.parametrize("nx,ny", [(64, 64), (33, 17), (5, 3)])
@pytest.mark.parametrize("adjoint", ["white", "contrast", "front", "tiny", "huge"])
@pytest.mark.parametrize("rho0,tau", [(1.0, 0.53), (1.0, 0.8), (3.0, 0.55)])
def test_adjoint_step_exact(nx, ny, adjoint, rho0, tau):
    import torch

    import paper_1809_06735_gb300 as P

    alpha, F0, kf = 1e-3, 2e-5, 2
    rng = np.random.default_rng(nx + ny)
    u = 0.05 * rng.standard_normal((2, ny, nx)).clip(-2, 2)
    f = np.stack([float(T[l]) * (1 + 3 * (CX[l] * u[0] + CY[l] * u[1])) for l in range(9)])
    f *= rho0 * (1 + 0.02 * rng.standard_normal((9, ny, nx)).clip(-2, 2))
    lam = rng.standard_normal((9, ny, nx))
    if adjoint == "contrast":  # cells of a warp 12 decades apart
        lam *= 10.0 ** rng.integers(-12, 1, size=(1, ny, nx))
    elif adjoint == "front":  # zero beyond the objective's reach
        lam[:, :, nx // 2:] = 0.0
    elif adjoint in ("tiny", "huge"):
        lam *= 1e-280 if adjoint == "tiny" else 1e280
    lat = P.Lattice([P.Member(nx, ny, tau, rho0, 1, kf, F0, alpha)], precision=64)
    out = torch.empty(9, ny, nx, dtype=torch.float64, device="cuda")
    dt, dF = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2))
    lat.adjoint_step(0, torch.from_numpy(f).cuda(), torch.from_numpy(lam).cuda(), out, 0.0, (0, 0),
                     1, dt, dF)
    ref, rt, rF, top, rho = _exact(f, lam, tau, alpha, F0, kf)
    # about 20 roundings of terms up to 3 times the cell's largest adjoint,
    # rho times that for dJ/dtau
    eps = 64 * 2.0 ** -53
    assert (np.abs(out.cpu().numpy() - ref) <= eps * top).all()
    assert abs(float(dt) - rt) <= eps * (top * np.maximum(rho, 1)).sum() / tau ** 2
    assert abs(float(dF) - rF) <= eps * top.sum()


@pytest.mark.parametrize("nx,ny,L,nstates,every", [
    (40, 28, 28, 13, 1),   # region = grid: five levels fit the scratch at once
    (40, 28, 20, 13, 5),   # batches with weighted, partly weighted and no levels
    (16, 12, 2, 300, 7),   # more levels than one batch may have
    (3, 2, 2, 9, 2)])
def test_objective_batches_match_single_steps(nx, ny, L, nstates, every):
    """A sweep whose levels take several batches against single steps: the
    adjoint bit for bit, the gradients to the rounding of their sums (2^-53
    per level and partial, 1e-12 covers 300 levels)."""
    import torch

    import paper_1809_06735_gb300 as P

    lat = P.Lattice([P.Member(nx, ny, 0.56, 1.0, 1, 1, 2e-4, 1e-3)], precision=64)
    rng = np.random.default_rng(nx)
    u = 0.03 * rng.standard_normal((2, ny, nx)).clip(-2, 2)
    lat.init_fields(0, np.ones((ny, nx)), u[0], u[1])
    states = torch.empty((nstates, 9, ny, nx), dtype=torch.float64, device="cuda")
    lat.record_trajectory(0, states)
    w = np.where(np.arange(nstates) % every == 0, 0.1 + np.arange(nstates) / nstates, 0.0)
    acc = torch.zeros(4, dtype=torch.float64, device="cuda")
    new = lambda: torch.empty((9, ny, nx), dtype=torch.float64, device="cuda")
    out, box = new(), (nx - 1, 1)
    lat.adjoint_sweep(0, states, None, out, new(), w, box, L, acc[0:1], acc[1:2])
    lam = None
    for k in range(nstates - 1, -1, -1):
        nxt = new()
        lat.adjoint_step(0, states[k], lam, nxt, float(w[k]), box, L, acc[2:3], acc[3:4])
        lam = nxt
    assert torch.equal(out, lam) and bool(out.isfinite().all())
    a = acc.cpu().numpy()
    assert abs(a[0] - a[2]) <= 1e-12 * abs(a[2]) and abs(a[1] - a[3]) <= 1e-12 * abs(a[3])
