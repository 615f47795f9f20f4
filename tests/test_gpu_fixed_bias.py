"""Fixed-point passes: roundings without a bias.  A bias of every frequency's
real part adds up at one place, azimuth 0 of every row (the row transforms) or
the first row of the axisymmetric part (the column transforms)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
EPS = 2.0**-52


def _plan(nu, nphi, dtype):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1509_01450_gb300 import Plan

    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    return torch, Plan(nu, nphi, u_min, du, 1.0, dtype).build()


@pytest.mark.parametrize("dtype", ["float64", "float32x2"])
def test_rows(dtype):
    """One Fourier mode of another phase in every row, and the same rolled by a
    third of the way round: the two agree to rounding, 10 eps of the rms a cell
    (FP64 transforms of this size), independent from row to row, so that a
    column's mean over 512 rows stays within 5 x 10 eps / sqrt(512) < 5e-16 of
    zero; twice that is allowed."""
    nu, nphi = 512, 4096
    torch, plan = _plan(nu, nphi, dtype)
    phase = np.random.default_rng(1).uniform(0.0, 2.0 * np.pi, (nu, 1))
    s = torch.tensor(np.cos(2.0 * np.pi * 3 * np.arange(nphi)[None] / nphi + phase), device="cuda")
    k = nphi // 3
    for a, b in zip(plan.forces(s), plan.forces(s.roll(k, 1).contiguous())):
        d = (a - b.roll(-k, 1)) / a.pow(2).mean().sqrt()
        assert float(d.mean(0).abs().max()) < 1e-15
    plan.check()


@pytest.mark.parametrize("nu", [512, 2048])
def test_columns(nu):
    """Axisymmetric densities, a Fourier mode in u of several phases, against the
    ring sums in extended precision.  Three roundings to FP64 of the column, the
    field and the spectrum leave about eps of the rms a row, the largest of 2048
    rows under 5 eps; the mean over the phases is held to that."""
    nphi = 64
    torch, plan = _plan(nu, nphi, "float64")
    kr, _ = plan.kernels()
    ring = np.asarray(kr, dtype=np.longdouble).reshape(2 * nu - 1, nphi).sum(1)
    i = np.arange(nu)
    M = ring[i[:, None] - i[None, :] + nu - 1]
    err = np.zeros(nu)
    phases = np.random.default_rng(3).uniform(0.0, 6.0, 16)
    for p in phases:
        x = np.cos(2.0 * np.pi * 5 * i / nu + p)
        F = plan.forces(torch.tensor(x[:, None] * np.ones((1, nphi)), device="cuda"))[0][:, 0].cpu().numpy()
        ref = M @ x.astype(np.longdouble)
        err += ((F - ref) / np.sqrt((ref**2).mean())).astype(np.float64)
    plan.check()
    assert np.abs(err).max() / len(phases) < 5 * EPS
