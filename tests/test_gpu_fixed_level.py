"""Fixed-point row passes on rows whose peak lies at azimuth 0: a periodic
convolution knows no first column, so a source of one cell (or of a Gaussian
one cell wide) there gives the forces, and as a seed the gradient, of the same
source a fifth of the way round, rolled.

Tolerance, relative to the norm over the rings.  The azimuthal mean of a ring
goes through three roundings to FP64 (its half spectrum, the column's result,
the field: eps / 2 each, the last relative to the ring's mean modulus) and
fixed-point transforms below them, on both sides: under 20 eps = 4.4e-15.  The
whole fields as in the other fixed-point tests: 3e-14.  Both runs use the same
kernel spectra, so compensated plans keep the same bounds."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
EPS = 2.0**-52


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def _source(nu, nphi, kind):
    s = np.zeros((nu, nphi))
    d = np.minimum(np.arange(nphi), nphi - np.arange(nphi))
    s[nu // 3] = 0.7310585786300049 * (d == 0 if kind == "cell" else np.exp(-0.5 * d * d))
    return s


@pytest.mark.parametrize("dtype", ["float64", "float32x2"])
@pytest.mark.parametrize("nu,nphi", [(128, 1024), (128, 2048), (64, 4096)])
@pytest.mark.parametrize("kind", ["cell", "gauss"])
def test_rolled(torch_cuda, nu, nphi, dtype, kind):
    torch = torch_cuda
    from paper_1509_01450_gb300 import Plan

    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    plan = Plan(nu, nphi, u_min, du, 1.0, dtype).build()
    s = torch.tensor(_source(nu, nphi, kind), device="cuda")
    k, zero = nphi // 5, torch.zeros_like(s)
    r = s.roll(k, 1).contiguous()
    at0 = [*plan.forces(s), plan.backward(s, zero), plan.backward(zero, s)]
    rolled = [*plan.forces(r), plan.backward(r, zero), plan.backward(zero, r)]
    plan.check()
    norm = lambda x: float(x.norm())  # noqa: E731
    for a, b in zip(at0, (x.roll(-k, 1) for x in rolled)):
        assert norm(a - b) < 3e-14 * norm(b)
    for n in (0, 2):  # F_r and the gradient of F_r (the azimuthal kernel has no mean)
        a, b = at0[n].mean(1), rolled[n].mean(1)
        assert norm(a - b) < 20 * EPS * norm(b)


def test_range(torch_cuda):
    """A cell of 0.73 2^1013 at azimuth 0, whose 4096-fold is beyond FP64's range:
    its forces are those of the unscaled cell, scaled, bit for bit."""
    torch = torch_cuda
    from paper_1509_01450_gb300 import Plan

    nu, nphi = 64, 4096
    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    plan = Plan(nu, nphi, u_min, du, 1.0, "float64").build()
    s = torch.tensor(_source(nu, nphi, "cell"), device="cuda")
    for a, b in zip(plan.forces(s * 2.0**1013), plan.forces(s)):
        assert torch.equal(a, b * 2.0**1013)
