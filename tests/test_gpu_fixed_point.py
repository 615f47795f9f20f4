"""The fixed-point passes of the FP64 and compensated plans at the edges of
their range: rows and columns of 256 .. 4096 points, alone and together with
the run-time-length passes, against numpy's convolution with the plan's own
folded kernels.

Tolerances.  The reference's rounding: numpy's FFT of n points errs by about
eps log2 n relative to the norm, three transforms along two axes; with eps =
1.1e-16 and n <= 8192 x 4096 points that stays under 10 eps log2(2^25) = 3e-14.
Compensated plans hold their spectra as double-floats (48 bits): 4e-15 per
entry more, under 1e-13 in all.
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
TOL = {"float64": 3e-14, "float32x2": 1e-13}
# (N_u, N_phi): both shortest, both longest, rows only, columns only, odd mode
# counts per column block, one row block of each length
SIZES = [(128, 256), (8, 256), (128, 64), (128, 4), (256, 512), (512, 1024), (64, 2048), (1024, 512), (2048, 256),
         (4, 4096), (2048, 4096)]


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def _case(torch, nu, nphi, dtype, **opts):
    from paper_1509_01450_gb300 import Plan

    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    plan = Plan(nu, nphi, u_min, du, 1.0, dtype).build(**opts)
    s = np.abs(workloads.random_field(nu, nphi, 3 * nu + nphi)) + 0.1
    return plan, s, torch.tensor(s, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("dtype", ["float64", "float32x2"])
@pytest.mark.parametrize("nu,nphi", SIZES)
def test_forward_and_adjoint(torch_cuda, nu, nphi, dtype):
    torch = torch_cuda
    plan, s, sd = _case(torch, nu, nphi, dtype)
    kr, kp = plan.kernels()
    Fr, Fp = (x.cpu().numpy() for x in plan.forces(sd))
    plan.check()
    assert oracle.rel_l2(Fr, Fp, *oracle.fft_conv(s, kr, kp)) < TOL[dtype]
    g = [workloads.random_field(nu, nphi, 7 + k) for k in range(2)]
    gs = plan.backward(*(torch.tensor(x, device="cuda") for x in g)).cpu().numpy()
    ref = oracle.fft_conv_T(*g, kr, kp)
    assert np.linalg.norm(gs - ref) < TOL[dtype] * np.linalg.norm(ref)


@pytest.mark.parametrize("nu,nphi", [(128, 256), (256, 1024)])
def test_exponents(torch_cuda, nu, nphi):
    """A density scaled by a power of two gives the forces scaled by it, bit
    for bit, over FP64's range (one exponent per block); zero gives zero; an
    infinity or NaN anywhere gives NaN everywhere, as FP64 sums do."""
    torch = torch_cuda
    plan, _, sd = _case(torch, nu, nphi, "float64")
    F = plan.forces(sd)
    for k in (-900, -30, 1, 900):
        for a, b in zip(plan.forces(sd * 2.0**k), F):
            assert torch.equal(a, b * 2.0**k)
    for a in plan.forces(torch.zeros_like(sd)):
        assert torch.equal(a, torch.zeros_like(a))
    for bad in (float("inf"), float("nan")):
        x = sd.clone()
        x[nu // 3, nphi // 5] = bad
        for a in (*plan.forces(x), plan.backward(x, sd)):
            assert torch.isnan(a).all()
