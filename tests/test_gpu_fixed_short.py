"""Fixed-point passes of 64 and 128 points (several transforms to a warp, each
with its own exponent), as rows, as columns and both, alone and beside the
longer and the run-time-length passes: against numpy's convolution with the
plan's folded kernels, and with rows 2^60 below their neighbours (whose own
rounding would show there if a warp's transforms shared an exponent).  The
tolerance is the reference's rounding: three
transforms along two axes of at most 2^19 points, 10 eps log2(2^19) < 3e-14
relative to the norm (compensated plans 1e-13)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
TOL = {"float64": 3e-14, "float32x2": 1e-13}
# 64, 128 points: both; rows only; columns only; beside other lengths; ragged mode counts per column block
SIZES = [(32, 64), (64, 128), (32, 128), (64, 64), (16, 64), (8, 128), (4, 128), (32, 4), (64, 16), (32, 32), (64, 2048),
         (512, 64), (1024, 128)]


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


@pytest.mark.parametrize("dtype", ["float64", "float32x2"])
@pytest.mark.parametrize("nu,nphi", SIZES)
def test_forward_and_adjoint(torch_cuda, nu, nphi, dtype):
    torch = torch_cuda
    from paper_1509_01450_gb300 import Plan

    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    plan = Plan(nu, nphi, u_min, du, 1.0, dtype).build()
    kr, kp = plan.kernels()
    s = np.abs(workloads.random_field(nu, nphi, 3 * nu + nphi)) + 0.1
    F = [x.cpu().numpy() for x in plan.forces(torch.tensor(s, device="cuda"))]
    plan.check()
    assert oracle.rel_l2(*F, *oracle.fft_conv(s, kr, kp)) < TOL[dtype]
    g = [workloads.random_field(nu, nphi, 7 + k) for k in range(2)]
    gs = plan.backward(*(torch.tensor(x, device="cuda") for x in g)).cpu().numpy()
    ref = oracle.fft_conv_T(*g, kr, kp)
    assert np.linalg.norm(gs - ref) < TOL[dtype] * np.linalg.norm(ref)


@pytest.mark.parametrize("nu,nphi", [(32, 64), (64, 128), (32, 2048)])
def test_exponents(torch_cuda, nu, nphi):
    """Scaling by powers of two is exact, zero gives zero, an infinity or NaN
    gives NaN everywhere; rows scaled apart by 2^60 transform each at its own
    exponent: the adjoint of forces in one row alone is the same, to rounding,
    as with the other rows 2^-60 of it (far below the tolerance)."""
    torch = torch_cuda
    from paper_1509_01450_gb300 import Plan

    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    plan = Plan(nu, nphi, u_min, du, 1.0, "float64").build()
    s = np.abs(workloads.random_field(nu, nphi, 5)) + 0.1
    sd = torch.tensor(s, device="cuda")
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
    one = torch.zeros_like(sd)
    one[nu // 2] = sd[nu // 2]
    small = sd * 2.0**-60
    small[nu // 2] = sd[nu // 2]
    zero = torch.zeros_like(sd)
    a, b = plan.backward(one, zero), plan.backward(small, zero)
    assert float((a - b).norm()) < 3e-14 * float(a.norm())
