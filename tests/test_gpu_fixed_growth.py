"""Fixed-point passes at the ends of what a block of values can grow by in a
pass: an impulse (no growth, so that the block is moved up before its twiddle
products), one Fourier mode and a constant along each axis (three bits a
pass), against numpy's convolution with the plan's folded kernels.  The
tolerance is the reference's rounding: three transforms along two axes of at
most 2^23 points in all, 10 eps log2(2^23) < 3e-14 relative to the norm
(compensated plans: 4e-15 per entry more, under 1e-13)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,tol", [("float64", 3e-14), ("float32x2", 1e-13)])
@pytest.mark.parametrize("nu,nphi", [(128, 256), (512, 512), (1024, 2048), (2048, 4096)])
@pytest.mark.parametrize("kind", ["impulse", "mode", "column", "row"])
def test_growth(nu, nphi, dtype, tol, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1509_01450_gb300 import Plan

    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    plan = Plan(nu, nphi, u_min, du, 1.0, dtype).build()
    kr, kp = plan.kernels()
    s = np.zeros((nu, nphi))
    if kind == "impulse":
        s[nu // 3, nphi // 5] = 1.0
    elif kind == "mode":
        s[:] = 2.0 + np.cos(2 * np.pi * (3 * np.arange(nphi)[None] / nphi + 5 * np.arange(nu)[:, None] / nu))
    elif kind == "column":
        s[:, nphi // 5] = 1.0
    else:
        s[nu // 3] = 1.0
    F = [x.cpu().numpy() for x in plan.forces(torch.tensor(s, device="cuda"))]
    plan.check()
    assert oracle.rel_l2(*F, *oracle.fft_conv(s, kr, kp)) < tol
    g = [s, s[::-1].copy()]
    gs = plan.backward(*(torch.tensor(x, device="cuda") for x in g)).cpu().numpy()
    ref = oracle.fft_conv_T(*g, kr, kp)
    assert np.linalg.norm(gs - ref) < tol * np.linalg.norm(ref)
