"""Persistent columns (FP32 columns of 8192 points, more modes than SMs) between
row passes that are not persistent, and the last size before them: against the
same plan's kernels in an FP64 convolution (FP32 rounding of an FFT
convolution: a few eps log2 n relative to the norm, eps = 6e-8, under 1e-5)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


# 152 SMs: 128 modes (one block a mode); 256 and 512 (the last round ragged); 1024 modes over several rounds
@pytest.mark.parametrize("nphi", [256, 512, 1024, 2048])
def test_forward_and_adjoint(nphi):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1509_01450_gb300 import Plan

    nu = 4096
    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    plan = Plan(nu, nphi, u_min, du, 1.0, "float32").build()
    kr, kp = plan.kernels()
    s = (np.abs(workloads.random_field(nu, nphi, 5)) + 0.1).astype(np.float32)
    F = plan.forces(torch.tensor(s, device="cuda"))
    plan.check()
    assert oracle.rel_l2(*(x.cpu().numpy() for x in F), *oracle.fft_conv(s.astype(np.float64), kr, kp)) < 1e-5
    g = [workloads.random_field(nu, nphi, 6 + k).astype(np.float32) for k in range(2)]
    gs = plan.backward(*(torch.tensor(x, device="cuda") for x in g)).cpu().numpy().astype(np.float64)
    plan.check()
    ref = oracle.fft_conv_T(*(x.astype(np.float64) for x in g), kr, kp)
    assert np.linalg.norm(gs - ref) < 1e-5 * np.linalg.norm(ref)
