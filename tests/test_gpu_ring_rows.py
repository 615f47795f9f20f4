"""Persistent row passes (FP32 rows of 8192 points, more units of rows than
SMs): the sizes around the line, against the same plan's kernels in an FP64
convolution (FP32 rounding of an FFT convolution: a few eps log2 n relative to
the norm, eps = 6e-8, under 1e-5), and the forward bit for bit against the
one-block-per-unit row pass, which pinned host densities take."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


# 152 SMs, units of 4 and 2 rows: no pass persistent, those of 2 rows, all (last round ragged, several rounds)
@pytest.mark.parametrize("nu", [256, 512, 1024, 2048])
def test_forward_and_adjoint(nu):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1509_01450_gb300 import Plan

    nphi = 8192
    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    plan = Plan(nu, nphi, u_min, du, 1.0, "float32").build()
    kr, kp = plan.kernels()
    s = (np.abs(workloads.random_field(nu, nphi, 5)) + 0.1).astype(np.float32)
    st = torch.tensor(s)
    F = plan.forces(st.cuda())
    plan.check()
    assert oracle.rel_l2(*(x.cpu().numpy() for x in F), *oracle.fft_conv(s.astype(np.float64), kr, kp)) < 1e-5
    g = [workloads.random_field(nu, nphi, 6 + k).astype(np.float32) for k in range(2)]
    gs = plan.backward(*(torch.tensor(x, device="cuda") for x in g)).cpu().numpy().astype(np.float64)
    ref = oracle.fft_conv_T(*(x.astype(np.float64) for x in g), kr, kp)
    assert np.linalg.norm(gs - ref) < 1e-5 * np.linalg.norm(ref)
    host = [st.pin_memory(), *(torch.empty_like(st).pin_memory() for _ in range(2))]
    plan.forces_host(*host)
    plan.check()
    assert torch.equal(host[1], F[0].cpu()) and torch.equal(host[2], F[1].cpu())
