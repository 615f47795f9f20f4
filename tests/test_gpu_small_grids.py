"""Row passes whose blocks shrink with the grid (FP32): the sizes where the
block shape changes, against the same plan's FP64 forces on the same density
(FP32 rounding of an FFT convolution: a few eps log2 n relative to the norm,
eps = 6e-8, under 1e-5) and bit for bit against the batched kernels, whose
blocks always hold 256 threads' worth of transforms."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


# run-time rows: one warp per block up to several blocks; fixed rows below and
# above one block per SM (152: 4 rows x 8 / 4 / 2 / 1 slots of 256 .. 2048 points)
@pytest.mark.parametrize("nu,nphi", [(4, 4), (64, 64), (4096, 32), (512, 128), (128, 256), (2048, 256), (256, 512),
                                     (512, 1024), (2048, 1024), (128, 2048), (1024, 2048)])
def test_forward_and_adjoint(torch_cuda, nu, nphi):
    torch = torch_cuda
    from paper_1509_01450_gb300 import Plan, forces_batched

    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    plan = Plan(nu, nphi, u_min, du, 1.0, "float32").build()
    kr, kp = plan.kernels()
    s = (np.abs(workloads.random_field(nu, nphi, 5)) + 0.1).astype(np.float32)
    sd = torch.tensor(s, device="cuda")
    F = plan.forces(sd)
    plan.check()
    assert oracle.rel_l2(*(x.cpu().numpy() for x in F), *oracle.fft_conv(s.astype(np.float64), kr, kp)) < 1e-5
    g = [workloads.random_field(nu, nphi, 6 + k).astype(np.float32) for k in range(2)]
    gs = plan.backward(*(torch.tensor(x, device="cuda") for x in g)).cpu().numpy().astype(np.float64)
    ref = oracle.fft_conv_T(*(x.astype(np.float64) for x in g), kr, kp)
    assert np.linalg.norm(gs - ref) < 1e-5 * np.linalg.norm(ref)
    B = [torch.empty_like(sd) for _ in range(2)]
    forces_batched([(plan, sd, *B)])
    assert torch.equal(B[0], F[0]) and torch.equal(B[1], F[1])
