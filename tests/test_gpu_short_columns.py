"""FP32 column passes of 64 and 128 points with fixed lengths, beside fixed-length
rows (256 points on) and tensor-core rows: plain, with one-sided edges and with
the origin wedge, forward and adjoint, against an FP64 plan of the same options
(FP32 rounding of an FFT convolution: a few eps log2 n relative to the norm,
eps = 6e-8, under 1e-5)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


# 64 and 128 points; the smallest and largest row blocks, rows fewer than a large block holds
@pytest.mark.parametrize("opts", [{}, {"radial_edges": 1}, {"radial_edges": 1, "wedge": 1}])
@pytest.mark.parametrize("nu,nphi,short", [(32, 256, 0), (64, 256, 0), (32, 1024, 0), (64, 2048, 0), (32, 4096, 0),
                                           (64, 64, 1), (32, 128, 1)])
def test_against_fp64(nu, nphi, short, opts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1509_01450_gb300 import Plan

    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    s = np.abs(workloads.random_field(nu, nphi, 5)) + 0.1
    w = np.abs(workloads.random_field(1, nphi, 9))[0] + 0.1
    g = [workloads.random_field(nu, nphi, 6 + k) for k in range(2)]
    got = {}
    for dtype in ("float64", "float32"):
        plan = Plan(nu, nphi, u_min, du, 1.0, dtype).build(short_dft=short if dtype == "float32" else 0, **opts)
        t = [torch.tensor(x, dtype=plan.dtype, device="cuda") for x in (s, w, *g)]
        if opts.get("wedge"):
            out = [*plan.forces_wedge(t[0], t[1]), *plan.backward_wedge(t[2], t[3])]
        else:
            out = [*plan.forces(t[0]), plan.backward(t[2], t[3])]
        plan.check()
        got[dtype] = [x.double().cpu() for x in out]
    norm = lambda v: float(torch.cat([x.flatten() for x in v]).norm())  # noqa: E731
    for part in ((0, 2), (2, 3), (3, 4)):
        a, b = (got[d][part[0]:part[1]] for d in ("float32", "float64"))
        if a:
            assert norm([x - y for x, y in zip(a, b)]) < 1e-5 * norm(b)
