"""Cases for the checked-build test of the persistent and the fixed-point passes
(tests/test_gpu_checked_persistent.py), laid out as checked_cases.py: run_all()
computes them with whichever library sg.lib() loads; run as a script (with
SG_LIBRARY_VARIANT=checked) it builds and loads the index-checked library and
saves the results to the .npz file named by its argument."""
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import workloads  # noqa: E402

# (N_u, N_phi, dtype, build options): persistent rows; persistent columns; both;
# fixed-point passes with double-float weights, and of one and of several
# transforms to a warp; rows in fixed point between edge updates
CASES = [
    (2048, 8192, "float32", {}),
    (4096, 512, "float32", {}),
    (4096, 8192, "float32", {}),
    (256, 512, "float32x2", {"weight_p": 1}),
    (64, 128, "float32x2", {}),
    (32, 64, "float64", {}),
    (128, 2048, "float64", {"radial_edges": 1}),
]


def run_all():
    import torch

    from paper_1509_01450_gb300 import Plan

    out = {}
    for nu, nphi, dtype, opts in CASES:
        u_min, du = workloads.grid_params(nu, 0.1, 10.0)
        plan = Plan(nu, nphi, u_min, du, 1.0, dtype).build(**opts)
        f = [torch.tensor(workloads.random_field(nu, nphi, 3 + k), dtype=plan.dtype, device="cuda") for k in range(3)]
        res = [*plan.forces(f[0].abs() + 0.1), plan.backward(f[1], f[2])]
        plan.check()  # raises SgError (SG_ERR_BOUNDS) if an index check failed
        for k, a in enumerate(res):
            out[f"{dtype}-{nu}x{nphi}/{k}"] = a.cpu().numpy()
        plan.close()
    return out


if __name__ == "__main__":
    assert os.environ.get("SG_LIBRARY_VARIANT") == "checked"
    from paper_1509_01450_gb300 import build, sg

    build.build(checked=True)
    assert sg.lib().sg_checked_build() == 1
    np.savez(sys.argv[1], **run_all())
