"""Device memory of compensated plans: those on the fixed-point passes hold
what an FP64 plan holds (same element sizes) and no double-float working
fields; with edges, the wedge or lengths without fixed-point passes they hold
the working fields and no fixed-point spectra.  Rebuilt with other options a
plan gives what a plan built so at once gives, and each allocation of a build
or load that fails gives SG_ERR_ALLOC and leaves nothing behind."""
import gc

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def _plan(nu, nphi, dtype):
    from paper_1509_01450_gb300 import Plan

    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    return Plan(nu, nphi, u_min, du, 1.0, dtype)


def _run(torch, plan, opts):
    nu, nphi = plan.nu, plan.nphi
    s, g, h = (torch.tensor(workloads.random_field(nu, nphi, 5 + k), device="cuda") for k in range(3))
    if opts.get("wedge"):
        w = torch.tensor(np.abs(workloads.random_field(1, nphi, 9))[0], device="cuda")
        return [*plan.forces_wedge(s, w), *plan.backward_wedge(g, h)]
    return [*plan.forces(s), plan.backward(g, h)]


OPTS = [{}, {"radial_edges": 1}, {"radial_edges": 1, "wedge": 1}]


@pytest.mark.parametrize("opts", OPTS)
@pytest.mark.parametrize("nu,nphi", [(128, 256), (32, 64), (16, 64), (64, 32)])
def test_bytes(torch_cuda, nu, nphi, opts):
    a, b = (_plan(nu, nphi, d).build(**opts) for d in ("float32x2", "float64"))
    fixed = nu >= 32 and nphi >= 64
    spectra = 2 * (nphi // 2 + 1) * (nu + 2) * 16 if nu >= 32 else 0  # the FP64 plan's, in fixed point
    more = 0 if fixed and not opts else 3 * nu * nphi * 8 - spectra + (2 * nphi * 8 if opts.get("wedge") else 0)
    assert a.device_bytes() == b.device_bytes() + more


def test_rebuilt_with_other_options(torch_cuda):
    torch = torch_cuda
    plan = _plan(128, 256, "float32x2")
    for opts in (OPTS[0], OPTS[2], OPTS[0], OPTS[1], OPTS[0]):
        got = _run(torch, plan.build(**opts), opts)
        plan.check()
        for a, b in zip(got, _run(torch, _plan(128, 256, "float32x2").build(**opts), opts)):
            assert torch.equal(a, b)


@pytest.mark.parametrize("opts", OPTS)
def test_failing_allocations(torch_cuda, opts, tmp_path):
    torch = torch_cuda
    from paper_1509_01450_gb300 import Plan, sg

    L = sg.lib()

    def count(fn):
        L.sg_test_fail_alloc(1 << 30)
        try:
            fn()
        finally:
            left = L.sg_test_fail_alloc(-1)
        return (1 << 30) - left

    def fails(k, fn):
        L.sg_test_fail_alloc(k)
        try:
            with pytest.raises(sg.SgError) as e:
                fn()
        finally:
            L.sg_test_fail_alloc(-1)
        assert e.value.status == sg.SG_ERR_ALLOC, k

    ref = _plan(64, 128, "float32x2").build(**opts)
    want = _run(torch, ref, opts)
    gc.collect()
    live = L.sg_test_live_allocations()
    plan = _plan(64, 128, "float32x2")
    n = count(lambda: plan.build(**opts))
    plan.close()
    for k in range(n):
        plan = _plan(64, 128, "float32x2")
        fails(k, lambda: plan.build(**opts))
        for a, b in zip(_run(torch, plan.build(**opts), opts), want):
            assert torch.equal(a, b)
        plan.close()
    if not opts:
        path = str(tmp_path / "plan.sg")
        ref.save(path)
        for k in range(count(lambda: Plan.load(path).close())):
            fails(k, lambda: Plan.load(path))
        plan = Plan.load(path)
        for a, b in zip(_run(torch, plan, opts), want):
            assert torch.equal(a, b)
        plan.close()
    gc.collect()
    assert L.sg_test_live_allocations() == live
