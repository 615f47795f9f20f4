"""Transforms of the fixed-point passes that share a warp, a block or a
transform with a much stronger row that has no part in what is compared."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


# rows of 64 and 128 points (several to a warp), of one and of several warps, of 4096
@pytest.mark.parametrize("dtype", ["float64", "float32x2"])
@pytest.mark.parametrize("nu,nphi", [(32, 64), (64, 128), (128, 256), (64, 1024), (32, 4096)])
def test_weak_row_beside_a_constant_one(nu, nphi, dtype):
    """Even rows constant, odd rows 2^-40 of them: a pair is one transform.  The
    azimuthal force knows nothing of the constant rows, and the gradient nothing
    of a constant gF_phi beside a weak gF_r: both are those of the weak rows
    alone, to the other fixed-point tests' 3e-14 of the norm (at one exponent a
    pair the weak rows are rounded at 2^-20 of themselves).  The mean modes of
    the strong rows leave their own rounding, 2^-53, in the axisymmetric part
    only, and the passes' 2^-59 of that, 2^-72 of the weak rows, beside it."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1509_01450_gb300 import Plan

    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    plan = Plan(nu, nphi, u_min, du, 1.0, dtype).build()
    even = (np.arange(nu) % 2 == 0)[:, None]
    weak = 2.0**-40 * np.where(even, 0.0, workloads.random_field(nu, nphi, 5))
    strong = np.where(even, 0.7310585786300049, 0.0) * np.ones((nu, nphi))
    w, s = (torch.tensor(x, device="cuda") for x in (weak, strong))
    g = torch.tensor(2.0**-40 * workloads.random_field(nu, nphi, 6), device="cuda")
    flat = torch.full_like(g, 0.7310585786300049)
    for a, b in ((plan.forces(w + s)[1], plan.forces(w)[1]),
                 (plan.backward(g, flat), plan.backward(g, torch.zeros_like(g)))):
        assert float((a - b).norm()) < 3e-14 * float(b.norm())
    plan.check()


# rows and columns of 64 and 128 points (several to a warp), one to a warp, one to several
@pytest.mark.parametrize("dtype", ["float64", "float32x2"])
@pytest.mark.parametrize("nu,nphi", [(32, 64), (64, 128), (32, 2048), (128, 256), (512, 64), (64, 1024)])
def test_weak_rows(nu, nphi, dtype):
    """Weak rows of 2^-80 beside pairs of constant rows of ones: what comes out of
    the azimuthal force and of the adjoint of it is the weak rows' alone, and at an
    exponent shared with a strong row, with the strong mode-0 column or with that
    column's rounding in the Nyquist mode, part or all of it would be lost.
    Compared with the weak rows alone, to 3e-14 of the norm."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1509_01450_gb300 import Plan

    u_min, du = workloads.grid_params(nu, 0.1, 10.0)
    plan = Plan(nu, nphi, u_min, du, 1.0, dtype).build()
    strong = (np.arange(nu) & 2 == 0)[:, None]  # in pairs: a pair of rows is one transform
    a, b = (2.0**-80 * np.where(strong, 0.0, workloads.random_field(nu, nphi, 5 + k)) for k in range(2))
    dev = lambda x: torch.tensor(x, device="cuda")  # noqa: E731
    ones = np.where(strong, 1.0, 0.0)

    def close(x, y):
        assert float(y.norm()) > 0.0
        assert float((x - y).norm()) < 3e-14 * float(y.norm())

    close(plan.forces(dev(a + ones))[1], plan.forces(dev(a))[1])
    close(plan.backward(dev(a), dev(b + ones)), plan.backward(dev(a), dev(b)))
    plan.check()
