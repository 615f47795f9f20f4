"""The framework's work as a user's program has it done, as measurable cases.

A case is one time step (or one gradient step) of a program that keeps a
prepared plan and calls the library on a new surface density: forces, their
adjoint, the differentiable step, the origin wedge, one-sided edges, the three
precisions, the tensor-core rows and the batched form.  `listed` names the
sizes of the repository's own workloads (the 64 x 64, 512 x 1024, 1024 x 2048
and 2048 x 4096 disks, the largest plan, the 256-disk batch); `draw` takes
others of the same ranges.  The library takes powers of two only, so ragged
work comes through the batch (any number of disks, mixed sizes) and through
grids that are far from square.

`exact` evaluates the same sums in 64 bits with plain torch and numpy: the
cell integrals by tensor Gauss-Legendre rules (graded toward the singular
point where a cell lies close to it, the own cell from its closed form in
eta), the slope terms folded, the convolution by torch.fft, and every
gradient by torch's own differentiation of that map.
"""
from __future__ import annotations

import math

import numpy as np
import torch

# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
# call: what a pass runs.  "forces", "adjoint" (plan.backward), "step"
# (self_gravity and the gradient of its outputs), "wedge" (forces_wedge and
# backward_wedge), "batch" (forces_batched over `disks` disks)


def _case(call, nu, nphi, dtype="float32", r_in=0.01, r_out=100.0, **more):
    c = {"call": call, "nu": nu, "nphi": nphi, "dtype": dtype, "r_in": r_in, "r_out": r_out, "weight_p": 0,
         "edges": 0, "short_dft": 0, "disks": 1}
    c.update(more)
    return c


def listed():
    out = [
        # the smallest disk in use (a test problem, or one ring of many): launches and host work count
        ("forces_64x64_f32", _case("forces", 64, 64, r_in=0.05, r_out=20.0)),
        # an ordinary simulation step with one-sided edge slopes
        ("edges_256x512_f32", _case("forces", 256, 512, edges=1)),
        # an ordinary simulation step, spiral and clump
        ("forces_512x1024_f32", _case("forces", 512, 1024)),
        # the headline step
        ("forces_2048x4096_f32", _case("forces", 2048, 4096)),
        # the largest plan the library takes
        ("forces_4096x8192_f32", _case("forces", 4096, 8192)),
        # the headline step's transpose, as a caller with its own chain rule uses it
        ("adjoint_2048x4096_f32", _case("adjoint", 2048, 4096)),
        # one differentiable evaluation: forward through autograd and the gradient
        ("step_1024x2048_f32", _case("step", 1024, 2048)),
        # a disk that reaches the origin: forces with the wedge and both gradients
        ("wedge_1024x2048_f32", _case("wedge", 1024, 2048, edges=1)),
        # many rings, few azimuths, on the tensor-core rows
        ("rows32_4096x32_f32", _case("forces", 4096, 32, r_in=1e-4, r_out=1e4, short_dft=1)),
        # reference precision
        ("forces_1024x2048_f64", _case("forces", 1024, 2048, dtype="float64")),
        # loss gradients in the compensated precision
        ("step_1024x2048_f32x2", _case("step", 1024, 2048, dtype="float32x2")),
        # an ensemble: 256 disks of 16 sizes in one call
        ("batch_256_f32", _case("batch", 0, 0, disks=256)),
    ]
    return [dict(c, name=n) for n, c in out]


def _pow2(rng, lo, hi):
    return 2 ** rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def draw(rng):
    kind = rng.choice(["forces", "forces", "adjoint", "step", "wedge", "edges", "rows", "f64", "f32x2", "batch"])
    if kind == "batch":
        return _case("batch", 0, 0, disks=rng.randint(2, 256), r_in=round(10 ** rng.uniform(-2.0, -1.0), 4))
    if kind == "rows":
        nu, nphi = _pow2(rng, 64, 4096), _pow2(rng, 32, 128)
        most = 4.0
    elif kind in ("f64", "f32x2", "wedge"):
        nu, nphi = _pow2(rng, 32, 1024), _pow2(rng, 64, 2048)
        most = 4.0
    else:
        nu, nphi = _pow2(rng, 32, 4096), _pow2(rng, 32, 8192)
        most = 4.0
        while nu * nphi > 2 ** 23:
            nu //= 2
    # the radial extent: cells from 1/64 to twice as long in u as in phi, within 10^-4 .. 10^4
    dphi = 2.0 * math.pi / nphi
    span = min(nu * dphi * 2.0, rng.uniform(1.0, most) * math.log(10.0))
    r_out = round(10 ** rng.uniform(0.0, 2.0), 4)
    r_in = float("%.6g" % (r_out * math.exp(-span)))
    p = rng.choice([0, 0, 1]) if span < 4.0 else 0  # p = 1 where r_out / r_in is small
    call = {"edges": "forces", "rows": "forces", "f64": rng.choice(["forces", "adjoint"]),
            "f32x2": rng.choice(["forces", "step"])}.get(kind, kind)
    return _case(call, nu, nphi, dtype={"f64": "float64", "f32x2": "float32x2"}.get(kind, "float32"), r_in=r_in,
                 r_out=r_out, weight_p=p, edges=1 if kind in ("edges", "wedge") else 0,
                 short_dft=1 if kind == "rows" else 0)


# ---------------------------------------------------------------------------
# inputs (from the seed alone)
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _grid(c):
    return math.log(c["r_in"]), math.log(c["r_out"] / c["r_in"]) / c["nu"]


def _centres(nu, nphi, u_min, du):
    i = torch.arange(nu, dtype=torch.float64, device=_device())
    r = 0.5 * (1.0 + math.exp(du)) * torch.exp(u_min + du * i)
    phi = (torch.arange(nphi, dtype=torch.float64, device=_device()) + 0.5) * (2.0 * math.pi / nphi)
    return r[:, None], phi[None, :]


def _random_field(nu, nphi, gen):
    """Unit-variance Gaussian field on the index torus with a k^-3 spectrum."""
    w = torch.randn((nu, nphi), generator=gen, device=_device(), dtype=torch.float32)
    ku = torch.fft.fftfreq(nu, device=_device())[:, None] * nu
    kp = torch.fft.rfftfreq(nphi, device=_device())[None, :] * nphi
    k2 = ku * ku + kp * kp
    k2[0, 0] = 1.0
    amp = k2 ** -0.75
    amp[0, 0] = 0.0
    g = torch.fft.irfft2(torch.fft.rfft2(w) * amp, s=(nu, nphi)).double()
    return g / g.std()


def _spiral(r, phi, rng):
    """A Kuzmin disk with a logarithmic spiral and an off-centre Kuzmin clump."""
    m, amp, pitch = rng.integers(1, 5), rng.uniform(0.05, 0.2), math.radians(rng.uniform(10.0, 30.0))
    s = (1.0 + amp * torch.cos(m * phi - torch.log(r) / math.tan(pitch))) / (2.0 * math.pi * (r * r + 1.0) ** 1.5)
    rc, pc = rng.uniform(1.0, 4.0), rng.uniform(0.0, 2.0 * math.pi)
    x, y = r * torch.cos(phi) - rc * math.cos(pc), r * torch.sin(phi) - rc * math.sin(pc)
    return s + 0.05 * 0.2 / (2.0 * math.pi * (x * x + y * y + 0.04) ** 1.5)


def _real(c):
    return torch.float32 if c["dtype"] == "float32" else torch.float64


def _sizes(c):
    """The batch's (N_u, N_phi) per disk: drawn from the sixteen sizes."""
    rng = np.random.default_rng(1450 + c["disks"])
    return [(int(rng.choice([128, 256, 512, 1024])), int(rng.choice([256, 512, 1024, 2048])))
            for _ in range(c["disks"])]


def _inputs(c, seed):
    """sigma, and by call gF_r, gF_phi and sigma_w, in the fields' type."""
    gen = torch.Generator(device=_device())
    gen.manual_seed(int(seed) * 7919 + 17)
    rng = np.random.default_rng(int(seed))
    dt = _real(c)
    if c["call"] == "batch":
        out, u_min = [], math.log(c["r_in"])
        for nu, nphi in _sizes(c):
            r, phi = _centres(nu, nphi, u_min, math.log(c["r_out"] / c["r_in"]) / nu)
            m, amp, pitch = int(rng.integers(1, 5)), rng.uniform(0.0, 0.2), math.radians(rng.uniform(10.0, 30.0))
            # an exponential disk with a log spiral; the phase comes from the seed
            ph = rng.uniform(0.0, 2.0 * math.pi)
            s = torch.exp(-r / 3.0) * (1.0 + amp * torch.cos(m * phi - torch.log(r) / math.tan(pitch) + ph))
            out.append(s.to(dt))
        return {"sigma": out}
    nu, nphi = c["nu"], c["nphi"]
    u_min, du = _grid(c)
    r, phi = _centres(nu, nphi, u_min, du)
    if nu * nphi >= 2 ** 21:  # log-normal disk
        sigma = torch.exp(0.5 * _random_field(nu, nphi, gen)) * torch.exp(-r / 3.0)
    else:
        sigma = _spiral(r, phi, rng)
    out = {"sigma": sigma.to(dt)}
    if c["call"] in ("adjoint", "step", "wedge"):
        # seeds of a loss on the forces, falling off with radius like the disk
        fall = 1.0 / (1.0 + r)
        out["g_r"] = (_random_field(nu, nphi, gen) * fall).to(dt)
        out["g_phi"] = (_random_field(nu, nphi, gen) * fall).to(dt)
    if c["call"] == "wedge":
        out["sigma_w"] = (sigma[0] * (1.0 + 0.1 * torch.cos(phi[0] - rng.uniform(0.0, 6.0)))).to(dt)
    return out


def _plan(c, nu, nphi, u_min, du):
    from paper_1509_01450_gb300 import Plan

    return Plan(nu, nphi, u_min, du, 1.0, c["dtype"]).build(
        weight_p=c["weight_p"], radial_edges=c["edges"], wedge=1 if c["call"] == "wedge" else 0,
        short_dft=c["short_dft"])


def prepare(case, seed):
    c = dict(case)
    s = _inputs(c, seed)
    s["call"] = c["call"]
    if c["call"] != "batch":
        s["plan"] = _plan(c, c["nu"], c["nphi"], *_grid(c))
        if c["call"] == "step":
            s["sigma"].requires_grad_(True)
        return s
    from paper_1509_01450_gb300 import sg

    plans, items, at = {}, [], 0
    total = sum(x.numel() for x in s["sigma"])
    s["F_r"], s["F_phi"] = (torch.empty(total, dtype=_real(c), device=_device()) for _ in range(2))
    for x in s["sigma"]:
        nu, nphi = x.shape
        if (nu, nphi) not in plans:
            plans[(nu, nphi)] = _plan(c, nu, nphi, math.log(c["r_in"]), math.log(c["r_out"] / c["r_in"]) / nu)
        views = [f[at:at + x.numel()].view(nu, nphi) for f in (s["F_r"], s["F_phi"])]
        items.append((plans[(nu, nphi)], x, *views))
        at += x.numel()
    s["items"] = items
    sg.batch_prepare(items)
    return s


def run(state):
    from paper_1509_01450_gb300 import sg

    call = state["call"]
    if call == "batch":
        sg.forces_batched(state["items"])
        return state["F_r"], state["F_phi"]
    plan = state["plan"]
    if call == "forces":
        return plan.forces(state["sigma"])
    if call == "adjoint":
        return plan.backward(state["g_r"], state["g_phi"])
    if call == "step":
        F_r, F_phi = sg.self_gravity(state["sigma"], plan)
        g, = torch.autograd.grad((F_r, F_phi), state["sigma"], (state["g_r"], state["g_phi"]))
        return F_r.detach(), F_phi.detach(), g
    F_r, F_phi = plan.forces_wedge(state["sigma"], state["sigma_w"])
    g, g_w = plan.backward_wedge(state["g_r"], state["g_phi"])
    return F_r, F_phi, g, g_w


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------
def _work(nu, nphi, e, passes, spectra=True):
    """passes: (fields in and out, row transforms, column transforms) summed
    over the directions.  Row transforms are real (2.5 n log2 n), column ones
    complex on 2 N_u points (5 n log2 n) for N_phi / 2 modes."""
    fields, rows, cols = passes
    by = fields * nu * nphi * e
    if spectra:  # both kernel spectra, kappa = 0 .. N_u
        by += 2 * (nphi // 2 + 1) * (nu + 1) * 2 * e
    fl = rows * nu * 2.5 * nphi * math.log2(nphi) + cols * (nphi // 2) * 5.0 * 2 * nu * math.log2(2 * nu)
    return by, fl


def work(case):
    c = case
    e = 4 if c["dtype"] == "float32" else 8
    if c["call"] == "batch":
        by = fl = 0.0
        seen = set()
        for nu, nphi in _sizes(c):
            b, f = _work(nu, nphi, e, (3, 3, 3), (nu, nphi) not in seen)
            seen.add((nu, nphi))
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    both = c["call"] in ("step", "wedge")
    by, fl = _work(c["nu"], c["nphi"], e, (6, 6, 6) if both else (3, 3, 3))
    half = c["nphi"] // 2 + 1
    if c["edges"]:  # both edge tables
        by += 2 * half * (2 * c["nu"] + 1) * e
    if c["call"] == "wedge":  # the four wedge tables, the wedge row and its gradient
        by += 4 * half * c["nu"] * e + 2 * c["nphi"] * e
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# the same in 64 bits: cell integrals
# ---------------------------------------------------------------------------
# eta = r' / r_i, xi = phi' - phi_j, F^2 = eta^2 - 2 eta cos xi + 1.  The six
# integrands over the source cell of offset (k, q):
#   -eta (1 - eta cos xi) / F^3  times  1, eta - beta^-k, xi + q dphi
#    eta^2 sin xi / F^3          times  the same
def _gl(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1.0), 0.5 * w  # on [0, 1]


def _integrands(e_off, x_off, e0, x0):
    """Radial and azimuthal integrands at eta = e0 + e_off, xi = x0 + x_off
    (torch or numpy); e0 and x0 are the cell's centre."""
    lib = torch if isinstance(e_off, torch.Tensor) else np
    eta, xi = e0 + e_off, x0 + x_off
    s2 = lib.sin(0.5 * xi) ** 2
    one = (1.0 - e0) - e_off  # 1 - eta
    f2 = one * one + 4.0 * eta * s2
    f3 = f2 * lib.sqrt(f2)
    a = -eta * (one + 2.0 * eta * s2) / f3
    b = eta * eta * lib.sin(xi) / f3
    return a, b


def _tensor_rule(e0, he, x0, hx, ne, nx):
    """[6, n]: the ne x nx Gauss-Legendre rule on cells centred at (e0, x0)
    (he, hx: half widths along eta and xi; all [n])."""
    acc = torch.zeros((6, e0.numel()), dtype=torch.float64, device=e0.device)
    (xe, we), (xx, wx) = _gl(ne), _gl(nx)
    for p, wp in zip(2.0 * xe - 1.0, 2.0 * we):
        eo = he * float(p)
        for z, wz in zip(2.0 * xx - 1.0, 2.0 * wx):
            xo = hx * float(z)
            a, b = _integrands(eo, xo, e0, x0)
            w = float(wp * wz)
            for c, f in ((0, a), (3, b)):
                acc[c] += w * f
                acc[c + 1] += w * f * eo
                acc[c + 2] += w * f * xo
    return acc * (he * hx)


def _order(dist):
    """Nodes for a cell whose nearest singular point lies dist cells away."""
    return np.where(dist >= 40, 4, np.where(dist >= 8, 6, 16))


def _panels(lo, hi, at, scale, ratio=3.0):
    """Edges of panels on [lo, hi] that shrink geometrically toward the point
    `at` of [lo, hi], down to about `scale`."""
    cuts = {lo, hi, min(max(at, lo), hi)}
    for side, end in ((-1.0, lo), (1.0, hi)):
        d = abs(end - at)
        while d > scale:
            d /= ratio
            if lo < at + side * d < hi:
                cuts.add(at + side * d)
    return sorted(cuts)


def _graded(e_lo, e_hi, e_c, x_lo, x_hi, x_c, e_scale, x_scale):
    """One cell near the singular point: panels graded toward eta = 1 (or the
    end nearest to it) and xi = 0, 16 nodes each way.  Offsets are measured
    from the cell's centre (e_c, x_c)."""
    t, w = _gl(16)
    out = np.zeros(6)
    ee = _panels(e_lo, e_hi, min(max(1.0, e_lo), e_hi), e_scale) if e_scale else [e_lo, e_hi]
    xx = _panels(x_lo, x_hi, min(max(0.0, x_lo), x_hi), x_scale) if x_scale else [x_lo, x_hi]
    for e1, e2 in zip(ee[:-1], ee[1:]):
        eo = (e1 - e_c) + (e2 - e1) * t
        for x1, x2 in zip(xx[:-1], xx[1:]):
            xo = (x1 - x_c) + (x2 - x1) * t
            a, b = _integrands(eo[:, None], xo[None, :], e_c, x_c)
            ww = w[:, None] * w[None, :] * (e2 - e1) * (x2 - x1)
            for c, f in ((0, a), (3, b)):
                out[c] += (ww * f).sum()
                out[c + 1] += (ww * f * eo[:, None]).sum()
                out[c + 2] += (ww * f * xo[None, :]).sum()
    return out


def _own_cell(du, dphi):
    """The singular cell: the eta integrals in closed form, with eta = cos xi
    + sin xi sinh t, and the xi integral on panels graded toward 0; K^{r,phi},
    K^{phi,0} and K^{phi,r} vanish by oddness."""
    L = np.longdouble
    t, w = _gl(24)
    t, w = t.astype(L), w.astype(L)
    h = L(np.tanh(L(du) / 2))  # 1 - eta_- = eta_+ - 1
    a = L(dphi) / 2
    edges = [a * L(3) ** -j for j in range(42)] + [L(0)]
    tot = np.zeros(3, dtype=L)
    for hi, lo in zip(edges[:-1], edges[1:]):
        xi = lo + (hi - lo) * t
        s, c, v = np.sin(xi), np.cos(xi), 2 * np.sin(xi / 2) ** 2  # v = 1 - c
        ends = []
        for sg in (-1, 1):
            d = sg * h + v  # eta - cos xi
            F = np.hypot(d, s)
            ends.append((np.arcsinh(d / s), d / F, F))
        (t1, th1, F1), (t2, th2, F2) = ends
        dt, dth, dF, dI = t2 - t1, th2 - th1, F2 - F1, 1 / F2 - 1 / F1
        r0 = c * (2 * dth - dt) + (c * c - s * s) * dI
        rr = -v * r0 + (-2 * c * s * s * dI - c * dF + (s * s - c * c) * (dt - dth))
        pp = xi / s * (c * c * dth - 2 * c * s * s * dI + s * s * (dt - dth))
        ww = w * (hi - lo)
        tot += np.array([-(ww * r0).sum(), -(ww * rr).sum(), (ww * pp).sum()]) * 2
    return np.array([tot[0], tot[1], 0.0, 0.0, 0.0, tot[2]], dtype=np.float64)


def _cells(nu, nphi, du):
    """The six kernels [6][2 N_u + 1][N_phi / 2 + 1], q = 0 .. N_phi / 2 (the
    others by symmetry)."""
    dev, dphi, nq = _device(), 2.0 * math.pi / nphi, nphi // 2 + 1
    half = math.tanh(0.5 * du)  # half width along eta over the centre
    out = torch.empty((6, 2 * nu + 1, nq), dtype=torch.float64, device=dev)
    k = torch.arange(-nu, nu + 1, dtype=torch.float64, device=dev)
    q = torch.arange(nq, dtype=torch.float64, device=dev)
    rows = max(1, (1 << 22) // nq)
    for r0 in range(0, 2 * nu + 1, rows):
        kk, qq = torch.meshgrid(k[r0:r0 + rows], q, indexing="ij")
        shape = kk.shape
        kk, qq = kk.reshape(-1), qq.reshape(-1)
        de = torch.maximum(kk.abs(), qq * (dphi / du))
        dx = torch.maximum(qq, kk.abs() * (du / dphi))
        bucket = lambda d: (d >= 8).long() + (d >= 40).long()  # noqa: E731
        zone = 3 * bucket(de) + bucket(dx)
        part = torch.empty((6, kk.numel()), dtype=torch.float64, device=dev)
        for z in range(9):
            at = (zone == z).nonzero()[:, 0]
            if at.numel() == 0:
                continue
            e0 = torch.exp(-kk[at] * du)
            part[:, at] = _tensor_rule(e0, half * e0, -qq[at] * dphi, torch.full_like(e0, 0.5 * dphi),
                                       (16, 6, 4)[z // 3], (16, 6, 4)[z % 3])
        out[:, r0:r0 + rows] = part.reshape(6, *shape)
    # the cells that lie closer to the singular point than their length
    near = [(0, j) for j in range(1, nq) if j * dphi < 1.5 * du]
    near += [(s * i, 0) for i in range(1, nu + 1) if i * du < 1.5 * dphi for s in (-1, 1)]
    for kk, qq in near:
        e0 = math.exp(-kk * du)
        v = _graded(e0 * (1 - half), e0 * (1 + half), e0, -(qq + 0.5) * dphi, -(qq - 0.5) * dphi, -qq * dphi,
                    0.25 * dphi * (qq - 0.5) if kk == 0 else 0.0, 0.25 * du * (abs(kk) - 0.5) if qq == 0 else 0.0)
        out[:, kk + nu, qq] = torch.from_numpy(v).to(dev)
    out[:, nu, 0] = torch.from_numpy(_own_cell(du, dphi)).to(dev)
    for c in (2, 3, 4):  # odd about xi = 0 and xi = pi
        out[c, :, 0] = out[c, :, -1] = 0.0
    return out


def _mirror(x, odd):
    """q = 0 .. N_phi / 2 extended to 0 .. N_phi - 1."""
    return torch.cat([x, (-1.0 if odd else 1.0) * x[..., 1:-1].flip(-1)], dim=-1)


ODD = (False, False, True, True, True, False)


def _kernels(nu, nphi, du):
    """Folded kernels (Kr, Kphi) [2 N_u - 1][N_phi] and the radial slope
    kernels (K^{r,r}, K^{phi,r}) [2 N_u + 1][N_phi]."""
    cells, dphi, bb = _cells(nu, nphi, du), 2.0 * math.pi / nphi, 2.0 * math.sinh(du)
    kk = torch.arange(-nu, nu + 1, dtype=torch.float64, device=cells.device)[:, None]
    folded, slopes = [], []
    for c in (0, 3):
        K = _mirror(cells[c], ODD[c])[1:-1]
        S = _mirror(cells[c + 1], ODD[c + 1])
        g = torch.exp(kk * du) * S
        K = K + (g[2:] - g[:-2]) / bb
        P = _mirror(cells[c + 2], ODD[c + 2])[1:-1]
        folded.append(K + (P.roll(-1, 1) - P.roll(1, 1)) / (2.0 * dphi))
        slopes.append(S)
    return folded, slopes


def _wedge_cells(nu, nphi, du):
    """The wedge [0, r_in] x one azimuthal cell seen from row i: the six
    integrals over eta in [0, eta_i], eta_i = r_in / r_i, with the slope
    factors from its centre eta_i / 2; [6][N_u][N_phi / 2 + 1]."""
    dev, dphi, nq = _device(), 2.0 * math.pi / nphi, nphi // 2 + 1
    out = torch.empty((6, nu, nq), dtype=torch.float64, device=dev)
    q = np.arange(nq)
    for i in range(nu):
        top = 2.0 * math.exp(-i * du) / (1.0 + math.exp(du))
        gap = 1.0 - top
        edges = _panels(0.0, top, top, gap) if top >= 0.4 else [0.0, top]
        dist = np.maximum(q, (i + 0.5) * du / dphi)
        orders = _order(dist)
        for n in sorted(set(orders.tolist())):
            at = torch.from_numpy(np.nonzero(orders == n)[0]).to(dev)
            x0 = -at.double() * dphi
            acc = torch.zeros((6, at.numel()), dtype=torch.float64, device=dev)
            te, we = _gl(16)
            eo = np.concatenate([a + (b - a) * te for a, b in zip(edges[:-1], edges[1:])]) - 0.5 * top
            ew = np.concatenate([(b - a) * we for a, b in zip(edges[:-1], edges[1:])])
            eo, ew = torch.from_numpy(eo).to(dev)[:, None], torch.from_numpy(ew).to(dev)[:, None]
            for z, wz in zip(*_gl(n)):
                xo = (z - 0.5) * dphi
                a, b = _integrands(eo, xo, 0.5 * top, x0[None, :])
                for c, f in ((0, a), (3, b)):
                    f = f * ew * (wz * dphi)
                    acc[c] += f.sum(0)
                    acc[c + 1] += (f * eo).sum(0)
                    acc[c + 2] += f.sum(0) * xo
            out[:, i, at] = acc
        if (i + 0.5) * du < 1.5 * dphi:  # q = 0: close to the singular point along xi
            v = _graded(0.0, top, 0.5 * top, -0.5 * dphi, 0.5 * dphi, 0.0, gap, 0.25 * gap)
            out[:, i, 0] = torch.from_numpy(v).to(dev)
    for c in (2, 3, 4):
        out[c, :, 0] = out[c, :, -1] = 0.0
    return out


# ---------------------------------------------------------------------------
# the same in 64 bits: the maps
# ---------------------------------------------------------------------------
def _forces64(sigma, K):
    """Zero-padded along u, periodic along phi (differentiable)."""
    nu, nphi = sigma.shape
    S = torch.fft.rfft2(sigma, s=(2 * nu, nphi))
    out = []
    for Kc in K:
        wrapped = torch.zeros((2 * nu, nphi), dtype=torch.float64, device=sigma.device)
        wrapped[:nu], wrapped[nu + 1:] = Kc[nu - 1:], Kc[:nu - 1]
        out.append(torch.fft.irfft2(S * torch.fft.rfft2(wrapped), s=(2 * nu, nphi))[:nu])
    return out


def _row_conv(rows, kernels):
    """Circular convolution along phi of one row with a kernel row per target row."""
    n = rows.shape[-1]
    prod = torch.fft.rfft(kernels, dim=-1) * torch.fft.rfft(rows, dim=-1)
    return torch.fft.irfft(prod, n=n, dim=-1)


def _edge_terms(sigma, slopes, u_min, du):
    """The change from ghost-row to one-sided radial slopes at the four edge rows."""
    nu = sigma.shape[0]
    r = [0.5 * math.exp(u_min + du * i) * (1.0 + math.exp(du)) for i in range(-2, nu + 2)]
    R = lambda i: r[i + 2]  # noqa: E731
    ghost = {-1: sigma[0] / (R(0) - R(-2)), 0: sigma[1] / (R(1) - R(-1)),
             nu - 1: -sigma[nu - 2] / (R(nu) - R(nu - 2)), nu: -sigma[nu - 1] / (R(nu + 1) - R(nu - 1))}
    side = {0: (sigma[1] - sigma[0]) / (R(1) - R(0)),
            nu - 1: (sigma[nu - 1] - sigma[nu - 2]) / (R(nu - 1) - R(nu - 2))}
    ri = torch.tensor(r[2:nu + 2], dtype=torch.float64, device=sigma.device)[:, None]
    out = []
    for S in slopes:
        acc = 0.0
        for a, g in ghost.items():
            d = (side[a] if a in side else 0.0) - g
            acc = acc + _row_conv(d, S[nu - a:2 * nu - a])  # K[i - a], i = 0 .. N_u - 1
        out.append(ri * acc)
    return out


def _wedge_terms(sigma, sigma_w, W, u_min, du):
    nu, nphi = sigma.shape
    r_in, dphi = math.exp(u_min), 2.0 * math.pi / nphi
    i = torch.arange(nu, dtype=torch.float64, device=sigma.device)
    ri = (0.5 * (1.0 + math.exp(du)) * torch.exp(u_min + du * i))[:, None]
    dr = (sigma[0] - sigma_w) / (0.5 * r_in * (1.0 + math.exp(du)) - 0.5 * r_in)
    dp = (sigma_w.roll(-1) - sigma_w.roll(1)) / (2.0 * dphi)
    out = []
    for c in (0, 3):
        w0, wr, wp = (_mirror(W[c + j], ODD[c + j]) for j in range(3))
        out.append(_row_conv(sigma_w, w0) + ri * _row_conv(dr, wr) + _row_conv(dp, wp))
    return out


def exact(case, seed):
    c = dict(case)
    s = _inputs(c, seed)
    if c["call"] == "batch":
        tables, F = {}, ([], [])
        for x in s["sigma"]:
            nu, nphi = x.shape
            if (nu, nphi) not in tables:
                tables[(nu, nphi)] = _kernels(nu, nphi, math.log(c["r_out"] / c["r_in"]) / nu)[0]
            for f, v in zip(F, _forces64(x.double(), tables[(nu, nphi)])):
                f.append(v.reshape(-1))
        return tuple(torch.cat(f) for f in F)
    u_min, du = _grid(c)
    K, slopes = _kernels(c["nu"], c["nphi"], du)
    sigma = s["sigma"].double().requires_grad_(True)
    ins = [sigma]
    F = _forces64(sigma, K)
    if c["edges"]:
        F = [f + e for f, e in zip(F, _edge_terms(sigma, slopes, u_min, du))]
    if c["call"] == "wedge":
        sigma_w = s["sigma_w"].double().requires_grad_(True)
        ins.append(sigma_w)
        F = [f + e for f, e in zip(F, _wedge_terms(sigma, sigma_w, _wedge_cells(c["nu"], c["nphi"], du), u_min, du))]
    if c["call"] == "forces":
        return tuple(f.detach() for f in F)
    g = torch.autograd.grad(F, ins, [s["g_r"].double(), s["g_phi"].double()])
    if c["call"] == "adjoint":
        return g[0]
    return (*(f.detach() for f in F), *g)
