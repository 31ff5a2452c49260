"""Performance cases of the Newton-step solver: the calls that a simulation, a
differentiation run and a batch of problems make, over the sizes they are
made at, with a plain 64-bit evaluation of the results that have a closed
definition (residual, energy, tangent applications, parameter gradients).

A case is a dict of plain values:

  kind      apply     one tangent application y = J v
            residual  residual and energy of a state
            tangent   a new state set, its residual, energy and tangent (all
                      levels), and one application of that tangent
            gradient  reverse-mode derivative of the residual with respect to
                      the state and the material parameters (torch.autograd)
            vcycle    one multigrid V-cycle z = M r
            newton    a Newton solve from the handle's state
            batch     one Newton correction of many small uneven problems
  nx ny nz  elements per axis (batch: problem count and edge range instead)
  prec      f32, f64, mixed (FP32 in, FP64 out), f16 (binary16 store)
  state     indent    the indentation load: prescribed spherical cap on the top
                      face, order parameters 1e-3 U[0, 1)
            smooth    smooth displacements (gradients up to 0.04) and order
                      parameters in [-0.02, 0.3], the penalty active in part
  material  sec51 (cubic, shared by all phases), table1 (anisotropic, per
            phase), nv12 (twelve variants, 15 unknowns per node)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2011_08802_gb300 import abi, autograd, binding, inputs

EDGE = inputs.CUBE_EDGE


# ---------------------------------------------------------------------------
# what is measured

def listed():
    return [
        # the smallest grid that the repository solves (8^3, 6,561 unknowns):
        # launch latency of one FP32 application, as a coarse level or a tiny
        # problem sees it
        dict(name="apply f32 8^3", kind="apply", nx=8, ny=8, nz=8, prec="f32", state="smooth", material="sec51"),
        # the product of differentiation and of the all-FP64 solve, odd box
        dict(name="apply f64 61x45x33", kind="apply", nx=61, ny=45, nz=33, prec="f64", state="smooth",
             material="sec51"),
        # FP64-class product of the mixed solve's outer FGMRES, odd box
        dict(name="apply mixed 93x77x61", kind="apply", nx=93, ny=77, nz=61, prec="mixed", state="smooth",
             material="sec51"),
        # the headline product: FP32 application on the largest grid
        dict(name="apply f32 128^3", kind="apply", nx=128, ny=128, nz=128, prec="f32", state="indent",
             material="sec51"),
        # residual and energy as a line search or a convergence test asks for
        # them, ragged box
        dict(name="residual 97x65x50", kind="residual", nx=97, ny=65, nz=50, prec="f64", state="smooth",
             material="sec51"),
        # everything a Newton iteration needs at a new iterate
        dict(name="tangent 80x72x56", kind="tangent", nx=80, ny=72, nz=56, prec="f32", state="smooth",
             material="sec51"),
        # the same with twelve variants (15 unknowns per node)
        dict(name="tangent nv12 36^3", kind="tangent", nx=36, ny=36, nz=36, prec="f32", state="smooth",
             material="nv12"),
        # differentiation at the size of the repository's configuration
        dict(name="gradient 32^3", kind="gradient", nx=32, ny=32, nz=32, prec="f64", state="smooth",
             material="sec51"),
        # preconditioner with the binary16 store on a grid whose levels do not
        # nest (75, 38, 19, 10, 5, 3)
        dict(name="vcycle f16 75^3", kind="vcycle", nx=75, ny=75, nz=75, prec="f16", state="indent",
             material="sec51"),
        # one mixed-precision Newton step of the benchmark problem (19.3 M
        # unknowns, six levels, relaxed products)
        dict(name="newton mixed 128^3", kind="newton", nx=128, ny=128, nz=128, prec="f32", state="indent",
             material="sec51"),
        # one load step of the 32^3 configuration: a full Newton solve to 1e-8,
        # all in FP64, four levels
        dict(name="newton f64 32^3", kind="newton", nx=32, ny=32, nz=32, prec="f64", state="indent",
             material="sec51"),
        # 64 independent problems of 8^3 to 24^3 elements solved together
        dict(name="batch 64", kind="batch", count=64, lo=8, hi=24, prec="f32", state="indent", material="sec51"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi, most):
    """Three edges, log-uniform in [lo, hi], at most `most` elements."""
    while True:
        n = [_log_int(rng, lo, hi) for _ in range(3)]
        if n[0] * n[1] * n[2] <= most:
            return dict(nx=n[0], ny=n[1], nz=n[2])


def draw(rng):
    kind = rng.choice(["apply", "apply", "residual", "tangent", "gradient", "vcycle", "newton", "batch"])
    material = rng.choice(["sec51", "sec51", "table1", "nv12"])
    if kind == "apply":
        prec = rng.choice(["f32", "f64", "mixed", "f16"])
        return dict(kind=kind, **_box(rng, 5, 128, 700_000 if material == "nv12" else 2_097_152), prec=prec,
                    state=rng.choice(["smooth", "indent"]), material=material)
    if kind == "residual":
        return dict(kind=kind, **_box(rng, 5, 110, 600_000), prec="f64", state=rng.choice(["smooth", "indent"]),
                    material=material)
    if kind == "tangent":
        return dict(kind=kind, **_box(rng, 5, 100, 80_000 if material == "nv12" else 500_000), prec="f32",
                    state="smooth", material=material)
    if kind == "gradient":
        return dict(kind=kind, **_box(rng, 5, 48, 60_000), prec="f64", state="smooth", material="sec51")
    if kind == "vcycle":
        n = _log_int(rng, 12, 128)
        return dict(kind=kind, nx=n, ny=n, nz=n, prec=rng.choice(["f32", "f16"]), state="indent", material="sec51")
    if kind == "newton":
        if rng.random() < 0.5:
            n = _log_int(rng, 10, 32)
            return dict(kind=kind, nx=n, ny=n, nz=n, prec="f64", state="indent", material="sec51")
        n = _log_int(rng, 16, 112)
        return dict(kind=kind, nx=n, ny=n, nz=n, prec=rng.choice(["f32", "f16"]), state="indent", material="sec51")
    lo = rng.randint(6, 12)
    return dict(kind=kind, count=_log_int(rng, 4, 64), lo=lo, hi=rng.randint(lo + 2, 24), prec="f32", state="indent",
                material="sec51")


# ---------------------------------------------------------------------------
# inputs (made on the GPU from the seed alone)

def _constants(case):
    return inputs.material_nv12() if case["material"] == "nv12" else dict(inputs.MATERIAL)


def _params(case, tau):
    if case["material"] == "table1":
        return abi.params_anisotropic(_constants(case), inputs.ELASTIC_TABLE1, tau, inputs.ORIENTATION_011)
    return abi.params_from_material(_constants(case), tau)


def _n_fields(case):
    return 15 if case["material"] == "nv12" else 9


def _lengths(case):
    """Box of cubic elements whose longest edge is EDGE."""
    h = EDGE / max(case["nx"], case["ny"], case["nz"])
    return h * case["nx"], h * case["ny"], h * case["nz"]


def _tau(case):
    return 0.128 if case["state"] == "indent" else 0.1


def _noise(gen, shape, cells, lo=-1.0, hi=1.0):
    """Smooth random field: values on a coarse grid of about `cells` cells per
    axis, interpolated trilinearly."""
    dims = [max(2, min(cells, s - 1)) + 1 for s in shape]
    g = torch.rand([1, 1] + dims, generator=gen, device="cuda", dtype=torch.float64) * (hi - lo) + lo
    return torch.nn.functional.interpolate(g, size=tuple(shape), mode="trilinear", align_corners=True)[0, 0]


def _smooth_state(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    nf, nn = _n_fields(case), (nx + 1) * (ny + 1) * (nz + 1)
    gen = torch.Generator("cuda").manual_seed(seed)
    shape = (nz + 1, ny + 1, nx + 1)
    h = EDGE / max(nx, ny, nz)
    z = torch.linspace(0.0, 1.0, nz + 1, device="cuda", dtype=torch.float64)[:, None, None]
    U = torch.empty(nf, *shape, device="cuda", dtype=torch.float64)
    for i in range(3):
        U[i] = z * _noise(gen, shape, 9)
    big = max(float((U[:3].diff(dim=a).abs() / h).max()) for a in (1, 2, 3))
    U[:3] *= 0.04 / big
    hi = 0.3 if nf == 9 else 0.15
    for k in range(3, nf):
        U[k] = _noise(gen, shape, 9, -0.02, hi)
    Un = U.clone()
    for k in range(3, nf):
        Un[k] -= 0.01 * _noise(gen, shape, 9)
    mask = torch.zeros(nf, *shape, device="cuda", dtype=torch.uint8)
    mask[:3, 0] = 1
    mask[:3, -1] = 1
    return U.reshape(nf, nn), Un.reshape(nf, nn), mask.reshape(nf, nn)


def _indent_state(case, seed, depth_frac=0.02):
    """First of ten load steps of the indentation ramp: bottom clamped, u_z of
    the top nodes within 0.3 L prescribed by a cap of depth depth_frac L / 10."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    nf, nn = _n_fields(case), (nx + 1) * (ny + 1) * (nz + 1)
    gen = torch.Generator("cuda").manual_seed(seed)
    Lx, Ly, Lz = _lengths(case)
    U = torch.zeros(nf, nz + 1, ny + 1, nx + 1, device="cuda", dtype=torch.float64)
    U[3:] = 1e-3 * torch.rand(nf - 3, nz + 1, ny + 1, nx + 1, generator=gen, device="cuda", dtype=torch.float64)
    mask = torch.zeros(U.shape, device="cuda", dtype=torch.uint8)
    mask[:3, 0] = 1
    x = torch.linspace(0.0, Lx, nx + 1, device="cuda", dtype=torch.float64) - Lx / 2
    y = torch.linspace(0.0, Ly, ny + 1, device="cuda", dtype=torch.float64) - Ly / 2
    r2 = (x[None, :] ** 2 + y[:, None] ** 2)
    radius, depth = 0.3 * Lx, 0.1 * depth_frac * Lz
    cap = (radius ** 2 + depth ** 2) / (2.0 * depth)
    under = r2 <= radius ** 2 * (1 + 1e-12)
    uz = -(depth - (cap - torch.sqrt(cap * cap - torch.where(under, r2, 0.0))))
    mask[2, -1] = under.to(torch.uint8)
    U[2, -1] = torch.where(under, uz, 0.0)
    Un = U.clone()
    Un[:3] = 0.0
    return U.reshape(nf, nn), Un.reshape(nf, nn), mask.reshape(nf, nn)


def _state(case, seed):
    return _smooth_state(case, seed) if case["state"] == "smooth" else _indent_state(case, seed)


def _direction(case, seed, mask, dtype):
    gen = torch.Generator("cuda").manual_seed(seed + 1_000_003)
    v = torch.randn(mask.shape, generator=gen, device="cuda", dtype=torch.float64).to(dtype)
    return v.masked_fill_(mask.bool(), 0.0)


def _batch_sizes(case, seed):
    """Edge lengths (fixed by the case) and final depths (by the seed)."""
    ns = np.random.default_rng(4).integers(case["lo"], case["hi"] + 1, size=case["count"])
    depths = np.random.default_rng(seed).uniform(0.005, 0.03, size=case["count"])
    return [int(n) for n in ns], [float(d) for d in depths]


def _problem(case, mask, U, Un, n_levels=0):
    P = binding.Problem(case["nx"], case["ny"], case["nz"], *_lengths(case), _params(case, _tau(case)), n_levels)
    P.set_dirichlet(mask)
    P.set_state(U, Un)
    if case["prec"] == "f16":
        P.set_preconditioner_store(True)
    return P


def _opts(case):
    """Solver options of the repository's benchmark for this kind of solve."""
    if case["prec"] == "f64":
        return abi.default_opts(abi.PFM_F64, max_newton=12, newton_rtol=1e-8, restart=30, lin_rtol=1e-8,
                                max_lin_it=400)
    return abi.default_opts(abi.PFM_F32, max_newton=1, restart=30, max_lin_it=400, lin_rtol=1e-8, krylov=1,
                            switch_rtol=1e-4)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        ns, depths = _batch_sizes(case, seed)
        probs, states = [], []
        for k, (n, d) in enumerate(zip(ns, depths)):
            c = dict(case, nx=n, ny=n, nz=n)
            U, Un, mask = _indent_state(c, seed + 7919 * (k + 1), d)
            probs.append(_problem(c, mask, U, Un, binding.levels_to(n, 2)))
            states.append(U)
        opts = abi.default_opts(abi.PFM_F32, max_newton=1, lin_rtol=1e-8, max_lin_it=400)
        return dict(kind=kind, B=binding.Batch(probs), U=states, opts=opts)
    U, Un, mask = _state(case, seed)
    P = _problem(case, mask, U, Un)
    s = dict(kind=kind, P=P, U=U, Un=Un, prec=case["prec"])
    if kind == "apply":
        P.linearize(abi.PFM_F64 if case["prec"] == "f64" else abi.PFM_F32)
        s["v"] = _direction(case, seed, mask, torch.float64 if case["prec"] == "f64" else torch.float32)
    elif kind == "tangent":
        s["v"] = _direction(case, seed, mask, torch.float32)
    elif kind == "gradient":
        m = inputs.MATERIAL
        s["theta"] = torch.tensor([m["C11"], m["C12"], m["C44"], 1.0], dtype=torch.float64, device="cuda",
                                  requires_grad=True)
        s["U"] = U.requires_grad_(True)
        s["g"] = _direction(case, seed, mask, torch.float64)
        s["constants"], s["tau"] = _constants(case), _tau(case)
    elif kind == "vcycle":
        r = P.residual()
        s["r"] = (-r / torch.linalg.norm(r)).to(torch.float32)
        P.linearize(abi.PFM_F32)
        s["opts"] = abi.default_opts(abi.PFM_F32)
    elif kind == "newton":
        s["opts"] = _opts(case)
    return s


def run(s):
    kind = s["kind"]
    if kind == "apply":
        if s["prec"] == "mixed":
            return s["P"].jacobian_apply_mixed(s["v"])
        return s["P"].jacobian_apply(s["v"])
    if kind == "residual":
        return s["P"].residual(energy=True)
    if kind == "tangent":
        P = s["P"]
        P.set_state(s["U"], s["Un"])
        R, e = P.linearize_residual(abi.PFM_F32, energy=True)
        return R, e, P.jacobian_apply(s["v"])
    if kind == "gradient":
        R = autograd.PFMResidual.apply(s["U"], s["theta"], s["P"], s["Un"], s["constants"], s["tau"])
        gU, gtheta = torch.autograd.grad(R, (s["U"], s["theta"]), s["g"])
        return R.detach(), gU, gtheta
    if kind == "vcycle":
        return s["P"].vcycle(s["r"], opts=s["opts"])
    if kind == "newton":
        U = s["U"].clone()
        s["P"].newton_solve(U, s["opts"])
        return U
    Us = [u.clone() for u in s["U"]]
    s["B"].newton_solve(Us, s["opts"])
    return torch.cat([u.reshape(-1) for u in Us])


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _apply_work(ne, nn, nf, prec):
    """One application: the stored tangent (n (n + 1) / 2 entries at 8 points
    per element), input and output vectors; the symmetric product per point."""
    nz = nf + 6
    entry = dict(f32=4, f64=8, mixed=8, f16=2)[prec]
    vec = dict(f32=8, f64=16, mixed=12, f16=8)[prec]
    return (ne * 8 * (nz * (nz + 1) // 2) * entry + nn * (nf * vec + 2),
            ne * 8 * (2 * nz * nz + 10 * nf))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        n = 0.5 * (case["lo"] + case["hi"])
        one = work(dict(case, kind="newton", nx=n, ny=n, nz=n))
        return {k: v * case["count"] for k, v in one.items()}
    nf = _n_fields(case)
    nz = nf + 6
    nx, ny, nzz = case["nx"], case["ny"], case["nz"]
    ne, nn = nx * ny * nzz, (nx + 1) * (ny + 1) * (nzz + 1)
    state = 3 * 8 * nf * nn                        # U, U_n read, R written
    point = 1500 + 40 * nf                         # energy and gradient per Gauss point
    hess = 25 * nz * nz                            # exact Hessian per Gauss point
    tangent = ne * 8 * (nz * (nz + 1) // 2) * 8    # stored once to FP64-class accuracy
    if kind == "apply":
        b, f = _apply_work(ne, nn, nf, case["prec"])
    elif kind == "residual":
        b, f = state, ne * 8 * point
    elif kind == "tangent":
        b, f = _apply_work(ne, nn, nf, "f32")
        b, f = b + state + tangent, f + ne * 8 * (point + hess)
    elif kind == "gradient":
        b, f = _apply_work(ne, nn, nf, "f64")
        b, f = b + state + tangent, f + ne * 8 * (2 * point + hess)
    else:
        # a V-cycle of 2 + 8 smoothing steps: ten finest-level applications and
        # eleven nodal block products (coarser levels: an eighth each)
        p = "f16" if case["prec"] == "f16" else case["prec"]
        ab, af = _apply_work(ne, nn, nf, p)
        size = 8 if p == "f64" else 4
        cb = nn * size * (nf * (nf + 1) // 2 + 7 * nf)
        b, f = 1.18 * (10 * ab + 11 * cb), 1.18 * (10 * af + 11 * nn * 2 * nf * nf)
        if kind == "newton":
            its = 10
            b, f = its * (b + ab), its * (f + af)
            b, f = b + 2 * state + tangent, f + ne * 8 * (2 * point + hess)
            if case["prec"] == "f64":
                b, f = 4 * b, 4 * f
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# 64-bit values: the discrete potential written down in torch, differentiated
# by torch.autograd

_CHUNK = 65536


def _shape_functions(h):
    """Values and gradients of the 8 trilinear functions at the 8 Gauss points
    (2-point rule per axis) of an element with edges h."""
    ga = 0.5 * (1.0 - 1.0 / math.sqrt(3.0))
    N, dN = np.zeros((8, 8)), np.zeros((8, 8, 3))
    for q in range(8):
        xi = [1.0 - ga if (q >> d) & 1 else ga for d in range(3)]
        for a in range(8):
            phi = [xi[d] if (a >> d) & 1 else 1.0 - xi[d] for d in range(3)]
            dphi = [(1.0 if (a >> d) & 1 else -1.0) / h[d] for d in range(3)]
            N[q, a] = phi[0] * phi[1] * phi[2]
            for d in range(3):
                dN[q, a, d] = math.prod(dphi[e] if e == d else phi[e] for e in range(3))
    return torch.tensor(N, device="cuda"), torch.tensor(dN, device="cuda")


def _mul3(a, b):
    return [[sum(a[i][k] * b[k][j] for k in range(3)) for j in range(3)] for i in range(3)]


def _inverse_sym(a):
    """Inverse (symmetric) and determinant of a symmetric 3x3 matrix of tensors."""
    c = [[None] * 3 for _ in range(3)]
    c[0][0] = a[1][1] * a[2][2] - a[1][2] * a[1][2]
    c[0][1] = c[1][0] = a[0][2] * a[1][2] - a[0][1] * a[2][2]
    c[0][2] = c[2][0] = a[0][1] * a[1][2] - a[0][2] * a[1][1]
    c[1][1] = a[0][0] * a[2][2] - a[0][2] * a[0][2]
    c[1][2] = c[2][1] = a[0][1] * a[0][2] - a[0][0] * a[1][2]
    c[2][2] = a[0][0] * a[1][1] - a[0][1] * a[0][1]
    det = a[0][0] * c[0][0] + a[0][1] * c[0][1] + a[0][2] * c[0][2]
    r = 1.0 / det
    return [[c[i][j] * r for j in range(3)] for i in range(3)], det


def _half_log(C):
    """1/2 log C of a symmetric 3x3 matrix of tensors by its integral over s of
    (C - I) (I + s (C - I))^-1 (14-point Gauss rule)."""
    x, w = np.polynomial.legendre.leggauss(14)
    X = [[C[i][j] - 1.0 if i == j else C[i][j] for j in range(3)] for i in range(3)]
    H = [[0.0] * 3 for _ in range(3)]
    for xk, wk in zip(x, w):
        s = 0.5 * (xk + 1.0)
        B, _ = _inverse_sym([[s * X[i][j] + (1.0 if i == j else 0.0) for j in range(3)] for i in range(3)])
        for i in range(3):
            for j in range(i, 3):
                H[i][j] = H[i][j] + 0.25 * wk * sum(X[i][k] * B[k][j] for k in range(3))
    for i in range(3):
        for j in range(i):
            H[i][j] = H[j][i]
    return H


def _energy(X, Xn, N, dN, w, p, theta):
    """Potential of a chunk of elements from its nodal values X, Xn
    [fields, 8, elements]; theta = (C11, C12, C44, s_gamma) or None for the
    parameter block's own stiffness and interface energies."""
    nv = X.shape[0] - 3
    nph = nv + 1
    F = torch.einsum("iae,qaJ->iJqe", X[:3], dN)
    F = [[F[i, j] + (1.0 if i == j else 0.0) for j in range(3)] for i in range(3)]
    eh = torch.einsum("kae,qa->kqe", X[3:], N)
    en = torch.einsum("kae,qa->kqe", Xn[3:], N)
    ge = torch.einsum("kae,qaJ->kJqe", X[3:], dN)
    eta = torch.cat([1.0 - eh.sum(0, keepdim=True), eh])
    etan = torch.cat([1.0 - en.sum(0, keepdim=True), en])
    geta = torch.cat([-ge.sum(0, keepdim=True), ge])
    Ut = np.array([list(p.Ut[i]) for i in range(nph)]).reshape(nph, 3, 3)
    Ft = [[sum(float(Ut[i, a, b]) * eta[i] for i in range(nph)) for b in range(3)] for a in range(3)]
    A, Jt = _inverse_sym(Ft)
    M = _mul3(F, A)
    C = [[sum(M[k][i] * M[k][j] for k in range(3)) for j in range(3)] for i in range(3)]
    H = _half_log(C)
    hv = [H[0][0], H[1][1], H[2][2], 2.0 * H[1][2], 2.0 * H[0][2], 2.0 * H[0][1]]
    if theta is None:
        W = 0.0
        for i in range(nph):
            L = np.array(list(p.Lvoigt[i])).reshape(6, 6)
            if i > 0 and np.array_equal(L, np.array(list(p.Lvoigt[0])).reshape(6, 6)):
                continue
            same = [k for k in range(nph) if list(p.Lvoigt[k]) == list(p.Lvoigt[i])]
            q = sum(float(L[a, b]) * hv[a] * hv[b] for a in range(6) for b in range(6) if L[a, b] != 0.0)
            W = W + (sum(eta[k] for k in same) if len(same) > 1 else eta[i]) * q
            if len(same) == nph:
                break
        gs = p.gamma_scale
    else:
        c11, c12, c44, gs = theta
        W = (c11 * (hv[0] ** 2 + hv[1] ** 2 + hv[2] ** 2)
             + 2.0 * c12 * (hv[0] * hv[1] + hv[1] * hv[2] + hv[0] * hv[2])
             + c44 * (hv[3] ** 2 + hv[4] ** 2 + hv[5] ** 2)) * eta.sum(0)
    W = 0.5 * Jt * W
    for i in range(nph):
        d = eta[i] - etan[i]
        neg = torch.clamp(eta[i], max=0.0)
        W = W + p.F0[i] * eta[i] + d * d / (2.0 * p.mobility[i] * p.tau) + 0.5 * p.eps_eta * neg * neg
    G = np.array([list(p.gamma[i]) for i in range(nph)])
    ell = np.array([list(p.ell[i]) for i in range(nph)])
    off = torch.tensor(np.where(np.eye(nph) > 0, 0.0, 4.0 * G / (math.pi * ell)), device="cuda")
    grad = off * torch.tensor(ell * ell, device="cuda")
    W = W + gs * 0.5 * (torch.einsum("iqe,ij,jqe->qe", eta, off, eta)
                        - torch.einsum("iJqe,ij,jJqe->qe", geta, grad, geta))
    return w * W.sum()


def _connectivity(nx, ny, nz):
    e = torch.arange(nx * ny * nz, device="cuda")
    ei, r = e % nx, e // nx
    ej, ek = r % ny, r // ny
    return torch.stack([(ei + (a & 1)) + (nx + 1) * ((ej + (a >> 1 & 1)) + (ny + 1) * (ek + (a >> 2)))
                        for a in range(8)])


def _derivatives(case, U, Un, mask, v=None, theta=None):
    """Energy, residual (zero at prescribed unknowns), and with a direction v
    the product J v (identity at prescribed unknowns) and v . dR/dtheta."""
    p = _params(case, _tau(case))
    h = [a / n for a, n in zip(_lengths(case), (case["nx"], case["ny"], case["nz"]))]
    N, dN = _shape_functions(h)
    w = h[0] * h[1] * h[2] / 8.0
    conn = _connectivity(case["nx"], case["ny"], case["nz"])
    fixed = mask.bool()
    nf, nn = U.shape
    energy, R = 0.0, torch.zeros_like(U)
    Jv = None if v is None else torch.zeros_like(U)
    vf = None if v is None else v.double().masked_fill(fixed, 0.0)
    gth = None if theta is None else torch.zeros(4, device="cuda", dtype=torch.float64)
    for c in range(0, conn.shape[1], _CHUNK):
        idx = conn[:, c:c + _CHUNK]
        flat = idx.reshape(-1)
        X = U[:, idx].detach().requires_grad_(True)
        th = None if theta is None else theta.detach().clone().requires_grad_(True)
        E = _energy(X, Un[:, idx], N, dN, w, p, th)
        energy += float(E.detach())
        g, = torch.autograd.grad(E, X, create_graph=v is not None)
        R.index_add_(1, flat, g.detach().reshape(nf, -1))
        if v is not None:
            s = (g * vf[:, idx]).sum()
            got = torch.autograd.grad(s, (X,) if th is None else (X, th))
            Jv.index_add_(1, flat, got[0].reshape(nf, -1))
            if th is not None:
                gth += got[1]
        del X, E, g
    R.masked_fill_(fixed, 0.0)
    if v is not None:
        Jv = torch.where(fixed, v.double(), Jv)
    return energy, R, Jv, gth


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("apply", "residual", "tangent", "gradient"):
        return None  # results of iterative processes: no closed 64-bit value
    U, Un, mask = _state(case, seed)
    if kind == "residual":
        energy, R, _, _ = _derivatives(case, U, Un, mask)
        return R, energy
    if kind == "apply":
        v = _direction(case, seed, mask, torch.float64 if case["prec"] == "f64" else torch.float32)
        return _derivatives(case, U, Un, mask, v)[2]
    if kind == "tangent":
        energy, R, Jv, _ = _derivatives(case, U, Un, mask, _direction(case, seed, mask, torch.float32))
        return R, energy, Jv
    m = inputs.MATERIAL
    theta = torch.tensor([m["C11"], m["C12"], m["C44"], 1.0], dtype=torch.float64, device="cuda")
    _, R, gU, gth = _derivatives(case, U, Un, mask, _direction(case, seed, mask, torch.float64), theta)
    return R, gU, gth
