"""Performance cases of the flux-reconstruction library: what a solver built on it calls, step after step.

A case is one handle (paper_2401_06132_gb300.fr.FRMesh) on a periodic box and one call on it: ``rhs``
evaluates du/dt = R(u) (a user's own time integrator, a steady or adjoint solver), ``rk4`` advances
the FP64 master state by one classical RK4 step (the stock time integrator, four RHS). Meshes:

  hex       N^3 uniform axis-aligned hexahedra          sheared   affine, full 3 x 3 metric
  curved    trilinear hexahedra, metric per point       mixed     half hexahedra, half prisms
  tet       six tetrahedra per cell                     pyr       hexahedra and six pyramids per cell
  ensemble  independent uniform boxes, edge, order, Mach and Reynolds numbers drawn per instance

Precisions are the library's: ``fp64``; ``fp32`` in its low-Mach form (reference pressure and density
given, as every reduced-precision user sets them); ``mixed_fp16``. ``aa``: "flux" (quadrature points
p + 2 per direction, the default), "off" (collocation), "full" (flux and surface flux).

The state is the Taylor-Green vortex at M = 0.1, shifted by phases drawn from the seed, with a
per-value perturbation, as a flow with interface jumps has.
"""
import functools
import math

import numpy as np
import torch

from paper_2401_06132_gb300 import fr, workloads

GAMMA, PRANDTL, BETA, TAU = 1.4, 0.71, 0.5, 0.1


def listed():
    def case(name, mesh, n, p, prec, call, aa="flux"):
        return dict(name=name, mesh=mesh, n=n, p=p, prec=prec, call=call, aa=aa)

    return [
        # a debugging-size box: a handful of elements, where launches and latency are all there is
        case("sheared3_p3_fp32_rhs", "sheared", 3, 3, "fp32", "rhs"),
        # the benchmark problem of the method, 35 M unknowns, double precision: the production run
        case("hex48_p3_fp64_rk4", "hex", 48, 3, "fp64", "rk4"),
        # the same in single precision, what a user takes once the accuracy has been checked
        case("hex48_p3_fp32_rk4", "hex", 48, 3, "fp32", "rk4"),
        # higher order at a middling size, a user's own integrator
        case("hex25_p4_fp64_rhs", "hex", 25, 4, "fp64", "rhs"),
        case("hex32_p4_fp32_rhs", "hex", 32, 4, "fp32", "rhs"),
        # mixed hexahedra and prisms: boundary-layer meshes
        case("mixed18_p3_fp64_rhs", "mixed", 18, 3, "fp64", "rhs"),
        case("mixed40_p3_fp32_rk4", "mixed", 40, 3, "fp32", "rk4"),
        # unstructured tetrahedra; pyramids between hexahedra and tetrahedra
        case("tet21_p3_fp32_rhs", "tet", 21, 3, "fp32", "rhs"),
        case("pyr11_p3_fp64_rk4", "pyr", 11, 3, "fp64", "rk4"),
        # a parameter study: many small boxes, both orders, in one handle
        case("ensemble14_fp32_rk4", "ensemble", 14, 0, "fp32", "rk4"),
        # full anti-aliasing for under-resolved flow; body-fitted (curved) hexahedra
        case("hex21_p3_fp32_full_rhs", "hex", 21, 3, "fp32", "rhs", "full"),
        case("curved17_p3_fp64_rhs", "curved", 17, 3, "fp64", "rhs"),
    ]


def draw(rng):
    """Sizes on a logarithmic scale between a few elements and what a workstation run holds; every
    mesh family, order, precision and anti-aliasing form that its family offers."""
    mesh = rng.choice(["hex", "hex", "sheared", "curved", "mixed", "mixed", "tet", "pyr", "ensemble"])
    prec = rng.choice(["fp64", "fp32", "fp32"] if mesh != "mixed" else ["fp64", "fp32", "mixed_fp16"])
    top = {"hex": 40, "sheared": 40, "curved": 36, "mixed": 32, "tet": 20, "pyr": 16, "ensemble": 12}[mesh]
    n = round(math.exp(rng.uniform(math.log(3), math.log(top))))
    if mesh == "mixed":
        n += n % 2
    p = rng.choice([3, 3, 4]) if mesh in ("hex", "sheared", "curved") else 0 if mesh == "ensemble" else 3
    if p == 4:
        n = max(3, n * 3 // 4)
    aa = rng.choice(["flux", "flux", "off", "full"]) if mesh in ("hex", "sheared") else "flux"
    return dict(mesh=mesh, n=n, p=p, prec=prec, call=rng.choice(["rhs", "rk4"]), aa=aa)


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


@functools.lru_cache(maxsize=4)
def _mesh(kind, n):
    if kind == "hex":
        return workloads.box_hex_mesh(n)
    if kind == "sheared":
        return workloads.sheared_box_mesh(n)
    if kind == "curved":
        return workloads.curved_box_mesh(n)
    if kind == "mixed":
        return workloads.mixed_box_mesh(n)
    if kind == "tet":
        return workloads.box_tet_mesh(n)
    return workloads.box_pyr_mesh(n, hex_below=n // 2)


def _instances(case):
    """(mesh kind, edge, order, Mach number, Reynolds number) of every instance of the handle."""
    if case["mesh"] == "ensemble":
        return [("hex", d["edge"], d["p"], d["mach"], d["re"]) for d in workloads.ensemble_draws(case["n"])]
    return [(case["mesh"], case["n"], case["p"], 0.1, 1600.0)]


def _p0(mach):
    return 1.0 / (GAMMA * mach * mach)


def _dt(case):
    """Well inside the acoustic stability limit (c = 10 at M = 0.1) of the finest instance."""
    return min(4.8e-3 / max(i[1] for i in _instances(case)), 5e-4)


def _state(case, seed):
    """The FP64 state in the library's layout: per instance and element type [element][variable][point]."""
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    eps = 1e-3 if case["call"] == "rhs" else 1e-4
    parts = []
    for kind, n, p, mach, _ in _instances(case):
        shift = (torch.rand(3, generator=g, device=dev, dtype=torch.float64) * 2 * math.pi).tolist()
        amp = 0.8 + 0.4 * float(torch.rand(1, generator=g, device=dev, dtype=torch.float64))
        for typ, verts in _blocks(_mesh(kind, n)):
            x = _map(typ, verts, _points(typ, p))[0]
            a, b, c = (x[..., d] + shift[d] for d in range(3))
            v = [amp * torch.sin(a) * torch.cos(b) * torch.cos(c), -amp * torch.cos(a) * torch.sin(b) * torch.cos(c)]
            pr = _p0(mach) + amp * amp / 16 * (torch.cos(2 * a) + torch.cos(2 * b)) * (torch.cos(2 * c) + 2)
            e = pr / (GAMMA - 1) + 0.5 * (v[0] * v[0] + v[1] * v[1])
            u = torch.stack([torch.ones_like(e), v[0], v[1], torch.zeros_like(e), e], dim=1)
            u *= 1 + eps * (2 * torch.rand(u.shape, generator=g, device=dev, dtype=torch.float64) - 1)
            parts.append(u.reshape(-1))
    return torch.cat(parts)


def prepare(case, seed):
    meshes, params = [], []
    for kind, n, p, mach, re in _instances(case):
        meshes.append(_mesh(kind, n))
        params.append(fr.make_params(p=p, prec=case["prec"], mu=1.0 / re, Pr=PRANDTL, beta=BETA, tau=TAU, p_ref=_p0(mach), rho_ref=1.0,
                                     nq1d=p + 1 if case["aa"] == "off" else 0, surface_aa=case["aa"] == "full"))
    m = fr.FRMesh(meshes, params)
    u = _state(case, seed)
    if case["call"] == "rhs":
        u = u.to(m.dtype)
    return dict(mesh=m, call=case["call"], dt=_dt(case), u=u, r=torch.empty_like(u) if case["call"] == "rhs" else None)


def run(state):
    m = state["mesh"]
    if state["call"] == "rhs":
        m.rhs(state["u"], state["r"])
        return state["r"]
    m.rk4_step(state["u"], state["dt"], 1)
    return state["u"]


def work(case):
    """State read and result written once; the arithmetic of the sum-factorised (hexahedra, prisms) or
    dense (tetrahedra, pyramids) operators, a multiply-add as two."""
    byts = flops = 0.0
    for kind, n, p, _, _ in _instances(case):
        m1 = p + 1 if case["aa"] == "off" else p + 2
        mesh = _mesh(kind, n)
        for typ in ("hex", "pri", "tet", "pyr"):
            ne = len(mesh.get(typ + "_v", ()))
            if not ne:
                continue
            n1 = p + 1
            nu = {"hex": n1 ** 3, "pri": 40, "tet": 20, "pyr": 30}[typ]
            nf = {"hex": 6 * n1 * n1, "pri": 68, "tet": 40, "pyr": 56}[typ]
            nq = m1 ** 3
            if typ == "hex":
                lines = n1 ** 3 * m1 + n1 ** 2 * m1 ** 2 + n1 * m1 ** 3
                ops = 35 * 2 * lines if case["aa"] != "off" else 30 * n1 ** 4
                ops += 30 * n1 ** 4 + 60 * n1 ** 3
                if case["aa"] == "full":
                    ops += 6 * (20 * 2 * (n1 * n1 * m1 + n1 * m1 * m1) + 10 * (n1 * m1 * m1 + n1 * n1 * m1) + 200 * m1 * m1)
            elif typ == "pri":
                ops = 35 * 2 * (40 * 5 + 10 * 25 * 5) + 5 * 2 * 40 * (10 + 10 + 4)
            else:
                ops = 20 * 2 * nq * nu + 5 * 2 * nu * 3 * nq + 3 * 10 * nu * nu
            line = n1 if typ in ("hex", "pri") else nu
            ops += nf * (5 * 2 * line + 20 * line + 130 // 2 + 120 + 10 * line) + 165 * nq
            size = 4 if case["call"] == "rhs" and case["prec"] != "fp64" else 8
            byts += ne * 5 * nu * 2 * size
            flops += ne * ops * (4 if case["call"] == "rk4" else 1)
    return {"bytes": byts, "flops": flops}


# ---------------------------------------------------------------------------------------------
# The same in plain 64-bit arithmetic: dense per-element operators from their definitions
# ---------------------------------------------------------------------------------------------
# Williams-Shunn triangle points as the paper prints them (Sec. 4.1)
_WS = np.array([
    [-0.333333333333333, -0.333333333333333], [-0.888871894660414, 0.777743789320828],
    [0.777743789320828, -0.888871894660414], [-0.888871894660414, -0.888871894660414],
    [0.268421495491446, -0.408932576528214], [-0.859488918963232, -0.408932576528214],
    [-0.408932576528214, -0.859488918963232], [0.268421495491446, -0.859488918963232],
    [-0.859488918963232, 0.268421495491446], [-0.408932576528214, 0.268421495491446]])
_CORNERS = {
    "hex": [[2 * (c & 1) - 1, 2 * (c >> 1 & 1) - 1, 2 * (c >> 2) - 1] for c in range(8)],
    "pri": [[-1, -1, -1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1], [1, -1, 1], [-1, 1, 1]],
    "tet": [[-1, -1, -1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]],
    "pyr": [[-1, -1, -1], [1, -1, -1], [-1, 1, -1], [1, 1, -1], [0, 0, 1]]}
_FACES = {  # corner numbers: three for a triangle, four (tensor order) for a quadrilateral
    "hex": [(0, 2, 4, 6), (1, 3, 5, 7), (0, 1, 4, 5), (2, 3, 6, 7), (0, 1, 2, 3), (4, 5, 6, 7)],
    "pri": [(0, 1, 2), (3, 4, 5), (0, 1, 3, 4), (1, 2, 4, 5), (0, 2, 3, 5)],
    "tet": [(0, 1, 2), (0, 1, 3), (0, 2, 3), (1, 2, 3)],
    "pyr": [(0, 1, 2, 3), (0, 1, 4), (1, 3, 4), (3, 2, 4), (2, 0, 4)]}


def _blocks(mesh):
    """(type, corner coordinates [element][corner][3]) of the mesh, in the library's element order."""
    verts = torch.as_tensor(mesh["verts"], dtype=torch.float64, device=_device())
    for typ in ("hex", "pri", "tet", "pyr"):
        v = mesh.get(typ + "_v")
        if v is not None and len(v):
            yield typ, verts[torch.as_tensor(np.asarray(v), dtype=torch.long, device=verts.device)]


def _gauss(n, alpha=0):
    """Gauss rule of the weight (1 - x)^alpha on [-1, 1] (Golub and Welsch)."""
    k = np.arange(n, dtype=np.float64)
    with np.errstate(invalid="ignore", divide="ignore"):
        a = -alpha * alpha / ((2 * k + alpha) * (2 * k + alpha + 2))
        a[0] = -alpha / (alpha + 2)
        s = 2 * k[1:] + alpha
        b = 4 * k[1:] ** 2 * (k[1:] + alpha) ** 2 / (s * s * (s * s - 1))
    a = np.nan_to_num(a)
    x, v = np.linalg.eigh(np.diag(a) + np.diag(np.sqrt(b), 1) + np.diag(np.sqrt(b), -1))
    return x, v[0] ** 2 * 2 ** (alpha + 1) / (alpha + 1)


def _grid(*rules):
    """Tensor product of 1D rules, the first fastest: coordinates and weights."""
    x = np.meshgrid(*[r[0] for r in rules[::-1]], indexing="ij")[::-1]
    w = np.meshgrid(*[r[1] for r in rules[::-1]], indexing="ij")
    return np.stack([c.ravel() for c in x], 1), np.prod([c.ravel() for c in w], axis=0)


def _tri_rule(k):
    x, w = _grid(_gauss(k), _gauss(k))
    return np.stack([0.5 * (1 + x[:, 0]) * (1 - x[:, 1]) - 1, x[:, 1]], 1), w * 0.5 * (1 - x[:, 1])


def _volume_rule(typ, k):
    if typ == "hex":
        return _grid(_gauss(k), _gauss(k), _gauss(k))
    if typ == "pri":
        (t, wt), (z, wz) = _tri_rule(k), _gauss(k)
        return np.concatenate([np.c_[t, np.full(len(t), c)] for c in z]), np.concatenate([wt * w for w in wz])
    if typ == "tet":
        x, w = _grid(_gauss(k), _gauss(k, 1), _gauss(k, 2))
        a, b, c = x.T
        return np.stack([0.25 * (1 + a) * (1 - b) * (1 - c) - 1, 0.5 * (1 + b) * (1 - c) - 1, c], 1), w / 8
    x, w = _grid(_gauss(k), _gauss(k), _gauss(k, 2))
    return np.stack([x[:, 0] * (1 - x[:, 2]) / 2, x[:, 1] * (1 - x[:, 2]) / 2, x[:, 2]], 1), w / 4


@functools.lru_cache(maxsize=None)
def _points(typ, p):
    """Solution points in the library's order."""
    if typ == "hex":
        return _volume_rule("hex", p + 1)[0]
    if typ == "pri":
        return np.concatenate([np.c_[_WS, np.full(10, z)] for z in _gauss(p + 1)[0]])
    out = []
    for c in range(p + 1):
        for b in range(p + 1 - c):
            for a in range(p + 1 - c - (b if typ == "tet" else 0)):
                if typ == "tet":
                    x = [-1 + 2 * t / p for t in (a, b, c)]
                    out.append([-0.5 + 0.8 * (t + 0.5) for t in x])
                else:
                    h, m = 1 - c / p, p - c
                    x, y = ((h * (-1 + 2 * t / m) if m else 0.0) for t in (a, b))
                    out.append([0.8 * x, 0.8 * y, -0.5 + 0.8 * (-1 + 2 * c / p + 0.5)])
    return np.array(out)


def _modes(typ, p):
    """The polynomial (pyramid: rational) space as exponents (i, j, r, k) of x^i y^j (1 - z)^r z^k."""
    r = range(p + 1)
    if typ == "hex":
        return [(i, j, 0, k) for k in r for j in r for i in r]
    if typ == "pri":
        return [(i, j, 0, k) for k in r for j in r for i in r if i + j <= p]
    if typ == "tet":
        return [(i, j, 0, k) for k in r for j in r for i in r if i + j + k <= p]
    return [(i, j, max(i, j) - i - j, k) for k in r for j in r for i in r if max(i, j) + k <= p]


def _evaluate(modes, x):
    """Modes and their three derivatives at points x: [1 + 3][point][mode]."""
    X, Y, Z = x.T
    pw = lambda b, n: b ** n if n > 0 else np.ones_like(b) if n == 0 else 1.0 / b ** -n  # noqa: E731
    out = np.zeros((4, len(x), len(modes)))
    for m, (i, j, r, k) in enumerate(modes):
        fx, fy, fr_, fz = pw(X, i), pw(Y, j), pw(1 - Z, r), pw(Z, k)
        out[0, :, m] = fx * fy * fr_ * fz
        out[1, :, m] = i * pw(X, i - 1) * fy * fr_ * fz if i else 0
        out[2, :, m] = j * fx * pw(Y, j - 1) * fr_ * fz if j else 0
        out[3, :, m] = fx * fy * ((-r * pw(1 - Z, r - 1) * fz if r else 0) + (k * fr_ * pw(Z, k - 1) if k else 0))
    return out


@functools.lru_cache(maxsize=None)
def _operators(typ, p, aa):
    """Dense operators of one element type as torch tensors on the device."""
    m1 = p + 1 if aa == "off" else p + 2
    modes, xs = _modes(typ, p), _points(typ, p)
    inv = np.linalg.inv(_evaluate(modes, xs)[0])
    nodal = lambda x: _evaluate(modes, x) @ inv  # noqa: E731  values and derivatives of the nodal basis
    xq, wq = _volume_rule(typ, m1)
    xe, we = _volume_rule(typ, p + 4)
    le = nodal(xe)
    minv = np.linalg.inv(le[0].T * we @ le[0])
    D = [minv @ (le[0].T * we) @ le[1 + d] for d in range(3)]
    M7 = nodal(xq)[0]
    M8 = minv @ (M7.T * wq)
    corners = np.array(_CORNERS[typ], dtype=np.float64)
    xf, nf, L = [], [], []
    for f in _FACES[typ]:
        c = corners[list(f)]
        du, dv = (c[1] - c[0]) / 2, (c[2] - c[0]) / 2
        at = lambda s: c[0] + (s[:, :1] + 1) * du + (s[:, 1:] + 1) * dv  # noqa: E731
        nrm = np.cross(du, dv)
        area = np.linalg.norm(nrm)
        nrm = nrm / area
        if nrm @ (c.mean(0) - corners.mean(0)) < 0:
            nrm = -nrm
        if len(f) == 4:   # tensor Gauss points: their own quadrature
            s, w = _grid(*[_gauss(p + 2 if aa == "full" else p + 1)] * 2)
            E = nodal(at(s))[0].T * w
        else:             # Williams-Shunn points: their nodal basis integrated exactly
            s = _WS
            sq, w = _tri_rule(p + 3)
            tri = [(i, j) for j in range(p + 1) for i in range(p + 1 - j)]
            val = lambda t: np.stack([t[:, 0] ** i * t[:, 1] ** j for i, j in tri], 1)  # noqa: E731
            E = nodal(at(sq))[0].T * w @ (val(sq) @ np.linalg.inv(val(s)))
        xf.append(at(s))
        nf.append(np.repeat(nrm[None], len(s), 0))
        L.append(minv @ E * area)
    xf, nf, L = np.concatenate(xf), np.concatenate(nf), np.concatenate(L, 1)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=_device())  # noqa: E731
    return dict(xs=xs, xq=xq, xf=xf, D=t(np.stack(D)), M0=t(nodal(xf)[0]), M7=t(M7), M8=t(M8), L=t(L), nf=t(nf))


def _map(typ, verts, x):
    """Physical coordinates [element][point][3], J^-1 (dxi_i/dx_j) and det J at reference points x."""
    t = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=verts.device)  # noqa: E731
    if typ == "hex":
        c = t(_CORNERS["hex"])
        h = 0.5 * (1 + t(x)[:, None, :] * c)               # [point][corner][direction]
        shape = h.prod(-1)
        grad = torch.stack([0.5 * c[:, d] * h[..., [k for k in range(3) if k != d]].prod(-1) for d in range(3)], -1)
        X = torch.einsum("pc,ecd->epd", shape, verts)
        J = torch.einsum("pci,ecd->epdi", grad, verts)     # dx_d / dxi_i
    else:
        c = t(_CORNERS[typ])
        last = {"pri": 3, "tet": 3, "pyr": 4}[typ]
        ref = torch.stack([c[1] - c[0], c[2] - c[0], c[last] - c[0]], 1)
        phy = torch.stack([verts[:, 1] - verts[:, 0], verts[:, 2] - verts[:, 0], verts[:, last] - verts[:, 0]], 2)
        A = phy @ torch.linalg.inv(ref)
        X = verts[:, None, 0] + torch.einsum("edi,pi->epd", A, t(x) - c[0])
        J = A[:, None].expand(-1, len(x), -1, -1)
    return X, J


def _pairs(x, period):
    """Partner of every flux point, matched by its coordinates modulo the periods."""
    per = torch.as_tensor(period, dtype=torch.float64, device=x.device)
    scale = 2.0 ** 19
    for off in (0.2371, 0.6173, 0.4419, 0.8837):
        k = torch.floor(torch.remainder(x / per + 0.013, 1.0) * scale + off).long()
        key = (k[:, 0] * (1 << 21) + k[:, 1]) * (1 << 21) + k[:, 2]
        key, order = torch.sort(key)
        a, b = order[0::2], order[1::2]
        if bool((key[0::2] == key[1::2]).all()) and bool((key[2::2] != key[1:-1:2]).all()):
            partner = torch.empty_like(order)
            partner[a], partner[b] = b, a
            return partner
    raise ValueError("flux points do not pair up")


def _flux(u, q, mu, pref):
    """Total flux f[direction][variable] of the state u [e, 5, pt] with gradient q [e, 5, 3, pt]; the
    viscous part alone beside it."""
    rho, E = u[:, 0], u[:, 4]
    v = u[:, 1:4] / rho[:, None]
    p = (GAMMA - 1) * (E - 0.5 * (u[:, 1:4] * v).sum(1))
    dv = (q[:, 1:4] - v[:, :, None] * q[:, :1]) / rho[:, None, None]        # dv_i / dx_d
    tau = mu * (dv + dv.transpose(1, 2))
    div = dv[:, 0, 0] + dv[:, 1, 1] + dv[:, 2, 2]
    for d in range(3):
        tau[:, d, d] -= 2.0 / 3.0 * mu * div
    eint = E / rho
    heat = mu * GAMMA / PRANDTL * ((q[:, 4] - eint[:, None] * q[:, 0]) / rho[:, None] - (v[:, :, None] * dv).sum(1))
    fv = torch.cat([torch.zeros_like(heat)[:, None], tau, ((v[:, :, None] * tau).sum(1) + heat)[:, None]], 1)
    fe = torch.cat([u[:, None, 1:4], u[:, 1:4, None] * v[:, None], (v * (E + p)[:, None])[:, None]], 1)
    for d in range(3):
        fe[:, 1 + d, d] += p - pref
    return fe - fv, fv


def _rhs(mesh, p, aa, mu, pref, u):
    """du/dt of one instance's state u (flat, the library's layout)."""
    blocks, off, elem = [], 0, 0
    for typ, verts in _blocks(mesh):
        op = _operators(typ, p, aa)
        ne, nu = len(verts), len(op["xs"])
        ub = u[off:off + ne * 5 * nu].reshape(ne, 5, nu)
        off += ub.numel()
        X, Jf = _map(typ, verts, op["xf"])
        ns = torch.einsum("epid,pi->epd", torch.linalg.inv(Jf), op["nf"]) * torch.linalg.det(Jf)[..., None]
        blocks.append(dict(typ=typ, verts=verts, op=op, u=ub, ns=ns, x=X, uf=ub @ op["M0"].T,
                           elem=elem + torch.arange(ne, device=u.device)[:, None].expand(-1, len(op["xf"]))))
        elem += ne
    flat = lambda k: torch.cat([b[k].reshape(-1) if b[k].dim() == 2 else b[k].reshape(-1, 3) for b in blocks])  # noqa: E731
    cat = lambda k: torch.cat([b[k].transpose(1, 2).reshape(-1, 5) for b in blocks])  # noqa: E731
    partner = _pairs(flat("x"), mesh["period"])
    el = flat("elem")
    left = (el < el[partner])[:, None]
    uf = cat("uf")
    up = uf[partner]
    uL, uR = torch.where(left, uf, up), torch.where(left, up, uf)
    common = (0.5 - BETA) * uL + (0.5 + BETA) * uR
    split = lambda a, k: (t.reshape(len(b["u"]), -1, k) for t, b in  # noqa: E731
                          zip(torch.split(a, [b["uf"].shape[0] * b["uf"].shape[2] for b in blocks]), blocks))
    for b, c in zip(blocks, split(common, 5)):
        op = b["op"]
        jump = c.transpose(1, 2) - b["uf"]
        qr = torch.stack([b["u"] @ op["D"][d].T + (jump * op["nf"][:, d]) @ op["L"].T for d in range(3)], 2)
        Js = torch.linalg.inv(_map(b["typ"], b["verts"], op["xs"])[1])
        b["q"] = torch.einsum("epid,evip->evdp", Js, qr)
        fv = _flux(b["uf"], b["q"] @ op["M0"].T, mu, pref)[1]
        n = b["ns"] / b["ns"].norm(dim=-1, keepdim=True)
        b["fvn"] = torch.einsum("evdp,epd->evp", fv, n)
    ns = flat("ns")
    mag = ns.norm(dim=-1, keepdim=True)
    n = torch.where(left, ns, -ns) / mag                     # outward from the left side
    fvn = cat("fvn")
    fp = fvn[partner]
    # own-normal viscous fluxes along the left normal: the right side's own normal is the opposite one
    fvL, fvR = torch.where(left, fvn, fp), torch.where(left, -fp, -fvn)

    def inviscid(w):
        pr = (GAMMA - 1) * (w[:, 4:] - 0.5 * (w[:, 1:4] ** 2).sum(1, keepdim=True) / w[:, :1])
        vn = (w[:, 1:4] * n).sum(1, keepdim=True) / w[:, :1]
        return torch.cat([w[:, :1] * vn, w[:, 1:4] * vn + (pr - pref) * n, vn * (w[:, 4:] + pr)], 1), vn.abs() + torch.sqrt(GAMMA * pr / w[:, :1])

    (feL, sL), (feR, sR) = inviscid(uL), inviscid(uR)
    F = 0.5 * (feL + feR) + (0.5 * torch.maximum(sL, sR) + TAU) * (uL - uR) - (0.5 + BETA) * fvL - (0.5 - BETA) * fvR
    F = torch.where(left, F, -F) * mag
    out = []
    for b, Fb in zip(blocks, split(F, 5)):
        op = b["op"]
        f = _flux(b["u"] @ op["M7"].T, b["q"] @ op["M7"].T, mu, pref)[0]
        Jq = _map(b["typ"], b["verts"], op["xq"])[1]
        Jq = torch.linalg.inv(Jq) * torch.linalg.det(Jq)[..., None, None]
        f = torch.einsum("epid,evdp->evip", Jq, f) @ op["M8"].T
        div = sum(f[:, :, d] @ op["D"][d].T for d in range(3))
        own = torch.einsum("evip,pi->evp", f @ op["M0"].T, op["nf"])
        div = div + (Fb.transpose(1, 2) - own) @ op["L"].T
        det = torch.linalg.det(_map(b["typ"], b["verts"], op["xs"])[1])
        out.append((-div / det[:, None]).reshape(-1))
    return torch.cat(out)


def exact(case, seed):
    u = _state(case, seed)
    if case["call"] == "rhs" and case["prec"] != "fp64":
        u = u.float().double()
    parts = [(_mesh(kind, n), p, mach, re) for kind, n, p, mach, re in _instances(case)]
    sizes = [sum(len(v) * 5 * len(_points(t, p)) for t, v in _blocks(mesh)) for mesh, p, _, _ in parts]

    def rhs(w):
        return torch.cat([_rhs(mesh, p, case["aa"], 1.0 / re, _p0(mach), x)
                          for (mesh, p, mach, re), x in zip(parts, torch.split(w, sizes))])

    if case["call"] == "rhs":
        return rhs(u)
    h = _dt(case)
    k = rhs(u)
    acc = k / 6
    for c, b in ((0.5, 1 / 3), (0.5, 1 / 3), (1.0, 1 / 6)):
        k = rhs(u + c * h * k)
        acc += b * k
    return u + h * acc
