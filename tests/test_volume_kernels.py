"""The FP64 block fixed-point kernels on prisms, tetrahedra and pyramids, and the four-element FP32
kernels on tetrahedra and pyramids, against the oracle.

FP64: states where a block scaled by its largest magnitude could lose small values (jumps inside an
element, values over twelve decades, units far from 1), on stretched meshes. Kernel and oracle compute
R = sum of operator rows times fluxes; each rounds at most C = 500 times (a row of the widest chain:
interpolation 30, gradient 90 + 60, projection 375, lift 60 terms, of which the projection's partial
sums count once per slice) at 2^-53 of the largest term, F S G with F the largest flux of the variable
(inviscid plus Rusanov dissipation; the viscous terms are far below), S the row sums of the divergence
and lift operators and G those of the inverse metric. The difference is held to twice that.

FP32: sizes on both sides of the line between one and four elements per CTA, with a last group that is
not full, at the FP32 forms' bounds on the FP32-rounded state (2e-5 relative L-infinity per variable
in the low-Mach form, 1e-3 without a reference state).
"""
import os

import numpy as np
import pytest

from oracle import oracle as O
from paper_2401_06132_gb300 import fr, workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
NU = {"hex": 64, "pri": 40, "tet": 20, "pyr": 30}
NCPU = max(1, min(16, (os.cpu_count() or 2) - 1))


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_06132_gb300 import build as B
    B.build()


def _blocks(m):
    return [(t, len(m[t + "_v"]), NU[t]) for t in NU if len(m.get(t + "_v", ()))]


def _state(kind, n, rng):
    """Conserved variables [variable][point] whose interpolants keep density and pressure positive."""
    rho, p = np.ones(n), 50.0 * np.ones(n)
    if kind == "decades":   # velocities over twelve decades inside every element
        v = [10.0 ** rng.uniform(-12, 0, n) * rng.choice([-1, 1], n) for _ in range(3)]
        p *= 1 + 1e-9 * rng.uniform(-1, 1, n)
    else:
        rho *= 1 + 0.05 * rng.uniform(-1, 1, n)
        p *= 1 + 0.05 * rng.uniform(-1, 1, n)
        v = [0.5 * rng.uniform(-1, 1, n) for _ in range(3)]
    if kind == "units":
        rho, p, v = rho * 1.2e-9, p * 3e5, [x * 1e7 for x in v]
    E = p / 0.4 + 0.5 * rho * sum(x * x for x in v)
    return np.stack([rho, rho * v[0], rho * v[1], rho * v[2], E])


@pytest.mark.parametrize("mesh", ["prisms", "tetrahedra", "pyramids"])
@pytest.mark.parametrize("kind", ["jumps", "decades", "units"])
@pytest.mark.parametrize("beta", [0.5, 0.2])
def test_fp64_matches_oracle_on_extreme_states(mesh, kind, beta):
    m = {"prisms": lambda: W.mixed_box_mesh(4), "tetrahedra": lambda: W.box_tet_mesh(2),
         "pyramids": lambda: W.box_pyr_mesh(2)}[mesh]()
    s = np.array([1.0, 7.0, 50.0])
    m = dict(m, verts=m["verts"] * s, period=tuple(np.array(m["period"]) * s))
    mu = 1e-5 if kind == "units" else 1e-3
    o = O.Oracle(m, 3, 5, mu=mu, beta=beta, threads=NCPU)
    rng = np.random.default_rng(7)
    U = [np.moveaxis(_state(kind, ne * nu, rng).reshape(5, ne, nu), 0, 1) for _, ne, nu in _blocks(m)]
    Uf = np.concatenate([u.reshape(-1) for u in U])
    Ro = o.rhs(Uf)
    f = fr.FRMesh(m, fr.make_params(p=3, beta=beta, mu=mu))
    u = torch.from_numpy(Uf).cuda()
    r = torch.empty_like(u)
    f.rhs(u, r)
    f.sync_status()
    diff = np.abs(r.cpu().numpy() - Ro)
    G = max(np.abs(o.geometry(e)[1]).sum() for e in range(sum(ne for _, ne, _ in _blocks(m))))
    ops = [t for t, key in enumerate(("hex", "pri", "tet", "pyr")) if len(m.get(key + "_v", ()))]
    S = L = 0.0
    for t in ops:
        A, P, M0 = np.abs(o.op(t, "Adiv")), np.abs(o.op(t, "M8")), np.abs(o.op(t, "M0"))
        n = np.linalg.norm(o.op(t, "nref"), axis=1)
        S = max(S, ((A @ P).sum(axis=(1, 2)) + np.abs(o.op(t, "lift")) @ n).max())
        L = max(L, M0.sum(1).max(), np.abs(o.op(t, "M7")).sum(1).max())
    amp = np.abs(np.concatenate([np.moveaxis(x, 1, 0).reshape(5, -1) for x in U], axis=1))
    rho = amp[0]
    v = (amp[1:4] / rho).max()
    pr = 0.4 * amp[4].max()
    w = (v + np.sqrt(1.4 * pr / rho.min())) * L
    start = 0
    for _, ne, nu in _blocks(m):
        d = diff[start:start + ne * 5 * nu].reshape(ne, 5, nu).max(axis=(0, 2))
        start += ne * 5 * nu
        for a in range(5):
            F = w * amp[a].max() * L + (pr if 1 <= a <= 3 else 0) + (w * pr if a == 4 else 0)
            assert d[a] <= 2 * 500 * 2.0 ** -53 * F * S * G, (a, d[a])


@pytest.mark.parametrize("lowmach", [True, False])
@pytest.mark.parametrize("mesh", ["tet2", "tet5", "tet7", "pyr2", "pyr7"])
@pytest.mark.parametrize("beta", [0.5, 0.2])
def test_fp32_dense_matches_oracle_on_both_sides_of_the_line(mesh, lowmach, beta):
    n = int(mesh[3:])
    m = W.box_tet_mesh(n) if mesh[:3] == "tet" else W.box_pyr_mesh(n)
    (t, ne, nu), = _blocks(m)
    p0 = W.tgv_p0()
    o = O.Oracle(m, 3, 5, beta=beta, p_ref=p0, threads=NCPU)
    U = W.tgv_state(o.sol_coords(), [(ne, nu)], perturb=1e-2).astype(np.float32)
    Ro = o.rhs(U.astype(np.float64)).reshape(ne, 5, nu)
    ref = dict(p_ref=p0, rho_ref=1.0) if lowmach else {}
    f = fr.FRMesh(m, fr.make_params(p=3, prec="fp32", beta=beta, **ref))
    u = torch.from_numpy(U).cuda()
    r = torch.empty_like(u)
    f.rhs(u, r)
    f.sync_status()
    err = np.abs(r.cpu().numpy().reshape(ne, 5, nu) - Ro).max(axis=(0, 2)) / np.abs(Ro).max(axis=(0, 2))
    assert err.max() <= (2e-5 if lowmach else 1e-3), err


@pytest.mark.parametrize("mesh", ["stretched", "sheared"])
@pytest.mark.parametrize("p", [3, 4])
@pytest.mark.parametrize("kind", ["jumps", "decades", "units"])
@pytest.mark.parametrize("beta", [0.5, 0.2])
def test_fp64_collocation_matches_oracle_on_extreme_states(mesh, p, kind, beta):
    """Hexahedra without anti-aliasing, at the bound of the first test (chains are shorter)."""
    m = W.sheared_box_mesh(3) if mesh == "sheared" else W.box_hex_mesh(3)
    s = np.array([1.0, 7.0, 50.0]) if mesh == "stretched" else np.ones(3)
    m = dict(m, verts=m["verts"] * s, period=tuple(np.array(m["period"]) * s))
    mu, ne, nu = 1e-5 if kind == "units" else 1e-3, 27, (p + 1) ** 3
    o = O.Oracle(m, p, p + 1, mu=mu, beta=beta, threads=NCPU)
    amp = _state(kind, ne * nu, np.random.default_rng(7))
    Uf = np.moveaxis(amp.reshape(5, ne, nu), 0, 1).reshape(-1).copy()
    Ro = o.rhs(Uf)
    f = fr.FRMesh(m, fr.make_params(p=p, nq1d=p + 1, beta=beta, mu=mu))
    u = torch.from_numpy(Uf).cuda()
    r = torch.empty_like(u)
    f.rhs(u, r)
    f.sync_status()
    d = np.abs(r.cpu().numpy() - Ro).reshape(ne, 5, nu).max(axis=(0, 2))
    G = max(np.abs(o.geometry(e)[1]).sum() for e in range(ne))
    S = (np.abs(o.op(0, "Adiv")).sum(axis=(1, 2)) + np.abs(o.op(0, "lift")) @ np.linalg.norm(o.op(0, "nref"), axis=1)).max()
    L = np.abs(o.op(0, "M0")).sum(1).max()
    amp = np.abs(amp)
    pr = 0.4 * amp[4].max()
    w = ((amp[1:4] / amp[0]).max() + np.sqrt(1.4 * pr / amp[0].min())) * L
    for a in range(5):
        F = w * amp[a].max() * L + (pr if 1 <= a <= 3 else 0) + (w * pr if a == 4 else 0)
        assert d[a] <= 2 * 500 * 2.0 ** -53 * F * S * G, (a, d[a])
