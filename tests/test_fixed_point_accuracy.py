"""Rounding errors of the FP64 kernels with block fixed-point operators, against the oracle in extended
precision, beside those of the oracle in FP64 on the same state: per element type and conserved variable
the largest error is held to K times the oracle's.

K: with every operator in FP64 arithmetic the kernels' errors were at most 2.5 (hexahedra), 1.6
(prisms), 14 (tetrahedra) and 8.2 (pyramids) times the oracle's on these states and on elements stretched
by 10^4 (other operator tables, other orders of the sums). K = 8 and 64 leave a factor of three or more,
the machines' libraries and the draws; a value that loses more than those few bits fails.

Stretched elements: the velocity component along the short direction s varies along the long direction l only,
the others vanish. Of the momentum along l that leaves the flux mu dv_s/dx_l through s, in which a
gradient resolved at the scale of the short direction would show up to 2^16 times larger than rounding.
"""
import os

import numpy as np
import pytest

import extended_oracle as X
from oracle import oracle as O
from paper_2401_06132_gb300 import fr, workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
K = {"hex": 8, "pri": 8, "tet": 64, "pyr": 64}
NCPU = max(1, min(16, (os.cpu_count() or 2) - 1))
MESHES = {"hex": lambda: W.box_hex_mesh(3), "sheared": lambda: W.sheared_box_mesh(3),
          "curved": lambda: W.curved_box_mesh(3), "mixed": lambda: W.mixed_box_mesh(4),
          "tet": lambda: W.box_tet_mesh(2), "pyr": lambda: W.box_pyr_mesh(2)}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_06132_gb300 import build as B
    B.build()


def _mesh(name, stretch):
    m = MESHES[name]()
    return dict(m, verts=m["verts"] * stretch, period=tuple(np.array(m["period"]) * stretch))


def _check(m, p, states, mu, p_ref=0.0, nq1d=None):
    q = nq1d or p + 2
    o = O.Oracle(m, p, q, mu=mu, p_ref=p_ref, threads=NCPU)
    nus = {"hex": (p + 1) ** 3, "pri": 40, "tet": 20, "pyr": 30}
    blocks = [(t, len(m[t + "_v"]), nu) for t, nu in nus.items() if len(m.get(t + "_v", ()))]
    x = o.sol_coords()
    U = [W.to_layout(s(x), [(ne, nu) for _, ne, nu in blocks]) for s in states]
    f = fr.FRMesh(m, fr.make_params(p=p, mu=mu, p_ref=p_ref, nq1d=q))
    for s, v, hi, lo in zip(states, U, *X.rhs(m, p, q, U, mu=mu, p_ref=p_ref, threads=NCPU)):
        plain = np.abs((o.rhs(v) - hi) - lo)
        u = torch.from_numpy(v).cuda()
        r = torch.empty_like(u)
        f.rhs(u, r)
        f.sync_status()
        err = np.abs((r.cpu().numpy() - hi) - lo)
        off = 0
        for t, ne, nu in blocks:
            e, b = (y[off:off + ne * 5 * nu].reshape(ne, 5, nu).max(axis=(0, 2)) for y in (err, plain))
            off += ne * 5 * nu
            assert (e <= K[t] * b).all(), (s.__name__, t, e / b)


def _conserved(rho, v, p):
    return np.stack([rho, rho * v[0], rho * v[1], rho * v[2], p / 0.4 + 0.5 * rho * sum(x * x for x in v)])


@pytest.mark.parametrize("mesh,p,nq1d", [(m, 3, None) for m in MESHES] + [("hex", 4, None), ("sheared", 3, 4)])
def test_errors_are_those_of_fp64_sums(mesh, p, nq1d):
    m = _mesh(mesh, np.array([1.0, 7.0, 50.0]) if mesh in ("mixed", "tet", "pyr") else np.ones(3))
    rng = np.random.default_rng(7)

    def vortex(x):
        a, b, c = (2 * np.pi * x[:, d] / m["period"][d] for d in range(3))
        v = [np.sin(a) * np.cos(b) * np.cos(c), -np.cos(a) * np.sin(b) * np.cos(c), 0 * a]
        return _conserved(np.ones_like(a), v, 71.4 + (np.cos(2 * a) + np.cos(2 * b)) * (np.cos(2 * c) + 2) / 16)

    def jumps(x):
        r = rng.uniform(-1, 1, (5, x.shape[0]))
        return _conserved(1 + 0.05 * r[0], 0.5 * r[1:4], 50 * (1 + 0.05 * r[4]))

    def decades(x):   # velocities over twelve decades inside every element
        v = 10.0 ** rng.uniform(-12, 0, (3, x.shape[0])) * rng.choice([-1, 1], (3, x.shape[0]))
        return _conserved(np.ones(x.shape[0]), v, 50 * (1 + 1e-9 * rng.uniform(-1, 1, x.shape[0])))

    _check(m, p, [vortex, jumps, decades], 1.0, nq1d=nq1d)


@pytest.mark.parametrize("s,both", [(0, False), (2, True)], ids=["one-long", "two-long"])
@pytest.mark.parametrize("mesh", list(MESHES))
def test_gradients_along_the_long_direction(mesh, s, both):
    l = (s + 1) % 3
    stretch = np.full(3, 2.0 ** 16 if both else 1.0)
    stretch[l], stretch[s] = 2.0 ** 16, 1.0
    m = _mesh(mesh, stretch)

    def long_variation(x):
        n = x.shape[0]
        v = [np.zeros(n) for _ in range(3)]
        v[s] = np.sin(2 * np.pi * x[:, l] / m["period"][l])
        return _conserved(np.ones(n), v, 50.0 * np.ones(n))

    _check(m, 3, [long_variation], 1.0, p_ref=50.0)
