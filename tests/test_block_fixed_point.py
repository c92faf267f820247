"""The FP64 volume kernels' block fixed-point operators against the plain FP64 form (one kernel per
paper kernel, every operator in FP64 arithmetic), over the states and metrics where a block scaled by
its largest magnitude could lose small values: jumps inside an element, values spread over decades,
stretched and curved elements, units far from 1, both sides weighted, fields that vanish; and the
handling of non-finite values.

Both forms compute R~ = sum of operator rows times fluxes; each rounds at most C = 100 times at 2^-53
of the largest term, F (3 directions) (row sum of the corrected derivative and the lift, below 16) 2/h,
with F the largest flux of the variable, inviscid plus Rusanov dissipation (|v| + c) |u| plus viscous
mu |grad u| terms (below the inviscid ones on these meshes). The difference is held to twice that.
"""
import numpy as np
import pytest

from paper_2401_06132_gb300 import fr, workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_06132_gb300 import build as B
    B.build()


def _mesh(name):
    if name == "curved":
        return W.curved_box_mesh(3)
    if name == "sheared":
        return W.sheared_box_mesh(3)
    m = W.box_hex_mesh(3)
    s = np.array([1.0, 20.0, 400.0])   # stretched
    return dict(m, verts=m["verts"] * s, period=tuple(np.array(m["period"]) * s))


def _state(kind, ne, nu, rng):
    """Conserved variables, [element][variable][point], whose traces and interpolants (row sums of the
    operators below 3.6) keep density and pressure positive."""
    shape = (ne, nu)
    rho = np.ones(shape)
    v = [0.3 * np.ones(shape), np.zeros(shape), -0.1 * np.ones(shape)]   # v_y vanishes
    p = 50.0 * np.ones(shape)
    if kind in ("jumps", "units"):
        rho *= 1 + 0.1 * rng.uniform(-1, 1, shape)
        p *= 1 + 0.1 * rng.uniform(-1, 1, shape)
        v = [0.5 * rng.uniform(-1, 1, shape) for _ in range(3)]
    elif kind == "decades":   # velocities over twelve decades inside every element
        v = [10.0 ** rng.uniform(-12, 0, shape) * rng.choice([-1, 1], shape) for _ in range(3)]
        p *= 1 + 1e-9 * rng.uniform(-1, 1, shape)
    if kind == "units":
        rho, p, v = rho * 1.2e-9, p * 3e5, [x * 1e7 for x in v]
    E = p / 0.4 + 0.5 * rho * sum(x * x for x in v)
    return np.stack([rho, rho * v[0], rho * v[1], rho * v[2], E], axis=1)


@pytest.mark.parametrize("mesh", ["stretched", "sheared", "curved"])
@pytest.mark.parametrize("p", [3, 4])
@pytest.mark.parametrize("kind", ["jumps", "decades", "units", "vanish"])
@pytest.mark.parametrize("beta", [0.5, 0.2])
def test_fixed_point_operators_match_plain_fp64(mesh, p, kind, beta):
    m = _mesh(mesh)
    nu = (p + 1) ** 3
    U = _state(kind, 27, nu, np.random.default_rng(7))
    prm = fr.make_params(p=p, beta=beta, mu=1e-3 * (1e-2 if kind == "units" else 1.0))
    f = fr.FRMesh(m, prm)
    u = torch.from_numpy(U.reshape(-1)).cuda()
    out = {}
    for form in ("fused", "unfused"):
        f.set_form(form)
        r = torch.empty_like(u)
        f.rhs(u, r)
        f.sync_status()
        out[form] = r.cpu().numpy().reshape(27, 5, nu)
    rho, E = U[:, 0], U[:, 4]
    v = U[:, 1:4] / rho[:, None]
    pr = 0.4 * (E - 0.5 * rho * (v * v).sum(1))
    # traces of jumping states exceed the nodal values by at most the row sum of the trace operator, 3.4
    w = (np.abs(v).max() + np.sqrt(1.4 * pr.max() / rho.min())) * 3.4
    h = np.linalg.norm(m["verts"][m["hex_v"][0, 1]] - m["verts"][m["hex_v"][0, 0]])
    for a in range(5):
        F = w * np.abs(U[:, a]).max() * 3.4 + (pr.max() if 1 <= a <= 3 else 0) + (w * pr.max() if a == 4 else 0)
        tol = 2 * 100 * 2.0 ** -53 * F * 3 * 16 * 2 / h
        assert np.abs(out["fused"][:, a] - out["unfused"][:, a]).max() <= tol, a


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("p", [3, 4])
def test_non_finite_values_are_reported(bad, p):
    """A non-finite value reaches R of its element as a non-finite value and the status word."""
    m = W.box_hex_mesh(3)
    nu = (p + 1) ** 3
    U = _state("jumps", 27, nu, np.random.default_rng(3))
    U[13, 2, 5] = bad
    f = fr.FRMesh(m, fr.make_params(p=p))
    u = torch.from_numpy(U.reshape(-1)).cuda()
    r = torch.empty_like(u)
    f.rhs(u, r)
    with pytest.raises(fr.FRError) as e:
        f.sync_status()
    assert e.value.status == fr.FR_ENONPHYS
    assert not np.isfinite(r.cpu().numpy().reshape(27, 5, nu)[13, 2]).any()
    f.rhs(torch.from_numpy(_state("jumps", 27, nu, np.random.default_rng(3)).reshape(-1)).cuda(), r)
    f.sync_status()
    assert torch.isfinite(r).all()
