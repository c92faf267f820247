"""Order on a stream of the phase kernels, each of which is set up while the last one drains: calls without a
synchronisation between them, each on a state that ordinary kernels write just before and into a result that
they read just after, equal the same calls with one after every step, bit for bit."""
import numpy as np
import pytest

from paper_2401_06132_gb300 import fr, workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("mesh", ["hex", "hex4", "full", "curved", "mixed", "tet", "pyr"])
def test_back_to_back_calls_equal_separate_ones(mesh, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_06132_gb300 import build as B
    B.build()
    m = {"curved": W.curved_box_mesh, "mixed": W.mixed_box_mesh, "tet": W.box_tet_mesh, "pyr": W.box_pyr_mesh}.get(
        mesh, W.box_hex_mesh)(4)
    p, p0 = 4 if mesh == "hex4" else 3, W.tgv_p0()
    f = fr.FRMesh(m, fr.make_params(p=p, prec=prec, p_ref=p0, rho_ref=1.0, surface_aa=mesh == "full"))
    nus = {"hex": (p + 1) ** 3, "pri": 40, "tet": 20, "pyr": 30}
    blocks = [(len(m[t + "_v"]), nu) for t, nu in nus.items() if len(m.get(t + "_v", ()))]
    u0 = torch.from_numpy(W.tgv_state(f.sol_coords(), blocks, perturb=1e-3)).cuda().to(f.dtype)
    w = torch.from_numpy(1 + 1e-3 * W.uniform_pm1(9, np.arange(u0.numel()))).cuda().to(f.dtype)

    def go(wait):
        u, r, out = u0.clone(), torch.empty_like(u0), []
        for _ in range(12):
            f.rhs(u, r)
            out.append(r.clone())
            u.copy_(u0).mul_(w).add_(r, alpha=1e-6)
            r.fill_(float("nan"))
            if wait:
                torch.cuda.synchronize()
        f.sync_status()
        return torch.stack(out)

    assert torch.equal(go(False), go(True))
