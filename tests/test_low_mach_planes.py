"""The low-Mach FP32 volume kernel on hexahedra (planes and columns, several elements per CTA): element
counts that do not fill a CTA, diagonal and full metrics, one and both sides weighted, and every launch
shape, against the oracle on the FP32-rounded state at the FP32 forms' bound (2e-5 relative L-infinity
per conserved variable); the shapes compute every value with the same operations, so their results are
equal bit for bit."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2401_06132_gb300 import fr, workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_06132_gb300 import build as B
    B.build()


@pytest.mark.parametrize("mesh", [lambda: W.box_hex_mesh(1), lambda: W.box_hex_mesh(3), lambda: W.sheared_box_mesh(3)],
                         ids=["one", "odd", "sheared"])
@pytest.mark.parametrize("p", [3, 4])
@pytest.mark.parametrize("beta", [0.5, 0.2])
def test_low_mach_rhs_matches_oracle_in_every_shape(mesh, p, beta):
    m = mesh()
    ne, nu, p0 = m["hex_v"].shape[0], (p + 1) ** 3, W.tgv_p0()
    o = O.Oracle(m, p, p + 2, beta=beta, p_ref=p0)
    U = W.tgv_state(o.sol_coords(), [(ne, nu)], perturb=1e-3).astype(np.float32)
    Ro = o.rhs(U.astype(np.float64)).reshape(ne, 5, nu)
    f = fr.FRMesh(m, fr.make_params(p=p, prec="fp32", beta=beta, p_ref=p0, rho_ref=1.0))
    u = torch.from_numpy(U).cuda()
    out = []
    for shape in range(3):
        f.set_volume_shape(shape)
        r = torch.empty_like(u)
        f.rhs(u, r)
        f.sync_status()
        out.append(r.cpu().numpy().reshape(ne, 5, nu))
        err = np.abs(out[-1] - Ro).max(axis=(0, 2)) / np.abs(Ro).max(axis=(0, 2))
        assert err.max() <= 2e-5, (shape, err)
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[2], out[1])
