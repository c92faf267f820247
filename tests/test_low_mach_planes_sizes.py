"""The low-Mach FP32 volume kernel on hexahedra above two elements per SM, where the default shape takes two
elements per CTA (p = 3; an odd count leaves the last CTA half full) or one of 128 threads (p = 4): every
launch shape against the oracle at the FP32 forms' bound (2e-5 relative L-infinity per conserved variable), and
the shapes against each other bit for bit."""
import os

import numpy as np
import pytest

from oracle import oracle as O
from paper_2401_06132_gb300 import fr, workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
NCPU = max(1, min(16, (os.cpu_count() or 2) - 1))


@pytest.mark.parametrize("p,n", [(3, 9), (4, 7)])
def test_every_shape_on_more_than_two_elements_per_sm(p, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_06132_gb300 import build as B
    B.build()
    m = W.box_hex_mesh(n)
    ne, nu, p0 = n ** 3, (p + 1) ** 3, W.tgv_p0()
    assert ne > 2 * torch.cuda.get_device_properties(0).multi_processor_count
    o = O.Oracle(m, p, p + 2, p_ref=p0, threads=NCPU)
    U = W.tgv_state(o.sol_coords(), [(ne, nu)], perturb=1e-3).astype(np.float32)
    Ro = o.rhs(U.astype(np.float64)).reshape(ne, 5, nu)
    f = fr.FRMesh(m, fr.make_params(p=p, prec="fp32", p_ref=p0, rho_ref=1.0))
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
