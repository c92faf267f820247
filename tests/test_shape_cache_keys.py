"""Keys of the stored volume-kernel shapes: handles whose shape index selects different kernels do not share
one, handles that run the same kernels do, and those of forms without kernels of their own are as before."""
import types

import pytest

from paper_2401_06132_gb300 import fr

torch = pytest.importorskip("torch")


@pytest.fixture
def key(monkeypatch):
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "GPU")
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_properties", lambda d: types.SimpleNamespace(multi_processor_count=152))

    def make(elements=1000, p=3, m=5, shapes=6, **kw):
        f = fr.FRMesh.__new__(fr.FRMesh)
        prm = [fr.make_params(p=p, **kw)]
        f.prec = prm[0].prec
        f._lowmach = f._is_lowmach(prm) if hasattr(f, "_is_lowmach") else None
        f.groups = lambda: [dict(type=0, p=p, m=m, elements=elements, shape=1, shapes=shapes)]
        return f._shape_keys()[0]

    return make


def test_forms_and_size_classes_have_their_own_keys(key):
    low = dict(prec="fp32", p_ref=71.4, rho_ref=1.0)
    keys = [key(**low), key(elements=304, **low), key(prec="fp32"), key(prec="fp64"), key(p=4, m=6, **low),
            key(prec="mixed_fp16", p_ref=71.4, rho_ref=1.0)]
    assert len(set(keys)) == len(keys)
    assert key(elements=305, **low) == keys[0] and key(elements=1, **low) == keys[1]


def test_other_keys_are_unchanged(key):
    assert key(prec="fp64") == key(prec="fp64", elements=8, p_ref=71.4, rho_ref=1.0) == "GPU|fp64|type0|p3|m5"
    assert key(prec="fp32") == key(prec="fp32", elements=8) == "GPU|fp32|type0|p3|m5"
    assert key(prec="fp32", m=4, p_ref=71.4, rho_ref=1.0) == "GPU|fp32|type0|p3|m4"
    assert key(prec="fp32", shapes=1) is None
