"""The tuner's cache keeps meshes of different size apart (no GPU: a mesh and the
library's entry points are stood in for)."""
import json

import pytest

from paper_2202_12477_gb300 import autotune as at
from paper_2202_12477_gb300 import hb

SIZES = [(8, 4096), (64, 32768), (125, 64000), (216, 110592), (4000, 2_048_000), (20000, 10_240_000),
         (249856, 127_926_272)]


def test_size_classes_are_ordered_and_distinct():
    names = [at.size_class(*s) for s in SIZES]
    assert len(set(names)) == len(SIZES)
    for e in (38, 76, 152, 1216):
        assert at.size_class(e, 512 * e) != at.size_class(e + 1, 512 * (e + 1))


class _Info:
    geo32 = 1


class _Mesh:
    def __init__(self, E, n_local):
        self.E, self.n_local, self.N, self.handle, self.info = E, n_local, 3, object(), _Info()


@pytest.fixture
def library(monkeypatch):
    calls = {"tuned": 0, "set": []}

    def tune(h, prec, screen, lam, reps):
        calls["tuned"] += 1
        return calls["best"], {3: 2.0, calls["best"]: 1.0}
    monkeypatch.setattr(at, "current_device_key", lambda: "gpu")
    monkeypatch.setattr(hb, "hb_autotune", tune)
    monkeypatch.setattr(hb, "hb_set_kernel_variant", lambda h, p, v: calls["set"].append(v))
    monkeypatch.setattr(hb, "hb_set_apply_variant", lambda h, p, v: calls["set"].append(("apply", v)))
    monkeypatch.setattr(hb, "hb_get_apply_variant", lambda h, p: calls["best"])
    return calls


def test_a_large_meshs_choice_is_not_used_on_a_small_one(tmp_path, library):
    path = str(tmp_path / "c.json")
    library["best"] = hb.HB_VARIANT_TC
    assert at.tune_mesh(_Mesh(1998848, 127_926_272), precs=(hb.HB_F64,), path=path)[hb.HB_F64] == hb.HB_VARIANT_TC
    library["best"] = 3
    assert at.tune_mesh(_Mesh(64, 4096), precs=(hb.HB_F64,), path=path)[hb.HB_F64] == 3
    assert library["tuned"] == 2
    # each size finds its own choice again
    assert at.tune_mesh(_Mesh(1900000, 121_600_000), precs=(hb.HB_F64,), path=path)[hb.HB_F64] == hb.HB_VARIANT_TC
    assert at.tune_mesh(_Mesh(60, 3840), precs=(hb.HB_F64,), path=path)[hb.HB_F64] == 3
    assert library["tuned"] == 2 and library["set"] == [hb.HB_VARIANT_TC, 3]


def test_entries_without_a_size_are_not_used(tmp_path, library):
    path = tmp_path / "c.json"
    path.write_text(json.dumps({"gpu": {at.entry_key(3, hb.HB_F64): {"variant": hb.HB_VARIANT_TC}}}))
    library["best"] = 3
    assert at.tune_mesh(_Mesh(64, 4096), precs=(hb.HB_F64,), path=str(path))[hb.HB_F64] == 3
    assert library["tuned"] == 1
