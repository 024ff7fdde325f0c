"""Plan.tune with a cache file: choices stored for other kernel tables are not applied (no GPU: a stand-in library)."""
import ctypes
import json

import torch

from paper_1506_07933_gb300 import afft


class Library:
    """Records the tuning calls of a plan."""

    def __init__(self):
        self.calls = []
        self.cfg = [0, 1, 1, 0, 0, 0]

    def afft_plan_tune(self, plan, stream):
        self.calls.append("tune")
        self.cfg = [2048, 1, 0, 0, 0, 0]
        return 0

    def afft_plan_set_tuning(self, plan, cfg):
        self.calls.append("set")
        self.cfg = [int(v) for v in cfg]
        return 0

    def afft_plan_get_tuning(self, plan, cfg):
        for i, v in enumerate(self.cfg):
            cfg[i] = v
        return 0


def plan(monkeypatch, lib):
    monkeypatch.setattr(afft, "load", lambda *a: lib)
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "GPU A")
    monkeypatch.setattr(afft, "_stream_handle", lambda s: 0)
    p = afft.Plan.__new__(afft.Plan)
    p.shape, p.kind, p.precision, p.batch = (64, 120, 240), afft.R2C, afft.F32, None
    p.device, p._p = torch.device("cpu"), ctypes.c_void_p()
    return p


def test_entries_of_other_kernel_tables_are_ignored(monkeypatch, tmp_path):
    path = str(tmp_path / "tune.json")
    bare = afft.tuning_key((64, 120, 240), afft.R2C, afft.F32, None, "GPU A")
    stale = [4096, 1, 1, 0, 0, 1]
    for key in (bare, "%s/tables%d" % (bare, afft.KERNEL_TABLES - 1)):
        afft.tuning_cache_store(path, key, stale)
    lib = Library()
    p = plan(monkeypatch, lib)
    assert p.tune(cache=path) is False
    assert lib.calls == ["tune"] and p.tuning == [2048, 1, 0, 0, 0, 0]
    assert json.load(open(path))["%s/tables%d" % (bare, afft.KERNEL_TABLES)] == [2048, 1, 0, 0, 0, 0]
    lib = Library()   # stored under the present tables: applied without tuning
    p = plan(monkeypatch, lib)
    assert p.tune(cache=path) is True
    assert lib.calls == ["set"] and p.tuning == [2048, 1, 0, 0, 0, 0]
