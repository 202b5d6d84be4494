"""What a cached launch is valid for, on the host."""
import pytest

from paper_1010_4135_gb300 import autotune


class FakeSim:
    def __init__(self, recovery=0.0, tau=1e-5):
        self.config = dict(nx=64, ny=32, nz=16, precision="fp32", scheme="nnd", bc_lo=(1, 0, 0), bc_hi=(2, 0, 0),
                           dt=1e-5, tau=tau)
        self.t_recovery = recovery
        self.launch = None

    def set_launch(self, variant, zchunk, ztail=0):
        self.launch = (variant, zchunk, ztail)


def _entry(sim=None, zchunks=autotune.ZCHUNKS):
    return autotune.entry_of([sim or FakeSim()], False, zchunks, device_name="d", sms=1)


def test_an_entry_is_of_its_candidates_and_kernel_form():
    names = {_entry(), _entry(zchunks=(0, 4, 8)), _entry(FakeSim(recovery=4.0)), _entry(FakeSim(tau=2e-5))}
    assert len(names) == 4
    assert all(n.startswith(autotune.key_of([FakeSim()], False, "d", 1)) for n in names)
    assert _entry() == _entry()


def test_an_entry_of_other_kernel_sources_is_not_used(tmp_path, monkeypatch):
    path = str(tmp_path / "launch.json")
    monkeypatch.setattr(autotune, "key_of", lambda *a, **k: "shape")
    monkeypatch.setattr(autotune, "measure", lambda *a, **k: {("tiled", 0, 0): 1.0})
    rec = {"variant": "tiled", "zchunk": 12, "ztail": 8, "ms": 0.5, "timings": {}}
    real = autotune.kernel_hash()
    monkeypatch.setattr(autotune, "kernel_hash", lambda: "other sources")
    autotune._store(path, autotune.entry_of([FakeSim()], False), rec)
    autotune._store(path, "shape", rec)  # a name without kernel and candidates
    s = FakeSim()
    assert autotune._tune([s], autotune.ZCHUNKS, 10, True, path, batched=False)["cached"]
    assert s.launch == ("tiled", 12, 8)
    monkeypatch.setattr(autotune, "kernel_hash", lambda: real)
    r = autotune._tune([s], autotune.ZCHUNKS, 10, True, path, batched=False)
    assert not r["cached"] and s.launch == ("tiled", 0, 0)
    assert autotune._tune([s], autotune.ZCHUNKS, 10, True, path, batched=False)["cached"]


@pytest.mark.parametrize("change", ["k_pair.cu", "lbm_internal.cuh"])
def test_the_hash_follows_the_sources(tmp_path, monkeypatch, change):
    for name in ("k_pair.cu", "lbm_internal.cuh"):
        (tmp_path / name).write_text("a")
    monkeypatch.setattr(autotune, "CSRC", str(tmp_path))
    autotune.kernel_hash.cache_clear()
    before = autotune.kernel_hash()
    (tmp_path / change).write_text("b")
    autotune.kernel_hash.cache_clear()
    assert autotune.kernel_hash() != before
    monkeypatch.undo()
    autotune.kernel_hash.cache_clear()
