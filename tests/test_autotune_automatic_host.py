"""The automatic launch (z chunk 0) among the tuner's candidates, on the host."""
from paper_1010_4135_gb300 import autotune


class FakeSim:
    config = dict(nx=64, ny=32, nz=16, precision="fp32", scheme="nnd", bc_lo=(1, 0, 0), bc_hi=(2, 0, 0))
    launch = None

    def set_launch(self, variant, zchunk, ztail=0):
        self.launch = (variant, zchunk, ztail)


def test_the_automatic_launch_is_measured_first():
    assert autotune.candidates()[0] == ("tiled", 0, 0)
    assert sum(1 for _, zc, _ in autotune.candidates(variants=("tiled",)) if zc == 0) == 1


def test_another_launch_has_to_beat_it_by_more_than_the_noise(tmp_path, monkeypatch):
    timings = {("tiled", 0, 0): 1.0, ("tiled", 8, 0): 0.985, ("tiled", 16, 8): 1.2}
    monkeypatch.setattr(autotune, "measure", lambda *a, **k: timings)
    s = FakeSim()
    r = autotune._tune([s], autotune.ZCHUNKS, 10, False, str(tmp_path / "a.json"), batched=False, key="K")
    assert s.launch == ("tiled", 0, 0) and (r["zchunk"], r["ztail"], r["ms"]) == (0, 0, 1.0)
    timings[("tiled", 8, 0)] = 0.9
    autotune._tune([s], autotune.ZCHUNKS, 10, False, str(tmp_path / "a.json"), batched=False, key="K")
    assert s.launch == ("tiled", 8, 0)


def test_without_it_the_fastest_is_chosen():
    assert autotune.choose({("tiled", 8, 0): 0.985, ("tiled", 16, 8): 0.99}) == ("tiled", 8, 0)
