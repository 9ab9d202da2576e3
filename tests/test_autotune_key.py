"""What a cached tuning result stands for (CPU): other render settings or other
kernels are tuned anew."""

import synth
from paper_2410_04974_gb300 import autotune


def test_other_settings_and_other_kernels_miss_the_cache(tmp_path, monkeypatch):
    cams = synth.ring_cameras(2, 64, 48)
    cache = str(tmp_path / "tune.json")
    seen = []

    def tune(**kw):
        return autotune.tune(None, 1000, 3, cams, cache=cache, measure=lambda c: seen.append(c) or 1.0,
                             device_name="fake", **kw)["cached"]

    assert not tune() and tune()
    assert not tune(store_aux=True) and tune(store_aux=True)
    assert not tune(store_aux=True, bg=(0.0, 0.0, 0.0)) and tune(bg=(0.0, 0.0, 0.0), store_aux=True)
    assert tune()
    csrc = tmp_path / "csrc"
    csrc.mkdir()
    (csrc / "raster.cu").write_text("// other kernels\n")
    monkeypatch.setattr(autotune._build, "CSRC", str(csrc))
    assert not tune() and tune()
