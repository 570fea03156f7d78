"""What the tuner and the geometry query say of FP64 passes, and cache lines of other versions."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1805_05821_gb300 import build
    build.build()


def test_reported_ctas_are_those_launched():
    """Two CTAs per SM up to j = 128 in the FP64 passes with column dots and at any j in pass C (as far as two
    stages fit half an SM's shared memory), one in the two-pass push; FP32 two until they do not fit."""
    from paper_1805_05821_gb300.foa_dmd import FoaDMD
    g = FoaDMD(100000, 300, "f64")
    assert g.tuned_geometry(0, 100)["ctas_per_sm"] == 2 and g.tuned_geometry(0, 200)["ctas_per_sm"] == 1
    assert g.tuned_geometry(2, 150)["ctas_per_sm"] == 2 and g.tuned_geometry(2, 290)["ctas_per_sm"] == 1
    assert g.tuned_geometry(3, 50)["ctas_per_sm"] == 1
    assert g.tuned_geometry(0, 100)["stage_bytes"] == 49152
    g.close()
    g = FoaDMD(100000, 500, "f32")
    assert g.tuned_geometry(1, 100)["ctas_per_sm"] == 2 and g.tuned_geometry(1, 499)["ctas_per_sm"] == 1
    g.close()


def test_stages_that_launch_alike_keep_the_default(tmp_path):
    """4096 values: every stage is cut to 8 KB, so all stage sizes are one launch and the tuner leaves the
    default's 48 KB.  A line of the format without a version is not used."""
    import torch
    from paper_1805_05821_gb300.foa_dmd import FoaDMD
    cache = tmp_path / "tune.txt"
    p = torch.cuda.get_device_properties(0)
    old = "".join(f"foa_dmd_tune {p.major * 10 + p.minor} 0 12 {k} {b} 16384 65536 1 0 0.001\n" for k in range(3) for b in range(5))
    cache.write_text(old)
    g = FoaDMD(4096, 100, "f64")
    g.autotune(cache)
    for k in range(3):
        for j in (4, 12, 24, 48, 96):
            t = g.tuned_geometry(k, j)
            assert t["tuned"] and t["stage_bytes"] == 49152, (k, j, t)
    assert len(cache.read_text().splitlines()) == 15 + 15
    h = FoaDMD(4096, 100, "f64")
    h.autotune(cache)
    for k in range(3):
        for j in (4, 48, 96):
            assert h.tuned_geometry(k, j) == g.tuned_geometry(k, j)
    g.close()
    h.close()
