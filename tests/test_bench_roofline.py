"""The benchmark's roofline of the inner iteration: its share of the memory's
bandwidth is that of a full iteration; the mean over a solve, whose incremental
iterations move a fraction of the bytes, is a rate only. The recorded traffic
depends on every file whose kernels a loop body holds."""
import os
import shutil
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_share_of_a_full_iteration():
    r = bench.iteration_roofline(m=30, np_=10, mp=35, full_s=2e-6, mean_s=1e-6, hbm=4.0)
    assert r["algorithmic_bytes_per_launch"] == 8 * 35 + 20 * 10
    assert abs(r["achieved"] - 0.24) < 1e-12 and abs(r["frac"] - 0.06) < 1e-12 and abs(r["avg_launch_us"] - 2) < 1e-9
    mean = r["mean_iteration"]
    assert abs(mean["us"] - 1) < 1e-9 and abs(mean["edges_per_s"] - 30e6) < 1
    assert not any("frac" in key for key in mean)
    r = bench.iteration_roofline(m=30, np_=10, mp=35, full_s=None, mean_s=1e-6, hbm=4.0)
    assert r["achieved"] is None and r["frac"] is None


def test_traffic_of_an_iteration_goes_stale_with_each_of_its_files(tmp_path, monkeypatch):
    csrc = os.path.join("paper_1705_02313_gb300", "csrc")
    shutil.copytree(os.path.join(ROOT, csrc), tmp_path / csrc)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = bench.kernel_source_hash("iteration")
    for name in ("pg_iter.cu", "pg_device.cuh", "pg_scan.cu", "pg_inc.cu"):
        path = tmp_path / csrc / name
        text = path.read_text()
        path.write_text(text + "\n// an edit\n")
        assert bench.kernel_source_hash("iteration") != before, name
        path.write_text(text)
    assert bench.kernel_source_hash("iteration") == before
