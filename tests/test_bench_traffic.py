"""The benchmark's stored DRAM traffic is tied to every file that makes up the kernel."""
import hashlib
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_traffic_of_a_kernel_in_several_files(tmp_path, monkeypatch):
    sys.path.insert(0, ROOT)
    import bench
    (tmp_path / "profiles").mkdir()
    (tmp_path / "a.cu").write_text("kernel")
    (tmp_path / "b.cuh").write_text("loads")
    sha = hashlib.sha256(b"kernelloads").hexdigest()[:16]
    (tmp_path / "profiles" / "traffic.txt").write_text(f"k w a.cu,b.cuh {sha} 123\n")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.stored_traffic("k", "w") == 123.0
    (tmp_path / "b.cuh").write_text("other loads")
    assert bench.stored_traffic("k", "w") is None
    (tmp_path / "b.cuh").unlink()
    assert bench.stored_traffic("k", "w") is None


def test_the_star_kernels_record_names_its_files():
    line = [v.split() for v in open(os.path.join(ROOT, "profiles", "traffic.txt")) if v.startswith("k_patch_apply_f32_fine")]
    names = {os.path.basename(f) for f in line[0][2].split(",")}
    assert names >= {"patches.cu", "star_blocks.cuh", "tma.cuh", "common.cuh"}
    assert all(os.path.exists(os.path.join(ROOT, f)) for f in line[0][2].split(","))
