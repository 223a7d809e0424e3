"""The bench quotes the captured DRAM traffic of the S apply only for the source that it was captured with."""
import os
import shutil



def test_traffic_goes_with_every_source_of_the_kernels(tmp_path, monkeypatch):
    import bench
    csrc = os.path.join(bench.ROOT, "paper_1809_00828_gb300", "csrc")
    kernels = [f for f in os.listdir(csrc) if f in ("fcm_schwarz.cu", "fcm_sym.cuh", "fcm_tma.cuh", "fcm_ff.cuh")]
    assert len(kernels) == 4
    real = bench._traffic_source_hash
    for f in kernels:
        shutil.copy(os.path.join(csrc, f), tmp_path)
    profile = tmp_path / "p.md"
    profile.write_text(f"traffic_bytes_per_s_apply: 123\nkernel_source_sha256: {real(str(tmp_path))}\n")
    monkeypatch.setattr(bench, "TRAFFIC_PROFILE", str(profile))
    monkeypatch.setattr(bench, "_traffic_source_hash", lambda: real(str(tmp_path)))
    assert bench._schwarz_traffic(bench.DEFAULT_WORKLOAD, "mixed") == 123.0
    for f in kernels:
        old = (tmp_path / f).read_bytes()
        (tmp_path / f).write_bytes(old + b"\n")
        assert bench._schwarz_traffic(bench.DEFAULT_WORKLOAD, "mixed") is None, f
        (tmp_path / f).write_bytes(old)
    assert bench._schwarz_traffic(bench.DEFAULT_WORKLOAD, "fp64") is None
