"""The benchmark names the kernel that its timed decode runs, and reports
recorded DRAM traffic only of the launch it was captured from."""
import bench


def test_kernel_of_the_resolved_plan():
    assert bench.deferred_kernel({"mode": 0, "flags": 0}).startswith("k_wave_copy")
    assert bench.deferred_kernel({"mode": 1, "flags": 1}).startswith("k_levels_persistent")
    # --mode persistent with short matches copies through registers
    assert bench.deferred_kernel({"mode": 1, "flags": 2}).startswith("k_ranges")


def test_mode_with_the_event():
    auto, waves, persistent = bench.MODE["auto"], bench.MODE["waves"], bench.MODE["persistent"]
    assert bench.timed_mode(auto, 128.0) == waves and bench.timed_mode(auto, 1024.0) == persistent
    assert bench.timed_mode(waves, 1024.0) == waves and bench.timed_mode(persistent, 32.0) == persistent


def test_traffic_of_the_captured_launch_only(tmp_path):
    launch = dict(G=32, block_size=32768, ctas_per_sm=2)
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / "traffic_k_levels_persistent_w.txt").write_text(
        "# comment\nkernel: k_levels_persistent<32>\nG: 32\nblock_size: 32768\nctas_per_sm: 2\n"
        f"kernel_sources_sha: {bench.kernel_sources_sha()}\ndram_bytes_read: 5\ndram_bytes_write: 7\n")

    def get(kernel="k_levels_persistent (x)", **kw):
        return bench.recorded_traffic("w", kernel, {**launch, **kw}, root=str(tmp_path))

    assert get() == 12
    assert get(G=16) is None and get(block_size=65536) is None and get(ctas_per_sm=1) is None
    assert get("k_ranges (x)") is None and get("k_lits (literals)") is None
    assert bench.recorded_traffic("other", "k_levels_persistent", launch, root=str(tmp_path)) is None
