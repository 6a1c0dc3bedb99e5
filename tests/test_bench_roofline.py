"""The bench's roofline figures: every workload counts bytes per launch, however
many steps it takes, and the headline's traffic comes from the summary of the
same steps per launch."""
import bench


def _fields(path):
    out = {}
    for line in open(path):
        if line.strip().startswith("- ") and ":" in line:
            k, v = line.strip()[2:].split(":", 1)
            out[k.strip()] = v.strip().strip("`")
    return out


def test_extras_count_bytes_per_launch():
    peak, _ = bench.measured_peak()
    one = bench._entry(1e9, 10, 1.0, 8, dict(tsteps=1))
    two = bench._entry(1e9, 10, 1.0, 8, dict(tsteps=2))
    assert one["glups"] == two["glups"] == 10.0
    assert abs(one["roofline_frac"] - 80.0 / peak) < 1e-12
    assert two["roofline_frac"] == one["roofline_frac"] / 2
    assert bench._entry(1e9, 10, 1.0, 8)["roofline_frac"] == one["roofline_frac"]


def test_traffic_of_both_step_counts(monkeypatch):
    for T in (1, 2):
        f = _fields(bench.PROFILE_FILES[T])
        assert int(f["tsteps"]) == T
        monkeypatch.setattr(bench, "kernel_sha", lambda: f["kernel_sha"])
        traffic, tun = bench.profiled_traffic(T, int(f["tile_q"]), int(f["tile_y"]))
        assert traffic == float(f["dram_bytes_per_launch"]) and tun["tsteps"] == T
        assert bench.profiled_traffic(T, int(f["tile_q"]), int(f["tile_y"]) + 2) == (None, None)
    assert bench.profiled_traffic(3, 16, 4) == (None, None)
