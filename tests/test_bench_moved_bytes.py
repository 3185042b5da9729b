"""The bench line's byte counts of what the sort's launches move: no stage claims
more than its time allows at the copy bandwidth it is compared with."""
import bench


def test_moved_bytes_beside_the_shared_basis(monkeypatch):
    monkeypatch.setattr(bench, "measured_peaks", lambda: (7000.0, "measured"))
    n = 1 << 24
    # milliseconds of 2^24 bodies at 60 % of that bandwidth, by what is moved
    moved = {"keys": 33 * n, "radix": (6 * 24 - 4) * n, "type_order": 5 * n}
    times = {k: b / (0.6 * 7000e9) * 1e3 for k, b in moved.items()}
    h = bench.hbm_block(times, n, 4, 0, passes=6)
    for k, b in moved.items():
        assert h[k]["moved_bytes"] == b
        assert h[k]["moved_frac"] == 0.6
        assert h[k].get("frac", 0.0) <= 1.0
    assert "frac" not in h["type_order"]         # its basis is seven times what it moves
    assert h["keys"]["bytes"] == 37 * n and h["radix"]["bytes"] == 6 * 32 * n
    assert "moved_bytes" not in bench.hbm_block({"gather": 1.0}, n, 4, 0)["gather"]


def test_passes_are_those_of_the_reported_radix_time():
    calls = [({"radix": 1.3, "keys": 0.2}, 8), ({"radix": 1.0, "keys": 0.3}, 6), ({"radix": 1.4, "keys": 0.1}, 8)]
    assert bench.best_stages(calls) == ({"radix": 1.0, "keys": 0.1}, 6)
