"""The benchmark's fraction of the operations a launch needs is given only for
the kernel sources on which the shares of drawn and propagated bunches were
counted; that of propagating every bunch always is."""
import bench


def test_shares_only_for_the_counted_sources(monkeypatch):
    monkeypatch.setattr(bench, "BUNCH_SHARES", {"vertical_1tev": (0.4, 0.025, "ab" * 8)})
    rl = bench.alu_roofline(6.4e7, 2e6, 0.3, 152, 2070.0)
    monkeypatch.setattr(bench, "_kernel_hash", lambda: "ab" * 8)
    got = bench.needed(rl, "vertical_1tev", 6.4e7, 2e6, 0.3)
    ops = 179 * 2e6 + (66 * 0.4 + 215 * 0.025) * 6.4e7
    assert abs(got["frac"] - ops / 0.3e-3 / 1e12 / rl["peak"]) < 1e-12
    assert got["all_bunches_frac"] == rl["frac"]
    monkeypatch.setattr(bench, "_kernel_hash", lambda: "0" * 16)        # sources changed
    got = bench.needed(rl, "vertical_1tev", 6.4e7, 2e6, 0.3)
    assert got["frac"] is None and got["achieved"] is None
    assert got["all_bunches_frac"] == rl["frac"] and got["peak"] == rl["peak"]
    assert bench.needed(rl, "no such workload", 6.4e7, 2e6, 0.3) == rl
