"""The autotuner times only what a size can tell apart (CPU): the V-cycles' settings do
nothing on sides that are solved directly."""
import workloads as W
from paper_2012_00881_gb300 import autotune as AT


def test_direct_sides_are_timed_once(monkeypatch):
    seen = []

    def timed(group, cand, n_slices, precision, cache):
        seen.append((group[0].n, dict(cand)))
        return 1.0 + len(seen) / 1e3

    monkeypatch.setattr(AT, "time_candidate", timed)
    wls = [W.Workload(name=str(n), n=n, half_width=3.0, n_xi=4, xi_len=1.0, ppc=1, beams=())
           for n in (7, 128, 4096)]
    tuned = AT.tune(wls, precision="fp32r")
    full = len(AT.candidates())
    assert [n for n, _ in seen].count(128) == 1 and [c for n, c in seen if n == 128] == [{}]
    assert [n for n, _ in seen].count(7) == full and [n for n, _ in seen].count(4096) == full
    assert AT.apply(wls[1], tuned) == {} and AT.apply(wls[2], tuned)["tile_x"] > 0


def test_other_settings_stay_apart():
    c = [dict(tile_x=32, tile_y=16, deposit_band_rows=r) for r in (0, -1)] + \
        [dict(tile_x=64, tile_y=32, deposit_band_rows=0), dict(tile_x=32, tile_y=16, cluster_size=8)]
    assert AT.distinct(c, 128, "fp32r") == [dict(deposit_band_rows=0), dict(deposit_band_rows=-1),
                                            dict(tile_x=32, tile_y=16, cluster_size=8)]
    assert AT.distinct(c, 2048, "fp64") == c
