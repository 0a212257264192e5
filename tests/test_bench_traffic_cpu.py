"""The DRAM traffic the benchmark's JSON line reports: the captured bytes a chain
times the chains of a launch (dominant pass) or of a step (all three passes), and
no figure where nothing was captured (CPU; no GPU needed)."""

import pytest

from tests.test_bench_cpu import _bench_module, _Plan, _res

PEAKS = {"hbm_gbs": 6688.8}
LOOP = {"ms": 1000.0, "phase_ms": {"to_real": 10.0, "to_sphere": 20.0, "energy": 0.0, "pair_fwd": 500.0,
                                   "pair_col": 600.0, "pair_inv": 700.0},
        "clocks": {"sm_mhz": 2070.0}, "stats": {"chains": 1000, "phase_launches": {}}}


@pytest.mark.parametrize("form", ["fp64", "df64", "mixed32"])
def test_reported_traffic_is_the_captures(form):
    b = _bench_module()
    assert {k[2] for k in b.DRAM_PER_CHAIN if k[0] == form} >= {8, 16}
    for (f, n, block), per in b.DRAM_PER_CHAIN.items():
        if f != form:
            continue
        assert n == 96 and set(per) == {"pair_fwd", "pair_col", "pair_inv"}
        one = b.reported(b.roofline(form, _Plan(), _res(10.0), 1, PEAKS, "measured", block), form, n, block)
        assert one["kernel"] == "pair_inv" and one["traffic"] == per["pair_inv"] * 38 and one["traffic_src"]
        loop = b.reported(b.roofline(form, _Plan(), LOOP, 1, PEAKS, "measured", block, streams=2), form, n, block)
        assert loop["traffic"] == sum(per.values()) * 1000
    none = b.reported(b.roofline(form, _Plan(), _res(10.0), 1, PEAKS, "measured", 4), form, 96, 4)
    assert none["traffic"] is None and none["traffic_src"] is None


def test_the_captures_lie_above_the_kept_columns():
    # each pass moves at least the columns it must read and write (mixed 4.34 MB, FP64
    # and double-float 8.68 MB a chain), some of which stays in L2 between passes
    b = _bench_module()
    for (form, _, _), per in b.DRAM_PER_CHAIN.items():
        columns = 4.34e6 if form == "mixed32" else 8.68e6
        assert per["pair_fwd"] > columns and 1.8 * columns < per["pair_col"] < 2.1 * columns
        assert per["pair_inv"] > columns
