"""The line bench.py prints stays readable in one piece: the autotuner's part
of it holds the forms chosen and the times taken, not the candidates that do
not exist or what the choice bits already say."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench

TIMES = ["m2l_rcr", "m2l_tensor", "m2m_l2l_rcr", "m2m_l2l_tensor", "m2l_staged", "m2m_l2l_staged", "m2l_staged_tc",
         "m2m_l2l_staged_tc", "m2l_staged_df", "m2m_l2l_staged_df", "m2l_tiles_df", "m2m_l2l_tiles_df",
         "m2l_staged_tcc", "m2m_l2l_staged_tcc"]


def test_tuning_summary_is_small_and_complete():
    def level(l):
        t = {k: (12.34567 if i % 2 else None) for i, k in enumerate(TIMES)}
        t.update({k + "_on": bool(i % 2) for i, k in enumerate(TIMES[1:])})
        return {**t, "choice": 1044 + l}

    tune = {op: {l: level(l) for l in range(2, 8)} for op in ("mixed", "inner", "fp64")}
    assert bench.tune_summary({"fp64_fixed_forms": "0,4"}) == {"fp64_fixed_forms": "0,4"}
    s = bench.tune_summary(tune)
    for op, levels in tune.items():
        for l, t in levels.items():
            assert s[op][l]["choice"] == t["choice"]
            assert {k: v for k, v in s[op][l].items() if k != "choice"} == {
                k: round(v, 3) for k, v in t.items() if k in TIMES and v is not None}
    assert len(json.dumps(s)) < 5000 < len(json.dumps(tune))


def test_folded_rotation_counts():
    """(n+1)^2 + n^2 = ((2n+1)^2 + 1) / 2: p (2p-1)(2p+1)/6 + p/2 over the degrees below p, 4 flops each."""
    for p in (1, 2, 12, 89, 159):
        assert bench.folded_rot_flops(p, p) == 4.0 * (p * (2 * p - 1) * (2 * p + 1) / 3 + p)
        assert bench.folded_rcr_flops(p, p) == bench.folded_rot_flops(p, p) + bench.coax_flops(p, p)
    assert bench.folded_rot_flops(5, 3) == 4.0 * ((1 + 5 + 13) + (1 + 5 + 13 + 25 + 41))


def test_rooflines_count_what_the_kernels_execute():
    tune = {6: {"choice": 256, "m2l_tiles_df": 2.0, "m2l_rcr": 3.0, "m2l_tensor": None}}
    form, ms, flops = bench.m2l_levels(tune, [0] * 6 + [12], [0] * 6 + [1000])[6]
    assert (form, ms, flops) == ("tiles_df", 2.0, 1000.0 * bench.folded_rcr_flops(12, 12))
