"""The line bench.py prints: the contract's fields whole, the side measures' figures
without the texts that go to the log, and short enough to be kept with its output."""
import json

import bench


def _roofline(v):
    return {"bound": "hbm", "achieved": v, "peak": 6779.0, "unit": "GB/s", "frac": v / 6779.0, "traffic": None,
            "bytes_per_launch": 17966877432, "kernel": "sweep_kernel<ByteState>", "peak_kind": "measured hbm_gbs (burst copy)",
            "step_bytes_alg": 18637966072, "step_frac": v / 6779.0}


def test_side_measures_are_cut_and_the_headline_is_not():
    v = 1234.56789012345
    layouts = {k: {"ms_per_step": v, "value": v, "unit": "GEdges/s", "roofline": _roofline(v), "how": "a" * 300}
               for k in ("u8", "u2", "u32")}
    line = {"metric": "m", "value": v, "config": {"workload": "w", "l2": "no flush"}, "roofline": _roofline(v),
            "layouts": layouts, "side_graphs": {"uniform27": {"n": 1 << 27, "layouts": layouts, "stats": [v, 1]}},
            "batched": None, "e2e": {"value": v, "how": "kept", "h2d_bytes_per_step": 3}}
    out = json.loads(json.dumps(bench.compact(line)))
    assert set(out) == set(line) and out["batched"] is None
    assert out["value"] == 1234.5679 and out["config"] == line["config"] and out["e2e"]["how"] == "kept"
    assert set(out["roofline"]) == set(line["roofline"])
    side = out["side_graphs"]["uniform27"]
    assert side["n"] == 1 << 27 and side["stats"] == [1234.57, 1]
    for lay in (*out["layouts"].values(), *side["layouts"].values()):
        assert lay == {"ms_per_step": 1234.57, "value": 1234.57, "unit": "GEdges/s",
                       "roofline": {"achieved": 1234.57, "frac": round(v / 6779.0, 6), "traffic": None}}
    assert len(json.dumps(bench.compact(line))) < 0.5 * len(json.dumps(line))
