"""The benchmark's line stays short enough to be read from the end of an output, however many variants it measures."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_variants_keep_their_values_only():
    measured = {"value": 830.89, "steps": 200, "ms_per_step": 2.58232, "launch": [1056, 8320],
                "roofline": {"kernel": "k", "peak_source": 300 * "x"}, "flux": {"launch_ms": 0.06958}}
    names = [f"{w}:{bench.variant_name(sc, dg, pr)}" for w in bench.WORKLOADS for sc in (0, 1) for dg in (2, 3) for pr in (0, 1)]
    result = {"metric": bench.METRIC, "value": 1046.6, "e2e": {"value": 900.0}, "clocks": {"sm_mhz": 2070.0},
              "variants": {n: dict(measured) for n in names}}
    line = bench.headline(result)
    assert line["variants"] == {w: {f"{x}_r{dg}": [830.89, 830.89] for x, dg in
                                    (("CTENO3", 2), ("CTENO4", 3), ("CTENOZ3", 2), ("CTENOZ4", 3))} for w in bench.WORKLOADS}
    assert {k: v for k, v in line.items() if k != "variants"} == {k: v for k, v in result.items() if k != "variants"}
    del result["variants"][names[0]]
    assert bench.headline(result)["variants"][names[0].split(":")[0]]["CTENO3_r2"] in ([None, 830.89], [830.89, None])
    assert len(json.dumps(line["variants"])) < 35 * len(names)
