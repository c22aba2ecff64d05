"""The benchmark's printed line stays short enough to be kept whole by what
collects it, and keeps every required key with its value."""
import json

import bench

REQUIRED = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks")


def record():
    text = "x" * 200
    out = {k: 1.2345678901234567 for k in bench.LINE_KEYS}
    out.update(metric=bench.METRIC, unit=bench.UNIT, vs_baseline=None, dtype=text, data=text,
               config={k: text for k in ("workload", "nsys_per_gpu", "method", "form", "l2", "parallelism")},
               e2e={"value": 8.0e6, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1},
               clocks={"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["none"]},
               cpu_baseline={"value": 5.0e4, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": text})
    out["roofline"] = {k: text[:40] for k in bench.LINE_ROOFLINE} | {"flops_model": text * 3, "traffic_source": text * 3}
    out["forms"] = {n: {"value": 1.0e6, "err_vs_fp64_oracle_p999": 1e-8, "form": text * 2} for n in bench.FORMS}
    out["target"] = {"bar": text, "chosen_meets": True}
    for leg in ("c0_vdp_rkck", "c1_bruss_rkc", "learned_proposal", "mixed_batch", "kinetics_ignition", "global_steps"):
        out[leg] = {f"k{i}": {"systems_per_s": 1.0, "note": text} for i in range(20)}
    out["c1_bruss_rkc"]["f2_lean"] = {"systems_per_s": 2.0e6}
    out["pleiades_rkck"] = {"systems_per_s": 3.0e5}
    return out


def test_line_is_short_and_whole():
    out = record()
    line = bench.short_line(out)
    assert "\n" not in line and len(line) < 6000
    d = json.loads(line)
    for k in REQUIRED:
        assert d[k] == out[k], k
    assert d["legs"] == {"c1_bruss_rkc.f2_lean": 2.0e6, "pleiades_rkck.systems_per_s": 3.0e5}
    assert d["forms"]["f2_lean"] == {"value": 1.0e6, "p999_err": 1e-8}
    assert set(d["roofline"]) == set(bench.LINE_ROOFLINE)


def test_line_of_a_record_without_legs():
    d = json.loads(bench.short_line({"metric": "m", "value": 1.0}))
    assert d == {"metric": "m", "value": 1.0}
