"""Host-side pieces of bench.py that need no GPU: the ncu record lookup keyed by
the kernel-source hash, the roofline helpers and the JSON shapes."""
import json

import pytest

import bench


def _records():
    with open(bench.NCU_RECORDS) as f:
        return json.load(f)["records"]


def test_ncu_records_are_well_formed():
    recs = _records()
    assert recs
    for tag, r in recs.items():
        assert len(r["source_hash"]) == 16 and r["elements"] > 0 and r["kernel"]
        assert any(k in r for k in ("dram_bytes", "fp64_pipe_inst_per_elem", "inst_per_elem")), tag


def test_ncu_record_needs_the_current_hash(monkeypatch):
    recs = _records()
    tag, r = next(iter(recs.items()))
    field = next(k for k in ("dram_bytes", "fp64_pipe_inst_per_elem", "inst_per_elem") if k in r)
    monkeypatch.setattr(bench, "kernel_source_hash", lambda: r["source_hash"])
    assert bench.ncu_record(tag, field) == pytest.approx(float(r[field]))
    monkeypatch.setattr(bench, "kernel_source_hash", lambda: "0000000000000000")
    assert bench.ncu_record(tag, field) is None
    assert bench.ncu_record("no such kernel", field) is None


def test_traffic_records_close_to_the_algorithmic_bytes():
    """Every DRAM-bytes record of a full-size capture is within a few percent of
    the algorithmic bytes of its launch (no re-reads)."""
    alg = {"tet_generic_mixed_aos": 256, "prism_generic_mixed_aos": 792, "tet_generic_fp64_aos": 416}
    for tag, r in _records().items():
        if "dram_bytes" in r and tag in alg and r.get("full_size", True):
            assert 0.9 * alg[tag] * r["elements"] <= r["dram_bytes"] <= 1.02 * alg[tag] * r["elements"], tag


def test_rooflines_of_the_alu_bound_forms():
    f = bench.pipe_roofline(7000.0, 77.0, 152, 2070.0, bench.FP64_PIPE_PER_CLK_SM, "FP64-pipe", "t")
    assert f["peak"] == pytest.approx(2 * 152 * 2.07e9 / 1e12)
    assert f["achieved"] == pytest.approx(7000e6 * 77 / 1e12)
    assert 0 < f["frac"] < 1 and f["bound"] == "alu"
    i = bench.pipe_roofline(19000.0, 1436.0, 152, 2070.0, bench.ISSUE_PER_CLK_SM, "thread", "t")
    assert i["peak"] == pytest.approx(4 * 32 * 152 * 2.07e9 / 1e12)
    assert i["frac"] == pytest.approx(19000e6 * 1436 / 1e12 / i["peak"])
    n = bench.pipe_roofline(19000.0, None, 152, 1900.0, bench.ISSUE_PER_CLK_SM, "thread", "t")
    assert n["frac"] is None and n["achieved"] is None and n["peak"] == pytest.approx(4 * 32 * 152 * 1.9e9 / 1e12)
    h = bench.hbm_roofline(6_000_000, 416, 1.0, 6781.1, "measured")
    assert h["achieved"] == pytest.approx(6e6 * 416 / 1e-3 / 1e9) and h["bound"] == "hbm"


def test_shape_and_context_records_are_json():
    assert bench.shape_dict((64, 0)) == {"elements_per_block": 64, "persistent": 0, "threads_per_element": 1}
    assert bench.shape_dict((32, 1, 2))["threads_per_element"] == 2
    ctx = bench.paper_context()
    json.dumps(ctx)
    assert ctx["melem_s"]["Tesla K20m"]["laplace_tet"] == pytest.approx(1000 / 2.02, abs=0.1)


def test_source_hash_ignores_comments_only():
    src = "template <int K> // bound\n__global__ void k(float *p) {\n    /* body */ p[0] = K; }\n"
    edited = src.replace("// bound", "// another note").replace("/* body */", "/* the\nbody */")
    assert bench.code_only(src) == bench.code_only(edited)
    assert bench.code_only(src) != bench.code_only(src.replace("p[0] = K", "p[0] = 2 * K"))


def test_printed_line_is_short_and_keeps_the_contract():
    """A full record of tens of kilobytes prints as one short line with every key that a
    reader of the benchmark needs, parsed from the last line of the output."""
    long = {"value": 12345.678901234567, "unit": "Melem/s", "roofline": {"note": "n" * 2000}, "workload": "w" * 500}
    clk = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 200, "samples_in_region": 190,
           "power_w_max": 1034.55}
    result = {"metric": bench.METRIC, "value": 11196.123456789012, "unit": "Melem/s", "n_gpus": 1, "steps": 8000,
              "warmup": 20, "ms_per_step": 0.5358832001686096, "higher_is_better": True, "scaling": "weak",
              "vs_baseline": None, "dtype": "f64", "data": "synthetic",
              "config": {"workload": bench.WORKLOAD, "n_elem_per_gpu": 6000000, "bytes_per_element": 416,
                         "launch_shape": bench.shape_dict((512, 1)),
                         "l2": "inputs larger than L2: 2.50 GB read+written per step per GPU",
                         "parallelism": "weak: 1 independent mesh(es), one per GPU"},
              "roofline": {"bound": "alu", "kernel": "k" * 70, "frac": 0.5, "note": "n" * 500,
                           "hbm": {"achieved": 4657.731384776873, "peak": 6677.2, "frac": 0.6975575667610485}},
              "gpu_launches": 8000, "clocks": clk,
              "e2e": {"value": 743.009764138675, "unit": "Melem/s", "h2d_bytes_per_step": 1536000000,
                      "d2h_bytes_per_step": 966000000, "ms_per_step": 8.07, "steps": 3, "dtype": "f64", "path": "p" * 300},
              "cpu_baseline": dict(long, cores=16, kind="oracle"),
              "serving": {"served": {"p50_ms": 0.2, "p99_ms": 0.5, "sustained_melem_s": 900.123}, "plain_fp64": long},
              "paper_context": {"melem_s": {"x" * 20: 1.0}}}
    for name in ("mixed_form", "double_word_form", "fp64_forms", "cfg1_stated", "threads_per_element", "prism_form",
                 "coef_function_form", "packed_form", "ordering_study", "indexed_form", "apply_form", "batched"):
        result[name] = dict(long)
    text = json.dumps(bench.summary_line(result, "/somewhere/bench_record.json"))
    assert len(json.dumps(result)) > 20000 and len(text) <= bench.LINE_LIMIT and "\n" not in text
    line = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "gpu_launches"):
        assert line[k] == result[k]
    assert line["clocks"] == clk and line["e2e"]["value"] == result["e2e"]["value"]
    assert line["e2e"]["h2d_bytes_per_step"] == 1536000000 and line["e2e"]["d2h_bytes_per_step"] == 966000000
    assert line["other_melem_s_and_ms"]["mixed_form"] == 12345.7
    assert bench.summary_line({k: result[k] for k in ("metric", "value", "unit")})["value"] == result["value"]
