"""bench.py's printed line stays short enough for whoever reads the end of its
output: the contract's keys unchanged, the rest of the record as far as it fits."""
import json

import bench


def record():
    served = [{"request": i, "nnz": 123456789, "fmt": "fp16", "solution_dose_max_frac_of_presc": 1.23456789e-6 * i,
               "outputs_letd_max_keV_um": 0.00123456789} for i in range(40)]
    r = {"metric": bench.METRIC, "value": 335.5108440700221, "unit": "iters/s", "n_gpus": 1, "steps": 20, "warmup": 5,
         "ms_per_step": 2.9805295944213865, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
         "dtype": "f32", "data": "synthetic", "config": bench.workload_config(6000000, 30000, 555627200, "fp32", 1),
         "timing_s": {"generate": 4.13, "load": 0.066},
         "roofline": {"bound": "hbm", "achieved": 6907.971097075139, "peak": 6784.8, "unit": "GB/s",
                      "frac": 1.0181539761046956, "traffic": 5650728624.0, "bytes_model": bench.BYTES_MODEL,
                      "forward": {"achieved": 6907.97, "deep": {"x": 1}}},
         "e2e": {"value": 300.1, "unit": "iters/s", "h2d_bytes_per_step": 1.0e7, "d2h_bytes_per_step": 9.6e4,
                 "what": "w" * 150},
         "gpu_launches": 160, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 1},
         "serving": {"served": {"plans_per_hour": 15063.83324443719}, "accuracy": {"accuracy_ok": True, "requests": served}}}
    for i in range(60):
        r[f"entry{i}"] = {f"number{j}": 1.0 / (1 + i + j) for j in range(20)}
    return r


def test_line_is_short_and_holds_the_contract():
    r = record()
    assert len(json.dumps(r)) > 20000
    text = bench.headline(r)
    assert len(text) <= bench.LINE_CHARS and "\n" not in text
    line = json.loads(text)
    for k in bench.LINE_KEYS:
        assert line[k] == r[k], k
    assert line["roofline"]["frac"] == 1.0182 and "bytes_model" not in line["roofline"]
    assert line["serving"]["served"]["plans_per_hour"] == 15064.0
    assert line["serving"]["accuracy"] == {"accuracy_ok": True}
    # a record that fits is there as a whole, shortened
    small = {k: r[k] for k in (*bench.LINE_KEYS, "timing_s")}
    assert json.loads(bench.headline(small)) == small


def test_record_file(tmp_path, capsys):
    r = record()
    path = str(tmp_path / "deep" / "record.json")
    bench.write_record(r, path)
    assert json.load(open(path)) == json.loads(json.dumps(r))
    bench.write_record(r, str(tmp_path / "deep" / "record.json" / "below_a_file.json"))  # reported, not raised
    assert "not written" in capsys.readouterr().err
