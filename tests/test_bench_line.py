"""The result line of bench.py stays short enough to be read whole: the sweep's single runs go to stderr."""
import json


def test_result_line_leaves_out_single_runs():
    import bench
    runs = [{"enc": "int8", "beta": 0.4 + 1e-3 * k, "note": "x" * 480} for k in range(72)]
    out = {"metric": "m", "value": 1.0, "e2e": {"value": 2.0}, "clocks": {"sm_mhz": 1}, "gpu_launches": 3,
           "config2": {"checks": 64, "failures": 0, "runs": runs}}
    assert len(json.dumps(out)) > 36000
    line, rest = bench.result_line(out)
    assert rest is runs
    assert line["config2"] == {"checks": 64, "failures": 0}
    assert {k: line[k] for k in out if k != "config2"} == {k: out[k] for k in out if k != "config2"}
    assert len(json.dumps(line)) < 1000
    for short in ({"metric": "m", "config2": None}, {"impl": "reference", "value": 1.0}):
        assert bench.result_line(short) == (short, None)
