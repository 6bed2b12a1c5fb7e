"""The bench's line on stdout stays short and whole (CPU only): a record of the
size the default run makes, cut to under 8 KB with every key it must have; and the
K3O rule that labels its batches is the library's."""
import json

import pytest

import bench

REQUIRED = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline")


def test_short_line_keeps_the_record_and_cuts_the_sections():
    line = {k: "x" for k in REQUIRED}
    line.update(value=2308.123456789, config={"workload": "w" * 500}, headline={"eval_rel_err_vs_fp64_oracle": 6.3e-14})
    wide = {"steps_per_s": 1234.56789012, "eval_rel_err_vs_fp64_oracle": 1.23456789e-13, "status": "OK",
            "kernel": "k" * 300, "traj_rel_err_after_77_steps": 1e-13}
    line["variants"] = {"v%d" % q: dict(wide) for q in range(24)}
    line["batched"] = {"B%d" % q: dict(wide, trajectory_steps_per_s=5.0e5) for q in range(30)}
    line["fitting"] = {"f%d" % q: dict(wide, s_per_iteration=3e-3, relative_residual=[0.1] * 5) for q in range(4)}
    line["serving"] = {"steps_per_s": 2.9e6, "p99_latency_s": 2.6, "per_rom": {"r%d" % q: dict(wide) for q in range(16)}}
    text = json.dumps(bench.short_line(line))
    got = json.loads(text)
    assert len(json.dumps(line)) > 20000 and len(text) < 8192 and "\n" not in text
    assert all(k in got for k in REQUIRED) and got["value"] == line["value"] and got["config"] == line["config"]
    assert got["variants"]["v3"] == {"steps_per_s": 1234.57, "eval_rel_err_vs_fp64_oracle": 1.23457e-13, "status": "OK"}
    assert got["serving"] == {"steps_per_s": 2.9e6, "p99_latency_s": 2.6}
    assert bench.short_line(dict(line, variants=None, serving=None))["variants"] == {}


@pytest.mark.parametrize("n,rank,batch,faster", [(1024, 1024, 16, True), (1024, 512, 15, False), (1024, 512, 16, True),
                                                 (128, 128, 768, True), (128, 128, 767, False), (128, 64, 2047, False),
                                                 (128, 64, 2048, True)])
def test_k3o_label_follows_the_rule(n, rank, batch, faster):
    assert bench.k3o_faster(n, rank, batch) is faster
