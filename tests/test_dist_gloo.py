"""The N>1 plumbing on CPU: two gloo ranks, max-over-ranks timing, per-rank token seeds."""
import os
import subprocess
import sys
import textwrap

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = textwrap.dedent("""
    import sys, json
    sys.path.insert(0, %r)
    from paper_2511_17885_b200 import dist as D
    rank, local, world = D.init("gloo")
    D.barrier()
    thr, t = D.aggregate_throughput(100.0 * (rank + 1), 1.0 + rank)
    seeds = D.token_seed_for_rank(5, rank)
    if rank == 0:
        print(json.dumps({"thr": thr, "t": t, "world": world, "seed": seeds}))
    D.barrier()
    D.shutdown()
""" % ROOT)


def test_two_gloo_ranks_aggregate(tmp_path):
    f = tmp_path / "w.py"
    f.write_text(SCRIPT)
    r = subprocess.run([sys.executable, "-m", "torch.distributed.run", "--nnodes=1", "--nproc-per-node", "2",
                        "--master-addr", "127.0.0.1", "--master-port", "29533", str(f)],
                       capture_output=True, text=True, timeout=180)
    assert r.returncode == 0, r.stderr[-2000:]
    import json
    line = [l for l in r.stdout.splitlines() if l.startswith("{")][-1]
    d = json.loads(line)
    assert d["world"] == 2 and abs(d["t"] - 2.0) < 1e-12 and abs(d["thr"] - 150.0) < 1e-9


def test_rank_seeds_differ():
    from paper_2511_17885_b200 import dist as D
    assert len({D.token_seed_for_rank(3, r) for r in range(8)}) == 8


def test_bench_reference_arm_runs_on_cpu():
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1",
                        "--warmup", "0", "--workload", "C0"], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    import json
    d = json.loads([l for l in r.stdout.splitlines() if l.startswith("{")][-1])
    assert d["impl"] == "reference" and d["value"] > 0 and d["cpu_baseline"]["kind"] == "oracle"


def test_bench_line_is_short_whatever_the_records_hold():
    """A reader that keeps a few KB of the output must find the whole line: the default run's (ten other workloads)."""
    import json
    sys.path.insert(0, ROOT)
    import bench
    text, x = "w" * 700, 1234567.890123456
    rec = {"value": x, "unit": "tokens/s", "ms_per_step": x, "timing": [x] * 50, "dtype": "bf16",
           "config": {"workload": text, "tokens_per_step": 14336, "l2": text, "routed_pairs": 61440, "tokens_per_layer": [1] * 24,
                      "parallelism": "replicas x1 (no collective)"},
           "clocks": {"sm_mhz": 1335.0, "sm_max_mhz": 1965, "reasons": ["sw_power_cap"], "samples": 1018, "power_w": x},
           "e2e": {"value": x, "unit": "tokens/s", "h2d_bytes_per_step": 10 ** 8, "d2h_bytes_per_step": 10 ** 8,
                   "batches_in_flight": 3, "timing": [x] * 50},
           "gpu_launches": 14000, "kernels": {f"k{i}": {"us_per_launch": x} for i in range(11)},
           "roofline": {"bound": "tensor", "achieved": x, "peak": x, "unit": "TFLOP/s", "frac": 0.7, "traffic": x, "kernel": "gemm1",
                        "us_per_launch": x, "peak_source": "measured (sustained bf16)", "note": text},
           "step_roofline": {"frac": 0.5, "bound": "tensor", "t_bound_us": x, "algorithmic_bytes": x},
           "cpu_baseline": {"value": x, "unit": "tokens/s", "cores": 16, "kind": "oracle", "sample": text}}
    line = dict(rec, metric=bench.METRIC, n_gpus=1, steps=20, warmup=5, higher_is_better=True, scaling="weak", vs_baseline=None,
                data="synthetic", configs={w: dict(rec) for w in bench.WORKLOADS if w not in ("all", bench.HEADLINE)})
    out = bench.short_line(line)
    assert len(json.dumps(out)) < 4000 and json.loads(json.dumps(out)) == out
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
              "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "roofline", "configs", "cpu_baseline"):
        assert k in out, k
    assert abs(out["value"] / x - 1) < 1e-5 and len(out["configs"]) == len(line["configs"])
