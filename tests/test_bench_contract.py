"""The bench's reference arm (the oracle timed on the host cores) prints the one
JSON line of the bench contract, with every key the contract names.  CPU only:
the reference arm never touches a GPU."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reference_arm_prints_the_contract_line():
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1",
                        "--warmup", "0", "--cpu-sample", "150000"],
                       cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [l for l in r.stdout.splitlines() if l.startswith("{")]
    assert len(lines) == 1
    d = json.loads(lines[0])
    for k in ("impl", "metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
              "scaling", "vs_baseline", "dtype", "data", "config", "cpu_baseline", "e2e"):
        assert k in d, k
    assert d["impl"] == "reference" and d["n_gpus"] == 1 and d["steps"] == 1 and d["value"] > 0
    assert d["higher_is_better"] is True and d["config"]["workload"].startswith("scaled:")
    cb = d["cpu_baseline"]
    assert cb["kind"] == "oracle" and cb["cores"] >= 1 and cb["value"] == d["value"] and cb["sample"]
    assert cb["host"]["nproc"] >= 1 and cb["host"]["cpu_model"]
    e = d["e2e"]
    assert (e["value"], e["unit"], e["h2d_bytes_per_step"], e["d2h_bytes_per_step"]) == (d["value"], d["unit"], 0, 0)


def _bench_module():
    import importlib.util
    spec = importlib.util.spec_from_file_location("bench_under_test", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_traffic_captures_match_the_kernel_code():
    """The committed DRAM-traffic captures name the kernel sources they were taken on by a
    digest of the code: comment edits keep it, any code edit changes it (and the bench then
    reports no traffic rather than a stale one)."""
    import tempfile
    bench = _bench_module()
    for name in ("expand_kernel_scaled_traffic.json", "expand_kernel_mid_traffic.json"):
        with open(os.path.join(ROOT, "profiles", name)) as f:
            t = json.load(f)
        assert bench.kernel_code_digest(t["kernel_sources"]) == t["kernel_code_sha256"], name
    with tempfile.TemporaryDirectory(dir=ROOT) as d:
        rel = os.path.relpath(os.path.join(d, "k.cuh"), ROOT)
        path = os.path.join(ROOT, rel)
        with open(path, "w") as f:
            f.write("int a = 1;  // one\n\n// a note\nint b = 2;\n")
        base = bench.kernel_code_digest([rel])
        with open(path, "w") as f:
            f.write("int a = 1;  // another note\n// more\nint b = 2;\n\n")
        assert bench.kernel_code_digest([rel]) == base
        with open(path, "w") as f:
            f.write("int a = 1;\nint b = 3;\n")
        assert bench.kernel_code_digest([rel]) != base


def test_guided_part_adds_a_summary_not_every_run():
    """The bench prints one line, which must stay short enough to be read back: 200 guided
    searches, 20 breadth-first ones and their networks add no more than their medians (on
    stand-ins for the GPU library and torch)."""
    from types import SimpleNamespace as NS

    import numpy as np
    bench = _bench_module()
    runs = []

    class Array(list):
        def cpu(self):
            return self

        def numpy(self):
            return np.array(self)

    def stats(_):
        return {"explored": 164441 + len(runs), "states": 2730458, "gpu_ms": 1.921, "expand_launches": 33,
                "first_deadlock_level": 32, "fill": 0.7561, "n_levels": 19}

    gx = NS(load_network=lambda n: n, guided_set_weights=lambda h, p: None, default_opts=lambda **k: k,
            guided_alloc_workspace=lambda h, o: None, alloc_workspace=lambda h, o: None, GX_DL_GUIDED=2, GX_DL_BFS_FIRST=0,
            find_deadlocks=lambda *a: runs.append(a) or (1, None), stats=stats, guided_trace=lambda h: [0] * 33,
            GxError=RuntimeError, MLP_PARAMS=1, mlp_init=lambda p, s: None, mlp_forward=lambda p, h: None)
    event = NS(record=lambda s: None, elapsed_time=lambda o: 2.0)
    torch = NS(cuda=NS(synchronize=lambda: None, empty_cache=lambda: None, current_stream=lambda: None,
                       Event=lambda enable_timing: event),
               empty=lambda *a, **k: None, randint=lambda *a, **k: None, float32=0, uint8=0)
    guide = NS(collect_examples=lambda nets, d: (np.zeros((5, 16)), None), train=lambda h, l, steps, lr: (None, Array([0.1] * 99)))
    inputs = NS(planted_network=lambda seed, n, n_traps=1: NS(name=f"planted_s{seed}_n{n}_k{n_traps}"))
    part = bench.guided_part(torch, gx, inputs, guide)
    assert len(runs) == 4 * 5 * (5 + 5 + 1 + 1)
    assert [s["guided_found"] for s in part["summary"]] == [25] * 4 and part["summary"][0]["bfs_median_ms"] == 1.921
    assert len(json.dumps(part)) < 4096
