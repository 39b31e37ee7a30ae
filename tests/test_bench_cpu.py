"""CPU-only checks of bench.py: the reference arm's JSON line, and the multi-process plumbing
(rendezvous, barrier, MAX all-reduce of the timing) with two gloo ranks."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(args, env_extra=None, timeout=300):
    env = dict(os.environ)
    env.update(env_extra or {})
    return subprocess.run([sys.executable, os.path.join(ROOT, "bench.py")] + args, capture_output=True, text=True,
                          env=env, timeout=timeout, cwd=ROOT)


def test_reference_arm_prints_one_json_line():
    res = run(["--impl", "reference", "--steps", "1", "--warmup", "0"])
    assert res.returncode == 0, res.stderr
    lines = [ln for ln in res.stdout.splitlines() if ln.strip()]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference" and d["unit"] == "TOPS" and d["higher_is_better"] is True
    assert d["value"] > 0 and d["ms_per_step"] > 0 and d["vs_baseline"] is None
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["cores"] >= 1
    assert d["e2e"]["h2d_bytes_per_step"] == 0 and d["e2e"]["d2h_bytes_per_step"] == 0
    assert d["config"]["workload"].startswith("config5") and "sample" in d["config"]


WORKER = r"""
import os, sys
sys.path.insert(0, {root!r})
import bench
rank, world, local = bench.dist_setup(2)
assert world == 2 and rank == int(os.environ["RANK"])
bench.barrier()
m = bench.max_over_ranks(10.0 + rank)          # rank 1 is the slow one
assert m == 11.0, m
bench.barrier()
print("rank", rank, "ok", m)
"""


def test_two_gloo_ranks_agree_on_the_max_time(tmp_path):
    script = tmp_path / "worker.py"
    script.write_text(WORKER.format(root=ROOT))
    procs = []
    for rank in range(2):
        env = dict(os.environ, RANK=str(rank), LOCAL_RANK=str(rank), WORLD_SIZE="2", MASTER_ADDR="127.0.0.1",
                   MASTER_PORT="29541", CUDA_VISIBLE_DEVICES="")
        procs.append(subprocess.Popen([sys.executable, str(script)], env=env, stdout=subprocess.PIPE,
                                      stderr=subprocess.PIPE, text=True))
    outs = [p.communicate(timeout=180) for p in procs]
    for p, (out, err) in zip(procs, outs):
        assert p.returncode == 0, err
        assert "ok 11.0" in out


def test_reference_arm_under_two_ranks_prints_once():
    """Under torchrun-style launch only rank 0 runs the oracle; the other rank exits 0 without output."""
    procs = []
    for rank in range(2):
        env = dict(os.environ, RANK=str(rank), LOCAL_RANK=str(rank), WORLD_SIZE="2", MASTER_ADDR="127.0.0.1",
                   MASTER_PORT="29542", CUDA_VISIBLE_DEVICES="")
        procs.append(subprocess.Popen([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--gpus", "2",
                                       "--steps", "1", "--warmup", "0"], env=env, stdout=subprocess.PIPE,
                                      stderr=subprocess.PIPE, text=True, cwd=ROOT))
    outs = [p.communicate(timeout=300) for p in procs]
    assert all(p.returncode == 0 for p in procs), [o[1] for o in outs]
    printed = [o[0].strip() for o in outs if o[0].strip()]
    assert len(printed) == 1 and json.loads(printed[0])["impl"] == "reference"


def test_printed_line_is_short_and_complete():
    """Whatever the record holds (per-layer lists of five workloads, long notes), the printed line stays under 4 KB and has
    every key of the headline."""
    import sys as _sys
    _sys.path.insert(0, ROOT)
    import bench
    x = 123.4567890123456
    layers = [{"name": f"l{i}", "us": x, "frac_of_roof": x, "roof": "tensor"} for i in range(64)]
    mode = {"conv_ms_cold": x, "conv_ms_warm": x, "outputs": "o" * 80, "algorithmic_bytes": 10 ** 10}
    res = {"modes": {"raw": mode, "fused": mode}, "per_layer": {"raw": layers, "fused": layers}}
    leg = {"ms_per_batch": x, "imgs_per_s": x, "e2e_imgs_per_s": x, "model": "m" * 300}
    roof = {k: x for k in ("achieved", "peak", "frac", "traffic", "conv_ms_per_step", "conv_launches_per_step", "hbm_peak_gbs",
                           "sum_layer_roofs_ms")}
    full = {"metric": bench.METRIC, "value": x, "unit": bench.UNIT, "n_gpus": 1, "steps": 100, "warmup": 10, "ms_per_step": x,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int32", "data": "synthetic",
            "config": {"workload": "w" * 300, "step": "s" * 300, "l2": "l" * 100}, "clocks": {"sm_mhz": 1965, "reasons": []},
            "gpu_launches": 10 ** 6, "device_wait_timeouts": 0,
            "roofline": dict(roof, bound="tensor", kernel="k" * 160, unit="TOPS", accounting="a" * 500),
            "per_config": {f"config{i}": res for i in range(1, 6)}, "network": dict(leg, fused=leg, resnet18_imagenet=leg),
            "streaming_kernels": {"note": "n" * 2000},
            "e2e": {"value": x, "unit": "TOPS", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1, "ms_per_step": x, "note": "n" * 400},
            "cpu_baseline": {"value": x, "unit": "TOPS", "cores": 16, "kind": "oracle", "sample": "s" * 500}}
    text = json.dumps(bench.short_line(full))
    line = json.loads(text)
    assert len(text) < 4096 < len(json.dumps(full))
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "clocks", "gpu_launches", "roofline", "e2e", "cpu_baseline"):
        assert key in line, key
    assert set(line["summary"]) == {f"config{i}" for i in range(1, 6)} | {"resnet20", "resnet20_fused", "resnet18_imagenet"}
