"""bench.py's reference arm (the FP64 oracle timed on the host cores): one JSON
line with the contract's keys on rank 0, nothing on the other ranks.  A tiny
pixel sample keeps it to a few seconds; no GPU is needed."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _run(env_extra):
    env = dict(os.environ)
    env.update(env_extra)
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1",
                        "--warmup", "0", "--cpu-sample-pixels", "64"],
                       cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return [ln for ln in r.stdout.splitlines() if ln.strip()]


def test_reference_arm_prints_one_contract_line():
    lines = _run({"RANK": "0", "WORLD_SIZE": "1"})
    assert len(lines) == 1, lines
    d = json.loads(lines[0])
    assert d["impl"] == "reference"
    assert d["unit"] == "patterns/s" and d["higher_is_better"] is True
    assert d["value"] > 0 and d["ms_per_step"] > 0 and d["steps"] == 1
    assert d["config"]["workload"] == "sh_l8_R48_grid128_det512_60deg"
    cb = d["cpu_baseline"]
    assert cb["kind"] == "oracle" and cb["cores"] >= 1 and cb["value"] == d["value"] and cb["sample"]
    e = d["e2e"]
    assert e["value"] == d["value"] and e["unit"] == d["unit"]
    assert e["h2d_bytes_per_step"] == 0 and e["d2h_bytes_per_step"] == 0


def test_reference_arm_other_ranks_print_nothing():
    assert _run({"RANK": "1", "WORLD_SIZE": "2"}) == []


def test_forward_path_names_the_kernels_that_run():
    """The roofline entry: only the single-product modes sum over every pixel on the
    tensor cores; the other modes' forward pass goes through the grid of directions."""
    sys.path.insert(0, ROOT)
    import bench
    for prec, bound, kernel in (("tc_bf16", "tensor", "msft_tc_kernel"), ("tc_f16", "tensor", "msft_tc_kernel"),
                                ("tc_bf16_split", "latency", "store mode"), ("fp32", "latency", "fg_y_kernel")):
        got = bench.forward_path(prec)
        assert got[0] == bound and kernel in got[1] and ("fg_pixels_out_kernel" in got[1]) == (bound != "tensor")
