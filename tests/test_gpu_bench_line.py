"""bench.py prints one JSON line with the keys its readers rely on.

Run on the small 4K workload in a process of its own (a few seconds): the line must carry the metric, the timed
region's figures, the roofline of the dominant kernel with its live CUDA-event time behind `achieved`, the same step
as a burst, the end-to-end figure through host buffers with its byte counts, the CPU baseline from the oracle, the
clock record and the launch count, and the figures must be consistent with one another.
"""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run_bench(*flags):
    res = subprocess.run([sys.executable, "bench.py", "--workload", "gqa4_4k", "--steps", "4", "--warmup", "3", *flags],
                         cwd=ROOT, capture_output=True, text=True, timeout=900)
    assert res.returncode == 0, res.stdout[-2000:] + res.stderr[-2000:]
    lines = [ln for ln in res.stdout.splitlines() if ln.startswith("{")]
    assert len(lines) == 1, res.stdout[-2000:]
    return json.loads(lines[0])


def test_bench_line_carries_the_contract_keys_and_consistent_figures():
    from bench import launches_per_step
    d = run_bench("--no-comparators")
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert key in d, key
    assert d["n_gpus"] == 1 and d["steps"] == 4 and d["warmup"] >= 3 and d["higher_is_better"] is True
    assert d["dtype"] == "bf16" and d["data"] == "synthetic" and d["vs_baseline"] is None
    assert d["config"]["workload"] == "gqa4_4k" and "model" not in d["config"]
    assert d["gpu_launches"] == 4 * launches_per_step(4096, 8)    # (which a test below holds against a profiler)
    lat = d["latency_ms"]
    assert lat["kap"] > 0 and lat["osk"] > 0 and abs(lat["kap"] + lat["osk"] - d["ms_per_step"]) < 0.25 * d["ms_per_step"]
    # value = visited-block work over the step time
    blocks = d["config"]["blocks_scored"] + d["config"]["blocks_computed"]
    assert abs(d["value"] - blocks * 2 * 128 ** 3 / (d["ms_per_step"] * 1e-3) / 1e12) < 1e-6 * d["value"] + 1e-9
    r = d["roofline"]
    for key in ("bound", "achieved", "peak", "unit", "frac", "traffic"):
        assert key in r, key
    assert r["bound"] == "tensor" and r["unit"] == "TFLOP/s" and abs(r["frac"] - r["achieved"] / r["peak"]) < 1e-9
    assert 0 < r["frac"] < 1.2
    burst = d["latency_ms_as_a_burst"]
    assert burst["kap"] > 0 and burst["osk"] > 0 and burst["osk"] < 1.5 * lat["osk"]
    e = d["e2e"]
    assert e["value"] > 0 and e["h2d_bytes_per_step"] > 0 and e["d2h_bytes_per_step"] > 0 and e["value"] < d["value"]
    c = d["cpu_baseline"]
    assert c["kind"] == "oracle" and c["value"] > 0 and c["cores"] >= 1 and c["sample"]
    assert "sm_mhz" in d["clocks"] and "reasons" in d["clocks"]


def test_bench_variants_run():
    for flags in (("--block-q", "256", "--osk-impl", "5"), ("--page-size", "16", "--pages-in-place"), ("--top-p", "0.95")):
        d = run_bench("--no-comparators", "--no-cpu-baseline", "--no-e2e", "--no-burst", *flags)
        assert d["value"] > 0 and d["latency_ms"]["osk"] > 0


@pytest.mark.parametrize("n,stride,page_size,in_place,osk_impl,block_q", [
    (1024, 8, 0, False, 0, 128), (4096, 8, 0, False, 0, 128), (8192, 8, 0, False, 0, 128), (24576, 8, 0, False, 0, 128),
    (4096, 8, 16, False, 0, 128), (4096, 8, 16, True, 0, 128), (8192, 8, 128, False, 0, 128), (8192, 8, 16, True, 4, 128),
    (8192, 8, 0, False, 5, 256), (16384, 16, 0, False, 0, 128), (8192, 4, 0, False, 0, 128)])
def test_launches_per_step_are_what_a_profiler_counts(n, stride, page_size, in_place, osk_impl, block_q):
    import torch
    import bench
    import paper_2607_25291_b200 as cosa
    nqb = n // 128
    q, k, v = (torch.randn(1, heads, n, 128, device="cuda").to(torch.bfloat16) for heads in (4, 1, 1))
    order = torch.empty(1, 4, nqb, nqb, dtype=torch.int32, device="cuda")
    count = torch.empty(1, 4, nqb, dtype=torch.int32, device="cuda")
    out, extra = torch.empty_like(q), {}
    if page_size:
        k, v = (t.view(1, n // page_size, page_size, 128).transpose(0, 1).contiguous() for t in (k, v))
        extra = dict(kv_page_table=torch.arange(n // page_size, dtype=torch.int32, device="cuda")[None].contiguous(),
                     kv_page_size=page_size, kv_num_pages=n // page_size, kv_pages_in_place=int(in_place))
    opt = cosa.default_options(stride=stride, skip_scale=n / 3, order_stride=nqb, impl=osk_impl, **extra)

    def step():
        cosa.cosa_kap_select(q, k, 0.3, order, count, opt=opt, block_q=block_q)
        cosa.cosa_osk_attention(q, k, v, order, count, 0.1, out, opt=opt)

    step()
    assert cosa.cosa_device_status() == 0
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        step()
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if "cosa" in e.name and e.device_type == torch.autograd.DeviceType.CUDA]
    if not any(e.device_type == torch.autograd.DeviceType.CUDA for e in prof.events()):
        pytest.skip("the profiler records no kernels here")
    assert len(names) == bench.launches_per_step(n, stride, page_size, in_place, osk_impl, block_q), names
