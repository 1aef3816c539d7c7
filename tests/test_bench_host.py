"""Host-side logic of bench.py: flop accounting, the reference arm's JSON line and
the multi-rank plumbing (world size 2 over gloo on the CPU)."""
import json
import os
import subprocess
import sys

import pytest
import torch
import torch.distributed as dist
import torch.multiprocessing as mp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_flop_accounting():
    f_ap, f_e2e = bench.step_flops()
    per_block = 202_375_168
    assert f_ap == 3 * 2 * 4096 * per_block          # 4.97 TFLOP per block and mode at 4096 tokens
    assert f_e2e == 3 * 2 * 16384 * per_block        # 19.89 TFLOP at 16384 tokens
    assert round(f_ap / 1e12, 2) == 4.97 and round(f_e2e / 1e12, 2) == 19.89


def test_peaks_have_a_source():
    p = bench.load_peaks()
    assert p["source"] in ("measured", "fallback")
    assert p["hbm_gbs"] > 1000 and p["bf16_tflops_sustained"] > 100


def test_traffic_figures_follow_the_kernel_sources(monkeypatch):
    """The ncu DRAM figures are reported only for the kernel sources they were captured from."""
    t = bench.traffic_per_launch("packed_fwd")
    if t is None:
        pytest.skip("gemm.cu or ptx.cuh changed since the last ncu capture (bench.py then reports traffic: null)")
    table = bench.NCU_TRAFFIC["packed_fwd"]
    assert t == pytest.approx((4 * table["qkvo"] + 2 * table["gate_up"] + table["down"]) / 7)
    assert 0.5 < t / 372.7e6 < 1.5                       # near the algorithmic bytes of a forward launch
    assert bench.traffic_per_launch("fakequant_fwd") is None
    monkeypatch.setitem(bench.NCU_TRAFFIC, "sources_sha256", "0" * 64)
    assert bench.traffic_per_launch("packed_fwd") is None


def _rank_main(rank, world, port, q):
    os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port), RANK=str(rank), WORLD_SIZE=str(world),
                      LOCAL_RANK=str(rank))
    dist.init_process_group("gloo", rank=rank, world_size=world)
    try:
        assert bench.dist_env() == (rank, rank, world)
        bench.barrier()
        slowest = bench.max_over_ranks(10.0 + rank, torch.device("cpu"))
        q.put((rank, slowest))
    finally:
        dist.destroy_process_group()


def test_max_over_ranks_world2_gloo():
    ctx = mp.get_context("spawn")
    q = ctx.Queue()
    port = 29500 + os.getpid() % 2000
    procs = [ctx.Process(target=_rank_main, args=(r, 2, port, q)) for r in range(2)]
    for p in procs:
        p.start()
    got = sorted(q.get(timeout=120) for _ in range(2))
    for p in procs:
        p.join(timeout=60)
        assert p.exitcode == 0
    assert got == [(0, 11.0), (1, 11.0)]             # every rank sees the slowest rank's time


def test_reference_arm_line_and_idle_ranks():
    env = dict(os.environ, RANK="0", WORLD_SIZE="1")
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1",
                          "--warmup", "0"], capture_output=True, text=True, env=env, timeout=600)
    assert out.returncode == 0, out.stderr
    line = json.loads(out.stdout.strip().splitlines()[-1])
    assert line["impl"] == "reference" and line["unit"] == "TFLOP/s" and line["value"] > 0
    assert line["cpu_baseline"]["kind"] == "oracle" and line["e2e"]["h2d_bytes_per_step"] == 0
    assert line["config"]["workload"] == bench.WORKLOAD
    assert line["cpu_baseline"]["cores"] >= 1 and line["cpu_baseline"]["threads"]["element-wise steps, group sums, bit packing"] == 1
    assert 0.0 < line["cpu_baseline"]["time_share_of_matrix_products"] < 1.0
    # under torchrun only rank 0 works; the others exit 0 silently
    env1 = dict(os.environ, RANK="1", WORLD_SIZE="2", LOCAL_RANK="1")
    out1 = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1",
                           "--warmup", "0", "--gpus", "2"], capture_output=True, text=True, env=env1, timeout=600)
    assert out1.returncode == 0 and out1.stdout.strip() == ""


def test_gpus_flag_spawns_the_ranks_itself():
    """`bench.py --gpus 2` with no launcher around it starts two ranks (here on the CPU, through the reference arm):
    exactly one line comes back, rank 0's, and it says n_gpus 2."""
    env = {k: v for k, v in os.environ.items() if k not in ("RANK", "LOCAL_RANK", "WORLD_SIZE", "MASTER_ADDR", "MASTER_PORT")}
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1",
                          "--warmup", "0", "--gpus", "2"], capture_output=True, text=True, env=env, timeout=600)
    assert out.returncode == 0, out.stderr
    lines = [l for l in out.stdout.strip().splitlines() if l.startswith("{")]
    assert len(lines) == 1
    line = json.loads(lines[0])
    assert line["impl"] == "reference" and line["n_gpus"] == 2


def test_rooflines_carry_every_denominator():
    peaks = bench.load_peaks()
    r = bench.tensor_roofline(1000.0, peaks, 0.4, 1500.0)
    assert r["peak"] == peaks["bf16_tflops"] and "burst" in r["peak_source"]            # a short timed region
    assert r["frac_vs_burst"] == pytest.approx(1000.0 / peaks["bf16_tflops"])
    assert r["frac_vs_sustained"] == pytest.approx(1000.0 / peaks["bf16_tflops_sustained"])
    assert r["frac_vs_nominal"] == pytest.approx(1000.0 / 2250.0)
    assert bench.tensor_roofline(1000.0, peaks, 5.0, 1400.0)["peak"] == peaks["bf16_tflops_sustained"]
    h = bench.hbm_roofline(4000.0, peaks)
    assert h["frac"] == pytest.approx(4000.0 / peaks["hbm_gbs"]) and h["frac_vs_nominal"] == pytest.approx(0.5)


def test_extra_configs_match_the_workload_table():
    from workloads import CONFIGS
    by_name = {c.name: c for c in CONFIGS}
    for name, spec in bench.EXTRA_CONFIGS.items():
        c = by_name[name]
        assert (spec["bits"], spec["group"]) == (c.bits, c.group)
        assert c.linears == bench.LINEARS[spec["model"]]
        assert {spec["t_ap"], spec["t_e2e"]} - {0} == {c.tokens}
        assert (spec["t_ap"] > 0) == ("block_ap" in c.modes) and (spec["t_e2e"] > 0) == ("e2e_qp" in c.modes)
        assert spec["w"] == (c.weight_dist, c.weight_scale, c.outlier_frac)


def test_the_line_on_standard_output_is_short(tmp_path, capsys):
    """The result's line holds the contract's keys in at most 2 KB, whatever else was measured; the rest goes elsewhere."""
    third = 1.0 / 3.0
    roof = dict(bench.tensor_roofline(1000.0 * third, bench.load_peaks(), 0.4, 1500.0), kernel="gemm_kernel (packed_bwd_dx)",
                traffic=1e9 * third, traffic_unit="x" * 200, algorithmic_bytes=1e9 * third)
    out = {"metric": "QLinear fwd+bwd TFLOP/s", "value": 1e3 * third, "unit": "TFLOP/s", "n_gpus": 8, "steps": 20, "warmup": 5,
           "ms_per_step": 20 * third, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
           "data": "synthetic", "config": {"workload": bench.WORKLOAD, "bits": 2, "group": 64, "tokens_block_ap": 4096,
                                           "tokens_e2e_qp": 16384, "l2": "inputs larger than L2 (working set > 2 GB per shape, weights per linear)"},
           "pct_of_bf16_peak": {k: 200 * third for k in ("vs_burst", "vs_sustained", "vs_nominal_dense")},
           "tflops_by_mode": {"block_ap": 1e3 * third, "e2e_qp": 1e3 * third}, "roofline": roof,
           "kernel_classes": {name: {"roofline": dict(roof), "ms": third} for name in
                              ("minmax_init", "fakequant_weight", "fakequant_fwd", "fakequant_bwd", "quantize_pack", "unpack", "packed_fwd",
                               "packed_bwd_dx", "packed_bwd_ds", "ste_bwd", "minmax_init_cold", "quantize_pack_cold", "unpack_cold")},
           "clocks": {"sm_mhz": 1300.0 + third, "sm_max_mhz": 1965.0, "power_w_max": 1000 * third, "samples": 145,
                      "reasons": ["hw_slowdown", "hw_thermal_slowdown", "sw_power_cap", "sw_thermal_slowdown"]},
           "e2e": {"value": 1e3 * third, "unit": "TFLOP/s", "ms_per_step": third, "steps": 20, "h2d_bytes_per_step": 10 ** 10,
                   "d2h_bytes_per_step": 10 ** 10}, "gpu_launches": 2940, "configs": {"x" * 50: "y" * 20000}, "streaming": ["z" * 9000],
           "cpu_baseline": {"value": 0.03 * third, "unit": "TFLOP/s", "kind": "oracle", "cores": 224, "sample": "s" * 500}}
    bench.report(out, str(tmp_path / "detail.json"))
    lines = capsys.readouterr().out.strip().splitlines()
    assert len(lines) == 1 and len(lines[0]) <= 2048
    line = json.loads(lines[0])
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
                "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "roofline"):
        assert key in line, key
    assert line["value"] == pytest.approx(out["value"], rel=1e-5) and line["roofline"]["traffic"] is not None
    assert json.load(open(tmp_path / "detail.json")) == out
    bench.report(out, None)
    both = capsys.readouterr()
    assert both.out.strip() == lines[0] and json.loads(both.err) == out
