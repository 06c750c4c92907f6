"""CPU-side checks of bench.py: the reference arm (the oracle timed on host cores) prints the contract's JSON
line, and the multi-rank aggregation (max of per-rank times over torch.distributed) works with two gloo ranks."""
import json
import os
import subprocess
import sys

import torch.multiprocessing as mp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reference_arm_prints_contract_line():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--workload", "1",
                          "--steps", "2", "--warmup", "1"], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert out.returncode == 0, out.stderr
    line = json.loads(out.stdout.strip().splitlines()[-1])
    assert line["impl"] == "reference" and line["unit"] == "agent-steps/s" and line["value"] > 0
    assert line["cpu_baseline"]["kind"] == "oracle" and line["cpu_baseline"]["cores"] >= 1
    assert line["e2e"]["h2d_bytes_per_step"] == 0 and line["e2e"]["d2h_bytes_per_step"] == 0
    assert line["config"]["workload"].startswith("cfg1_") and line["higher_is_better"] is True
    for key in ("metric", "n_gpus", "steps", "warmup", "ms_per_step", "scaling", "vs_baseline", "dtype", "data"):
        assert key in line


def _rank_main(rank, world, port, out_dir):
    os.environ.update(RANK=str(rank), WORLD_SIZE=str(world), LOCAL_RANK=str(rank), MASTER_ADDR="127.0.0.1",
                      MASTER_PORT=str(port))
    sys.path.insert(0, ROOT)
    import bench
    r, w, _ = bench.dist_setup(world)
    assert (r, w) == (rank, world)
    bench.dist_barrier(w)
    got = bench.dist_max(10.0 + rank, w, device="cpu")    # every rank must see the slowest rank's time
    with open(os.path.join(out_dir, f"r{rank}.txt"), "w") as f:
        f.write(str(got))
    import torch.distributed as dist
    dist.destroy_process_group()


def test_two_rank_time_aggregation_gloo(tmp_path):
    mp.spawn(_rank_main, args=(2, 29533, str(tmp_path)), nprocs=2, join=True)
    assert [float(open(tmp_path / f"r{k}.txt").read()) for k in range(2)] == [11.0, 11.0]


def test_algorithmic_bytes_formula():
    sys.path.insert(0, ROOT)
    import bench
    from paper_2205_05248_b200 import workloads
    cfg = workloads.config(5)
    assert abs(bench.algorithmic_bytes_per_agent_step(cfg, 64) - 737.25) < 1e-9
    assert abs(bench.flops_per_agent_step(cfg) - (2 * 64 * (80 + 384 + 14) + 25 * 64)) < 1e-9


def test_roofline_of_each_kernel():
    """The bound follows the kernel that ran: HBM or tensor cores, in fp32 six bf16 products a product on the split-operand
    kernel, plain FFMA on the CUDA-core kernel."""
    sys.path.insert(0, ROOT)
    import bench
    from paper_2205_05248_b200 import workloads
    peaks = {"hbm_gbs": 6500.0, "bf16_tflops": 1600.0, "bf16_tflops_sustained": 1400.0}
    cfg = workloads.config(5, E=4096, precision="fp32")
    steps = 4096 * 8 * 64
    flops = bench.flops_per_agent_step(cfg)
    r = bench.step_roofline(cfg, "actor_tcs_kernel", 1.1, 64, steps, peaks, "measured")
    assert r["bound"] == "tensor" and r["kernel"] == "actor_tcs_kernel" and r["peak"] == 1400.0
    assert abs(r["achieved"] - 6 * flops * steps / 1.1e-3 / 1e12) < 1e-6 and r["frac"] < 1.0
    r = bench.step_roofline(cfg, "actor_ffma_kernel", 4.9, 64, steps, peaks, "measured", ffma_peak=72.0)
    assert r["bound"] == "alu" and r["peak"] == 72.0 and abs(r["achieved"] - flops * steps / 4.9e-3 / 1e12) < 1e-6
    r = bench.step_roofline(workloads.config(5), "actor_tcp_kernel", 5.7, 64, 65536 * 8 * 64, peaks, "measured")
    assert r["bound"] == "hbm" and abs(r["achieved"] - 737.25 * 65536 * 8 * 64 / 5.7e-3 / 1e9) < 1e-6
