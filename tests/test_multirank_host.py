"""The N > 1 arm of the benchmark without GPUs: two gloo ranks on CPU.

Prompts are independent, so ranks share nothing on the data path; what has to
be right is that every rank draws different prompts and that the whole-job
figure is (sum of units) / (slowest rank's time)."""
import os
import sys

import numpy as np
import torch
import torch.distributed as dist
import torch.multiprocessing as mp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def _worker(rank, world, port, out):
    import bench
    from paper_2503_05330_b200 import synth
    os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port))
    dist.init_process_group("gloo", rank=rank, world_size=world)
    w = synth.WORKLOADS[1]
    tokens, _ = synth.make_streams(w, bench.rank_seed(w, rank))
    times, units = bench.whole_job([10.0 + rank, 5.0 - rank], [100.0 * (rank + 1), 7.0], "cpu")
    out[rank] = (int(tokens.sum()), times, units)
    dist.barrier()
    dist.destroy_process_group()


def test_two_ranks_draw_different_prompts_and_reduce_max_time_sum_units():
    world = 2
    port = 29500 + os.getpid() % 2000
    with mp.Manager() as m:
        out = m.dict()
        mp.spawn(_worker, args=(world, port, out), nprocs=world, join=True)
        res = dict(out)
    assert res[0][0] != res[1][0]                       # different streams per rank
    for r in range(world):
        assert res[r][1] == [11.0, 5.0]                 # MAX over ranks
        assert res[r][2] == [300.0, 14.0]               # SUM over ranks


def test_single_process_passthrough():
    import bench
    assert bench.whole_job([3.0], [4.0], "cpu") == ([3.0], [4.0])


def test_the_printed_line_stays_short_and_keeps_what_the_contract_names():
    import json
    import bench
    k = {"us": 1.23456789, "p10_us": 1.0, "p90_us": 2.0, "kernel_us": {"dag": 1.0}, "get_beams_us": 3.0}
    builds = {"workspace_bytes": 1, "build_by_k": {str(n): dict(k) for n in range(1, 9)}}
    scale = {"store_bytes": 1, "gbs": 2.0, "frac": 0.5, "groups": 64}
    line = {"metric": bench.METRIC, "value": 1234567.891, "unit": bench.UNIT, "n_gpus": 1, "steps": 2, "warmup": 3, "ms_per_step": 0.1,
            "e2e": {"value": 1.0, "unit": bench.UNIT, "h2d_bytes_per_step": 5, "d2h_bytes_per_step": 6, "how": "x" * 500},
            "gpu_launches": 9, "clocks": {"sm_mhz": 1965.0, "reasons": []}, "kernels": {"step": {"us_per_launch": 15.0, "gbs": 1.0}},
            "roofline": {"steady_state_full_history": builds, "by_config": {f"config {n}": builds for n in range(10)},
                         "match_at_scale": scale, "gather_at_scale": scale, "bytes_model": "x" * 300, "note": "x" * 300},
            "dag_export": {"us_per_sdms_get_dag_call": 60.0}, "fuzzy_epsilon_1": {"us_per_step": 1.0}, "backoff_from_k_max": None,
            "cpu_baseline": {"value": 1.0, "by_threads": {}, "sample": "x" * 300}}
    text = json.dumps(bench.printed(line))
    assert len(text) < 6000
    out = json.loads(text)
    assert out["value"] == 1234570.0 and out["e2e"]["h2d_bytes_per_step"] == 5 and out["gpu_launches"] == 9
    assert out["roofline"]["by_config"]["config 3"]["us_by_k"]["8"] == 1.23457
    line["roofline"].update(steady_state_full_history=None, by_config=None, match_at_scale=None, gather_at_scale=None)
    assert json.loads(json.dumps(bench.printed(line)))["roofline"]["by_config"] is None       # several ranks: those passes are left out
