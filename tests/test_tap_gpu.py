"""Device pool planner (tiles, Algorithm 2, exchange volumes) == oracle, bit for bit, through the C ABI."""
import numpy as np
import pytest
import torch

import oracle
from oracle import schedule as osched
from paper_2607_23250_b200 import pools

pytestmark = pytest.mark.gpu


def _compare(cu, seq_off, cp, B, H, hq, hkv, d, tau=(3, 100)):
    from paper_2607_23250_b200 import binding as lb
    got = lb.libra_tap_plan(torch.from_numpy(np.asarray(cu, np.int32)).cuda(), seq_off, cp, B, H, hq, hkv, d, *tau)
    L = oracle.tap_layout(cu, seq_off, cp, B, H, hq, hkv, d)
    W = L["n_workers"]
    want = oracle.tap_place(L["f"], L["q_home"], L["v_qo"], L["kv_off"], L["kv_grp"], L["v_g"], L["resident"], W, *tau)
    fwd, bwd = oracle.tap_exchange(cu, seq_off, cp, H, hkv, d, want["sigma"], L["q_home"], L["v_qo"], want["C"],
                                   L["resident"])
    torch.cuda.synchronize()
    assert int(got["status"].item()) == 0
    assert np.array_equal(got["sigma"].cpu().numpy(), want["sigma"])
    assert np.array_equal(got["loads"].cpu().numpy(), want["loads"])
    assert int(got["comm_total"].item()) == want["comm_total"]
    assert np.array_equal(got["fwd_bytes"].cpu().numpy(), fwd)
    assert np.array_equal(got["bwd_bytes"].cpu().numpy(), bwd)
    # the transfer records of the same assignment, and of one that scatters the tiles, equal the oracle's list
    if len(want["sigma"]) <= 4096:
        cu_dev = torch.from_numpy(np.asarray(cu, np.int32)).cuda()
        scattered = np.array([(5 * t + 3) % W for t in range(len(want["sigma"]))], np.int32)
        for sigma in (want["sigma"], scattered):
            rec = lb.libra_tap_schedule(cu_dev, seq_off, torch.from_numpy(sigma).cuda(), cp, B, H, hq, hkv, d)
            assert np.array_equal(rec.cpu().numpy().reshape(-1, 6), osched.schedule(cu, seq_off, cp, B, H, sigma))
    return want, fwd


def test_tiny_hand_checked_layout():
    _compare([0, 5, 6, 16, 20, 32], [0, 16, 32], 2, 4, 2, 4, 2, 8)


@pytest.mark.parametrize("seed", range(12))
def test_random_pools(seed):
    rng = np.random.default_rng(seed)
    P, CP = int(rng.integers(1, 6)), int(rng.choice([1, 2, 4, 8]))
    seqs = [pools.random_layout(rng, int(rng.integers(50, 3000)), int(rng.integers(1, 400))) for _ in range(P)]
    cu = pools.cu_seqlens([x for s in seqs for x in s])
    seq_off = np.concatenate([[0], np.cumsum([sum(s) for s in seqs])]).astype(np.int32)
    H, hkv = [(1, 4), (2, 4), (4, 4), (8, 4), (4, 2)][seed % 5]
    tau = [(3, 100), (0, 1), (50, 100)][seed % 3]
    _compare(cu, seq_off, CP, int(rng.choice([16, 64, 100, 256])), H, 8, hkv, 64, tau)


@pytest.mark.parametrize("P,CP,B,H", [(2, 4, 2048, 2), (8, 2, 1024, 4), (4, 16, 2048, 8)])
def test_long_tailed_pools(P, CP, B, H):
    """Pools of 32768-token sequences of the 30B shape (config 3: Hq 32, Hkv 4, d 128, Pareto-tailed samples)."""
    spec = pools.config(3)
    seqs = [pools.sequence_lengths(spec, i) for i in range(P)]
    cu = pools.cu_seqlens([x for s in seqs for x in s])
    seq_off = np.concatenate([[0], np.cumsum([sum(s) for s in seqs])]).astype(np.int32)
    want, fwd = _compare(cu, seq_off, CP, B, H, spec.hq, spec.hkv, spec.head_dim)
    loads = want["loads"]
    assert loads.max() <= 1.03 * loads.mean() + max(1, oracle.tap_layout(cu, seq_off, CP, B, H, spec.hq, spec.hkv, spec.head_dim)["f"].max())


@pytest.mark.parametrize("P,CP,max_len", [(3, 11, 90), (4, 17, 300), (8, 16, 200), (8, 17, 200), (8, 16, 5)])
def test_worker_counts_around_the_one_warp_placement(P, CP, max_len):
    """33, 68 and 128 workers (two to four per lane), 136 (a thread each) and samples so short that the residency rows
    do not fit shared memory."""
    rng = np.random.default_rng(P * CP + max_len)
    seqs = [pools.random_layout(rng, 1500, max_len) for _ in range(P)]
    cu = pools.cu_seqlens([x for s in seqs for x in s])
    _compare(cu, np.arange(P + 1, dtype=np.int32) * 1500, CP, 100, 2, 8, 4, 64)


@pytest.mark.parametrize("P,CP,H,hq,hkv,max_len,total", [
    (2, 4, 8, 8, 4, 400, 3000),            # a byte of residency per group; a full step of shards
    (3, 3, 16, 16, 4, 60, 3000),           # two steps a block, nine workers
    (2, 20, 24, 24, 8, 150, 2000),         # three steps a block, two workers a lane
    (2, 4, 20, 20, 5, 100, 2000),          # the last step half full
    (2, 2, 2, 1 << 17, 1 << 17, 900, 20000),   # volumes beyond 32 bits
    (2, 40, 1, 1 << 18, 1 << 18, 900, 5000),   # the same with four workers a lane
    (4, 2, 8, 8, 8, 3, 3000),              # tables beyond the shared memory a block has without opting in
    (4, 4, 32, 32, 8, 2, 6000),            # tables beyond shared memory
])
def test_steps_of_the_one_block_placement(P, CP, H, hq, hkv, max_len, total):
    rng = np.random.default_rng(P * CP + H)
    seqs = [pools.random_layout(rng, total, max_len) for _ in range(P)]
    cu = pools.cu_seqlens([x for s in seqs for x in s])
    for tau in ((3, 100), (0, 1)):
        _compare(cu, np.arange(P + 1, dtype=np.int32) * total, CP, 128, H, hq, hkv, 8, tau)


@pytest.mark.parametrize("blocks", [1024, 1025, 2500])
def test_blocks_beyond_a_batch_of_the_rank_sort(blocks):
    rng = np.random.default_rng(blocks)
    total = blocks * 4 - 1
    cu = pools.cu_seqlens(pools.random_layout(rng, 2 * total, 300))
    _compare(cu, [0, total, 2 * total], 4, 8, 1, 2, 1, 8)


@pytest.mark.parametrize("P", [255, 256, 300, 1024])
def test_many_sequences(P):
    """As many sequences as the smaller tables hold, more, and as many as there can be workers."""
    rng = np.random.default_rng(P)
    seqs = [pools.random_layout(rng, int(rng.integers(3, 20)), 9) for _ in range(P)]
    cu = pools.cu_seqlens([x for s in seqs for x in s])
    seq_off = np.concatenate([[0], np.cumsum([sum(s) for s in seqs])]).astype(np.int32)
    _compare(cu, seq_off, 1, 16, 1, 2, 1, 8)


@pytest.mark.parametrize("P", [3, 300])
def test_replays_of_a_captured_call_need_nothing_of_the_host(P):
    """A graph captured around the planner gives the eager call's results after the host memory of that time has been used
    for something else."""
    from paper_2607_23250_b200 import binding as lb
    rng = np.random.default_rng(P)
    seqs = [pools.random_layout(rng, 24, 9) for _ in range(P)]
    cu = torch.from_numpy(pools.cu_seqlens([x for s in seqs for x in s])).cuda()
    seq_off = [24 * i for i in range(P + 1)]
    want = lb.libra_tap_plan(cu, seq_off, 1, 16, 1, 2, 1, 8)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = lb.libra_tap_plan(cu, seq_off, 1, 16, 1, 2, 1, 8)
    junk = [np.full(2 * (P + 1), -1, np.int32) for _ in range(4096)]
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        for name in want:
            assert torch.equal(got[name], want[name]), name
    assert int(want["status"].item()) == 0 and len(junk) == 4096


def test_zero_length_samples_and_short_tail():
    _compare([0, 0, 3, 3, 3, 40, 40, 41], [0, 41], 2, 16, 2, 4, 2, 8)
    _compare([0, 7, 7, 30, 30], [0, 7, 30], 1, 4, 1, 2, 2, 8)


def test_bad_arguments():
    from paper_2607_23250_b200 import binding as lb
    cu = torch.tensor([0, 9], dtype=torch.int32).cuda()
    with pytest.raises(Exception):
        lb.libra_tap_plan(cu, [0, 9], 1, 4, 3, 4, 2, 8)    # 3 shards do not divide 4 heads
    with pytest.raises(Exception):
        lb.libra_tap_plan(cu, [0, 9], 0, 4, 2, 4, 2, 8)


def test_planner_as_the_first_call_of_a_process_under_capture():
    """The exchange planner allocates in stream order, which a capture allows, also before anything else of the library has
    run on the device (a child process, since this one has long called it)."""
    import os
    import subprocess
    import sys
    code = """
import torch
from paper_2607_23250_b200 import binding as lb
cu = torch.tensor([0, 3000, 8192], dtype=torch.int32).cuda()
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    lb.libra_tap_plan(cu, [0, 8192], 2, 1024, 2, 4, 2, 128)
res = lb.libra_tap_plan(cu, [0, 8192], 2, 1024, 2, 4, 2, 128)
torch.cuda.synchronize()
assert int(res["status"].item()) == 0
"""
    subprocess.run([sys.executable, "-c", code], check=True, timeout=300, cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
