"""The work a training or evaluation program has this library do, as cases that can be timed.

A case is a dict of plain values.  `prepare(case, seed)` makes what the program holds before the call (tensors, the
plan of a layout that is already in use, workspaces), `run(state)` is one pass through the public binding, `work(case)`
the operations and bytes of that pass and `tolerance(case)` how far two correct results may lie apart.

Kinds of pass:
  fwd         attention forward of one layer, plan in hand (evaluation, activation recomputation)
  bwd         attention backward of one layer, plan in hand, out and lse from the forward
  step        forward and backward of one layer, plan in hand (one layer of a training step)
  microbatch  plan, forward and backward: the first layer of a micro-batch, whose layout is new
  vrsp        sequence placement of one optimizer-step window (squared-length work, then pools)
  tap         pool planning across workers: tiles, destinations, exchange volumes, transfer records
"""
import math

import numpy as np
import torch

from paper_2607_23250_b200 import binding as lb
from paper_2607_23250_b200 import pools


def attention(name, kind, n_seqs, seq_len, hq, hkv, d, form, layout="lognormal", param=0.0, weights="pairs", draw=0):
    """layout: lognormal (median 644), pareto (one long-tailed sample per sequence besides), frac (one sample of
    param * seq_len per sequence besides), short (uniform lengths up to param).  form: the backward the plan selects,
    fused (pair tiles) or two-kernel (bit-reproducible; the library's default plan)."""
    case = dict(kind=kind, n_seqs=n_seqs, seq_len=seq_len, hq=hq, hkv=hkv, d=d, form=form, layout=layout,
                param=param, weights=weights, draw=draw)
    return dict(name=name, **case) if name else case


def listed():
    return [
        # one 4096-token sequence, 4 heads of 64: a small model's evaluation call, all latency
        attention("fwd_4k_d64", "fwd", 1, 4096, 4, 4, 64, "two-kernel"),
        # the same layer in training
        attention("step_4k_d64", "step", 1, 4096, 4, 4, 64, "two-kernel"),
        # a ragged pool of short samples (chat turns), odd token count, few heads
        attention("step_short_10k", "step", 1, 10007, 8, 2, 128, "fused", "short", 400),
        # first layer of a new micro-batch: one packed 32768-token sequence, 32 / 8 heads, planned on arrival
        attention("microbatch_32k", "microbatch", 1, 32768, 32, 8, 128, "fused"),
        # forward alone of the 8B-shaped pool (evaluation, recomputation of a checkpointed layer)
        attention("fwd_131k", "fwd", 4, 32768, 32, 8, 128, "fused"),
        # the benchmark's default workload: one training layer of the 8B-shaped pool
        attention("step_131k", "step", 4, 32768, 32, 8, 128, "fused"),
        # one rank's slice when the 8B-shaped pool is split over 8 GPUs by heads, bit-reproducible backward
        attention("bwd_slice_131k", "bwd", 4, 32768, 4, 1, 128, "two-kernel", weights="blocks"),
        # 30B-shaped pool with long-tailed samples, eight query heads per kv head
        attention("step_262k_pareto", "step", 8, 32768, 32, 4, 128, "fused", "pareto"),
        # long context: each sequence is one 65536-token sample (largest)
        attention("step_65k_long", "step", 2, 65536, 32, 8, 128, "fused", "frac", 1.0),
        # micro-benchmark head shape: 128 / 4 heads of 256
        attention("step_32k_d256", "step", 1, 32768, 128, 4, 256, "fused"),
        # placement of a 1024-sequence window into pools of 8
        dict(name="vrsp_1024", kind="vrsp", n_seqs=1024, pool=8, seq_len=32768),
        # planning of a pool of eight 32768-token sequences over 16 workers, 1024-token blocks, 4 head shards
        dict(name="tap_8x2", kind="tap", n_seqs=8, seq_len=32768, cp=2, block=1024, shards=4, hq=32, hkv=4, d=128),
    ]


LARGEST_FLOPS = 2.5e14      # step_65k_long
HEADS = {64: [(4, 4), (8, 2), (16, 4)], 128: [(32, 8), (32, 4), (64, 4), (8, 2), (8, 1), (4, 1)], 256: [(128, 4), (32, 1)]}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fwd", "fwd", "bwd", "step", "step", "step", "microbatch", "microbatch", "vrsp", "tap"])
    if kind == "vrsp":
        pool = rng.choice([2, 4, 8, 16, 32])
        return dict(kind=kind, n_seqs=pool * _log_int(rng, 8, 64), pool=pool, seq_len=rng.choice([8192, 32768, 65536]))
    if kind == "tap":
        return dict(kind=kind, n_seqs=rng.randint(1, 8), seq_len=rng.randint(8192, 65536), cp=rng.choice([2, 4, 8]),
                    block=rng.choice([1024, 2048]), shards=rng.choice([1, 2, 4, 8]), hq=32, hkv=rng.choice([4, 8]), d=128)
    d = rng.choice([64, 128, 128, 128, 256])
    hq, hkv = rng.choice(HEADS[d])
    layout = rng.choice(["lognormal", "lognormal", "pareto", "frac", "short"])
    param = {"frac": rng.choice([0.25, 0.5, 1.0]), "short": float(_log_int(rng, 16, 1024))}.get(layout, 0.0)
    form = "two-kernel" if d == 64 else rng.choice(["fused", "fused", "two-kernel"])
    total = _log_int(rng, 1000, 262144)
    n_seqs = rng.choice([1, 2, 4, 8])
    case = attention(None, kind, n_seqs, max(256, total // n_seqs), hq, hkv, d, form, layout, param,
                     rng.choice(["pairs", "pairs", "blocks"]), rng.randint(1, 1 << 20))
    while work(case)["flops"] > LARGEST_FLOPS or case["n_seqs"] * case["seq_len"] * hq * d > 1.1e9:
        case["seq_len"] = int(case["seq_len"] * 0.7)
    return case


# ---- layouts ---------------------------------------------------------------------------------------

def _spec(case, seed):
    big = {"pareto": "pareto", "frac": "frac"}.get(case.get("layout"), "none")
    # index 3 of the generator's streams; `seed` is what sets layouts apart
    return pools.PoolSpec("case", 3, case["n_seqs"], case["seq_len"], case.get("hq", 1), case.get("hkv", 1),
                          case.get("d", 64), big=big, big_frac=float(case.get("param", 0.0)), seed=seed)


def lengths_of(case):
    if case["layout"] == "short":
        rng = np.random.default_rng([case["draw"], 9])
        return [x for _ in range(case["n_seqs"]) for x in pools.random_layout(rng, case["seq_len"], int(case["param"]))]
    return pools.pool_lengths(_spec(case, case["draw"]))


def tap_tiles(case):
    return case["n_seqs"] * -(-case["seq_len"] // case["block"]) * case["shards"]


# ---- one pass ----------------------------------------------------------------------------------------

def _plan(case, cu):
    directions = lb.LIBRA_DIR_Q | lb.LIBRA_DIR_PAIR if case["form"] == "fused" else 0
    blocks = case["weights"] == "blocks"
    return lb.libra_plan_tiles(cu, case["hq"], 256, directions=directions, tile_kv=128, n_heads_kv=case["hkv"],
                               total_tokens=case["n_seqs"] * case["seq_len"],
                               weight_model=lb.LIBRA_WEIGHT_BLOCKS if blocks else lb.LIBRA_WEIGHT_PAIRS,
                               unit_cost_q=12 if blocks else 0, unit_cost_kv=6 if blocks else 0)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "vrsp":
        seqs = [pools.sequence_lengths(_spec(dict(case, layout="pareto"), seed), i % 64) for i in range(64)]
        rng = np.random.default_rng([seed, 1])
        seqs = [seqs[j] for j in rng.integers(0, 64, case["n_seqs"])]
        offs = pools.cu_seqlens([x + int(rng.integers(0, 9)) for s in seqs for x in s])   # no two sequences quite alike
        first = pools.cu_seqlens([len(s) for s in seqs])
        return dict(case=case, offs=torch.from_numpy(offs).cuda(), first=torch.from_numpy(first).cuda())
    if kind == "tap":
        lens = pools.pool_lengths(_spec(dict(case, layout="pareto"), seed))
        seq_off = [i * case["seq_len"] for i in range(case["n_seqs"] + 1)]
        # the executor's record buffer holds any assignment of such a pool, unused rows are zero
        rows = tap_tiles(case) + case["n_seqs"] * case["cp"] * case["shards"] * (sum(lens) // 256)
        return dict(case=case, cu=torch.from_numpy(pools.cu_seqlens(lens)).cuda(), seq_off=seq_off,
                    records=torch.zeros((rows, 6), dtype=torch.int32, device="cuda"))
    T, hq, hkv, d = case["n_seqs"] * case["seq_len"], case["hq"], case["hkv"], case["d"]
    names = ("q", "k", "v") if kind == "fwd" else ("q", "k", "v", "dout")
    s = pools.make_tensors(T, hq, hkv, d, seed=seed, device="cuda", names=names)
    s["case"] = case
    s["cu"] = torch.from_numpy(pools.cu_seqlens(lengths_of(case))).cuda()
    if kind == "microbatch":
        return s                                         # plan, results and workspace are made on arrival
    s["plan"] = _plan(case, s["cu"])
    s["out"] = torch.empty_like(s["q"])
    s["lse"] = torch.empty((hq, T), dtype=torch.float32, device="cuda")
    if kind != "fwd":
        s.update(dq=torch.empty_like(s["q"]), dk=torch.empty_like(s["k"]), dv=torch.empty_like(s["v"]))
        s["ws"] = torch.empty(lb.libra_attn_pool_bwd_workspace_bytes(s["plan"], s["q"], s["k"]), dtype=torch.uint8,
                              device="cuda")
    if kind == "bwd":
        lb.libra_attn_pool_fwd(s["q"], s["k"], s["v"], s["plan"], out=s["out"], lse=s["lse"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "vrsp":
        work_dev = lb.libra_vrsp_work(s["offs"], s["first"])
        return dict(lb.libra_vrsp_place(work_dev, case["pool"]), work=work_dev)
    if kind == "tap":
        geom = (case["cp"], case["block"], case["shards"], case["hq"], case["hkv"], case["d"])
        res = lb.libra_tap_plan(s["cu"], s["seq_off"], *geom)
        rec = lb.libra_tap_schedule(s["cu"], s["seq_off"], res["sigma"], *geom)[:len(s["records"])]
        s["records"][:len(rec)] = rec
        s["records"][len(rec):].zero_()
        return dict(res, records=s["records"])
    if kind == "microbatch":
        plan = _plan(case, s["cu"])
        out, lse = lb.libra_attn_pool_fwd(s["q"], s["k"], s["v"], plan)
        dq, dk, dv = lb.libra_attn_pool_bwd(s["q"], s["k"], s["v"], out, lse, s["dout"], plan)
        plan.destroy()
        return dict(out=out, lse=lse, dq=dq, dk=dk, dv=dv)
    res = {}
    if kind in ("fwd", "step"):
        res["out"], res["lse"] = lb.libra_attn_pool_fwd(s["q"], s["k"], s["v"], s["plan"], out=s["out"], lse=s["lse"])
    if kind in ("bwd", "step"):
        res["dq"], res["dk"], res["dv"] = lb.libra_attn_pool_bwd(
            s["q"], s["k"], s["v"], s["out"], s["lse"], s["dout"], s["plan"], dq=s["dq"], dk=s["dk"], dv=s["dv"],
            workspace=s["ws"])
    return res


# ---- what a pass cannot do without ---------------------------------------------------------------------

def work(case):
    if case["kind"] == "vrsp":
        D, K = case["n_seqs"], case["n_seqs"] // case["pool"]
        samples = D * case["seq_len"] / 1800.0           # about what the generator draws per sequence
        return dict(bytes=4 * samples + 4 * D + 16 * D + 8 * K, flops=2 * samples)
    if case["kind"] == "tap":
        W = case["n_seqs"] * case["cp"]
        tiles = tap_tiles(case)
        return dict(bytes=4.0 * tiles + 8 * W + 16 * W * W + 24 * tiles, flops=4.0 * tiles * W)
    ln = np.asarray(lengths_of(case), dtype=np.int64)
    pairs = int((ln * (ln + 1) // 2).sum())
    T, hq, hkv, d = int(ln.sum()), case["hq"], case["hkv"], case["d"]
    q, kv, rows = 2 * T * hq * d, 2 * T * hkv * d, 4 * T * hq
    fwd = dict(bytes=2 * q + 2 * kv + rows, flops=4 * d * hq * pairs)                # q k v in, out lse out
    bwd = dict(bytes=4 * q + 4 * kv + rows, flops=10 * d * hq * pairs)               # q k v out dout lse in, dq dk dv out
    parts = {"fwd": [fwd], "bwd": [bwd]}.get(case["kind"], [fwd, bwd])
    return {key: float(sum(p[key] for p in parts)) for key in ("bytes", "flops")}


def tolerance(case):
    if case["kind"] in ("vrsp", "tap"):
        return "exact"                                   # integers
    # bf16 operands and results, fp32 sums; P and dS are rounded to bf16 between the two products.  Against 64-bit
    # references both backward forms show up to 3.5e-3 and 0.13 (dq, dk), against each other 4.0e-3 and 0.13.
    return {"rel": 0.01, "max": 0.4}
