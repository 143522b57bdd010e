"""Fused backward on pairs of CTAs (256-key tiles; pools with few cells that only one of two neighbouring key blocks sees)
against the CPU oracle's gradient.  The call and the plan are the fused backward's; a chunk is asked for where the planner
would take single CTAs for so small a pool."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_23250_b200 import pools
from test_attn_bwd_fused_gpu import _check, _run

pytestmark = pytest.mark.gpu


def _plan(lengths, hq, hkv, W=0, chunk=0):
    from paper_2607_23250_b200 import binding as lb
    return lb.libra_plan_tiles(torch.from_numpy(pools.cu_seqlens(lengths)).cuda(), hq, 256, n_workers=W,
                               directions=lb.LIBRA_DIR_Q | lb.LIBRA_DIR_PAIR, tile_kv=128, n_heads_kv=hkv, pair_chunk=chunk)


def _ctas(lengths, hq, hkv, W=0, chunk=0):
    plan = _plan(lengths, hq, hkv, W, chunk)
    n = plan.fused_ctas()
    plan.destroy()
    return n


def _run_on_pairs(lengths, hq, hkv, W=0, chunk=0, **kw):
    assert _ctas(lengths, hq, hkv, W, chunk) == 2
    return _run(lengths, hq, hkv, W=W, chunk=chunk, **kw)


@pytest.mark.parametrize("lengths,W,chunk,ctas", [
    ([1024, 1024], 0, 512, 2), ([1500, 1700], 0, 512, 1),        # cells past the ends of a lower key block's samples
    ([2700, 1800], 0, 512, 2), ([2500, 2300], 0, 512, 1),        # the same close to the line on either side
    ([600], 0, 512, 1), ([1000], 0, 512, 2),                     # cells at the diagonal
    ([0, 4000, 0, 0, 0], 0, 512, 2),                             # empty samples change nothing
    ([1100], 0, 0, 1), ([1100], 0, 128, 2),                      # a chunk of one row block, unless it was asked for
    ([3000], 0, 0, 1), ([3000], 0, 256, 2), ([4000], 0, 0, 2),   # few tiles a worker
    ([4000], 2, 0, 2), ([4000], 1, 0, 1),                        # two workers at least
    ([4000], 3, 0, 1), ([4000], 37, 512, 1), ([4000], 147, 0, 2),   # an odd one stays idle
])
def test_which_pools_run_on_pairs(lengths, W, chunk, ctas):
    plan = _plan(lengths, 8, 2, W, chunk)
    assert plan.fused_ctas() == ctas
    plan.destroy()


def test_no_form_without_pair_tiles():
    from paper_2607_23250_b200 import binding as lb
    plan = lb.libra_plan_tiles(torch.tensor([0, 3000], dtype=torch.int32).cuda(), 2, 256)
    with pytest.raises(lb.LibraError) as err:
        plan.fused_ctas()
    assert err.value.code == lb.ERR_PLAN_MISMATCH
    plan.destroy()


@pytest.mark.parametrize("lengths", [
    [1024],                      # whole key blocks, an even number
    [1100],                      # nine key blocks: the last pair lacks its upper half; a ragged end
    [1025, 1153],                # a sample that starts inside a key block
    [128 * 9 + 1, 128 * 7 - 1, 2500],   # samples that end just past and just before a block's edge
    [300, 2000, 100],            # a sample that ends in the lower half of a wide key block
    [2900, 1, 1900, 40],         # short ones between long ones
])
@pytest.mark.parametrize("hq,hkv,chunk", [(4, 2, 256), (2, 2, 512), (8, 1, 512)])
def test_edges_of_the_key_blocks(lengths, hq, hkv, chunk):
    got, ref, cu, _ = _run_on_pairs(lengths, hq, hkv, seed=hq, chunk=chunk)
    _check(got, ref, cu)


@pytest.mark.parametrize("chunk", [128, 384, 512, 4096])
def test_query_chunk_sizes(chunk):
    """One row block a chunk makes tiles of which a half sees nothing; an odd number of them lets a chunk begin at the upper
    key block."""
    got, ref, cu, _ = _run_on_pairs([3000, 1100], 4, 2, seed=1, chunk=chunk)
    _check(got, ref, cu)


@pytest.mark.parametrize("W", [2, 4, 147, 148])
def test_worker_counts(W):
    """A pair of CTAs for every two workers; an odd one stays idle."""
    got, ref, cu, _ = _run_on_pairs([1300, 1200], 4, 1, seed=W, W=W, chunk=512)
    _check(got, ref, cu)


def test_repeat_agrees_to_rounding():
    got, ref, cu, again = _run_on_pairs([2600, 2100], 8, 2, seed=9, repeat=True, chunk=512)
    _check(got, ref, cu)
    for g, a in zip(got, again):
        assert np.abs(g - a).max() <= 2.0 ** -7 * np.abs(g).max()     # one bf16 step of the largest values


def test_tile_times_cover_every_tile():
    from paper_2607_23250_b200 import binding as lb
    lengths, hq, hkv = [3000, 1100], 4, 2
    cu_np = pools.cu_seqlens(lengths)
    t = pools.make_tensors(int(cu_np[-1]), hq, hkv, 128, seed=5, device="cuda")
    plan = _plan(lengths, hq, hkv, chunk=512)
    assert plan.fused_ctas() == 2
    out, lse = lb.libra_attn_pool_fwd(t["q"], t["k"], t["v"], plan)
    lb.libra_attn_pool_bwd(t["q"], t["k"], t["v"], out, lse, t["dout"], plan)
    ns, busy = plan.tile_times(lb.KERNEL_BWD_FUSED), plan.busy_times(lb.KERNEL_BWD_FUSED)
    assert len(ns) == plan.info(lb.LIBRA_DIR_PAIR)["n_tiles"] and (ns > 0).all()
    assert int(ns.max()) <= int(busy.max()) and int(ns.astype(np.int64).sum()) <= int(busy.astype(np.int64).sum())
    # two neighbouring key blocks of a chunk share the pair's time by their live cells
    kb, qc, _ = plan.export_pairs()
    cells, compared = plan.export(lb.LIBRA_DIR_PAIR)["weight"], 0
    for u in range(len(kb) - 1):
        if kb[u] % 2 == 0 and kb[u + 1] == kb[u] + 1 and qc[u + 1] == qc[u] and cells[u] != cells[u + 1]:
            a, b = ns[u] / cells[u], ns[u + 1] / cells[u + 1]
            assert abs(a - b) <= 0.15 * max(a, b), (u, ns[u], ns[u + 1], cells[u], cells[u + 1])   # (each CTA reads its own clock)
            compared += 1
    assert compared >= 8
    plan.destroy()


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_values_that_are_not_finite_stay_in_their_block(value):
    """The pair streams row blocks that only one of its key blocks sees: what is not finite there reaches no key of the other,
    and a key or value that is not finite no row that does not see its block."""
    from paper_2607_23250_b200 import binding as lb
    T, hq, hkv, at = 1100, 2, 1, {"v": 700, "k": 200, "q": 300, "dout": 800}
    plan = _plan([T], hq, hkv, chunk=256)
    assert plan.fused_ctas() == 2
    clean = pools.make_tensors(T, hq, hkv, 128, seed=3, device="cuda")
    out0, lse0 = lb.libra_attn_pool_fwd(clean["q"], clean["k"], clean["v"], plan)
    for name, row in at.items():
        t = {n: x.clone() for n, x in clean.items()}
        t[name][row, 0, 5] = value
        first, behind = row // 128 * 128, row // 128 * 128 + 128
        dq, dk, dv = lb.libra_attn_pool_bwd(t["q"], t["k"], t["v"], out0, lse0, t["dout"], plan)
        if name in ("k", "v"):
            assert torch.isfinite(dq[:first].float()).all(), name
            assert not torch.isfinite(dq[row:].float()).all()
        else:
            assert torch.isfinite(dk[behind:].float()).all() and torch.isfinite(dv[behind:].float()).all(), name
            assert not torch.isfinite(dk[first:row].float()).all()
    plan.destroy()


@pytest.mark.parametrize("lengths,W", [([1200], 0), ([1300, 1200], 4)])
def test_gives_up_cleanly_when_one_producer_stalls(lengths, W):
    """The odd CTAs' producers issue no loads (a flag that nothing sets): TIMEOUT is reported, the context stays usable, and
    the next launch with the injection off is correct."""
    from paper_2607_23250_b200 import binding as lb
    hq, hkv = 4, 2
    cu_np = pools.cu_seqlens(lengths)
    t = pools.make_tensors(int(cu_np[-1]), hq, hkv, 128, seed=4)
    q, k, v, dout = (t[n].cuda() for n in ("q", "k", "v", "dout"))
    plan = _plan(lengths, hq, hkv, W, chunk=512)
    assert plan.fused_ctas() == 2
    out, lse = lb.libra_attn_pool_fwd(q, k, v, plan)
    plan.set_wait_limit_ns(200_000)
    plan.inject_stall(True)
    lb.libra_attn_pool_bwd(q, k, v, out, lse, dout, plan)
    with pytest.raises(lb.LibraError) as err:
        plan.busy_times(lb.KERNEL_BWD_FUSED)
    assert err.value.code == lb.ERR_TIMEOUT
    plan.inject_stall(False)
    plan.set_wait_limit_ns(0)
    got = [x.float().cpu().numpy() for x in lb.libra_attn_pool_bwd(q, k, v, out, lse, dout, plan)]
    plan.busy_times(lb.KERNEL_BWD_FUSED)
    f = {n: t[n].float().numpy() for n in t}
    o_ref, l_ref = oracle.attn_fwd(f["q"], f["k"], f["v"], cu_np)
    _check(got, oracle.attn_bwd(f["q"], f["k"], f["v"], o_ref, l_ref, f["dout"], cu_np), cu_np)
    plan.destroy()
