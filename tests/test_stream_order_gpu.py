"""Passes that follow one another on a stream without a wait in between: the library's kernels start before the one ahead
has finished and some run side by side, so every pass must still see its own inputs and statistics only.  The two-kernel
forms are bit-reproducible and are compared bit for bit with passes that were waited for; the accumulating forms by the
rounding bound 2^-7 of their fp32 sums in another order (bf16 results)."""
import numpy as np
import pytest
import torch

from paper_2607_23250_b200 import pools

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,hq,hkv,pairs", [(64, 4, 2, False), (128, 4, 2, False), (128, 4, 2, True), (256, 2, 1, False),
                                            (256, 2, 1, True)])
@pytest.mark.parametrize("T", [130, 3000, 50000])     # one tile, tiles on a part of the SMs, more tiles than run side by side
def test_back_to_back_passes(d, hq, hkv, pairs, T):
    from paper_2607_23250_b200 import binding as lb
    if T == 50000 and d == 256:
        T = 20000
    rng = np.random.default_rng(T + d)
    cu = torch.from_numpy(pools.cu_seqlens(pools.random_layout(rng, T, 700))).cuda()
    directions = lb.LIBRA_DIR_Q | (lb.LIBRA_DIR_PAIR if pairs else lb.LIBRA_DIR_KV)
    plan = lb.libra_plan_tiles(cu, hq, 256, directions=directions, tile_kv=128, n_heads_kv=hkv, pair_chunk=256 if T < 50000 else 0)
    ins = [pools.make_tensors(T, hq, hkv, d, seed=s, device="cuda") for s in (1, 2)]
    out, lse = torch.empty_like(ins[0]["q"]), torch.empty((hq, T), dtype=torch.float32, device="cuda")
    grads = [torch.empty_like(ins[0][n]) for n in ("q", "k", "v")]
    ws = torch.empty(lb.libra_attn_pool_bwd_workspace_bytes(plan, ins[0]["q"], ins[0]["k"]), dtype=torch.uint8, device="cuda")

    def step(i):
        x = ins[i]
        lb.libra_attn_pool_fwd(x["q"], x["k"], x["v"], plan, out=out, lse=lse)
        lb.libra_attn_pool_bwd(x["q"], x["k"], x["v"], out, lse, x["dout"], plan, dq=grads[0], dk=grads[1], dv=grads[2], workspace=ws)
        return [t.clone() for t in (out, lse, *grads)]

    want = []
    for i in (0, 1):
        want.append(step(i))
        torch.cuda.synchronize()
    got = [(i, step(i)) for i in (0, 1, 0, 1, 1, 0)]
    torch.cuda.synchronize()
    plan.busy_times(lb.KERNEL_FWD)
    plan.busy_times(lb.KERNEL_BWD_FUSED if pairs else lb.KERNEL_BWD_DKDV)     # raises on a kernel timeout status
    for i, res in got:
        for k, (a, b) in enumerate(zip(res, want[i])):
            if pairs and k >= 2:
                assert (a.float() - b.float()).abs().max() <= 2.0 ** -7 * b.float().abs().max()
            else:
                assert torch.equal(a, b), k
    plan.destroy()


@pytest.mark.parametrize("d,hq,hkv,T", [(64, 4, 4, 4096), (128, 8, 2, 9000), (128, 4, 1, 300), (256, 4, 1, 3000)])
@pytest.mark.parametrize("name", ["q", "dout"])
def test_dq_in_place(d, hq, hkv, T, name):
    """dq written over q or over dout, with few enough tiles that the dQ kernel could run beside the kernel ahead of it, which
    reads all of both.  Bit for bit the results of a call with buffers of its own (the two-kernel forms are reproducible)."""
    from paper_2607_23250_b200 import binding as lb
    cu = torch.from_numpy(pools.cu_seqlens([T])).cuda()
    plan = lb.libra_plan_tiles(cu, hq, 256, tile_kv=128, n_heads_kv=hkv)
    t = pools.make_tensors(T, hq, hkv, d, seed=5, device="cuda")
    out, lse = lb.libra_attn_pool_fwd(t["q"], t["k"], t["v"], plan)
    want = lb.libra_attn_pool_bwd(t["q"], t["k"], t["v"], out, lse, t["dout"], plan)
    for _ in range(3):
        x = {n: v.clone() for n, v in t.items()}
        got = lb.libra_attn_pool_bwd(x["q"], x["k"], x["v"], out, lse, x["dout"], plan, dq=x[name])
        for a, b in zip(got, want):
            assert torch.equal(a, b)
    plan.destroy()


@pytest.mark.parametrize("side_stream", [False, True])
@pytest.mark.parametrize("d", [64, 256])
def test_plans_destroyed_behind_their_last_pass(d, side_stream):
    """Plan, forward, backward, destroy, over and over with another layout each time and no wait on the host: on the
    legacy stream the plan's memory is given back in the stream's order, and the next plan takes it; a plan whose passes ran
    on another stream is waited for.  Bit for bit the results of passes that were waited for."""
    from paper_2607_23250_b200 import binding as lb
    T, hq, hkv = 6000, 4, 2
    rng = np.random.default_rng(d)
    cus = [torch.from_numpy(pools.cu_seqlens(pools.random_layout(rng, T, int(m)))).cuda() for m in (6000, 200, 2000, 700)]
    t = pools.make_tensors(T, hq, hkv, d, seed=5, device="cuda")
    other = torch.cuda.Stream() if side_stream else None
    torch.cuda.synchronize()

    def once(cu):
        plan = lb.libra_plan_tiles(cu, hq, 256, tile_kv=128, n_heads_kv=hkv, total_tokens=T)
        if other is None:
            out, lse = lb.libra_attn_pool_fwd(t["q"], t["k"], t["v"], plan)
            res = (out, lse, *lb.libra_attn_pool_bwd(t["q"], t["k"], t["v"], out, lse, t["dout"], plan))
        else:
            other.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(other):
                out, lse = lb.libra_attn_pool_fwd(t["q"], t["k"], t["v"], plan)
                res = (out, lse, *lb.libra_attn_pool_bwd(t["q"], t["k"], t["v"], out, lse, t["dout"], plan))
        plan.destroy()
        return res

    want = []
    for cu in cus:
        want.append(once(cu))
        torch.cuda.synchronize()
    got = [(i % 4, once(cus[i % 4])) for i in range(16)]
    torch.cuda.synchronize()
    for i, res in got:
        for a, b in zip(res, want[i]):
            assert torch.equal(a, b)


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
def test_plan_built_while_a_stream_is_captured(mode):
    """A plan outlives the call that builds it, so its memory may not belong to a graph: where the capture forbids an ordinary
    allocation the plan is refused, in relaxed mode it is good from the graph's first replay on, and after the graph is gone."""
    import oracle
    from paper_2607_23250_b200 import binding as lb
    cu_np = np.array([0, 300, 1000], np.int32)
    cu = torch.from_numpy(cu_np).cuda()
    lb.libra_plan_tiles(cu, 2, 256, total_tokens=1000).destroy()     # what a first call sets up is there
    torch.cuda.synchronize()
    graph, plans, refused = torch.cuda.CUDAGraph(), [], False
    try:
        with torch.cuda.graph(graph, capture_error_mode=mode):
            try:
                plans.append(lb.libra_plan_tiles(cu, 2, 256, total_tokens=1000))
            except lb.LibraError as err:
                refused = err.code == lb.ERR_CUDA
    except RuntimeError:
        assert refused          # the capture is void after a call that it forbids
    if mode == "relaxed":
        graph.replay()
        torch.cuda.synchronize()
        del graph
        got, want = plans[0].export(), oracle.plan(cu_np, 2, 256, plans[0].info()["n_workers"], 0)
        assert plans[0].status() == 0 and np.array_equal(got["loads"], want["loads"])
        plans[0].destroy()
    else:
        assert refused and not plans
    assert torch.ones(4, device="cuda").sum().item() == 4
