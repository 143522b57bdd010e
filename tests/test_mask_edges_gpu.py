"""Sample bounds at, before and after the edges of the 32-column mask words, of the 64- and 128-row blocks and of the
256-row tiles, in every kernel that masks; the pool ends inside a 32-row output tile.  Tolerances: the forward's and the
gradients' stated bounds (max-abs error relative to the tensor's maximum)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_23250_b200 import pools
from parity import band_errors, rel_to_max

pytestmark = pytest.mark.gpu

# starts at 31, 63, 96, 128, 161, 225, 256, 352, 479, 512, 513, 545, 642, 768, 1023, 1025
LENGTHS = [31, 32, 33, 32, 33, 64, 31, 96, 127, 33, 1, 32, 97, 126, 255, 2]


@pytest.mark.parametrize("tail", [1, 31, 32, 33, 160])
@pytest.mark.parametrize("d,pairs", [(64, False), (128, False), (128, True), (256, False), (256, True)])
def test_sample_bounds_at_word_and_block_edges(d, pairs, tail):
    from paper_2607_23250_b200 import binding as lb
    hq, hkv = 2, 1
    cu_np = pools.cu_seqlens(LENGTHS + [tail])
    t = pools.make_tensors(int(cu_np[-1]), hq, hkv, d, seed=tail)
    q, k, v, dout = (t[n].cuda() for n in ("q", "k", "v", "dout"))
    directions = lb.LIBRA_DIR_Q | (lb.LIBRA_DIR_PAIR if pairs else lb.LIBRA_DIR_KV)
    plan = lb.libra_plan_tiles(torch.from_numpy(cu_np).cuda(), hq, 256, directions=directions, tile_kv=128, n_heads_kv=hkv)
    out, lse = lb.libra_attn_pool_fwd(q, k, v, plan)
    grads = lb.libra_attn_pool_bwd(q, k, v, out, lse, dout, plan)
    torch.cuda.synchronize()
    plan.busy_times(lb.KERNEL_FWD)                           # raises on a kernel timeout status
    plan.busy_times(lb.KERNEL_BWD_FUSED if pairs else lb.KERNEL_BWD_DKDV)
    f = {n: t[n].float().numpy() for n in t}
    o_ref, l_ref = oracle.attn_fwd(f["q"], f["k"], f["v"], cu_np)
    g_ref = oracle.attn_bwd(f["q"], f["k"], f["v"], o_ref, l_ref, f["dout"], cu_np)
    assert rel_to_max(out.float().cpu().numpy(), o_ref) <= 2e-2
    assert np.abs(lse.cpu().numpy() - l_ref).max() <= 1e-3
    for g, r in zip(grads, g_ref):
        g = g.float().cpu().numpy()
        assert rel_to_max(g, r) <= 5e-2
        assert band_errors(g, r, cu_np, band=32) <= 5e-2
    plan.destroy()
