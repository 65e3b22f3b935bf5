"""The unit-length limit of decode schedules: calls that do not fill the GPU are
cut finer, cover the same tokens exactly once, and keep units at least four
blocks long (eight once there are enough units). CPU, through the ABI; the
GPU test checks that the static-scratch entry point still takes every call it
took without the limit."""
import numpy as np
import pytest

import oracle
import paper_2508_17445_gb300 as tp
import workloads
from test_host import BT, _built, check_schedule, meta_forest  # noqa: F401

# blocks around one per SM (152), around one and several per resident CTA
SHAPES = [((1216 - 160,), (40, 40, 40, 40)), ((1216,), (40, 40, 40, 40)), ((1217,), (33, 1, 64, 65)),
          ((5000,), (8, 900, 2000, 31)), ((9000, 3), (4000, 4000, 4000, 4001))]


@pytest.mark.parametrize("flags", [0, tp.TP_DECODE_NO_SHARE, tp.TP_MMA_SYNC, tp.TP_DECODE_TCGEN05,
                                   tp.TP_DECODE_CUDA_CORE_SMALL])
@pytest.mark.parametrize("prompt,leaf_tokens", SHAPES)
def test_units_of_calls_that_do_not_fill_the_gpu(prompt, leaf_tokens, flags):
    heads = workloads.Heads(28, 4, 128)
    s = workloads.shared_prompt(seed=1, prompt=sum(prompt), n_leaves=4, leaf_tokens=leaf_tokens, heads=heads)
    f = meta_forest(heads=heads, pool_blocks=1 << 12)
    ids = f.replay(s.ops)
    m = oracle.OracleForest(block_tokens=BT, pool_blocks=1 << 12).replay(s)
    S = check_schedule(f, ids, m, s, s.leaves, flags)
    lens = {}
    for u in S["units"]:
        lens[int(u[0])] = int(u[1])
    blocks = sum(lens.values()) * heads.num_kv_heads
    if blocks < 152 or flags & tp.TP_DECODE_NO_SHARE:  # not limited
        return
    limit = max(4 if blocks < 4 * 304 else 8, -(-blocks // 608))
    assert max(lens.values()) <= limit
    # only a node's own remainder is shorter than half the limit
    node_blocks = {-(-t // BT) for t in (sum(prompt), *leaf_tokens)}
    assert all(2 * n >= limit or n in node_blocks for n in lens.values())


@pytest.mark.gpu
def test_noalloc_takes_calls_whose_finer_schedule_does_not_fit():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    # 64 query heads: 33 KB of partials per slot, so 32 MiB hold about 1000
    h = workloads.Heads(64, 1, 128)
    s = workloads.shared_prompt(seed=2, prompt=9000, n_leaves=64, leaf_tokens=(600,) * 64, heads=h)
    f = tp.Forest(h.num_q_heads, h.num_kv_heads, h.head_dim, pool_blocks=s.upper_bound_blocks(32) + 8, device="cuda:0")
    ids = f.replay(s.ops, kv_fn=lambda i: s.kv(i, "cuda:0"))
    leaves = [ids[x] for x in s.leaves]
    S = tp.tp_debug_schedule(f.handle, leaves)
    assert S["n_slots"] * h.num_q_heads * (h.head_dim + 1) * 4 > 32 << 20
    Q = s.q("cuda:0")
    O_ref, LSE_ref = f.decode(leaves, Q)
    O, LSE = torch.full_like(O_ref, float("nan")), torch.full_like(LSE_ref, float("nan"))
    tp.tp_decode_noalloc(f.handle, leaves, Q, O, LSE)
    f.sync()
    assert np.isfinite(O.float().cpu().numpy()).all()
    assert (O.float() - O_ref.float()).abs().max().item() <= 1e-2
    assert (LSE - LSE_ref).abs().max().item() <= 5e-5
    f.close()
