"""Where prefill row blocks are split: schedules on both sides of the rule's
edges cover every visible token once (CPU), and the kernels, which derive each
row's occurrence and visible length from its unit, agree with the oracle on
split and unsplit blocks of both head sizes, to O's own rounding where a call's
probabilities are held in two terms (GPU)."""
import numpy as np
import pytest

import oracle
import paper_2508_17445_gb300 as tp
import workloads
from test_prefill_host import check_prefill_coverage, metadata_forest

# one row block (18 queries of a 7-row group at most) on either side of the lengths that are split: 8 + 20 tiles on
# tcgen05 and 4 + 4 on mma.sync, a little longer with more rows
EDGES = [(8 * 32, 1, False, False), (8 * 32 + 1, 1, False, True), (28 * 32, 1, False, True), (28 * 32 + 1, 1, True, True),
         (28 * 32 + 1, 18, False, True), (30 * 32, 40, False, True), (31 * 32, 40, True, True), (72 * 32, 1, True, True),
         (72 * 32 + 1, 1, True, True), (73 * 32, 18, True, True), (128 * 32 + 1, 5, True, True), (40 * 32, 40, True, True),
         (9000, 40, True, True)]


@pytest.mark.parametrize("flags", [0, tp.TP_MMA_SYNC])
@pytest.mark.parametrize("tokens,queries,split,split_mma", EDGES)
def test_split_edges(tokens, queries, split, split_mma, flags):
    s = workloads.single_path(seed=1, lengths=(tokens,), heads=workloads.Heads(28, 4, 128))
    f, ids = metadata_forest(s)
    model = oracle.OracleForest(block_tokens=32, pool_blocks=1 << 10).replay(s)
    check_prefill_coverage(f, model, ids, [s.leaves[0]], [queries], flags)
    d = tp.tp_debug_prefill_schedule(f.handle, [ids[s.leaves[0]]], [queries], flags)
    assert (d["n_slots"] > 0) == (split_mma if flags else split)


# whole prompts, whose partials cost more than the tail they save, and calls whose units fill the GPU, stay whole
@pytest.mark.parametrize("heads,tokens,paths,queries", [(workloads.Heads(28, 4, 128), 1100, 1, 1100),
                                                        (workloads.Heads(28, 4, 128), 2600, 1, 2600),
                                                        (workloads.Heads(16, 2, 64), 1800, 1, 1800),
                                                        (workloads.Heads(28, 4, 128), 2048, 32, 4),
                                                        (workloads.Heads(28, 4, 128), 2048, 8, 64)])
def test_blocks_left_whole(heads, tokens, paths, queries):
    f = tp.Forest(heads.num_q_heads, heads.num_kv_heads, heads.head_dim, pool_blocks=paths * 82 + 8)
    nodes = [f.add_root() for _ in range(paths)]
    for x in nodes:
        f.append(x, n_tokens=tokens)
    assert tp.tp_debug_prefill_schedule(f.handle, nodes, [queries] * paths)["n_slots"] == 0
    f.close()


@pytest.mark.gpu
@pytest.mark.parametrize("flags", [0, tp.TP_MMA_SYNC])
@pytest.mark.parametrize("heads", [workloads.Heads(28, 4, 128), workloads.Heads(16, 2, 64), workloads.Heads(12, 1, 128)])
@pytest.mark.parametrize("tokens,queries", [e[:2] for e in EDGES])
def test_split_edges_against_the_oracle(tokens, queries, heads, flags):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from test_gpu_parity import _kv_source, build_forest, check
    s = workloads.single_path(seed=2, lengths=(31, tokens - 31), heads=heads)  # the last node holds the queries
    f, ids = build_forest(s)
    Q = s.q("cuda:0", n=queries)
    O, LSE = f.prefill([ids[s.leaves[0]]], [queries], Q, flags)
    f.sync()
    src = _kv_source(s)
    model = oracle.OracleForest(block_tokens=32, pool_blocks=f.cfg.pool_blocks).replay(s)
    o_ref, lse_ref = model.prefill([s.leaves[0]], [queries], Q.cpu(), src)
    abs_src = lambda i: (src(i)[0], oracle.bf16_bits(src(i)[1]) & np.uint16(0x7FFF))  # noqa: E731
    a_ref, _ = model.prefill([s.leaves[0]], [queries], Q.cpu(), abs_src)
    check(O, LSE, o_ref, lse_ref, a_ref)
    f.close()


# schedules of a little under and over 512 and 4096 words (4 units of 10 words per 18 queries): two parameter sizes of
# the launch, then an upload; calls back to back, each with a schedule of its own
@pytest.mark.gpu
def test_schedule_words_with_the_launch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from test_gpu_parity import _kv_source, build_forest, check
    heads = workloads.Heads(28, 4, 128)
    sizes = [18, 198, 216, 217, 1782, 1800, 1818, 1900, 1, 217]
    cases = []
    for i, n in enumerate(sizes):
        s = workloads.single_path(seed=20 + i, lengths=(n,), heads=heads)
        f, ids = build_forest(s)
        cases.append((s, f, ids[s.leaves[0]], n, s.q("cuda:0", n=n)))
    torch.cuda.synchronize()
    words = [len(tp.tp_debug_prefill_schedule(f.handle, [x], [n])["units"]) * 10 + 16 for _, f, x, n, _ in cases]
    assert min(words) < 512 < words[3] < 4096 < max(words)
    outs = [f.prefill([x], [n], Q) for _, f, x, n, Q in cases]
    torch.cuda.synchronize()
    for (s, f, x, n, Q), (O, LSE) in zip(cases, outs):
        f.sync()
        rows = sorted({0, n // 2, n - 1} | set(range(0, n, 97)))
        model = oracle.OracleForest(block_tokens=32, pool_blocks=f.cfg.pool_blocks).replay(s)
        o_ref, lse_ref = model.prefill([s.leaves[0]], [n], Q.cpu(), _kv_source(s), indices=rows)
        check(O, LSE, o_ref, lse_ref, rows=rows)
        f.close()


# whole prompts at the edges of a tile, a stage and two stages: every causal mask of the last stage
@pytest.mark.gpu
@pytest.mark.parametrize("heads", [workloads.Heads(28, 4, 128), workloads.Heads(16, 2, 64)])
@pytest.mark.parametrize("tokens", [1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129])
def test_masked_last_stages(tokens, heads):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from test_gpu_parity import _kv_source, build_forest
    s = workloads.single_path(seed=40 + tokens, lengths=(tokens,), heads=heads)
    f, ids = build_forest(s)
    Q = s.q("cuda:0", n=tokens)
    O, LSE = f.prefill([ids[s.leaves[0]]], [tokens], Q)
    f.sync()
    src = _kv_source(s)
    model = oracle.OracleForest(block_tokens=32, pool_blocks=f.cfg.pool_blocks).replay(s)
    o_ref, lse_ref = model.prefill([s.leaves[0]], [tokens], Q.cpu(), src)
    abs_src = lambda i: (src(i)[0], oracle.bf16_bits(src(i)[1]) & np.uint16(0x7FFF))  # noqa: E731
    a_ref, _ = model.prefill([s.leaves[0]], [tokens], Q.cpu(), abs_src)
    # rows that see a few tokens have |O| up to the values' own size (4 and more), where the two bf16 roundings (of P and
    # of O, 2^-8 each) alone exceed the absolute bar of 1e-2: the derived bound 2^-8 (|O| + A) + 1e-5 holds everywhere
    d_o = np.abs(O.float().cpu().numpy().astype(np.float64) - o_ref)
    assert (d_o <= 2.0 ** -8 * (np.abs(o_ref) + a_ref) + 1e-5).all()
    assert np.abs(LSE.cpu().numpy().astype(np.float64) - lse_ref).max() <= 5e-5
    f.close()


# Calls of few units hold each probability in two bf16 terms, split rows or not: what they leave out is 2^-16 of the
# probability (2^-8 of a second term below 2^-7 of it, halved by rounding), so O is off by its own rounding (half a unit in the last of its 8 places) and, with what fp32 sums and exp2
# add to the scores and the sums, 2^-15 of A = sum p |v|. (One bf16 term leaves out up to 2^-8 of each probability, in sum
# ~2^-13 A over some hundred tokens.)
# Schedules of both parameter sizes, uploaded, and with split rows
@pytest.mark.gpu
@pytest.mark.parametrize("flags", [0, tp.TP_MMA_SYNC])
@pytest.mark.parametrize("heads", [workloads.Heads(28, 4, 128), workloads.Heads(16, 2, 64)])
@pytest.mark.parametrize("tokens,queries", [(33, 33), (100, 100), (717, 717), (2000, 2000), (1000, 1), (2100, 40), (9000, 40)])
def test_probabilities_in_two_terms(tokens, queries, heads, flags):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from test_gpu_parity import _kv_source, build_forest
    s = workloads.single_path(seed=60 + tokens, lengths=(tokens,), heads=heads)
    f, ids = build_forest(s)
    Q = s.q("cuda:0", n=queries)
    O, LSE = f.prefill([ids[s.leaves[0]]], [queries], Q, flags)
    f.sync()
    rows = sorted({0, queries // 3, queries - 1} | set(range(0, queries, 131)))
    src = _kv_source(s)
    model = oracle.OracleForest(block_tokens=32, pool_blocks=f.cfg.pool_blocks).replay(s)
    o_ref, lse_ref = (x[rows] for x in model.prefill([s.leaves[0]], [queries], Q.cpu(), src, indices=rows))
    abs_src = lambda i: (src(i)[0], oracle.bf16_bits(src(i)[1]) & np.uint16(0x7FFF))  # noqa: E731
    a_ref = model.prefill([s.leaves[0]], [queries], Q.cpu(), abs_src, indices=rows)[0][rows]
    d_o = np.abs(O[rows].float().cpu().numpy().astype(np.float64) - o_ref)
    assert (d_o <= 2.0 ** (np.floor(np.log2(np.abs(o_ref))) - 8) + 2.0 ** -15 * a_ref).all()
    assert np.abs(LSE[rows].cpu().numpy().astype(np.float64) - lse_ref).max() <= 5e-5
    f.close()


# Infinite values come through as in calls with one term: both terms of a probability are above 0 where it is (rows that do
# not see the value are left out: a masked probability of 0 times infinity is NaN there, as in every tensor-core product;
# whole tiles, since what a short one leaves of its slot is multiplied by 0 too)
@pytest.mark.gpu
@pytest.mark.parametrize("flags", [0, tp.TP_MMA_SYNC])
@pytest.mark.parametrize("tokens,queries", [(128, 128), (704, 704), (2112, 40)])
def test_infinite_values(tokens, queries, flags):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = torch.Generator(device="cuda:0").manual_seed(tokens)
    K, V = (torch.randn((tokens, 2, 128), generator=g, device="cuda:0").to(torch.bfloat16) for _ in range(2))
    V[10, 0, 5], V[20, 1, 7] = float("inf"), float("-inf")
    Q = torch.randn((queries, 8, 128), generator=g, device="cuda:0").to(torch.bfloat16)
    f = tp.Forest(8, 2, 128, pool_blocks=128, device="cuda:0")
    r = f.add_root()
    f.append(r, K, V)
    O, _ = f.prefill([r], [queries], Q, flags)
    f.sync()
    see = O[-min(queries, tokens - 20):]
    assert (see[:, :4, 5] == float("inf")).all() and (see[:, 4:, 7] == float("-inf")).all()
    see[:, :4, 5], see[:, 4:, 7] = 0, 0
    assert torch.isfinite(see.float()).all()
    f.close()
