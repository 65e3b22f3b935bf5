"""Kernels that start while their predecessor still runs: calls back to back
without waiting give the results of the same calls run one at a time -- two
trees on one stream, appends between decodes, every routing (tcgen05 units
first, last, none), prefill between decodes, a replayed CUDA graph, and the
tcgen05 units' results over many repeats of a call."""
import pytest
import torch

import paper_2508_17445_gb300 as tp
import workloads
from test_gpu_parity import _built, build_forest  # noqa: F401

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _setup(script, seed):
    f, ids = build_forest(script)
    leaves = [ids[x] for x in script.leaves]
    g = torch.Generator(device=DEV).manual_seed(seed)
    h = script.heads
    return f, leaves, [torch.randn((len(leaves), h.num_q_heads, h.head_dim), generator=g, device=DEV).to(torch.bfloat16)
                       for _ in range(3)]


# tcgen05 and mma.sync units together; tcgen05 last (1792 tcgen05 units); mma.sync alone
@pytest.mark.parametrize("script", [workloads.qwen7b(seed=1, n_prompts=3, segment=64),
                                    workloads.qwen7b(seed=2, n_prompts=64, segment=64, prompt_range=(32, 96)),
                                    workloads.no_sharing(seed=3, n_seqs=9, segments=2)],
                         ids=["both", "tcgen05-last", "mma-alone"])
def test_calls_back_to_back(script):
    sets = [_setup(script, 5), _setup(workloads.tiny(seed=4), 6)]
    if script.name == "qwen7b" and len(script.leaves) == 1024:
        assert tp.tp_debug_schedule(sets[0][0].handle, sets[0][1])["n_tc_units"] >= 1672
    want = []
    for f, leaves, Qs in sets:
        for Q in Qs:
            O, LSE = f.decode(leaves, Q)
            torch.cuda.synchronize()
            want.append((O, LSE))
    for _ in range(5):
        got = []
        for f, leaves, Qs in sets:
            for Q in Qs:
                got.append(f.decode(leaves, Q))
        torch.cuda.synchronize()
        for (O, LSE), (O2, LSE2) in zip(want, got):
            assert torch.equal(O, O2) and torch.equal(LSE, LSE2)
    for f, _, _ in sets:
        f.sync()
        f.close()


def test_decodes_with_prefill_and_appends_between():
    script = workloads.qwen7b(seed=7, n_prompts=3, segment=48)

    def run(wait):
        f, leaves, Qs = _setup(script, 8)
        g = torch.Generator(device=DEV).manual_seed(9)
        h = script.heads
        out = []
        for step in range(6):
            K, V = (torch.randn((len(leaves), h.num_kv_heads, h.head_dim), generator=g, device=DEV).to(torch.bfloat16)
                    for _ in range(2))
            Qp = torch.randn((len(leaves) * 40, h.num_q_heads, h.head_dim), generator=g, device=DEV).to(torch.bfloat16)
            torch.cuda.synchronize()
            f.append_tokens(leaves, K, V)
            if wait:
                torch.cuda.synchronize()
            out.append(f.decode(leaves, Qs[0]))
            if wait:
                torch.cuda.synchronize()
            out.append(f.prefill(leaves, [40] * len(leaves), Qp))
            if wait:
                torch.cuda.synchronize()
            out.append(f.decode(leaves, Qs[1]))
            if wait:
                torch.cuda.synchronize()
        f.sync()
        f.close()
        return out
    for (O, LSE), (O2, LSE2) in zip(run(True), run(False)):
        assert torch.equal(O, O2) and torch.equal(LSE, LSE2)


def test_captured_decode_replays():
    f, leaves, Qs = _setup(workloads.qwen7b(seed=1, n_prompts=2, segment=64), 3)
    stream = torch.cuda.Stream()
    tp.tp_set_stream(f.handle, stream.cuda_stream)
    torch.cuda.synchronize()
    want = [f.decode(leaves, Q) for Q in Qs]  # caches the schedule
    torch.cuda.synchronize()
    got = [(torch.zeros_like(O), torch.zeros_like(LSE)) for O, LSE in want]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for Q, out in zip(Qs, got):
            f.decode(leaves, Q, out=out)
    for _ in range(3):
        for O, LSE in got:
            O.zero_(), LSE.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        for (O, LSE), (O2, LSE2) in zip(want, got):
            assert torch.equal(O, O2) and torch.equal(LSE, LSE2)
    f.sync()
    f.close()


# An operand that the tensor core reads before it has landed shows as a result that differs from one repeat to the next:
# short units (a few stages each, every one started by the copies' arrival) and long ones, decode and prefill
@pytest.mark.parametrize("heads", [workloads.Heads(28, 4, 128), workloads.Heads(16, 2, 64)])
@pytest.mark.parametrize("tokens,queries", [(40, 40), (717, 717), (2000, 130)])
def test_tcgen05_results_repeat(heads, tokens, queries):
    s = workloads.single_path(seed=6, lengths=(tokens,), heads=heads)
    f, ids = build_forest(s)
    leaf = ids[s.leaves[0]]
    Q, Qd = s.q(DEV, n=queries), s.q(DEV, n=200)
    outs = [(f.prefill([leaf], [queries], Q), f.decode([leaf] * 200, Qd, flags=tp.TP_DECODE_ALL_TCGEN05))
            for _ in range(60)]
    f.sync()
    for pre, dec in outs[1:]:
        for a, b in zip(pre + dec, outs[0][0] + outs[0][1]):
            assert torch.equal(a, b)
    f.close()
