"""Host-buffer decode calls whose results the merge writes to pinned memory
itself, or leaves to a download: bit-identical to the device-buffer call in
either case -- waiting after each call, back to back, small and large results,
one pinned and one pageable buffer, buffers at odd offsets, and the same pinned
buffers as before a call with others; and tp_sync covers them after the tree
has been given another stream."""
import pytest
import torch

import paper_2508_17445_gb300 as tp
import workloads
from test_gpu_parity import _built, build_forest  # noqa: F401

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


# O of 16 leaves is 115 KB, of 48 344 KB: below and above the 128 KB line
@pytest.mark.parametrize("prompts", [1, 3])
def test_results_written_to_the_host(prompts):
    script = workloads.qwen7b(seed=3, n_prompts=prompts, segment=64)
    f, ids = build_forest(script)
    leaves = [ids[x] for x in script.leaves]
    n = len(leaves)
    g = torch.Generator(device=DEV).manual_seed(5)
    Qs = [torch.randn((n, 28, 128), generator=g, device=DEV).to(torch.bfloat16) for _ in range(6)]
    want = []
    for Q in Qs:
        O, LSE = f.decode(leaves, Q)
        f.sync()
        want.append((O.cpu(), LSE.cpu()))
    pinned = [Q.cpu().pin_memory() for Q in Qs]
    shape = (n, 28, 128)

    def buffers(kind):
        if kind == "pinned":
            return torch.zeros(shape, dtype=torch.bfloat16).pin_memory(), torch.zeros(shape[:2]).pin_memory()
        if kind == "pageable lse":
            return torch.zeros(shape, dtype=torch.bfloat16).pin_memory(), torch.zeros(shape[:2])
        raw = torch.zeros(n * 28 * 128 + 1, dtype=torch.bfloat16).pin_memory()  # O two bytes off
        return raw[1:].view(shape), torch.zeros(shape[:2]).pin_memory()

    for wait in (True, False):
        for kind in ("pinned", "pageable lse", "offset"):
            outs = [buffers(kind) for _ in Qs]
            for Q, out in zip(pinned, outs):
                tp.tp_decode_host(f.handle, leaves, Q, out[0], out[1])
                if wait:
                    f.sync()
            f.sync()
            for (O, LSE), (Oh, Lh) in zip(want, outs):
                assert torch.equal(O, Oh) and torch.equal(LSE, Lh)
    # one O for calls of both kinds: the last call's results stay
    O, lse_pinned, lse_plain = *buffers("pinned"), torch.zeros(shape[:2])
    for rep in range(10):
        for k, lse in ((0, lse_plain), (1, lse_pinned), (2, lse_plain), (3, lse_pinned)):
            tp.tp_decode_host(f.handle, leaves, pinned[k], O, lse)
        f.sync()
        assert torch.equal(O, want[3][0]) and torch.equal(lse_pinned, want[3][1]) and torch.equal(lse_plain, want[2][1])
    f.close()


# the kernels of the call sit behind ~50 ms of other work on the stream that the tree had then
@pytest.mark.parametrize("n", [1, 8])
def test_sync_after_the_stream_changed(n):
    script = workloads.no_sharing(seed=4, n_seqs=n, segments=1)
    f, ids = build_forest(script)
    h, leaves = script.heads, [ids[x] for x in script.leaves]
    Q = script.q(DEV)
    O_ref, LSE_ref = f.decode(leaves, Q, flags=tp.TP_MMA_SYNC)
    f.sync()
    want = O_ref.cpu(), LSE_ref.cpu()
    Qh = Q.cpu().pin_memory()
    old, new = torch.cuda.Stream(), torch.cuda.Stream()
    tp.tp_set_stream(f.handle, old.cuda_stream)
    outs = [(torch.zeros((n, h.num_q_heads, h.head_dim), dtype=torch.bfloat16).pin_memory(),
             torch.zeros((n, h.num_q_heads)).pin_memory()) for _ in range(3)]
    tp.tp_decode_host(f.handle, leaves, Qh, *outs[0], tp.TP_MMA_SYNC)  # first buffers made, everything idle
    f.sync()
    torch.cuda.synchronize()
    with torch.cuda.stream(old):
        torch.cuda._sleep(100_000_000)
    tp.tp_decode_host(f.handle, leaves, Qh, *outs[1], tp.TP_MMA_SYNC)
    tp.tp_set_stream(f.handle, new.cuda_stream)
    f.sync()  # the new stream is idle: the results are still on the old one
    assert torch.equal(outs[1][0], want[0]) and torch.equal(outs[1][1], want[1])
    # a call on the new stream into the buffers of one still waiting on the old: the later call's results stay
    tp.tp_set_stream(f.handle, old.cuda_stream)
    with torch.cuda.stream(old):
        torch.cuda._sleep(100_000_000)
    other = torch.zeros_like(Qh).pin_memory()
    tp.tp_decode_host(f.handle, leaves, other, *outs[2], tp.TP_MMA_SYNC)
    tp.tp_set_stream(f.handle, new.cuda_stream)
    tp.tp_decode_host(f.handle, leaves, Qh, *outs[2], tp.TP_MMA_SYNC)
    f.sync()
    assert torch.equal(outs[2][0], want[0]) and torch.equal(outs[2][1], want[1])
    f.close()
