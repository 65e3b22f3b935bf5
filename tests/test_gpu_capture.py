"""Calls that carry host state into their launches (pool slots, tile words) are
refused while the tree's stream is captured into a CUDA graph, as they were
while that state went up in copies of its own: a replay would write a token's
old slot again, or read blocks that have changed hands. Refused, they launch
nothing and change nothing, and work again after the capture."""
import gc

import pytest
import torch

import paper_2508_17445_gb300 as tp
from test_gpu_parity import _built  # noqa: F401
from test_gpu_token_words import forest

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def refused(f, call):
    """`call` inside a capture of the tree's stream: refused, nothing of it in the graph."""
    side, x, graph = torch.cuda.Stream(), torch.zeros(1, device=DEV), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    tp.tp_set_stream(f.handle, side.cuda_stream)
    gc.collect()
    with torch.cuda.graph(graph, stream=side):
        x.add_(1)
        with pytest.raises(tp.TreepoError) as e:
            call()
    tp.tp_set_stream(f.handle, torch.cuda.current_stream().cuda_stream)
    assert e.value.code == "INVALID_ARG" and "captured" in str(e.value)
    del e  # (its traceback's frames hold the graph, which must not be collected inside a later capture)
    graph.replay()
    torch.cuda.synchronize()
    assert x.item() == 1.0


@pytest.mark.parametrize("n", [3, 5000])  # words in the launch, words in a device buffer
@pytest.mark.parametrize("first", [31, 32])  # inside the last block, and one more block each
def test_append_tokens(n, first):
    f, leaves, draw = forest(n, first)
    K, V = draw(n, 1), draw(n, 1)
    before = f.stats()["free_blocks"]
    refused(f, lambda: tp.tp_append_tokens(f.handle, leaves, K, V))
    assert f.stats()["free_blocks"] == before and f.node_info(leaves[0])["n_tokens"] == first
    f.append_tokens(leaves, K, V)
    Kg, Vg = (torch.empty((5 + first + 1, 1, 64), dtype=torch.bfloat16, device=DEV) for _ in range(2))
    assert tp.tp_debug_gather(f.handle, leaves[-1], Kg, Vg) == len(Kg)
    f.sync()
    assert torch.equal(Kg[-1], K[-1]) and torch.equal(Vg[-1], V[-1])
    f.close()


# a schedule that travels with the launch, and ones that are uploaded (the second with split rows)
@pytest.mark.parametrize("tokens,queries", [(40, 40), (3000, 3000), (9000, 2)])
def test_prefill(tokens, queries):
    f = tp.Forest(2, 1, 64, pool_blocks=512, device=DEV)
    g = torch.Generator(device=DEV).manual_seed(tokens)
    draw = lambda m, h: torch.randn((m, h, 64), generator=g, device=DEV).to(torch.bfloat16)  # noqa: E731
    r = f.add_root()
    f.append(r, draw(tokens, 1), draw(tokens, 1))
    Q = draw(queries, 2)
    want = f.prefill([r], [queries], Q)
    out = torch.empty_like(want[0]), torch.empty_like(want[1])
    refused(f, lambda: tp.tp_prefill(f.handle, [r], [queries], Q, *out))
    before = f.decode([r], Q[:1])
    refused(f, lambda: (tp.tp_prefill(f.handle, [r], [0], Q, *out),  # no queries: nothing to do, captured or not
                        f.decode([r], Q[:1], flags=tp.TP_DECODE_NO_CACHE, out=before)))
    tp.tp_prefill(f.handle, [r], [queries], Q, *out)
    f.sync()
    assert torch.equal(out[0], want[0]) and torch.equal(out[1], want[1])
    f.close()


def test_decode_that_has_to_change_the_schedule():
    f, leaves, draw = forest(4, 3)
    Q = draw(4, 2)
    f.decode(leaves, Q)
    out = torch.empty_like(Q), torch.empty((4, 2), device=DEV)
    for change in ("patch", "build"):
        if change == "patch":  # a segment append leaves the cached schedule's tile words one token behind
            f.append(leaves[1], draw(1, 1), draw(1, 1))
            which = leaves
        else:
            which = leaves[::-1]
        refused(f, lambda: f.decode(which, Q, out=out))
        f.decode(which, Q, out=out)
        want = f.decode(which, Q, flags=tp.TP_DECODE_NO_CACHE)
        f.decode(leaves, Q)
        f.sync()
        assert torch.equal(out[0], want[0]) and torch.equal(out[1], want[1])
    f.close()
