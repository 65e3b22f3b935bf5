"""Token steps whose words (pool slots, schedule patches) travel with the launch:
numbers of leaves on both sides of each parameter size (512 and 4096 words,
then a device buffer), block boundaries, a leaf list other than the cached
schedule's, and a stream changed between a decode and the next append."""
import numpy as np
import pytest
import torch

import paper_2508_17445_gb300 as tp
from test_gpu_parity import _built  # noqa: F401

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def forest(n, first, heads=(2, 1, 64)):
    """n leaves of `first` tokens under one root of 5 tokens."""
    f = tp.Forest(*heads, pool_blocks=3 * n + 64, device=DEV)
    g = torch.Generator(device=DEV).manual_seed(n)
    draw = lambda m, h: torch.randn((m, h, heads[2]), generator=g, device=DEV).to(torch.bfloat16)  # noqa: E731
    r = f.add_root()
    f.append(r, draw(5, heads[1]), draw(5, heads[1]))
    leaves = f.fork(r, n)
    for x in leaves:
        f.append(x, draw(first, heads[1]), draw(first, heads[1]))
    return f, leaves, draw


# 3 n and 4 n words against 512 and 4096
@pytest.mark.parametrize("n", [1, 2, 128, 129, 170, 171, 1024, 1025, 1365, 1366])
@pytest.mark.parametrize("first", [1, 30])
def test_appended_tokens_and_patched_schedule(n, first):
    f, leaves, draw = forest(n, first)
    Q = draw(n, 2)
    f.decode(leaves, Q)  # caches the schedule
    last = []
    for step in range(4):  # first = 30: crosses into a new block
        K, V = draw(n, 1), draw(n, 1)
        f.append_tokens(leaves, K, V)
        last.append((K, V))
        O, LSE = f.decode(leaves, Q)
        O2, LSE2 = f.decode(leaves, Q, flags=tp.TP_DECODE_NO_CACHE)
        f.decode(leaves, Q)  # back to the cached flags
        f.sync()
        assert torch.equal(O, O2) and torch.equal(LSE, LSE2)
    for i in {0, n // 2, n - 1}:
        Kg, Vg = (torch.empty((5 + first + 4, 1, 64), dtype=torch.bfloat16, device=DEV) for _ in range(2))
        assert tp.tp_debug_gather(f.handle, leaves[i], Kg, Vg) == len(Kg)
        f.sync()
        for step, (K, V) in enumerate(last):
            assert torch.equal(Kg[5 + first + step], K[i]) and torch.equal(Vg[5 + first + step], V[i])
    f.close()


def test_append_to_other_leaves_than_the_cached_ones():
    f, leaves, draw = forest(40, 3)
    Q = draw(40, 2)
    f.decode(leaves, Q)
    for some in (leaves[:7], leaves[::-1], [leaves[3]], leaves):
        f.append_tokens(some, draw(len(some), 1), draw(len(some), 1))
        O, LSE = f.decode(leaves, Q)
        O2, LSE2 = f.decode(leaves, Q, flags=tp.TP_DECODE_NO_CACHE)
        f.decode(leaves, Q)
        f.sync()
        assert torch.equal(O, O2) and torch.equal(LSE, LSE2)
    f.close()


# The decode still waits on the old stream while the new one appends: its schedule must not change under it, so the
# append carries no patch, and the next decode makes up for it.
def test_stream_changed_between_decode_and_append():
    f, leaves, draw = forest(64, 3)
    Q = draw(64, 2)
    streams = torch.cuda.Stream(), torch.cuda.Stream()
    new = lambda: (torch.empty_like(Q), torch.empty((64, 2), device=DEV))  # noqa: E731
    tp.tp_set_stream(f.handle, streams[0].cuda_stream)
    for k in range(6):
        old, s = streams[k & 1], streams[~k & 1]
        K, V = draw(64, 1), draw(64, 1)
        want, got = new(), new()
        torch.cuda.synchronize()
        f.decode(leaves, Q, out=want)  # caches or patches the schedule for the tokens of now
        f.sync()
        with torch.cuda.stream(old):
            torch.cuda._sleep(20_000_000)
        f.decode(leaves, Q, out=got)
        tp.tp_set_stream(f.handle, s.cuda_stream)
        f.append_tokens(leaves, K, V)
        s.wait_stream(old)
        after, fresh = new(), new()
        f.decode(leaves, Q, out=after)
        f.decode(leaves, Q, flags=tp.TP_DECODE_NO_CACHE, out=fresh)
        torch.cuda.synchronize()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        assert torch.equal(after[0], fresh[0]) and torch.equal(after[1], fresh[1])
        assert not torch.equal(after[0], want[0])
    f.close()


# rollout token steps: 4 words a row, rows up to prompts x 16
@pytest.mark.parametrize("prompts", [8, 9, 64, 65])
def test_rollout_steps(prompts):
    def run(flags):
        rows = prompts * 16
        f = tp.Forest(2, 1, 64, pool_blocks=prompts * 16 * 8, device=DEV)
        O = torch.zeros((rows, 2, 64), dtype=torch.bfloat16, device=DEV)
        L = torch.zeros((rows, 2), device=DEV)
        nr = np.zeros(1, np.int32)
        p = tp.rollout_params([7] * prompts, width=16, max_depth=2, seg_tokens=5, arity=1, init_branches=16, decode=1,
                              decode_flags=flags, seed=3)
        probe = tp.TpRolloutProbe(call=4, cap=rows, o=O.data_ptr(), lse=L.data_ptr(), n_rows=nr.ctypes.data)
        ev, _ = f.rollout(p, probe=probe)
        f.sync()
        f.close()
        assert nr[0] == rows
        return ev, O, L
    a, b = run(0), run(tp.TP_DECODE_NO_CACHE)
    np.testing.assert_array_equal(a[0], b[0])
    assert torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
