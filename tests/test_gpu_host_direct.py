"""Host-buffer decode calls whose results the merge writes to pinned memory
itself, or leaves to a download: bit-identical to the device-buffer call in
either case -- waiting after each call, back to back, small and large results,
one pinned and one pageable buffer, buffers at odd offsets, and the same pinned
buffers as before a call with others."""
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
