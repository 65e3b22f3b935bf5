"""GPU parity of the LSE merge over its whole range of partials per row: one
warp per row, rows shared by 2, 4 and 8 warps, fixed-size records (up to 15
partials) and the CSR, shares that are empty or longer than one 32-slot
chunk, partials that are infinite. Same oracle, bars and derived tolerance as test_gpu_parity.py."""
import pytest
import torch

import paper_2508_17445_gb300 as tp
import workloads
from test_gpu_parity import _built, run_and_compare  # noqa: F401  (the fixture builds the library)

pytestmark = pytest.mark.gpu


# paths of these many tokens: 1 partial up to several hundred per row
LENGTHS = [1, 127, 129, 640, 1152, 15 * 128, 15 * 128 + 1, 2177, 33 * 128, 8500, 40000]


@pytest.mark.parametrize("tokens", LENGTHS)
@pytest.mark.parametrize("heads", [workloads.Heads(4, 1, 64), workloads.Heads(12, 1, 128), workloads.Heads(64, 8, 128)])
def test_one_path(tokens, heads):
    run_and_compare(workloads.single_path(seed=tokens, lengths=(tokens,), heads=heads))


# several rows per block with different numbers of partials (a share of a row
# with fewer partials than warps is empty)
@pytest.mark.parametrize("heads", [workloads.Heads(4, 1, 64), workloads.Heads(28, 4, 128)])
@pytest.mark.parametrize("leaf_tokens", [(1, 1, 1), (5000, 3, 700), (2500, 2500, 2500, 1, 60)])
def test_rows_with_different_partials(heads, leaf_tokens):
    run_and_compare(workloads.shared_prompt(seed=3, prompt=900, n_leaves=len(leaf_tokens), leaf_tokens=leaf_tokens,
                                            heads=heads))


# whole tiles only, and infinite values in the first one: 2 partials up to several hundred, so full and short batches of
# them in every share of a row
@pytest.mark.parametrize("tokens", [192, 640, 1152, 2176, 8512, 40000])
@pytest.mark.parametrize("flags", [0, tp.TP_MMA_SYNC, tp.TP_DECODE_NO_SHARE])
def test_infinite_partials(tokens, flags):
    g = torch.Generator(device="cuda:0").manual_seed(tokens)
    K, V = (torch.randn((tokens, 2, 128), generator=g, device="cuda:0").to(torch.bfloat16) for _ in range(2))
    V[10, 0, 5], V[20, 1, 7] = float("inf"), float("-inf")
    f = tp.Forest(8, 2, 128, pool_blocks=tokens // 32 + 8, device="cuda:0")
    r = f.add_root()
    f.append(r, K, V)
    for n in (1, 3, 40):  # rows shared by eight warps down to one
        Q = torch.randn((n, 8, 128), generator=g, device="cuda:0").to(torch.bfloat16)
        O, _ = f.decode([r] * n, Q, flags=flags)
        f.sync()
        assert (O[:, :4, 5] == float("inf")).all() and (O[:, 4:, 7] == float("-inf")).all()
        O[:, :4, 5], O[:, 4:, 7] = 0, 0
        assert torch.isfinite(O.float()).all()
    f.close()
