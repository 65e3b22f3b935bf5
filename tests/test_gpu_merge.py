"""GPU parity of the LSE merge over its whole range of partials per row: one
warp per row, rows shared by 2, 4 and 8 warps, fixed-size records (up to 15
partials) and the CSR, shares that are empty or longer than one 32-slot
chunk. Same oracle, bars and derived tolerance as test_gpu_parity.py."""
import pytest

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
