"""The tree advantage over the sizes where its launch changes: one cluster (up
to 1024 outputs) and a grid, the last output of a CTA, one to four warps of
outputs per CTA, and more outputs than the grid has threads (then four
launches); paths deeper than the ancestors a thread keeps; node tables far
larger than what the outputs reach; rewards that are not finite. Oracle and
tolerance of test_gpu_rollout.py (fp64 accumulation, fp32 output: 1e-6
(|adv| + 1))."""
import numpy as np
import pytest
import torch

import paper_2508_17445_gb300 as tp
from test_gpu_parity import _built  # noqa: F401
from test_gpu_rollout import check_advantage, run_advantage

pytestmark = pytest.mark.gpu


def flat_trees(n_out, width, depth, seed):
    """Prompts of `width` trajectories: a shared chain of depth // 2, then one of its own each."""
    rng = np.random.default_rng(seed)
    parent, leaf = [], []
    while len(leaf) < n_out:
        parent.append(-1)
        top = len(parent) - 1
        for _ in range(depth // 2):
            parent.append(top)
            top = len(parent) - 1
        for _ in range(min(width, n_out - len(leaf))):
            x = top
            for _ in range(max(1, depth - depth // 2)):
                parent.append(x)
                x = len(parent) - 1
            leaf.append(x)
    return np.array(parent, np.int32), leaf, rng.random(n_out).round(2)


@pytest.mark.parametrize("n_out", [1, 2, 31, 32, 33, 128, 256, 257, 1023, 1024, 1025, 9728, 9729, 19457, 38912, 38913])
def test_outputs_per_launch(n_out):
    check_advantage(*flat_trees(n_out, 16, 3, n_out))


@pytest.mark.parametrize("depth", [1, 63, 64, 65, 66, 200])
def test_deep_paths(depth):
    check_advantage(*flat_trees(100, 7, depth, depth))
    check_advantage(*flat_trees(1100, 7, depth, depth))


def test_all_equal_and_negative_rewards():
    parent, leaf, reward = flat_trees(64, 16, 4, 1)
    check_advantage(parent, leaf, np.full(64, 0.25))
    reward = np.where(np.arange(64) < 16, -3.5, reward - 0.5)  # the first prompt's are all equal
    check_advantage(parent, leaf, reward)


# one output of depth 600 among shallow ones whose A_i are all equal: the mean of A_i is ~sqrt(n) times its spread, where
# one-pass statistics lose most
@pytest.mark.parametrize("n_out", [1000, 1100, 20000])
def test_one_deep_output_among_shallow_ones(n_out):
    parent, leaf = [-1], []
    for _ in range(n_out - 1):
        parent.append(0)
        leaf.append(len(parent) - 1)
    x = 0
    for _ in range(600):
        parent.append(x)
        x = len(parent) - 1
    check_advantage(parent, leaf + [x], [0.0] * (n_out - 1) + [1.0])


# the four launches' answer, whichever launch a call takes: no advantages once a counted A_i is not finite, the deviation
# says so, and a query whose rewards are all the same value stays left out
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("n_out", [64, 1100, 38913])
def test_rewards_that_are_not_finite(n_out, value):
    parent, leaf, reward = flat_trees(n_out, 16, 4, 2)
    reward[:16] = value  # the first prompt's are all equal: rejected
    if not np.isnan(value):
        check_advantage(parent, leaf, reward)
    reward[20] = value
    adv, stats = run_advantage(parent, leaf, reward)
    assert (adv == 0).all() and np.isnan(stats[2]) and stats[3] == 0
    # alone in every group of its own: beside an output that ends at the root and forms no group
    parent, leaf, reward = list(parent) + [-1], list(leaf), list(np.where(np.isfinite(reward), reward, 0.0))
    parent.append(len(parent) - 1)
    adv, stats = run_advantage(parent, leaf + [len(parent) - 2, len(parent) - 1], reward + [0.0, value])
    assert (adv == 0).all() and np.isnan(stats[2])


# the outputs reach a small part of the table, and the workspace holds another call's remains
@pytest.mark.parametrize("n_out", [1, 40, 1024, 1025, 9000])
def test_large_node_table(n_out):
    rng = np.random.default_rng(n_out)
    parent, leaf, reward = flat_trees(n_out, 16, 5, n_out)
    n_nodes = 300_000
    ids = rng.permutation(n_nodes)[:len(parent)].astype(np.int32)
    table = np.full(n_nodes, -1, np.int32)
    table[ids] = np.where(parent < 0, -1, ids[parent])
    want = check_advantage(table, ids[leaf], reward)
    P, L = torch.from_numpy(table).cuda(), torch.from_numpy(ids[leaf]).cuda()
    R = torch.tensor(reward, dtype=torch.float32, device="cuda:0")
    ws = torch.full((tp.tp_advantage_workspace_bytes(n_nodes, n_out),), 255, dtype=torch.uint8, device="cuda:0")
    adv, stats = torch.zeros(n_out, device="cuda:0"), torch.zeros(4, dtype=torch.float64, device="cuda:0")
    for _ in range(2):
        tp.tp_tree_advantage(P, L, R, adv, stats, ws)
        torch.cuda.synchronize()
        # the sums' order differs from call to call: fp64 rounding
        assert np.abs(adv.cpu().numpy() - want).max() <= 1e-6
