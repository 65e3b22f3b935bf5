"""The work that users of this library have it do, as measurable cases.

Each case goes through the public binding the way a sampling or training
program does: decode attention over a forest (one call per layer and token),
a segment's token loop (append one token per leaf, decode), decode with host
buffers, prefill of appended segments and of new prompts, a whole rollout of
Algorithm 1, and the tree advantage of a finished batch. Tree shapes, head
counts and lengths are those of the repository's workloads and tests, or
generic; K, V, Q are N(0, 1) in bf16, with the queries scaled by ``peak`` where
a case stands for the peaked attention of trained models.
"""
import math

import numpy as np
import torch

import paper_2508_17445_gb300 as tp

DEV = "cuda:0"
BLOCK = 32  # tokens per pool block
MAX_EVENTS = 1 << 13  # of a rollout


# ------------------------------------------------------------------ forests --
def _forest(prompts, lo, hi, branch, depth, segment, private=0, tail=0, heads=(28, 4, 128), shape="full", peak=1.0):
    """Case keys of a forest: ``prompts`` roots of lo..hi tokens; "full": every node forks into ``branch`` down to
    ``depth`` (segments of ``segment`` tokens), then ``private`` more segments on each leaf; "diverging": at each of
    ``depth`` boundaries a path forks into 1..4 (0.4/0.3/0.2/0.1, at most 32 alive) and stops with p = 0.1 after a
    segment. ``tail``: the last segment holds 1..tail tokens instead."""
    hq, hkv, hd = heads
    return dict(prompts=prompts, lo=lo, hi=hi, branch=branch, depth=depth, segment=segment, private=private, tail=tail,
                hq=hq, hkv=hkv, hd=hd, shape=shape, peak=peak)


def _trees(case):
    """The case's forest: per prompt (parent per node, tokens per node, leaves); node 0 is the root."""
    rng = np.random.default_rng(case["prompts"] * 7919 + case["segment"])
    out = []
    for _ in range(case["prompts"]):
        parent, tokens = [-1], [int(rng.integers(case["lo"], case["hi"] + 1))]
        if case["shape"] == "full":
            live = [0]
            for _d in range(case["depth"]):
                nxt = []
                for x in live:
                    for _k in range(case["branch"]):
                        parent.append(x)
                        tokens.append(case["segment"])
                        nxt.append(len(parent) - 1)
                live = nxt
            for x in live:
                tokens[x] += case["private"] * case["segment"]
        else:
            def fork(paths):
                draws = rng.choice(4, size=len(paths), p=[0.4, 0.3, 0.2, 0.1]) + 1
                res = []
                for i, (x, d) in enumerate(zip(paths, draws)):
                    k = max(1, min(int(d), 32 - len(res) - (len(paths) - i - 1)))
                    if k == 1:
                        res.append(x)
                        continue
                    for _k in range(k):
                        parent.append(x)
                        tokens.append(0)
                        res.append(len(parent) - 1)
                return res
            live = fork([0])
            for s in range(1, case["depth"] + 1):
                for x in live:
                    tokens[x] += case["segment"]
                if s == case["depth"]:
                    break
                keep = [x for x in live if rng.random() >= 0.1] or live[:1]
                live = fork(keep)
            # drop what no living path holds
            need = set()
            for x in live:
                while x != -1 and x not in need:
                    need.add(x)
                    x = parent[x]
            new = {x: i for i, x in enumerate(sorted(need))}
            parent, tokens, live = ([new.get(parent[x], -1) for x in sorted(need)], [tokens[x] for x in sorted(need)],
                                    [new[x] for x in live])
        if case["tail"]:
            for x in live:
                tokens[x] += int(rng.integers(1, case["tail"] + 1)) - (case["segment"] if case["depth"] else 0)
        out.append((parent, [max(t, 1 if p == -1 else 0) for p, t in zip(parent, tokens)], live))
    return out


def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + stream * 7919 + 17) % (1 << 62))


def _randn(shape, gen, scale=1.0):
    x = torch.randn(shape, generator=gen, device=DEV, dtype=torch.float32)
    return (x * scale if scale != 1.0 else x).to(torch.bfloat16)


def _tree_kv(case, seed, t, tokens):
    g = _gen(seed, 100 + t)
    shape = (sum(tokens), case["hkv"], case["hd"])
    return _randn(shape, g), _randn(shape, g)


def _queries(case, seed, n):
    return _randn((n, case["hq"], case["hd"]), _gen(seed, 1), case["peak"])


def _grow(case, seed, spare_blocks=8):
    """The forest on the GPU; returns it, the leaves and each tree's node ids."""
    trees = _trees(case)
    blocks = sum(-(-t // BLOCK) for _, tok, _ in trees for t in tok)
    f = tp.Forest(case["hq"], case["hkv"], case["hd"], pool_blocks=blocks + spare_blocks, device=DEV)
    leaves = []
    for t, (parent, tokens, live) in enumerate(trees):
        K, V = _tree_kv(case, seed, t, tokens)
        kids, ids, at = {}, {}, 0
        for x, p in enumerate(parent):
            kids.setdefault(p, []).append(x)
        for x, p in enumerate(parent):
            if p == -1:
                ids[x] = f.add_root()
            elif x not in ids:
                ids.update(zip(kids[p], f.fork(ids[p], len(kids[p]))))
            if tokens[x]:
                f.append(ids[x], K[at:at + tokens[x]], V[at:at + tokens[x]])
            at += tokens[x]
        leaves += [ids[x] for x in live]
    return f, leaves


def _paths(trees):
    """(tree, node rows' index ranges root first, path length) of every leaf."""
    for t, (parent, tokens, live) in enumerate(trees):
        start = np.concatenate([[0], np.cumsum(tokens)])
        for x in live:
            chain = []
            while x != -1:
                chain.append(x)
                x = parent[x]
            chain.reverse()
            yield t, [(int(start[c]), int(start[c + 1])) for c in chain], int(sum(tokens[c] for c in chain))


def _attend(q, k, v, vis=None):
    """fp64 attention: q [m][hq][hd] over k, v [s][hkv][hd]; vis [m]: row i sees the first vis[i] tokens."""
    m, hq, hd = q.shape
    hkv = k.shape[1]
    qd = q.double().view(m, hkv, hq // hkv, hd).permute(1, 0, 2, 3).reshape(hkv, -1, hd)
    s = qd @ k.double().permute(1, 2, 0) / math.sqrt(hd)
    if vis is not None:
        hide = torch.arange(k.shape[0], device=q.device)[None, :] >= vis[:, None]
        s = s.masked_fill(hide.repeat_interleave(hq // hkv, 0)[None], -math.inf)
    lse = torch.logsumexp(s, -1)
    o = torch.exp(s - lse[..., None]) @ v.double().permute(1, 0, 2)
    back = lambda x: x.view(hkv, m, hq // hkv, -1).permute(1, 0, 2, 3).reshape(m, hq, -1)  # noqa: E731
    return back(o), back(lse).squeeze(-1)


def _cat(outs):
    return tuple(torch.cat(x) for x in zip(*outs))


# -------------------------------------------------------------------- cases --
def listed():
    """One case per line of use; the forest cases are one layer's call."""
    return [
        # the smallest call: a prompt's eight short paths, single kv head (launches and host work)
        dict(name="decode_small", path="decode", **_forest(1, 128, 128, 2, 3, 32, tail=32, heads=(4, 1, 64))),
        # the end of a batch: the last four paths of one prompt, 14 segments long (few rows, long context)
        dict(name="decode_last_paths", path="decode", **_forest(1, 1000, 1000, 4, 1, 512, private=13, tail=512, peak=2.0)),
        # a 64-prompt batch, binary trees of 16 leaves, paths of ~2700 tokens
        dict(name="decode_batch", path="decode", **_forest(64, 256, 1024, 2, 4, 512)),
        # 14 segments of 512 with random branching and early stops: the largest decode call
        dict(name="decode_diverging", path="decode", **_forest(32, 1024, 1024, 0, 14, 512, shape="diverging")),
        # 64 leaves per prompt over a wide shared prefix, 64 query heads (stacked rows dominate)
        dict(name="decode_wide_prefix", path="decode", **_forest(8, 2048, 2048, 4, 3, 256, private=2, heads=(64, 8, 128), peak=2.0)),
        # a segment's token loop over 64 paths: fork, 40 x (append one token per leaf, decode), prune
        dict(name="token_loop", path="loop", steps=40, **_forest(4, 256, 1024, 2, 4, 128)),
        # a caller whose queries and results live in pinned host memory, 16-prompt batch
        dict(name="decode_host", path="decode_host", **_forest(16, 256, 1024, 2, 4, 512)),
        # one new prompt of an odd length: append and causal attention over it
        dict(name="prompt", path="prompt", **_forest(1, 717, 717, 0, 0, 0)),
        # a batch's new 512-token segments, 16 per prompt of 1024: the largest prefill call
        dict(name="segment_prefill", path="prefill", queries=512, **_forest(32, 1024, 1024, 16, 1, 512)),
        # ragged short segments (re-computed tails of different lengths) at head_dim 64
        dict(name="ragged_prefill", path="prefill", queries=0, **_forest(24, 33, 700, 3, 2, 150, tail=150, heads=(16, 2, 64), peak=2.0)),
        # a training step's rollout batch on a fresh forest, decode after every token
        dict(name="rollout", path="rollout", width=16, max_depth=4, steps=64, **_forest(8, 256, 1024, 2, 0, 64)),
        # the advantages of a 64-prompt batch of 16 trajectories each
        dict(name="advantage", path="advantage", prompts=64, width=16, depth=14),
    ]


_HEADS = [(4, 1, 64), (8, 2, 64), (16, 2, 64), (16, 2, 128), (28, 4, 128), (64, 8, 128), (12, 1, 128)]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)) )))))


def _cost(case):
    w = work(case)
    return w["bytes"] / 6e12 + w["flops"] / 1e15


def draw(rng):
    most = max(_cost(dict(c)) for c in listed() if c["name"] in ("decode_diverging", "segment_prefill"))
    while True:
        path = rng.choice(["decode", "decode", "decode", "decode", "loop", "decode_host", "prompt", "prefill", "prefill",
                           "rollout", "advantage"])
        heads = rng.choice(_HEADS)
        peak = rng.choice([1.0, 2.0, 3.0])
        if path == "advantage":
            return dict(path=path, prompts=_log(rng, 1, 256), width=rng.choice([4, 8, 16, 32]), depth=rng.randint(2, 28))
        lo = _log(rng, 1, 2048)
        hi = lo + rng.randrange(0, lo + 1)
        if path == "prompt":
            n = _log(rng, 1, 8192)
            return dict(path=path, **_forest(1, n, n, 0, 0, 0, heads=heads, peak=peak))
        if path == "rollout":
            return dict(path=path, width=rng.choice([4, 8, 16]), max_depth=rng.randint(1, 4), steps=_log(rng, 8, 64),
                        **_forest(_log(rng, 1, 16), lo, hi, rng.choice([1, 2, 4]), 0, 64, heads=heads))
        branch, depth = rng.choice([(1, 0), (1, 1), (2, 1), (2, 3), (2, 4), (3, 2), (4, 2), (4, 3), (16, 1)])
        seg = _log(rng, 16, 512)
        private = rng.choice([0, 0, 1, 3, 13]) if depth else 0
        shape = "diverging" if path == "decode" and rng.random() < 0.25 else "full"
        case = dict(path=path, **_forest(_log(rng, 1, 64), lo, hi, branch, rng.randint(3, 14) if shape == "diverging" else depth,
                                         seg, private, rng.choice([0, seg]) if depth and shape == "full" else 0, heads, shape, peak))
        if path == "loop":
            case["steps"] = _log(rng, 4, 64)
        if path == "prefill":
            case["queries"] = rng.choice([0, 1, seg])
        n_leaves = sum(len(t[2]) for t in _trees(case))
        if _cost(case) <= most and n_leaves <= (256 if path == "loop" else 2048):
            return case


# ------------------------------------------------------------ the token loop --
def _loop_prepare(case, seed):
    n = sum(len(t[2]) for t in _trees(case))
    steps, hq, hkv, hd = case["steps"], case["hq"], case["hkv"], case["hd"]
    f, parents = _grow(case, seed, spare_blocks=n * (-(-steps // BLOCK) + 1))
    for x in parents:
        f.fork(x, 1)  # another path stays below every parent, so pruning the loop's own frees only its tokens
    g = _gen(seed, 2)
    K, V = _randn((steps, n, hkv, hd), g), _randn((steps, n, hkv, hd), g)
    Q = _randn((steps, n, hq, hd), g, case["peak"])
    return dict(case=case, f=f, parents=parents, K=K, V=V, Q=Q, O=torch.empty_like(Q),
                LSE=torch.empty((steps, n, hq), dtype=torch.float32, device=DEV))


def _loop_run(s):
    f = s["f"]
    leaves = [f.fork(x, 1)[0] for x in s["parents"]]
    for t in range(s["case"]["steps"]):
        f.append_tokens(leaves, s["K"][t], s["V"][t])
        f.decode(leaves, s["Q"][t], out=(s["O"][t], s["LSE"][t]))
    for x in leaves:
        f.prune(x)
    return s["O"], s["LSE"]


# --------------------------------------------------------------- prefill rows --
def _prefill_counts(case, trees):
    """Query tokens of every leaf: ``queries`` > 0: that many, else a different odd count each (at most it holds)."""
    rng = np.random.default_rng(case["segment"] + 3)
    out = []
    for _, tokens, live in trees:
        for x in live:
            want = case["queries"] or int(rng.integers(1, tokens[x] + 1))
            out.append(min(want, tokens[x]))
    return out


# ------------------------------------------------------------------- rollout --
def _rollout_prompts(case):
    rng = np.random.default_rng(case["prompts"])
    return [int(x) for x in rng.integers(case["lo"], case["hi"] + 1, case["prompts"])]


def _rollout_levels(case):
    """Paths per depth of a prompt whose paths all run to the end (early stops and refills change it per seed)."""
    return [min(2 * case["branch"] ** d, case["width"]) for d in range(case["max_depth"])]


# ----------------------------------------------------------------- advantage --
def _advantage_table(case, seed):
    """Node table of a finished batch: per prompt ``width`` trajectories through binary trees ``depth`` deep, some
    stopped early; rewards 0 / 1, all equal for some prompts."""
    rng = np.random.default_rng(seed)
    parent, leaf, reward = [], [], []
    for _ in range(case["prompts"]):
        parent.append(-1)
        live, mine = [len(parent) - 1], []
        p = rng.choice([0.0, 0.3, 0.5, 0.8, 1.0])
        for d in range(case["depth"]):
            nxt = []
            room = case["width"] - len(mine)
            for i, x in enumerate(live):
                for _k in range(2 if len(nxt) + (len(live) - i) < room else 1):
                    parent.append(x)
                    nxt.append(len(parent) - 1)
            stop = [x for x in nxt if d + 1 == case["depth"] or rng.random() < 0.03]
            mine += stop
            live = [x for x in nxt if x not in set(stop)]
            if not live:
                break
        leaf += mine
        reward += [float(rng.random() < p) for _ in mine]
    return np.array(parent, np.int32), np.array(leaf, np.int32), np.array(reward, np.float32)


def _advantage_exact(parent, leaf, reward):
    total, count = np.zeros(len(parent)), np.zeros(len(parent))
    chains, root = [], []
    for x, r in zip(leaf, reward):
        chain, y = [], parent[x]
        while y != -1:
            chain.append(y)
            y = parent[y]
        chains.append(chain)
        root.append(chain[-1] if chain else -1)
        total[chain] += float(r)
        count[chain] += 1
    seen = {}
    for y, r in zip(root, reward):
        lo, hi = seen.get(y, (r, r))
        seen[y] = (min(lo, r), max(hi, r))
    ok = np.array([bool(c) and seen[y][0] != seen[y][1] for c, y in zip(chains, root)])
    a = np.array([np.mean(float(r) - total[c] / count[c]) if g else 0.0 for c, r, g in zip(chains, reward, ok)])
    n = int(ok.sum())
    mean, std = (float(a[ok].mean()), float(a[ok].std())) if n else (0.0, 0.0)
    adv = np.where(ok, a / std, 0.0) if std > 0 else np.zeros(len(a))
    return adv, np.array([n, mean, std, 0.0])


# ----------------------------------------------------------------- interface --
def prepare(case, seed):
    path = case["path"]
    if path == "loop":
        return _loop_prepare(case, seed)
    if path == "advantage":
        parent, leaf, reward = (torch.from_numpy(x).to(DEV) for x in _advantage_table(case, seed))
        ws = torch.empty(tp.tp_advantage_workspace_bytes(len(parent), len(leaf)), dtype=torch.uint8, device=DEV)
        return dict(case=case, parent=parent, leaf=leaf, reward=reward, ws=ws, adv=torch.empty_like(reward),
                    stats=torch.zeros(4, dtype=torch.float64, device=DEV))
    if path == "rollout":
        prompts = _rollout_prompts(case)
        blocks = sum(-(-p // BLOCK) for p in prompts)
        blocks += case["prompts"] * case["width"] * (3 * case["max_depth"]) * (-(-case["steps"] // BLOCK) + 1)
        params = tp.rollout_params(prompts, width=case["width"], max_depth=case["max_depth"], seg_tokens=case["steps"],
                                   arity=case["branch"], init_branches=2, p_eos=1 / 2048, p_boxed=0.03, p_fail=0.03,
                                   decode=1, seed=int(seed) & 0xffffffff)
        rows = case["prompts"] * case["width"]
        O = torch.zeros((rows, case["hq"], case["hd"]), dtype=torch.bfloat16, device=DEV)
        L = torch.zeros((rows, case["hq"]), dtype=torch.float32, device=DEV)
        # one decode call's outputs are copied out: the first segment's last token but two
        probe = tp.TpRolloutProbe(call=max(0, case["steps"] - 3), cap=rows, o=O.data_ptr(), lse=L.data_ptr())
        return dict(case=case, blocks=blocks, params=params, probe=probe, O=O, LSE=L)
    if path == "prompt":
        n = case["lo"]
        K, V = _tree_kv(case, seed, 0, [n])
        f = tp.Forest(case["hq"], case["hkv"], case["hd"], pool_blocks=-(-n // BLOCK) + 8, device=DEV)
        return dict(case=case, f=f, K=K, V=V, Q=_queries(case, seed, n))
    f, leaves = _grow(case, seed)
    s = dict(case=case, f=f, leaves=leaves)
    if path == "prefill":
        s["counts"] = _prefill_counts(case, _trees(case))
        s["Q"] = _queries(case, seed, sum(s["counts"]))
    else:
        s["Q"] = _queries(case, seed, len(leaves))
    if path == "decode_host":
        s["Q"] = s["Q"].cpu().pin_memory()
        s["out"] = (torch.empty(s["Q"].shape, dtype=torch.bfloat16).pin_memory(),
                    torch.empty(s["Q"].shape[:2], dtype=torch.float32).pin_memory())
    return s


def run(s):
    path = s["case"]["path"]
    if path == "decode":
        return s["f"].decode(s["leaves"], s["Q"])
    if path == "loop":
        return _loop_run(s)
    if path == "decode_host":
        out = s["f"].decode_host(s["leaves"], s["Q"], out=s["out"])
        s["f"].sync()  # the host results are valid only then
        return out
    if path == "prefill":
        return s["f"].prefill(s["leaves"], s["counts"], s["Q"])
    if path == "prompt":
        f = s["f"]
        r = f.add_root()
        f.append(r, s["K"], s["V"])
        out = f.prefill([r], [int(s["K"].shape[0])], s["Q"])
        f.prune(r)
        return out
    if path == "rollout":
        c = s["case"]
        with tp.Forest(c["hq"], c["hkv"], c["hd"], pool_blocks=s["blocks"], device=DEV) as f:
            events, stats = f.rollout(s["params"], cap_events=MAX_EVENTS, probe=s["probe"])
        log = np.zeros((MAX_EVENTS, 8), np.int64)  # how many there are depends on the draws
        log[:len(events)] = events
        return log, stats, s["O"], s["LSE"]
    tp.tp_tree_advantage(s["parent"], s["leaf"], s["reward"], s["adv"], s["stats"], s["ws"],
                         torch.cuda.current_stream().cuda_stream)
    return s["adv"], s["stats"]


def work(case):
    path = case["path"]
    if path == "advantage":
        t = _advantage_table(case, 0)
        return {"bytes": 4 * len(t[0]) + 12 * len(t[1]) + 32, "flops": 0}
    hq, hkv, hd = case["hq"], case["hkv"], case["hd"]
    token, query = 2 * hkv * hd * 2, hq * (hd * 2 + hd * 2 + 4)  # K and V of a token; Q, O and LSE of a query
    if path == "rollout":
        # a batch whose paths all reach the last depth: the decode calls read every living token once, and the prompts
        # and generated tokens are written once
        nbytes = flops = 0
        for p in _rollout_prompts(case):
            shared, above = p, p
            nbytes += p * token
            for n in _rollout_levels(case):
                for t in range(1, case["steps"] + 1):
                    nbytes += (shared + n * t) * token + n * (query + token)
                    flops += 4 * hd * hq * n * (above + t)
                shared += n * case["steps"]
                above += case["steps"]
        return {"bytes": nbytes, "flops": flops}
    trees = _trees(case)
    unique = sum(sum(t[1]) for t in trees)
    lengths = [n for _, _, n in _paths(trees)]
    if path == "loop":
        n, steps = len(lengths), case["steps"]
        nbytes = sum((unique + n * t) * token + n * (query + 2 * token) for t in range(1, steps + 1))
        return {"bytes": nbytes, "flops": sum(4 * hd * hq * (sum(lengths) + n * t) for t in range(1, steps + 1))}
    if path == "prompt":
        n = case["lo"]
        return {"bytes": n * (2 * token + query), "flops": 4 * hd * hq * (n * (n + 1) // 2)}
    if path == "prefill":
        counts = _prefill_counts(case, trees)
        seen = sum(m * n - m * (m - 1) // 2 for m, n in zip(counts, lengths))
        return {"bytes": unique * token + sum(counts) * query, "flops": 4 * hd * hq * seen}
    return {"bytes": unique * token + len(lengths) * query, "flops": 4 * hd * hq * sum(lengths)}


def tolerance(case):
    if case["path"] == "advantage":
        # fp64 sums in any order, rounded to fp32 once
        return {"rel": 1e-6, "max": 1e-5}
    # O is bf16 and its probabilities are rounded to bf16 before P.V (2e-3 to 3e-3 from 64 bits); the largest element is
    # one where terms cancel, against the output's root mean square. A rollout's events and counts are the same.
    return {"rel": 1e-2, "max": 0.1, "differ": 0.0}


def exact(case, seed):
    path = case["path"]
    if path == "rollout":
        return None  # the sampler's own draws decide what is attended to
    if path == "advantage":
        return _advantage_exact(*_advantage_table(case, seed))
    if _cost(case) > 0.02:
        return None
    trees = _trees(case)
    kv, outs = {}, []
    if path == "prompt":
        K, V = _tree_kv(case, seed, 0, [case["lo"]])
        Q = _queries(case, seed, case["lo"])
        return _cat([_attend(Q[i:i + 512], K, V, torch.arange(i + 1, min(i + 512, len(Q)) + 1, device=DEV))
                     for i in range(0, len(Q), 512)])
    if path == "loop":
        n, steps, hkv, hd = sum(len(t[2]) for t in trees), case["steps"], case["hkv"], case["hd"]
        g = _gen(seed, 2)
        LK, LV = _randn((steps, n, hkv, hd), g), _randn((steps, n, hkv, hd), g)
        Q = _randn((steps, n, case["hq"], hd), g, case["peak"])
    else:
        counts = _prefill_counts(case, trees) if path == "prefill" else None
        Q = _queries(case, seed, sum(counts) if counts else sum(len(t[2]) for t in trees))
    at = 0
    for i, (t, parts, n) in enumerate(_paths(trees)):
        if t not in kv:
            kv = {t: _tree_kv(case, seed, t, trees[t][1])}
        K, V = (torch.cat([x[a:b] for a, b in parts]) for x in kv[t])
        if path == "loop":
            K, V = torch.cat([K, LK[:, i]]), torch.cat([V, LV[:, i]])
            outs.append(_attend(Q[:, i], K, V, torch.arange(n + 1, n + steps + 1, device=DEV)))
        elif path == "prefill":
            m = counts[i]
            outs.append(_attend(Q[at:at + m], K, V, torch.arange(n - m + 1, n + 1, device=DEV)))
            at += m
        else:
            outs.append(_attend(Q[i:i + 1], K, V))
    if path == "loop":
        return tuple(torch.stack(x, 1) for x in zip(*outs))
    return _cat(outs)
