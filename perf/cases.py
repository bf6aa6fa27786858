"""The work a decode loop gives this library, as cases that can be timed and compared.

A round of entropy-guided speculative decoding expands a tree of draft tokens from vocabulary-sized logits,
verifies it with tree-masked attention over a paged bf16 cache, accepts the longest matching path and compacts
the cache.  The cases below are those calls as a program makes them: outputs and workspaces kept between calls,
everything on the current stream, no host round trip.  Two are whole rounds.

A case's `kind`:
  expand     sage_expand_topk (draft side with the token gather, or target side without), or its static variant
  grow       dynamic tree construction level by level, acceptance and the acceptance history
  attention  sage_tree_attention for one layer (a model's forward calls it once per layer) or stacked layers
  compact    sage_accept followed by sage_compact_kv
  round      all of the above in order, the tree from a template hand-over or grown on the device

Shapes are those of the repository's workloads: 64 query heads over 8 KV heads (a target of 72B parameters) or
fewer query heads per group (a draft-sized model), head dimension 128, pages of 64 tokens, vocabulary 152064 or
32000, trees of (depth, width, nodes) = (8, 2, 24), (6, 3, 36), (4, 6, 48), (3, 10, 60), chains, up to 64 nodes.
"""
import heapq
import math

import numpy as np
import torch

import paper_2602_00523_b200 as sage

HEAD_DIM, PAGE, CAP = 128, 64, sage.SAGE_MAX_NODES
TEMPLATES = [(8, 2, 24), (6, 3, 36), (4, 6, 48), (3, 10, 60)]
THRESHOLDS = [0.8, 0.4, 0.1]
MAX_PATH = 9


def listed():
    return [
        # --- logits side
        # Smallest call: the draft's candidates for a 15-node tree over a small vocabulary.
        dict(name="expand_tiny", kind="expand", rows=15, vocab=32000, k=4, k_entropy=4, trees="8x2x15", batch=1,
             style="mixed", static=False),
        # A draft's expansion in every round: 60 nodes, ten candidates each, and the tokens of the tree.
        dict(name="expand_draft_60", kind="expand", rows=60, vocab=152064, k=10, k_entropy=10, trees="3x10x60",
             batch=1, style="high", static=False),
        # The target's greedy tokens for a batch of sixteen trees of 24 to 60 nodes (672 rows).
        dict(name="expand_target_serving", kind="expand", rows=672, vocab=152064, k=1, k_entropy=1, trees="",
             batch=0, style="mixed", static=False),
        # --- trees
        # Growing sixteen sequences' trees level by level between draft passes, and the history of acceptance.
        dict(name="grow_batch16", kind="grow", batch=16, levels=8, k=10, n_max=60),
        # --- attention, one layer at a time
        # Draft-side attention: small group of query heads, short context, a tree of ten nodes.
        dict(name="attention_draft_2k", kind="attention", layers=1, batch=1, ctx_min=2048, ctx_max=2048,
             trees="4x3x10", q_heads=32, kv_heads=8, capacity=False),
        # One layer of the target at a video-length context with the widest template.
        dict(name="attention_layer_16k", kind="attention", layers=1, batch=1, ctx_min=16384, ctx_max=16384,
             trees="3x10x60", q_heads=64, kv_heads=8, capacity=False),
        # One layer of batched serving: sixteen ragged sequences, each with its own template.
        dict(name="attention_serving16", kind="attention", layers=1, batch=16, ctx_min=1024, ctx_max=8192,
             trees="mix", q_heads=64, kv_heads=8, capacity=False),
        # --- attention, all layers of the target in one launch
        # A chain of nine (draft depth eight) in node arrays of full capacity, as the device-side loop keeps them.
        dict(name="attention_chain_80", kind="attention", layers=80, batch=1, ctx_min=16384, ctx_max=16384,
             trees="8x1x9", q_heads=64, kv_heads=8, capacity=True),
        # The deep and narrow template.
        dict(name="attention_deep_80", kind="attention", layers=80, batch=1, ctx_min=16384, ctx_max=16384,
             trees="8x2x24", q_heads=64, kv_heads=8, capacity=False),
        # --- acceptance and cache update for four sequences and all layers
        dict(name="compact_batch4", kind="compact", layers=80, batch=4, ctx_min=1000, ctx_max=3000, trees="mix",
             kv_heads=8),
        # --- whole rounds
        # A chat-length context; the tree is grown on the device within node arrays of full capacity.
        dict(name="round_grown_4k", kind="round", layers=80, ctx=4096, trees="grown", rows=CAP, vocab=152064),
        # A video-length context with the widest template; the next tree is handed over by the entropy.
        dict(name="round_16k_video", kind="round", layers=80, ctx=16384, trees="3x10x60", rows=60, vocab=152064),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _some_tree(rng):
    depth, width = rng.randint(1, 8), rng.randint(1, 10)
    return "%dx%dx%d" % (depth, width, rng.randint(depth + 1, CAP))


def draw(rng):
    kind = rng.choice(["expand", "expand", "expand", "grow", "attention", "attention", "attention", "attention",
                       "compact", "round"])
    if kind == "expand":
        vocab = rng.choice([32000, 128256, 152064, _log_int(rng, 1000, 160000)])
        k, k_entropy = rng.choice([(1, 1), (2, 10), (4, 4), (10, 10), (rng.randint(1, 16), rng.randint(1, 16))])
        style = rng.choice(["low", "high", "mixed", "steps"])
        if rng.random() < 0.5:
            tree = _some_tree(rng)
            batch = _log_int(rng, 1, 16)
            rows = batch * len(_tree(tree)[0])
            return dict(kind=kind, rows=rows, vocab=vocab, k=max(k, int(tree.split("x")[1])), k_entropy=k_entropy,
                        trees=tree, batch=batch, style=style, static=False)
        rows = _log_int(rng, 1, 960)
        return dict(kind=kind, rows=rows, vocab=vocab, k=k, k_entropy=k_entropy, trees="", batch=0, style=style,
                    static=rows <= 600 and rng.random() < 0.25)
    if kind == "grow":
        return dict(kind=kind, batch=_log_int(rng, 1, 64), levels=rng.randint(2, 8), k=rng.choice([4, 8, 10, 16]),
                    n_max=rng.randint(16, CAP))
    if kind == "attention":
        q_heads, kv_heads = rng.choice([(64, 8), (64, 8), (64, 8), (32, 8), (16, 8), (8, 8), (8, 1), (28, 7), (32, 16)])
        batch = rng.choice([1, 1, _log_int(rng, 1, 40)])
        layers = rng.choice([1, 1, 1, _log_int(rng, 1, 80)])
        ctx_max = _log_int(rng, 64, 32768)
        while layers * batch * ctx_max * kv_heads > 80 * 16384 * 8:       # no dearer than the largest listed case
            layers, batch = max(1, layers // 2), (batch if layers > 1 else max(1, batch // 2))
        ctx_min = ctx_max if batch == 1 else max(16, ctx_max // rng.randint(1, 8))
        trees = "mix" if batch > 1 and rng.random() < 0.6 else _some_tree(rng)
        return dict(kind=kind, layers=layers, batch=batch, ctx_min=ctx_min, ctx_max=ctx_max, trees=trees,
                    q_heads=q_heads, kv_heads=kv_heads, capacity=batch == 1 and rng.random() < 0.3)
    if kind == "compact":
        batch, layers = _log_int(rng, 1, 32), _log_int(rng, 1, 80)
        ctx_max = _log_int(rng, 64, min(8192, 80 * 8192 // (batch * layers) + 128))
        return dict(kind=kind, layers=layers, batch=batch, ctx_min=max(16, ctx_max // 2), ctx_max=ctx_max,
                    trees=rng.choice(["mix", _some_tree(rng)]), kv_heads=rng.choice([8, 8, 1, 4]))
    trees = rng.choice(["grown", "%dx%dx%d" % rng.choice(TEMPLATES)])
    return dict(kind=kind, layers=rng.choice([28, 32, 48, 64, 80]), ctx=_log_int(rng, 500, 16384), trees=trees,
                rows=CAP if trees == "grown" else int(trees.split("x")[2]), vocab=rng.choice([152064, 128256, 32000]))


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _tree(shape):
    """(parent, rank) of a "depth x width x nodes" tree: the chain of first candidates down to `depth`, then the
    likeliest further nodes (a candidate of rank r counts 0.6 ** r), level by level."""
    depth, width, nodes = (int(v) for v in shape.split("x"))
    chosen, heap = {(0,) * i: 1.0 for i in range(min(depth, nodes - 1) + 1)}, []

    def offer(path):
        if len(path) < depth:
            for r in range(width):
                if path + (r,) not in chosen:
                    heapq.heappush(heap, (-chosen[path] * 0.6 ** r, path + (r,)))

    for path in list(chosen):
        offer(path)
    while len(chosen) < nodes and heap:
        score, path = heapq.heappop(heap)
        if path not in chosen:
            chosen[path] = -score
            offer(path)
    order = sorted(chosen, key=lambda p: (len(p), p))
    at = {p: i for i, p in enumerate(order)}
    return [-1] + [at[p[:-1]] for p in order[1:]], [0] + [p[-1] for p in order[1:]]


def _trees(shape, batch):
    return [_tree("%dx%dx%d" % TEMPLATES[b % 4] if shape == "mix" else shape) for b in range(batch)]


def _i32(values):
    return torch.tensor(values, dtype=torch.int32, device="cuda")


def _packed(trees):
    offsets = [0]
    for t in trees:
        offsets.append(offsets[-1] + len(t[0]))
    return {"parent": _i32([v for t in trees for v in t[0]]), "rank": _i32([v for t in trees for v in t[1]]),
            "node_offsets": _i32(offsets)}


def _lengths(case):
    """Prefix lengths of a batch, spread over [ctx_min, ctx_max], the same for every seed."""
    r = np.random.RandomState(case["batch"] * 7 + case["ctx_max"])
    lens = r.randint(case["ctx_min"], case["ctx_max"] + 1, case["batch"])
    lens[0] = case["ctx_max"]
    return [int(v) for v in lens]


def _logits(gen, rows, vocab, style):
    x = torch.randn(rows, vocab, generator=gen, device="cuda")
    kind = torch.randint(0, 3, (rows, 1), generator=gen, device="cuda") if style == "mixed" else torch.full(
        (rows, 1), {"low": 0, "high": 1, "steps": 2}[style], device="cuda")
    x = torch.where(kind == 1, x * 0.5, x)
    # peaks: one far above the rest (a confident draft), none, or eight in steps of one
    n = min(8, vocab)
    at = torch.randint(0, vocab // n, (rows, n), generator=gen, device="cuda") + torch.arange(n, device="cuda") * (vocab // n)
    top = x.amax(dim=1, keepdim=True)
    lone = top + 6 + 4 * torch.rand(rows, 1, generator=gen, device="cuda")
    steps = top + 10 - torch.arange(n, device="cuda")
    first = torch.arange(n, device="cuda") == 0
    old = x.gather(1, at)
    return x.scatter_(1, at, torch.where((kind == 0) & first, lone, torch.where(kind == 2, steps, old)))


def _target_logits(gen, draft, k):
    """The target agrees with the draft's first candidate of a node four times in five, else with another one or none."""
    rows, vocab = draft.shape
    best = torch.topk(draft, max(k, 2), dim=1).indices
    u = torch.rand(rows, generator=gen, device="cuda")
    other = torch.randint(0, vocab, (rows,), generator=gen, device="cuda")
    want = torch.where(u < 0.8, best[:, 0], torch.where(u < 0.92, best[:, 1], other))
    x = torch.randn(rows, vocab, generator=gen, device="cuda")
    return x.scatter_(1, want[:, None], x.amax(dim=1, keepdim=True) + 6)


def _cache(gen, layers, lengths, nodes, kv_heads):
    """Paged pools with an eighth of spare pages, pages in random order, the first two fifths of every sequence
    visual tokens of larger magnitude."""
    need = [-(-(l + n) // PAGE) for l, n in zip(lengths, nodes)]
    pages = int(math.ceil(sum(need) * 1.125))
    order = torch.randperm(pages, generator=gen, device="cuda").to(torch.int32)
    table = torch.full((len(need), max(need)), -1, dtype=torch.int32, device="cuda")
    visual, at = [], 0
    for b, n in enumerate(need):
        table[b, :n] = order[at:at + n]
        visual.append(order[at:at + int(0.4 * n)].long())
        at += n
    pools = []
    for _ in range(2):
        pool = torch.empty(layers, pages, kv_heads, PAGE, HEAD_DIM, dtype=torch.bfloat16, device="cuda")
        for layer in range(layers):
            pool[layer].normal_(generator=gen)
            pool[layer, torch.cat(visual)] *= 1.5
        pools.append(pool)
    return {"k": pools[0], "v": pools[1], "table": table, "seq_len": _i32(lengths), "prefix": _i32(lengths)}


def _bytes(n):
    return torch.empty(max(16, n), dtype=torch.uint8, device="cuda")


def _expand_out(rows, k, tree_nodes):
    o = {"topk_idx": torch.empty(rows, k, dtype=torch.int32, device="cuda"),
         "topk_logprob": torch.empty(rows, k, device="cuda")}
    for name in ("entropy_full", "entropy_topk", "alpha", "lse"):
        o[name] = torch.empty(rows, device="cuda")
    if tree_nodes:
        o["draft_token"] = torch.empty(tree_nodes, dtype=torch.int32, device="cuda")
    return o


def _grown(batch):
    """Node slots of trees that are grown on the device; node 0 of every sequence is its root."""
    t = {n: torch.zeros(batch * CAP, dtype=torch.int32, device="cuda") for n in ("parent", "rank", "depth", "token")}
    t["parent"].fill_(-1)
    t["cum_logprob"] = torch.zeros(batch * CAP, device="cuda")
    t["n_nodes"], t["frontier_begin"] = _i32([1] * batch), _i32([0] * batch)
    return t


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = {"case": case, "status": sage.new_status()}
    kind = case["kind"]
    if kind == "expand":
        rows, vocab, k = case["rows"], case["vocab"], case["k"]
        trees = _trees(case["trees"], case["batch"]) if case["trees"] else []
        s.update(logits=_logits(gen, rows, (vocab + 3) // 4 * 4, case["style"])[:, :vocab], tree={},
                 ws=_bytes(sage.sage_expand_topk_workspace_size(rows, vocab)),
                 out=_expand_out(rows, k, sum(len(t[0]) for t in trees)))
        if trees:
            s["tree"] = dict(_packed(trees), root_token=torch.randint(0, vocab, (len(trees),), generator=gen, device="cuda",
                                                                      dtype=torch.int32))
    elif kind == "grow":
        batch, k = case["batch"], case["k"]
        rows = batch * CAP
        lp = torch.log_softmax(torch.randn(rows, k, generator=gen, device="cuda") * 2, dim=1)
        s.update(idx=torch.randint(0, 152064, (rows, k), generator=gen, device="cuda", dtype=torch.int32),
                 logprob=lp.sort(dim=1, descending=True).values.contiguous(),
                 alpha=torch.rand(batch, generator=gen, device="cuda"), policy=sage.make_policy(THRESHOLDS), tree=_grown(batch),
                 history=sage.make_history_policy(), window=torch.zeros(batch, 10, dtype=torch.int32, device="cuda"),
                 count=_i32([0] * batch), d_max=torch.full((batch,), 8.0, device="cuda"),
                 path_len=torch.randint(1, MAX_PATH + 1, (batch,), generator=gen, device="cuda", dtype=torch.int32))
    elif kind == "attention":
        trees = _trees(case["trees"], case["batch"])
        s.update(_packed(trees))
        nodes = [len(t[0]) for t in trees]
        s.update(_cache(gen, case["layers"], _lengths(case), nodes, case["kv_heads"]))
        held = CAP if case["capacity"] else sum(nodes)
        if held > sum(nodes):
            s["parent"] = torch.cat([s["parent"], torch.full((held - sum(nodes),), -1, dtype=torch.int32, device="cuda")])
        q = torch.empty(case["layers"], held, case["q_heads"], HEAD_DIM, dtype=torch.bfloat16, device="cuda")
        s.update(q=q.normal_(generator=gen), out=torch.zeros_like(q),
                 ws=_bytes(sage.sage_tree_attention_workspace_size(case["layers"], case["batch"], held, case["q_heads"],
                                                                   case["kv_heads"], HEAD_DIM, s["table"].shape[1])))
    elif kind == "compact":
        trees = _trees(case["trees"], case["batch"])
        s.update(_packed(trees))
        nodes = [len(t[0]) for t in trees]
        s.update(_cache(gen, case["layers"], _lengths(case), nodes, case["kv_heads"]))
        # the target takes the first or the second candidate of most nodes: siblings carry their rank as token
        s.update(draft=s["rank"].clone(), out={},
                 target=(torch.rand(sum(nodes), generator=gen, device="cuda") * 1.5).to(torch.int32))
    else:
        rows, vocab, layers, k = case["rows"], case["vocab"], case["layers"], 10
        grown = case["trees"] == "grown"
        trees = [] if grown else [_tree(case["trees"])]
        s.update(_cache(gen, layers, [case["ctx"]], [rows], 8))
        draft = _logits(gen, rows, vocab, "steps" if grown else "mixed")
        q = torch.empty(layers, rows, 64, HEAD_DIM, dtype=torch.bfloat16, device="cuda")
        s.update(draft=draft, target=_target_logits(gen, draft, k), q=q.normal_(generator=gen), attention=torch.zeros_like(q),
                 policy=sage.make_policy(THRESHOLDS), alpha_row=_i32([0]), root=_i32([seed % 1000]),
                 ws_topk=_bytes(sage.sage_expand_topk_workspace_size(rows, vocab)),
                 ws=_bytes(sage.sage_tree_attention_workspace_size(layers, 1, rows, 64, 8, HEAD_DIM, s["table"].shape[1])),
                 out_draft=_expand_out(rows, k, 0 if grown else rows), out_target=_expand_out(rows, 1, 0), out_accept={},
                 alpha_before=torch.rand(1, generator=gen, device="cuda"), history=sage.make_history_policy(),
                 window=torch.zeros(1, 10, dtype=torch.int32, device="cuda"), count=_i32([0]),
                 d_max=torch.full((1,), 8.0, device="cuda"))
        if grown:
            s.update(tree=_grown(1), node_offsets=_i32([0, 1]))
            s["tree"]["token"][0] = seed % 1000
        else:
            bank = [_tree("%dx%dx%d" % t) for t in TEMPLATES]
            pad = lambda v, fill: v + [fill] * (CAP - len(v))                                   # noqa: E731
            s.update(_packed(trees), bank_parent=_i32([pad(t[0], -1) for t in bank]),
                     bank_rank=_i32([pad(t[1], 0) for t in bank]), bank_n=_i32([len(t[0]) for t in bank]),
                     out_next={"next_parent": _i32([-1] * CAP), "next_rank": _i32([0] * CAP), "next_node_offsets": _i32([0, 0])})
    return s


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------
def run(s):
    return {"expand": _run_expand, "grow": _run_grow, "attention": _run_attention, "compact": _run_compact,
            "round": _run_round}[s["case"]["kind"]](s)


def _run_expand(s):
    c = s["case"]
    if c["static"]:
        return sage.sage_expand_topk_static(s["logits"], c["k"], c["k_entropy"], out=s["out"], status=s["status"], **s["tree"])
    return sage.sage_expand_topk(s["logits"], c["k"], c["k_entropy"], out=s["out"], ws=s["ws"], status=s["status"], **s["tree"])


def _grow(s, levels, idx, logprob, alpha, n_max):
    s["tree"]["n_nodes"].fill_(1)
    s["tree"]["frontier_begin"].zero_()
    for _ in range(levels):
        sage.sage_grow_tree(idx, logprob, alpha, s["policy"], s["tree"], n_max=n_max, d_max_seq=s["d_max"], status=s["status"])


def _run_grow(s):
    c = s["case"]
    _grow(s, c["levels"], s["idx"], s["logprob"], s["alpha"], c["n_max"])
    sage.sage_update_history(s["path_len"], s["history"], s["window"], s["count"], s["d_max"], status=s["status"])
    return [s["tree"], s["window"], s["count"], s["d_max"]]


def _run_attention(s):
    return sage.sage_tree_attention(s["q"], s["k"], s["v"], s["table"], s["seq_len"], s["parent"], s["node_offsets"],
                                    1.0 / math.sqrt(HEAD_DIM), out=s["out"], ws=s["ws"], status=s["status"])


def _run_compact(s):
    s["seq_len"].copy_(s["prefix"])                       # every pass starts from the same prefix
    a = sage.sage_accept(s["parent"], s["draft"], s["target"], s["node_offsets"], MAX_PATH, out=s["out"], status=s["status"])
    sage.sage_compact_kv(s["k"], s["v"], s["table"], s["seq_len"], a["path"], a["path_len"], status=s["status"])
    return [a, s["seq_len"], s["k"], s["v"]]


def _run_round(s):
    st, grown = s["status"], s["case"]["trees"] == "grown"
    s["seq_len"].copy_(s["prefix"])                       # every pass starts from the same prefix
    if grown:
        d = sage.sage_expand_topk(s["draft"], 10, 10, out=s["out_draft"], ws=s["ws_topk"], status=st)
        _grow(s, 8, d["topk_idx"], d["topk_logprob"], s["alpha_before"], CAP)
        s["node_offsets"][1:].copy_(s["tree"]["n_nodes"])
        parent, tokens, out_next = s["tree"]["parent"], s["tree"]["token"], {}
    else:
        d = sage.sage_expand_topk(s["draft"], 10, 10, parent=s["parent"], rank=s["rank"], node_offsets=s["node_offsets"],
                                  root_token=s["root"], out=s["out_draft"], ws=s["ws_topk"], status=st)
        out_next = sage.sage_select_tree(d["alpha"], s["policy"], alpha_row=s["alpha_row"], bank_parent=s["bank_parent"],
                                         bank_rank=s["bank_rank"], bank_n_nodes=s["bank_n"], handover=True, out=s["out_next"],
                                         status=st)
        parent, tokens = s["parent"], d["draft_token"]
    sage.sage_tree_attention(s["q"], s["k"], s["v"], s["table"], s["seq_len"], parent, s["node_offsets"],
                             1.0 / math.sqrt(HEAD_DIM), out=s["attention"], ws=s["ws"], status=st)
    t = sage.sage_expand_topk(s["target"], 1, 1, out=s["out_target"], ws=s["ws_topk"], status=st)
    a = sage.sage_accept(parent, tokens, t["topk_idx"], s["node_offsets"], MAX_PATH, out=s["out_accept"], status=st)
    sage.sage_compact_kv(s["k"], s["v"], s["table"], s["seq_len"], a["path"], a["path_len"], status=st)
    if grown:
        sage.sage_update_history(a["path_len"], s["history"], s["window"], s["count"], s["d_max"], status=st)
    return [d, out_next, s["attention"], t, a, s["seq_len"], s["d_max"], s["k"], s["v"]]


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without, and how exact it is
# ---------------------------------------------------------------------------------------------
def _expand_work(rows, vocab, k):
    return {"bytes": 4.0 * rows * vocab + rows * (8.0 * k + 16), "flops": 6.0 * rows * vocab}


def _attention_work(layers, lengths, nodes, q_heads, kv_heads):
    kv = sum(l + n for l, n in zip(lengths, nodes)) * kv_heads * HEAD_DIM * 4.0
    qo = sum(nodes) * q_heads * HEAD_DIM * 4.0
    return {"bytes": layers * (kv + qo),
            "flops": layers * sum(4.0 * n * q_heads * (l + n) * HEAD_DIM for l, n in zip(lengths, nodes))}


def _sum(*parts):
    return {n: sum(p[n] for p in parts) for n in ("bytes", "flops")}


def work(case):
    kind = case["kind"]
    if kind == "expand":
        return _expand_work(case["rows"], case["vocab"], case["k"])
    if kind == "grow":
        return {"bytes": case["batch"] * (case["n_max"] * (20.0 + 8 * case["k"]) + 60), "flops": case["batch"] * case["n_max"] * 10.0}
    if kind == "compact":
        # about three of an accepted path's rows are not yet in place
        return {"bytes": case["batch"] * (case["layers"] * 3 * case["kv_heads"] * HEAD_DIM * 8.0 + 64 * 12), "flops": 64.0 * case["batch"]}
    if kind == "attention":
        return _attention_work(case["layers"], _lengths(case), [len(t[0]) for t in _trees(case["trees"], case["batch"])],
                               case["q_heads"], case["kv_heads"])
    nodes = 12 if case["trees"] == "grown" else case["rows"]          # a grown tree has about a dozen nodes
    return _sum(_expand_work(case["rows"], case["vocab"], 10), _expand_work(case["rows"], case["vocab"], 1),
                _attention_work(case["layers"], [case["ctx"]], [nodes], 64, 8),
                {"bytes": case["layers"] * 3 * 8 * HEAD_DIM * 8.0, "flops": 0.0})


def tolerance(case):
    kind = case["kind"]
    if kind in ("grow", "compact"):
        return "exact"
    if kind == "expand":
        # 32-bit sums over up to 152064 terms, merged in 64 bits: 5e-8 (largest 2.4e-7) from the same path in 64 bits; sums
        # merged in 32 bits would be right too.  The candidates themselves are exact.
        return {"rel": 1e-6, "max": 1e-5}
    # probabilities and outputs rounded to bf16: 2.3e-3 (largest 2.9e-2) from the same path in 64 bits
    return {"rel": 9e-3, "max": 0.12}
