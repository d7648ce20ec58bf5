"""Performance cases of the tree-verification library: what a decoding loop has it do, through the public calls.

Five kinds of pass, each the work between two host decisions of a speculative-decoding loop:

  step    one verification step of the target model: falcon_tree_attn for every layer, falcon_tree_accept on the
          logits, falcon_kv_compact with the accepted tokens and features recorded in the same launch
  draft   one drafter pass: falcon_tree_attn of one layer under caller-supplied mask rows, the tree's K/V still in
          buffers of their own, then falcon_topm on the nodes' logits (the children the tree is grown by)
  head    the greedy decision without a logits matrix: falcon_lm_head_argmax, falcon_tree_accept from its argmax,
          falcon_feature_gather
  sample  the non-greedy decision: falcon_tree_accept with a temperature
  grow    child selection alone: falcon_topm

A case is a dict of plain values.  Tree sizes and prefix lengths of a batch are drawn inside the case's bounds by a
generator seeded with the case's own numbers; tokens, trees, logits, q, K and V come from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2412_12639_b200 as falcon
from paper_2412_12639_b200 import binding, synth

PATH_STRIDE = synth.T_MAX
P_ACCEPT = 0.7      # probability that greedy decoding takes one of a node's children
LOGITS_STD = 2.0
HEAD_STD = 0.02     # LM-head weights; features have unit variance

_contexts = {}


def _context():
    """One context per device, kept by the program."""
    dev = torch.cuda.current_device()
    if dev not in _contexts:
        _contexts[dev] = falcon.Context(dev)
    return _contexts[dev]


# --------------------------------------------------------------------------- the cases
def _step(name, batch, layers, hq, hkv, d, vocab, prefix, tree, depth, branch, pad=0):
    return {"name": name, "kind": "step", "batch": batch, "layers": layers, "hq": hq, "hkv": hkv, "d": d, "vocab": vocab,
            "pad": pad, "prefix_lo": prefix[0], "prefix_hi": prefix[1], "tree_lo": tree[0], "tree_hi": tree[1],
            "depth": depth, "branch": branch}


def _spec_step(name):
    """The step of one of the repository's own configurations."""
    s = synth.SPECS[name]
    return _step("step_" + name, s.batch, s.n_layers, s.n_q_heads, s.n_kv_heads, s.head_dim, s.vocab,
                 s.prefix_range or (s.prefix, s.prefix), s.tree_range or (s.tree, s.tree), s.max_depth, s.branch)


def _draft(name, batch, hq, hkv, d, vocab, prefix, tree, m, pad=0):
    return {"name": name, "kind": "draft", "batch": batch, "hq": hq, "hkv": hkv, "d": d, "vocab": vocab, "pad": pad,
            "prefix_lo": prefix[0], "prefix_hi": prefix[1], "tree_lo": tree[0], "tree_hi": tree[1], "depth": 6,
            "branch": 4, "m": m}


def _head(name, batch, hidden, vocab, tree):
    return {"name": name, "kind": "head", "batch": batch, "hidden": hidden, "vocab": vocab, "tree_lo": tree[0],
            "tree_hi": tree[1], "depth": 6, "branch": 4}


def listed():
    return [
        # one small layer on a short prefix: three launches, nothing to hide them behind
        _spec_step("tiny"),
        # single-user decoding on 7B-, 13B- and 70B-shaped models: multi-head attention with 1k and 2k prefixes,
        # grouped heads with a 4k prefix
        _spec_step("v7b"),
        _spec_step("l13b"),
        _spec_step("l70b"),
        # a serving batch of eight sequences of very different lengths
        _spec_step("ragged"),
        # a larger serving batch with grouped heads
        _step("step_serve16", 16, 32, 32, 8, 128, 32000, (256, 4096), (20, 64), 6, 4),
        # a drafter pass (one layer, relaxed mask, tree K/V in its own buffers) for one sequence, and for a small
        # batch with 64-wide heads and longer prefixes
        _draft("draft_one", 1, 32, 32, 128, 32000, (1024, 1024), (60, 60), 20),
        _draft("draft_batch", 4, 16, 16, 64, 32000, (512, 4096), (20, 60), 8),
        # the greedy tokens of one tree and of a serving batch straight from the LM head
        _head("head_one", 1, 4096, 32000, (60, 60)),
        _head("head_batch", 8, 5120, 32000, (20, 80)),
        # non-greedy decoding of a serving batch
        {"name": "sample_batch", "kind": "sample", "batch": 8, "vocab": 32000, "pad": 0, "tree_lo": 20, "tree_hi": 80,
         "depth": 8, "branch": 4, "temperature": 1.0},
        # the first children of a tree: one row, the smallest call
        {"name": "grow_root", "kind": "grow", "rows": 1, "vocab": 32000, "pad": 0, "m": 20},
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], its logarithm spread evenly."""
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def _span(rng, lo, hi, batch):
    """Bounds for a batch: one value for a single sequence, a range otherwise."""
    a = _log_int(rng, lo, hi)
    if batch == 1:
        return a, a
    b = _log_int(rng, lo, hi)
    return min(a, b), max(a, b)


def _vocab(rng):
    v = _log_int(rng, 1000, 131072)
    return v if rng.random() < 0.5 else max(1000, v // 64 * 64)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "draft", "draft", "head", "sample", "grow"])
    # rows of the logits follow one another directly, or with a pitch rounded up to 16 bytes
    vocab, pad = _vocab(rng), rng.choice([0, 4])
    depth, branch = rng.randint(3, 8), rng.randint(3, 8)  # holds more than 39 nodes at least
    tree_max = min(synth.T_MAX, synth.tree_capacity(depth, branch))
    if kind == "step":
        top = max((c for c in listed() if c["kind"] == "step"), key=lambda c: work(c)["bytes"])
        most = work(top)
        d = rng.choice([128, 128, 128, 64])
        while True:
            batch = _log_int(rng, 1, 16)
            hkv, group = rng.choice([4, 8, 8, 16, 32, 40]), rng.choice([1, 1, 2, 4, 8])
            case = _step("", batch, _log_int(rng, 1, 80), hkv * group, hkv, d, vocab, _span(rng, 16, 8192, batch),
                         _span(rng, 4, tree_max, batch), depth, branch, pad)
            # the cost of a step: its bytes, and the scores it has to form (64-wide heads do less work for each)
            w = work(case)
            if hkv * group <= 64 and w["bytes"] <= 0.5 * most["bytes"] and w["flops"] / d <= 0.5 * most["flops"] / top["d"]:
                break
        case.pop("name")
        return case
    if kind == "draft":
        batch = _log_int(rng, 1, 8)
        hkv, group = rng.choice([4, 8, 16, 32]), rng.choice([1, 1, 2, 4])
        case = _draft("", batch, min(64, hkv * group), hkv, rng.choice([64, 128]), vocab, _span(rng, 16, 4096, batch),
                      _span(rng, 4, tree_max, batch), rng.randint(1, 32), pad)
        case.update(depth=depth, branch=branch)
    elif kind == "head":
        batch = _log_int(rng, 1, 8)
        case = _head("", batch, 8 * _log_int(rng, 32, 1024), vocab, _span(rng, 4, tree_max, batch))
        case.update(depth=depth, branch=branch)
    elif kind == "sample":
        batch = _log_int(rng, 1, 16)
        lo, hi = _span(rng, 4, tree_max, batch)
        case = {"kind": "sample", "batch": batch, "vocab": vocab, "pad": pad, "tree_lo": lo, "tree_hi": hi, "depth": depth,
                "branch": branch, "temperature": round(rng.uniform(0.5, 1.2), 2)}
    else:
        case = {"kind": "grow", "rows": _log_int(rng, 1, 512), "vocab": vocab, "pad": pad, "m": rng.randint(1, 32)}
    case.pop("name", None)
    return case


# --------------------------------------------------------------------------- sizes, bytes and operations
def _sizes(case):
    """(tree sizes, prefix lengths) of the batch: a function of the case alone."""
    lo, hi = case.get("prefix_lo", 0), case.get("prefix_hi", 0)
    rng = np.random.default_rng([case["batch"], case["tree_lo"], case["tree_hi"], lo, hi, case["vocab"]])
    trees = rng.integers(case["tree_lo"], case["tree_hi"] + 1, size=case["batch"])
    prefix = rng.integers(lo, hi + 1, size=case["batch"])
    return [int(t) for t in trees], [int(x) for x in prefix]


def _pitch(case):
    return (case["vocab"] + case["pad"]) // 4 * 4 if case["pad"] else case["vocab"]


def _expected_path(T, depth):
    """Nodes on the accepted path, root included, when each node's child is taken with probability P_ACCEPT."""
    return sum(P_ACCEPT ** k for k in range(min(depth, T - 1) + 1))


def _attn_work(case, trees, prefix):
    hq, hkv, d = case["hq"], case["hkv"], case["d"]
    b = sum(4 * hkv * (L + T) * d + 4 * T * hq * d for T, L in zip(trees, prefix))
    f = sum(4 * hq * d * T * (L + min(T, 1 + case["depth"])) for T, L in zip(trees, prefix))
    return b, f


def work(case):
    kind = case["kind"]
    if kind == "grow":
        return {"bytes": 4 * case["rows"] * case["vocab"] + 8 * case["rows"] * case["m"], "flops": 0}
    trees, prefix = _sizes(case)
    n = sum(trees)
    on_path = sum(_expected_path(T, case["depth"]) for T in trees)
    if kind == "sample":
        return {"bytes": 4 * n * case["vocab"] + 16 * n, "flops": 0}
    if kind == "head":
        return {"bytes": 2 * case["hidden"] * (case["vocab"] + n) + 16 * n + 4 * case["hidden"] * on_path,
                "flops": 2 * n * case["hidden"] * case["vocab"]}
    b, f = _attn_work(case, trees, prefix)
    if kind == "draft":
        return {"bytes": b + 16 * n + 4 * n * case["vocab"] + 8 * n * case["m"], "flops": f}
    moved = 8 * case["layers"] * case["hkv"] * case["d"] * on_path + 4 * case["hq"] * case["d"] * on_path
    return {"bytes": case["layers"] * b + 4 * n * case["vocab"] + 16 * n + moved, "flops": case["layers"] * f}


def tolerance(case):
    if case["kind"] in ("step", "draft"):
        # attention outputs are bf16 with bf16 weights inside; tokens, paths, lengths and moved rows are exact
        return {"rel": 1e-2, "max": 0.1}
    if case["kind"] == "head":
        return {"rel": 2e-5, "max": 2e-4}  # the logits of the chosen tokens: fp32 sums of up to 8192 terms
    return "exact"


# --------------------------------------------------------------------------- inputs
def _i32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()


class _Batch:
    """Packed trees with drafted tokens, and which child (if any) the target takes at each node."""

    def __init__(self, case, seed):
        sizes, prefix = _sizes(case)
        rng = np.random.default_rng([seed, 1])
        parents = [synth.random_tree(rng, T, case["depth"], case["branch"]) for T in sizes]
        self.sizes, self.prefix = sizes, prefix
        self.host_off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
        self.host_prefix = np.array(prefix, dtype=np.int32)
        self.parents = parents
        self.n = int(self.host_off[-1])
        self.host_token = synth.random_tokens(rng, self.n, case["vocab"])
        rows, toks = [], []
        for off, par in zip(self.host_off, parents):
            for u, ch in enumerate(synth.children_lists(par)):
                if ch and rng.random() < P_ACCEPT:
                    rows.append(int(off) + u)
                    toks.append(int(self.host_token[int(off) + ch[int(rng.integers(0, len(ch)))]]))
        self.taken_rows = torch.tensor(rows, dtype=torch.int64, device="cuda")
        self.taken_tokens = torch.tensor(toks, dtype=torch.int64, device="cuda")
        self.node_off, self.parent, self.token = _i32(self.host_off), _i32(np.concatenate(parents)), _i32(self.host_token)
        self.prefix_len = _i32(self.host_prefix)
        self.status = torch.zeros(len(sizes), dtype=torch.int32, device="cuda")
        self.desc = binding.tree_desc(len(sizes), self.n, max(sizes), max(prefix), self.node_off, self.parent,
                                      self.prefix_len, token=self.token, prefix_len_host=self.host_prefix,
                                      node_off_host=self.host_off, status=self.status)


def _logits(case, gen, rows, batch=None):
    """fp32 [rows, pitch]; at nodes whose child the target takes, that child's token leads by one."""
    x = torch.randn((rows, _pitch(case)), dtype=torch.float32, device="cuda", generator=gen).mul_(LOGITS_STD)
    if batch is not None and batch.taken_rows.numel():
        top = x[batch.taken_rows, :case["vocab"]].amax(dim=1)
        x[batch.taken_rows, batch.taken_tokens] = top + 1.0
    return x


def _path_outputs(n_seq):
    return {"path": torch.zeros((n_seq, PATH_STRIDE), dtype=torch.int32, device="cuda"),
            "n_path": torch.zeros(n_seq, dtype=torch.int32, device="cuda"),
            "next_token": torch.zeros(n_seq, dtype=torch.int32, device="cuda")}


def _features_out(case, s, batch, hidden, gen):
    """Feature matrix of the nodes and where the accepted nodes' rows and tokens go."""
    rows = max(batch.sizes)
    s["features"] = torch.randn((batch.n, hidden), dtype=torch.bfloat16, device="cuda", generator=gen)
    s["out"]["features"] = torch.zeros((len(batch.sizes), rows, hidden), dtype=torch.bfloat16, device="cuda")
    s["out"]["tokens"] = torch.zeros((len(batch.sizes), rows), dtype=torch.int32, device="cuda")
    o = s["out"]
    return binding.gather_args(batch.desc, hidden, s["features"], hidden, o["path"], PATH_STRIDE, o["n_path"], rows,
                               o["features"], o["tokens"])


def _prepare_step(case, seed, gen):
    t = _Batch(case, seed)
    B, NL, Hq, Hkv, D, V = len(t.sizes), case["layers"], case["hq"], case["hkv"], case["d"], case["vocab"]
    s_cap = max(t.prefix) + max(t.sizes)
    # every layer's cache in one allocation; the tree's rows follow the prefix of each sequence
    cache = torch.empty((NL, 2, B, Hkv, s_cap, D), dtype=torch.bfloat16, device="cuda").normal_(generator=gen)
    q = torch.empty((NL, t.n, Hq, D), dtype=torch.bfloat16, device="cuda").normal_(generator=gen)
    out = torch.zeros_like(q)
    logits = _logits(case, gen, t.n, t)
    g = torch.zeros(t.n, dtype=torch.int32, device="cuda")
    new_len = torch.zeros(B, dtype=torch.int32, device="cuda")
    o = _path_outputs(B)
    s = {"batch": t, "cache": cache, "q": q, "logits": logits, "out": o}
    gather = _features_out(case, s, t, Hq * D, gen)
    kptr = torch.tensor([cache[l, 0].data_ptr() for l in range(NL)], dtype=torch.int64, device="cuda")
    vptr = torch.tensor([cache[l, 1].data_ptr() for l in range(NL)], dtype=torch.int64, device="cuda")
    strides = tuple(int(x) for x in cache[0, 0].stride()[:3])
    # From the second layer on the prefix was written long before the preceding kernel; the first layer follows the
    # previous step's compaction.  Each call names the caches of the next layer.
    s["attn"] = [binding.attn_args(t.desc, Hq, Hkv, D, 1.0 / math.sqrt(D), q[l], out[l], cache[l, 0], cache[l, 1], strides,
                                   s_cap, flags=binding.ATTN_PREFIX_STABLE if l else 0,
                                   next_k_cache=cache[l + 1, 0] if l + 1 < NL else None,
                                   next_v_cache=cache[l + 1, 1] if l + 1 < NL else None) for l in range(NL)]
    s["accept"] = binding.accept_args(t.desc, V, logits, logits.shape[1], g, o["path"], PATH_STRIDE, o["n_path"],
                                      o["next_token"])
    s["compact"] = binding.compact_args(t.desc, NL, Hkv, D, kptr, vptr, strides, s_cap, o["path"], PATH_STRIDE,
                                        o["n_path"], new_len, gather=gather)
    s["keep"] = (kptr, vptr, gather)
    o.update(attn=out, argmax=g, new_len=new_len)
    for b, (T, L) in enumerate(zip(t.sizes, t.prefix)):  # the rows the compaction works on
        o["tree_rows_%d" % b] = cache[:, :, b, :, L:L + T]
    return s


def _relaxed_mask(t):
    """Mask rows of the drafter's block-wise relaxed causal mask: ancestors-or-self and the siblings numbered before."""
    rows = []
    for par in t.parents:
        anc = []
        for i, p in enumerate(par):
            row = (anc[p] if p >= 0 else 0) | (1 << i)
            anc.append(row)
        for i, p in enumerate(par):
            sib = sum(1 << j for j in range(i) if par[j] == p) if p >= 0 else 0
            row = anc[i] | sib
            rows.append([row & ((1 << 64) - 1), row >> 64])
    return torch.from_numpy(np.array(rows, dtype=np.uint64).view(np.int64)).cuda()


def _prepare_draft(case, seed, gen):
    t = _Batch(case, seed)
    B, Hq, Hkv, D, V, m = len(t.sizes), case["hq"], case["hkv"], case["d"], case["vocab"], case["m"]
    s_cap = max(t.prefix) + max(t.sizes)

    def bf16(*shape):
        return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(generator=gen)

    k, v, k_tree, v_tree, q = bf16(B, Hkv, s_cap, D), bf16(B, Hkv, s_cap, D), bf16(t.n, Hkv, D), bf16(t.n, Hkv, D), bf16(t.n, Hq, D)
    out, mask = torch.zeros_like(q), _relaxed_mask(t)
    logits = _logits(case, gen, t.n)
    val = torch.zeros((t.n, m), dtype=torch.float32, device="cuda")
    idx = torch.zeros((t.n, m), dtype=torch.int32, device="cuda")
    return {"batch": t, "keep": (k, v, k_tree, v_tree, q, mask, logits),
            "attn": binding.attn_args(t.desc, Hq, Hkv, D, 1.0 / math.sqrt(D), q, out, k, v, tuple(int(x) for x in k.stride()[:3]),
                                      s_cap, k_tree=k_tree, v_tree=v_tree, tree_mask=mask),
            "topm": binding.topm_args(t.n, V, logits, logits.shape[1], m, val, idx),
            "out": {"attn": out, "top_val": val, "top_idx": idx}}


def _prepare_head(case, seed, gen):
    t = _Batch(case, seed)
    hidden, V = case["hidden"], case["vocab"]
    head = torch.empty((V, hidden), dtype=torch.bfloat16, device="cuda").normal_(std=HEAD_STD, generator=gen)
    s = {"batch": t, "head": head, "out": _path_outputs(len(t.sizes))}
    s["gather"] = _features_out(case, s, t, hidden, gen)
    if t.taken_rows.numel():  # the taken child's logit leads the others' spread by far
        lead = 16.0 * HEAD_STD * math.sqrt(hidden) / (hidden * HEAD_STD * HEAD_STD)
        s["features"][t.taken_rows] += (lead * head[t.taken_tokens].float()).bfloat16()
    o = s["out"]
    o["argmax"] = torch.zeros(t.n, dtype=torch.int32, device="cuda")
    o["top_logit"] = torch.zeros(t.n, dtype=torch.float32, device="cuda")
    s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    s["lm"] = binding.lm_argmax_args(t.n, hidden, V, s["features"], hidden, head, hidden, o["argmax"], max_out=o["top_logit"],
                                     status=s["status"])
    s["accept"] = binding.accept_args(t.desc, 0, None, 0, o["argmax"], o["path"], PATH_STRIDE, o["n_path"], o["next_token"])
    return s


def _prepare_sample(case, seed, gen):
    t = _Batch(case, seed)
    V = case["vocab"]
    logits = _logits(case, gen, t.n, t)
    u = torch.rand(t.n, device="cuda", generator=gen)
    # A draw within the rounding of fp32 sums of a token's boundary may go to either side: such numbers are moved to
    # the middle of a likely token's interval, so that what is right does not hang on the order of a sum.
    for lo in range(0, t.n, 64):
        cdf = torch.softmax(logits[lo:lo + 64, :V].double() / case["temperature"], dim=1).cumsum(dim=1)
        x = u[lo:lo + 64].double()
        j = torch.searchsorted(cdf, x[:, None]).clamp_(max=V - 1)
        hi = cdf.gather(1, j)[:, 0]
        below = torch.where(j[:, 0] > 0, cdf.gather(1, (j - 1).clamp_(min=0))[:, 0], torch.zeros_like(hi))
        near = torch.minimum(hi - x, x - below) < 2e-5
        p = torch.diff(cdf, dim=1, prepend=torch.zeros_like(cdf[:, :1]))
        top = p.argmax(dim=1, keepdim=True)
        mid = (cdf.gather(1, top) - 0.5 * p.gather(1, top))[:, 0]
        u[lo:lo + 64] = torch.where(near, mid, x).float()
    g = torch.zeros(t.n, dtype=torch.int32, device="cuda")
    o = _path_outputs(len(t.sizes))
    s = {"batch": t, "logits": logits, "u": u, "out": o}
    s["accept"] = binding.accept_args(t.desc, V, logits, logits.shape[1], g, o["path"], PATH_STRIDE, o["n_path"], o["next_token"],
                                      temperature=case["temperature"], uniforms=u)
    o["drawn"] = g
    return s


def _prepare_grow(case, seed, gen):
    rows, m = case["rows"], case["m"]
    logits = _logits(case, gen, rows)
    val = torch.zeros((rows, m), dtype=torch.float32, device="cuda")
    idx = torch.zeros((rows, m), dtype=torch.int32, device="cuda")
    return {"logits": logits, "topm": binding.topm_args(rows, case["vocab"], logits, logits.shape[1], m, val, idx),
            "out": {"top_val": val, "top_idx": idx}}


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    s = {"step": _prepare_step, "draft": _prepare_draft, "head": _prepare_head, "sample": _prepare_sample,
         "grow": _prepare_grow}[case["kind"]](case, int(seed), gen)
    s["kind"], s["ctx"] = case["kind"], _context()
    return s


# --------------------------------------------------------------------------- one pass
def run(s):
    ctx, kind = s["ctx"], s["kind"]
    if kind == "step":
        for a in s["attn"]:
            ctx.falcon_tree_attn(a)
        ctx.falcon_tree_accept(s["accept"])
        ctx.falcon_kv_compact(s["compact"])
    elif kind == "draft":
        ctx.falcon_tree_attn(s["attn"])
        ctx.falcon_topm(s["topm"])
    elif kind == "head":
        ctx.falcon_lm_head_argmax(s["lm"])
        ctx.falcon_tree_accept(s["accept"])
        ctx.falcon_feature_gather(s["gather"])
    elif kind == "sample":
        ctx.falcon_tree_accept(s["accept"])
    else:
        ctx.falcon_topm(s["topm"])
    return s["out"]
