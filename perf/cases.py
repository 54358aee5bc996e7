"""What is measured: decode steps, tree-masked prefills and LSE merges of the
fork-tree attention library, through the calls a serving program makes.

A decode case is one step of every live branch of a forest of requests: each
request has a prefix, optionally a level of subtask nodes under it, and trial
branches under the prefix (or under each subtask) with private suffixes.  A
prefill case is one pass of a join (a chain of finished threads and new text
after it) or of thread openings under a shared prefix.  A merge case combines
two attention results over disjoint key sets.

A program keeps the plan, the KV pools, and its out / lse buffers between
steps, so they are part of the prepared state; the node lengths depend on the
case alone, the page order and the values on the seed.
"""
import math

import numpy as np
import torch

from paper_2608_24658_gb300 import workloads as W
from paper_2608_24658_gb300.api import Plan, lse_merge

KV_BYTES = {"bf16": 2, "fp8": 1, "fp32": 4}


def _decode(name, mode, q_heads, kv_heads, head_dim, requests, prefix_lo, prefix_hi, subtasks,
            subtask_len, trials, suffix_lo, suffix_hi, permuted, small_q, shape):
    case = dict(op="decode", mode=mode, q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim,
                requests=requests, prefix_lo=prefix_lo, prefix_hi=prefix_hi, subtasks=subtasks,
                subtask_len=subtask_len, trials=trials, suffix_lo=suffix_lo, suffix_hi=suffix_hi,
                permuted=permuted, small_q=small_q, shape=shape)
    return dict(case, name=name) if name else case


def _prefill(name, mode, q_heads, kv_heads, prefix, joined, thread_lo, thread_hi, chunks,
             chunk_lo, chunk_hi, permuted, shape):
    case = dict(op="prefill", mode=mode, q_heads=q_heads, kv_heads=kv_heads, head_dim=128,
                prefix=prefix, joined=joined, thread_lo=thread_lo, thread_hi=thread_hi,
                chunks=chunks, chunk_lo=chunk_lo, chunk_hi=chunk_hi, permuted=permuted,
                shape=shape)
    return dict(case, name=name) if name else case


def _merge(name, dtype, head_dim, rows):
    case = dict(op="merge", dtype=dtype, head_dim=head_dim, rows=rows)
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest step: one short request that has just forked; launches
        # and latency count
        _decode("tiny_fork", "bf16", 8, 2, 64, 1, 256, 256, 0, 0, 4, 32, 64, False, False, 0),
        # one request with 16 trials of ragged length, the common single-user step
        _decode("trials16", "bf16", 32, 8, 128, 1, 2048, 2048, 0, 0, 16, 512, 4096, False, True, 1),
        # the same step with 32-bit tensors, as a program runs it to check numerics
        _decode("trials16_fp32", "fp32", 32, 8, 128, 1, 2048, 2048, 0, 0, 16, 512, 4096, False,
                True, 1),
        # nested regions: 8 subtasks with 8 trials each under one prefix
        _decode("two_level", "bf16", 64, 8, 128, 1, 4096, 4096, 8, 1024, 8, 256, 2048, False,
                False, 2),
        # a smaller model's heads (head_dim 64): a few requests with wide forks
        # over long prefixes, pages in the order an allocator hands them out
        _decode("forks_d64", "bf16", 32, 8, 64, 4, 2048, 8192, 0, 0, 32, 64, 1024, True, False, 7),
        # serving at full load: 32 requests, 1024 branches, permuted pages, 18 GB of KV
        _decode("batched", "bf16", 32, 8, 128, 32, 1024, 8192, 0, 0, 32, 256, 8192, True, False, 3),
        # long reasoning: 128 branches of up to 16k tokens under a 32k prefix
        _decode("long", "bf16", 64, 8, 128, 1, 32768, 32768, 0, 0, 128, 4096, 16384, False, False, 4),
        # the same with the KV cache in e4m3
        _decode("long_e4m3", "fp8", 64, 8, 128, 1, 32768, 32768, 0, 0, 128, 4096, 16384, False,
                False, 4),
        # thread openings: 16 chunks of 64 tokens prefilled under a shared prefix
        _prefill("fork_prefill", "bf16", 32, 8, 2048, 0, 0, 0, 16, 64, 64, False, 6),
        # the join: new text prefilled over the prefix and 16 finished threads
        _prefill("join_prefill", "bf16", 32, 8, 2048, 16, 512, 4096, 1, 1024, 1024, False, 1),
        # the join with the KV cache in e4m3
        _prefill("join_prefill_e4m3", "fp8", 32, 8, 2048, 16, 512, 4096, 1, 1024, 1024, False, 1),
        # two results over disjoint keys of a long prefill combined: 8192 tokens x 32 heads
        _merge("lse_merge", "bf16", 128, 8192 * 32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.random()
    if kind < 0.12:
        return _merge(None, rng.choice(["bf16", "fp32"]), rng.choice([64, 128]),
                      _log(rng, 16, 8192 * 32))
    shape = rng.randrange(1 << 30)
    if kind < 0.35:
        q_heads, kv_heads = rng.choice([(32, 8), (64, 8), (16, 2), (28, 4), (16, 16)])
        chunks = rng.choice([1, 1, 2, _log(rng, 2, 32)])
        lo = _log(rng, 1, 1024 // chunks)
        joined = rng.choice([0, 0, _log(rng, 1, 16)])
        tlo = _log(rng, 16, 1024) if joined else 0
        return _prefill(None, rng.choice(["bf16", "bf16", "fp8"]), q_heads, kv_heads,
                        _log(rng, 1, 8192), joined, tlo, _log(rng, tlo, 2048) if joined else 0,
                        chunks, lo, _log(rng, lo, 1024 // chunks), rng.random() < 0.5, shape)
    mode = rng.choice(["bf16", "bf16", "bf16", "fp8", "fp32"])
    q_heads, kv_heads = rng.choice([(8, 2), (32, 8), (64, 8), (16, 2), (28, 4), (16, 16)])
    head_dim = 128 if mode == "fp8" else rng.choice([64, 128, 128])
    plo = _log(rng, 64, 16384)
    slo = _log(rng, 1, 4096)
    case = _decode(None, mode, q_heads, kv_heads, head_dim, _log(rng, 1, 16), plo,
                   _log(rng, plo, 32768), rng.choice([0, 0, _log(rng, 2, 8)]), _log(rng, 16, 2048),
                   _log(rng, 1, 64), slo, _log(rng, slo, 8192), rng.random() < 0.5,
                   rng.random() < 0.3, shape)
    # no larger than the listed cases (the 32-bit step runs without tensor cores)
    top_b, top_f = (4e8, 4e9) if mode == "fp32" else (6e9, 1e11)
    while True:
        w = work(case)
        if w["bytes"] <= top_b and w["flops"] <= top_f:
            return case
        key = max(("requests", "trials", "suffix_hi", "prefix_hi"),
                  key=lambda k: case[k] / {"requests": 8, "trials": 8}.get(k, 256))
        case[key] = max(1, int(case[key] * 0.7))
        case["suffix_lo"] = min(case["suffix_lo"], case["suffix_hi"])
        case["prefix_lo"] = min(case["prefix_lo"], case["prefix_hi"])


def _forest(case):
    """(parent, node lengths, leaf or chunk nodes) of a case."""
    rng = np.random.default_rng(case["shape"])

    def between(lo, hi):
        return int(rng.integers(lo, hi + 1))

    parent, lens, leaves = [], [], []

    def node(up, n):
        parent.append(up)
        lens.append(n)
        return len(parent) - 1

    if case["op"] == "prefill":
        up = node(-1, case["prefix"])
        for _ in range(case["joined"]):
            up = node(up, between(case["thread_lo"], case["thread_hi"]))
        leaves = [node(up, between(case["chunk_lo"], case["chunk_hi"]))
                  for _ in range(case["chunks"])]
        return parent, lens, leaves
    for _ in range(case["requests"]):
        if case["prefix_lo"] == case["prefix_hi"]:
            n = case["prefix_lo"]
        else:       # prefixes of concurrent requests: lognormal, clipped
            n = int(min(case["prefix_hi"], max(case["prefix_lo"], round(
                math.exp(math.log(2 * case["prefix_lo"]) + 0.5 * float(rng.standard_normal()))))))
        root = node(-1, n)
        forks = [node(root, case["subtask_len"]) for _ in range(case["subtasks"])] or [root]
        for f in forks:
            for _ in range(case["trials"]):
                leaves.append(node(f, between(case["suffix_lo"], case["suffix_hi"])))
    return parent, lens, leaves


def _tree(case, seed):
    """The case's tree with its q, K and V on the GPU."""
    parent, lens, leaves = _forest(case)
    small = case["op"] == "prefill" or case["small_q"]
    build = W.build_prefill if case["op"] == "prefill" else W.build_tree
    return build("case", parent, lens, leaves, num_q_heads=case["q_heads"],
                 num_kv_heads=case["kv_heads"], head_dim=case["head_dim"], mode=case["mode"],
                 seed=seed, permute_pages=case["permuted"], device="cuda",
                 q_std=1.0 / math.sqrt(case["head_dim"]) if small else 1.0)


def _merge_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rows, d = case["rows"], case["head_dim"]
    dtype = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16
    o = [torch.randn((rows, d), generator=gen, device="cuda").to(dtype) for _ in range(2)]
    # lse of a few thousand keys each; a few rows have an empty side
    lse = [8.0 + torch.randn(rows, generator=gen, device="cuda") for _ in range(2)]
    for k in range(2):
        lse[k][torch.rand(rows, generator=gen, device="cuda") < 0.01] = -math.inf
    return o[0], lse[0], o[1], lse[1]


def prepare(case, seed):
    if case["op"] == "merge":
        o_a, lse_a, o_b, lse_b = _merge_inputs(case, seed)
        return dict(merge=(o_a, lse_a, o_b, lse_b, torch.empty_like(o_a), torch.empty_like(lse_a)))
    tree = _tree(case, seed)
    plan = Plan.for_prefill(tree) if case["op"] == "prefill" else Plan.for_tree(tree)
    out = torch.empty_like(tree.q)
    lse = torch.empty(tree.q.shape[:2], dtype=torch.float32, device="cuda")
    return dict(plan=plan, tree=tree, out=out, lse=lse, workspace=plan.workspace(tree.k_pages.device))


def run(state):
    if "merge" in state:
        return lse_merge(*state["merge"])
    t = state["tree"]
    return state["plan"].decode(t.q, t.k_pages, t.v_pages, out=state["out"], lse=state["lse"],
                                workspace=state["workspace"], k_scale=t.k_scale,
                                v_scale=t.v_scale)


def work(case):
    if case["op"] == "merge":
        elem = 4 if case["dtype"] == "fp32" else 2
        return {"bytes": case["rows"] * (3 * case["head_dim"] * elem + 12),
                "flops": case["rows"] * case["head_dim"] * 4}
    parent, lens, leaves = _forest(case)
    h_q, h_kv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    under = [0] * len(parent)
    for n in leaves:
        under[n] = lens[n] if case["op"] == "prefill" else 1
    queries = sum(under)
    for n in range(len(parent) - 1, 0, -1):
        if parent[n] >= 0:
            under[parent[n]] += under[n]
    if case["op"] == "prefill":     # causal in the chunk itself
        own = set(leaves)
        keys = sum(lens[n] * (lens[n] + 1) // 2 if n in own else lens[n] * under[n]
                   for n in range(len(parent)))
    else:
        keys = sum(lens[n] * under[n] for n in range(len(parent)))
    elem = KV_BYTES[case["mode"]]
    q_elem = 4 if case["mode"] == "fp32" else 2
    return {"bytes": sum(lens) * 2 * h_kv * d * elem + queries * h_q * (2 * d * q_elem + 4),
            "flops": keys * h_q * 4 * d}


def tolerance(case):
    # relative error of out and of lse, four times what `exact` shows: bf16
    # results carry the rounding of P and of out to 8 bits (2.3e-3), with e4m3
    # KV P has 11 (1.7e-3), a merge rounds once (1.6e-3); 32-bit sums 2.3e-7
    if case["op"] == "merge":
        return {"rel": 1e-6 if case["dtype"] == "fp32" else 7e-3}
    return {"rel": {"bf16": 9e-3, "fp8": 7e-3, "fp32": 1e-6}[case["mode"]]}


def _node_kv(tree, n):
    """K and V of node n in 64 bits, [H_kv, tokens, d]."""
    lo, hi = int(tree.node_page_ptr[n]), int(tree.node_page_ptr[n + 1])
    ids = torch.as_tensor(tree.page_ids[lo:hi].astype(np.int64), device="cuda")
    kv = []
    for pages, scale in ((tree.k_pages, tree.k_scale), (tree.v_pages, tree.v_scale)):
        raw = pages.view(torch.uint8)[ids].view(pages.dtype) if pages.element_size() == 1 else pages[ids]
        x = raw.to(torch.float32).to(torch.float64)
        if scale is not None:
            x = x * scale.to(torch.float64).view(1, -1, 1, 1)
        kv.append(x.permute(1, 0, 2, 3).reshape(x.shape[1], -1, x.shape[3])[:, :int(tree.node_len[n])])
    return kv


def _attend(q, k, v, sm_scale, mask=None):
    """q [H_kv, rows, d] over k, v [H_kv, keys, d]: (o, lse)."""
    s = torch.matmul(q, k.transpose(1, 2)) * sm_scale
    if mask is not None:
        s = s.masked_fill(mask, -math.inf)
    lse = torch.logsumexp(s, dim=-1)
    return torch.matmul(torch.exp(s - lse.unsqueeze(-1)), v), lse


def exact(case, seed):
    if case["op"] == "merge":
        o_a, lse_a, o_b, lse_b = (x.to(torch.float64) for x in _merge_inputs(case, seed))
        lse = torch.logaddexp(lse_a, lse_b)
        w_a, w_b = (torch.exp(x - lse).nan_to_num(0.0).unsqueeze(1) for x in (lse_a, lse_b))
        return w_a * o_a + w_b * o_b, lse
    tree = _tree(case, seed)
    h_q, h_kv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    g = h_q // h_kv
    sm_scale = 1.0 / math.sqrt(d)
    out = torch.empty(tree.q.shape, dtype=torch.float64, device="cuda")
    lse = torch.empty(tree.q.shape[:2], dtype=torch.float64, device="cuda")
    row = 0
    inner = {}
    for b in range(len(tree.leaf_node)):
        path = tree.path(b)
        for n in list(inner):
            if n not in path:
                del inner[n]
        for n in path[:-1]:
            if n not in inner:
                inner[n] = _node_kv(tree, n)
        kv = [inner[n] for n in path[:-1]] + [_node_kv(tree, path[-1])]
        k, v = (torch.cat([x[i] for x in kv], dim=1) for i in range(2))
        if case["op"] == "decode":
            o, l = _attend(tree.q[b].to(torch.float64).view(h_kv, g, d), k, v, sm_scale)
            out[b], lse[b] = o.reshape(h_q, d), l.reshape(h_q)
            continue
        own = int(tree.node_len[path[-1]])
        before = k.shape[1] - own
        seen = torch.arange(own, device="cuda") + before
        for t0 in range(0, own, 256):
            t1 = min(own, t0 + 256)
            q = tree.q[row + t0:row + t1].to(torch.float64).view(t1 - t0, h_kv, g, d)
            hidden = torch.arange(k.shape[1], device="cuda")[None, :] > seen[t0:t1, None]
            hidden = hidden.repeat_interleave(g, dim=0)
            for j in range(h_kv):
                o, l = _attend(q[:, j].reshape(1, -1, d), k[j:j + 1], v[j:j + 1], sm_scale, hidden)
                out[row + t0:row + t1, j * g:(j + 1) * g] = o.view(t1 - t0, g, d)
                lse[row + t0:row + t1, j * g:(j + 1) * g] = l.view(t1 - t0, g)
        row += own
    return out, lse
