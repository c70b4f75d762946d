"""What a user of this library has it do, as measurable cases.

A case is one call sequence of a serving loop on one batch: a speculative round (verify, greedy acceptance,
commit), the fused commit-and-verify round, a plain decode step, or the draft-side utilities of a round.  Shapes are
those of the repository's benchmark workloads (``bench.py``, ``synth.config``) or generic ones between them; value
distributions are those of ``synth`` (state ~ N(0, 0.02^2), normalised keys, sigmoid gates, 75 % matchable tokens).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_16673_b200 import binding as speca
from paper_2607_16673_b200 import synth

DEV = "cuda"
P_MATCH = 0.75


def listed():
    # op: round | fused | decode | draft; L layers, B sequences, H heads; nodes lo..hi per sequence
    # kind: chain (lo nodes), tree (random, <= 4 children), proposal (top-k beam shape), mixed (half chains of 8,
    # half trees of hi nodes), chains+proposals (half chains of 8, half proposals of lo..hi nodes)
    def c(name, op, L, B, H, dk, dv, kind="chain", lo=1, hi=1, depth=8, tf32=False):
        return dict(name=name, op=op, L=L, B=B, H=H, dk=dk, dv=dv, kind=kind, lo=lo, hi=hi, depth=depth, tf32=tf32)

    return [
        # smallest call there is: one layer of a small model drafting a chain of four for one user, call by call
        c("chain4_1layer", "round", 1, 1, 4, 64, 64, "chain", 4, 4),
        # one interactive user, whole 24-layer stack, chain drafter with eight tokens
        c("chain8_1user", "round", 24, 1, 16, 128, 128, "chain", 8, 8),
        # one interactive user, tree drafter with a 32-node budget
        c("tree32_1user", "round", 24, 1, 16, 128, 128, "tree", 32, 32, 6),
        # one interactive user at d_k = d_v = 256, narrow deep proposal tree (top-2, 16 levels)
        c("proposal_deep_1user", "round", 24, 1, 8, 256, 256, "proposal", 32, 32, 16),
        # a small model with 64-wide heads served to a handful of users, ragged draft trees
        c("ragged_d64", "round", 24, 12, 16, 64, 64, "tree", 5, 40),
        # ordinary serving batch: 32 users, ragged trees of 8..64 nodes
        c("ragged_b32", "round", 24, 32, 16, 128, 256, "tree", 8, 64),
        # the same heads with 64-node trees drafted up to 16 levels deep
        c("deep64_b16", "round", 24, 16, 16, 128, 256, "tree", 40, 64, 16),
        # full serving batch: 128 users, half chains of 8, half 64-node trees (the benchmark's default workload)
        c("mixed_b128", "round", 24, 128, 16, 128, 256, "mixed", 8, 64),
        # wide heads, 64 users, chains of 8 and top-4 proposals, the commit of a round delayed into the next one's call
        c("fused_wide_b64", "fused", 24, 64, 8, 256, 256, "chains+proposals", 16, 32),
        # the same call for a user who trades accuracy for time (single TF32 pass, one pass over the state)
        c("fused_tf32_b32", "fused", 24, 32, 16, 128, 256, "tree", 8, 64, 8, True),
        # rounds without a draft: one token per sequence at the full serving batch
        c("decode_b128", "decode", 24, 128, 16, 128, 256),
        # what surrounds the verification of a tree round at the full batch: proposal conversion, pruning, chain
        # decomposition, stochastic acceptance, convolution-state commit
        c("draft_b128", "draft", 24, 128, 16, 128, 256, "tree", 24, 64),
    ]


def draw(rng):
    """One more case of the ranges above; cost bounded by the largest listed case's."""
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    op = rng.choice(["round"] * 6 + ["fused"] * 2 + ["decode"] * 2 + ["draft"])
    dk, dv = rng.choice([(64, 64), (128, 128), (128, 128), (128, 256), (128, 256), (128, 256), (256, 256)])
    H = rng.choice([3, 4, 8, 12, 16, 16])
    L = rng.choice([1, 6, 12, 24, 24, 24])
    B = log_int(1, 128)
    kind, lo, hi, depth, tf32 = "chain", 1, 1, 8, False
    if op != "decode":
        kind = rng.choice(["chain", "tree", "tree", "proposal", "mixed"]) if op != "draft" else "tree"
        top = 32 if dk == 256 else 64
        depth = rng.choice([8, 8, 16]) if op == "round" else 8
        if kind == "chain":
            lo = hi = rng.randint(2, depth)
        else:
            hi = rng.randint(9, top)
            lo = rng.randint(max(1, hi // 4), hi)
        tf32 = op == "fused" and dk > 64 and rng.random() < 0.5
    # 64-wide heads and trees that are wide and deep at once are what smaller models and batches use
    if dk == 64 or (depth == 16 and hi > 32):
        B = min(B, 24)
    return dict(op=op, L=L, B=B, H=H, dk=dk, dv=dv, kind=kind, lo=lo, hi=hi, depth=depth, tf32=tf32)


# ---------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------
def _parents(case, rng):
    kind, lo, hi, depth = case["kind"], case["lo"], case["hi"], case["depth"]

    def tree(n):
        return synth.random_tree_parent(n, depth, 4, rng)

    # node counts spread evenly over lo..hi, handed to the sequences in random order
    half = case["B"] // 2 if kind == "chains+proposals" else 0
    sizes = [8] * half + list(rng.permutation(np.linspace(lo, hi, case["B"] - half).round().astype(int)))
    out = []
    for b in range(case["B"]):
        n = int(sizes[b])
        if kind == "chain":
            out.append(synth.chain_parent(lo))
        elif kind == "tree":
            out.append(tree(n))
        elif kind == "proposal":
            # narrow shapes use every level, wide ones (top-4) half of them
            narrow = depth > 8
            out.append(synth.proposal_tree_parent(2 if narrow else 4, depth if narrow else int(rng.integers(4, 9)), n, rng, depth))
        elif kind == "mixed":
            out.append(synth.chain_parent(min(8, hi)) if 2 * b < case["B"] else tree(hi))
        else:                                   # chains+proposals
            out.append(synth.chain_parent(8) if b < half else
                       synth.proposal_tree_parent(4, int(rng.integers(4, 9)), n, rng, depth))
    return out


def _tokens(rng, offs, parent):
    """Token ids by the rule of synth.draw_tokens (siblings distinct, a node's target matches one of its children
    with probability P_MATCH), drawn without a Python loop over the vocabulary."""
    T, B = len(parent), len(offs) - 1
    seq = np.repeat(np.arange(B), np.diff(offs))
    local = np.arange(T) - offs[seq]
    draft = ((rng.integers(0, 400, T) * 64 + local) % synth.VOCAB).astype(np.int32)     # distinct inside a sequence
    target = rng.integers(0, synth.VOCAB, T).astype(np.int32)
    root = rng.integers(0, synth.VOCAB, B).astype(np.int32)
    order = rng.permutation(T)                  # the child that matches: the last one in a random order
    node = np.where(parent < 0, T + seq, offs[seq] + parent)[order]
    pick = np.full(T + B, -1, np.int64)
    pick[node] = order
    pick[rng.random(T + B) >= P_MATCH] = -1
    both = np.concatenate([target, root])
    both[pick >= 0] = draft[pick[pick >= 0]]
    return draft, both[:T].copy(), both[T:].copy()


def _draft(case, seed):
    """One draft of the batch: topology, token ids, factor records, on the GPU."""
    rng = np.random.default_rng(seed)
    parents = _parents(case, rng)
    offs = np.concatenate([[0], np.cumsum([len(p) for p in parents])]).astype(np.int32)
    parent = np.concatenate(parents).astype(np.int32)
    depth = np.concatenate([synth.depth_of(p) for p in parents]).astype(np.int32)
    draft, target, root = _tokens(rng, offs, parent)
    q, k, v, alpha, beta = synth.device_records(seed, case["L"], len(parent), case["H"], case["dk"], case["dv"], DEV)
    d = dict(q=q, k=k, v=v, alpha=alpha, beta=beta, total_nodes=len(parent), parents=parents)
    for name, a in (("node_offsets", offs), ("parent", parent), ("depth", depth), ("draft_tok", draft),
                    ("target_tok", target), ("root_tok", root)):
        d[name] = torch.from_numpy(a).to(DEV)
    return d


def _paths(B, depth):
    i32 = dict(dtype=torch.int32, device=DEV)
    return dict(path_idx=torch.zeros(B, depth, **i32), path_len=torch.zeros(B, **i32), next_tok=torch.zeros(B, **i32))


def _accept(st, d, out):
    speca.greedy_accept(st["dims"].batch, st["dims"].max_depth, d["node_offsets"], d["parent"], d["draft_tok"],
                        d["target_tok"], d["root_tok"], out["path_idx"], out["path_len"], out["next_tok"], st["status"])


def prepare(case, seed):
    L, B, H, dk, dv, op = (case[x] for x in ("L", "B", "H", "dk", "dv", "op"))
    seed = (int(seed) * 1009 + 17) % (1 << 31)
    st = dict(op=op, kind=case["kind"], status=torch.zeros(1, dtype=torch.int32, device=DEV))
    if op == "draft":
        return _prepare_draft(case, seed, st)
    budget = max(case["hi"], 8) if case["kind"] != "chain" else case["lo"]
    route = speca.ROUTE_TF32 if case["tf32"] else speca.ROUTE_AUTO
    st["dims"] = dims = speca.Dims(L, B, H, dk, dv, 1.0, case["depth"], budget, route)
    st["S"] = synth.device_state(seed + 1, L, B, H, dk, dv, 0.02, DEV)
    if op == "decode":
        q, k, v, alpha, beta = synth.device_records(seed + 2, L, B, H, dk, dv, DEV)
        st.update(q=q, k=k, v=v, alpha=alpha, beta=beta, o=torch.zeros(L, B, H, dv, device=DEV))
        return st
    st["d"] = d = _draft(case, seed + 2)
    st["o"] = torch.zeros(L, d["total_nodes"], H, dv, device=DEV)
    st["ws"] = speca.alloc_workspace(dims, d["total_nodes"])
    st["out"] = _paths(B, case["depth"])
    if op == "fused":
        # the round before: its draft, what its verification left, and the paths accepted from it
        st["prev"] = p = _draft(case, seed + 3)
        st["pending"] = _paths(B, case["depth"])
        ws = speca.alloc_workspace(dims, p["total_nodes"])
        o = torch.zeros(L, p["total_nodes"], H, dv, device=DEV)
        p["u"] = torch.zeros_like(o) if case["tf32"] else None
        st["u"] = torch.zeros_like(st["o"]) if case["tf32"] else None
        speca.verify_tree(dims, st["S"], p["q"], p["k"], p["v"], p["alpha"], p["beta"], p["node_offsets"],
                          p["total_nodes"], p["parent"], p["depth"], o, p["u"], ws, st["status"])
        _accept(st, p, st["pending"])
    return st


CONV_CHANNELS, CONV_WIDTH = 8192, 3             # q, k and v of 16 heads at d_k = 128, d_v = 256; kernel size 4


def _prepare_draft(case, seed, st):
    rng = np.random.default_rng(seed)
    B, N, L = case["B"], case["hi"], case["L"]
    parents = _parents(case, rng)
    offs = np.concatenate([[0], np.cumsum([len(p) for p in parents])]).astype(np.int32)
    T = int(offs[-1])
    mask = np.zeros((B, N, N), np.uint8)
    for b, p in enumerate(parents):
        for i, a in enumerate(p):
            if a >= 0:
                mask[b, i] = mask[b, a]
            mask[b, i, i] = 1
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    i32 = dict(dtype=torch.int32, device=DEV)
    st.update(B=B, N=N, L=L, T=T, depth=case["depth"], mask=torch.from_numpy(mask).to(DEV),
              node_offsets=torch.from_numpy(offs).to(DEV), parent=torch.zeros(T, **i32),
              logp=torch.log(torch.rand(T, generator=g, device=DEV).clamp_min(1e-3)),
              p_target=torch.rand(T, generator=g, device=DEV), p_draft=torch.rand(T, generator=g, device=DEV),
              uniform=torch.rand(T, generator=g, device=DEV), out_offsets=torch.zeros(B + 1, **i32),
              out_parent=torch.zeros(T, **i32), out_index=torch.zeros(T, **i32), chain_head=torch.zeros(T, **i32),
              n_chains=torch.zeros(B, **i32), out=_paths(B, case["depth"]),
              C=torch.randn(L, B, CONV_WIDTH, CONV_CHANNELS, generator=g, device=DEV).to(torch.bfloat16),
              x=torch.empty(L, T, CONV_CHANNELS, dtype=torch.bfloat16, device=DEV).normal_(generator=g))
    return st


# ---------------------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------------------
def run(st):
    if st["op"] == "draft":
        return _run_draft(st)
    dims, S = st["dims"], st["S"]
    if st["op"] == "decode":
        speca.decode_step(dims, S, st["q"], st["k"], st["v"], st["alpha"], st["beta"], st["o"])
        return st["o"], S
    d, out, T = st["d"], st["out"], st["d"]["total_nodes"]
    rec = (d["q"], d["k"], d["v"], d["alpha"], d["beta"], d["node_offsets"], T)
    if st["op"] == "fused":
        speca.commit_verify_tree(dims, S, st["prev"], st["pending"]["path_idx"], st["pending"]["path_len"], *rec,
                                 d["parent"], d["depth"], st["o"], st["u"], st["ws"], st["status"])
        _accept(st, d, out)
        return (st["o"], S, out["path_idx"], out["path_len"], out["next_tok"], st["status"]) + \
            (() if st["u"] is None else (st["u"],))
    if st["kind"] == "chain":
        speca.verify_chain(dims, S, *rec, st["o"], None, st["ws"], st["status"])
    else:
        speca.verify_tree(dims, S, *rec, d["parent"], d["depth"], st["o"], None, st["ws"], st["status"])
    _accept(st, d, out)
    speca.commit(dims, S, d["k"], d["v"], d["alpha"], d["beta"], d["node_offsets"], T, d["parent"], out["path_idx"],
                 out["path_len"], st["status"])
    return st["o"], S, out["path_idx"], out["path_len"], out["next_tok"], st["status"]


TAU, BUDGET = 1e4, 20                       # the budget decides: 20 nodes of every tree are kept


def _run_draft(st):
    B, N, offs, out = st["B"], st["N"], st["node_offsets"], st["out"]
    speca.tree_mask_to_parent(st["mask"], offs, st["parent"], st["status"])
    speca.prune_tree(N, TAU, BUDGET, offs, st["parent"], st["logp"], st["out_offsets"], st["out_parent"],
                     st["out_index"], st["status"])
    speca.chain_decompose(N, offs, st["parent"], st["chain_head"], st["n_chains"], st["status"])
    speca.stochastic_accept(B, st["depth"], offs, st["parent"], st["p_target"], st["p_draft"], st["uniform"],
                            out["path_idx"], out["path_len"], st["status"])
    speca.commit_conv(st["C"], st["x"], offs, st["T"], out["path_idx"], out["path_len"], st["status"])
    kept = int(st["out_offsets"][B])            # the host needs the number of kept nodes to size the next call
    return (st["parent"], st["out_offsets"], st["out_parent"][:kept], st["out_index"][:kept], st["chain_head"],
            st["n_chains"], out["path_idx"], out["path_len"], st["C"], st["status"])


# ---------------------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far correct results may lie apart
# ---------------------------------------------------------------------------------------------------------------
def _mean_nodes(case):
    if case["kind"] == "chain":
        return float(case["lo"])
    mid = 0.5 * (case["lo"] + case["hi"])
    if case["kind"] == "mixed":
        return 0.5 * (min(8, case["hi"]) + case["hi"])
    return 0.5 * (8 + mid) if case["kind"] == "chains+proposals" else mid


def work(case):
    L, B, H, dk, dv, op = (case[x] for x in ("L", "B", "H", "dk", "dv", "op"))
    units, state = float(L * B * H), 4.0 * dk * dv
    if op == "decode":
        return dict(bytes=units * (2 * state + 4 * dk + 2 * dv + 8 + 4 * dv), flops=units * 8 * dk * dv)
    T = B * _mean_nodes(case)
    if op == "draft":
        # masks, per-node words of the five calls, and the register rows that move (3 in 4 sequences accept)
        rows = P_MATCH * L * B * CONV_WIDTH * 2
        return dict(bytes=B * case["hi"] ** 2 + 4.0 * 14 * T + rows * CONV_CHANNELS * 2, flops=0.0)
    # an accepted path is empty for one sequence in four and about three nodes long otherwise
    hit = P_MATCH * units
    verify = units * state + T * L * H * (4 * dk + 2 * dv + 8 + 4 * dv)
    commit = hit * (2 * state + 3 * (2 * dk + 2 * dv + 8))
    if op == "fused":
        commit -= hit * state                   # one read serves both
    return dict(bytes=verify + commit, flops=T * L * H * 8.0 * dk * dv + hit * 3 * 4.0 * dk * dv)


def tolerance(case):
    if case["op"] == "draft":
        return "exact"                          # whole numbers and copied 16-bit patterns
    if case["tf32"]:
        # one pass over the state at 10 mantissa bits, truncated: 3.6e-5 and 1.1e-3 from the fp64 oracle
        return {"rel": 1.5e-4, "max": 5e-3}
    # fp32 sums of up to 256 + 16 products: at most 6.7e-7 and 4.6e-6 from the fp64 oracle over these cases
    return {"rel": 2.7e-6, "max": 2e-5}
