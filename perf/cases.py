"""The work that a rollout engine has this library do, as cases that can be timed.

A speculative round is a proposal, one attention call per layer of the packed target forward, a verification, and
the bookkeeping that turns the round into the next one.  Each case is one such piece (or a whole round), called
through the binding as a step loop calls it: device tensors, work plans and workspaces are made once and kept, the
outputs go into tensors that are made once where the entry point takes them.

Shapes are those of the repository's workloads (heads, hidden size, vocabulary, node budget), batch sizes run from
the last straggling sequences of a rollout to its full concurrency.  Inputs are drawn on the device with the
distributions of ``paper_2608_04962_b200.inputs``: Gaussian weights and activations, log-normal cache lengths, the
best-first tree, target logits with one boosted mode token per node.
"""
import math
from statistics import NormalDist

import numpy as np
import torch

from paper_2608_04962_b200 import binding as S
from paper_2608_04962_b200 import inputs as I

DEV = "cuda"
BF16, F32, I32 = torch.bfloat16, torch.float32, torch.int32
PAGE = S.PAGE_TOKENS
SUPPORT = 48        # feedback support budget
RANK = 24           # sketch rank
SEVERITY_MIN = 0.03  # observations below it are discarded


# ------------------------------------------------------------------------------------------ the cases


def _case(name, op, model, B, N, **kw):
    w = I.WORKLOADS[model]
    c = {"op": op, "model": model, "B": B, "N": N, "k": w.k, "V": w.V, "T": 1.0, "kv": w.kv_a, "layers": 1}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a toy model's whole round: every launch and every host call shows
        _case("round_tiny", "round", "tiny", 4, 8, kv=160, layers=2, clip=0.1, paged=False),
        # the tail of a rollout: two sequences are left, ten nodes each, all layers of the model
        _case("round_tail_b2", "round", "qwen1.5b", 2, 10, kv=1500, layers=28, clip=0.0, paged=False),
        # the same model at full concurrency, all layers
        _case("round_full_b256", "round", "qwen1.5b", 256, 16, kv=1500, layers=28, clip=0.0, paged=False),
        # proposal for a handful of long sequences: the weights are streamed for 32 rows
        _case("propose_b8", "propose", "qwen7b", 8, 64, clip=0.0, affine=False, pre_head=False),
        # proposal of the largest shape, where the projection is a full contraction with a ragged last row block
        _case("propose_b64", "propose", "qwen14b", 64, 48, clip=0.0, affine=False, pre_head=False),
        # attention layers over a paged cache, odd batch and tree
        _case("attn_paged_b37", "attn", "qwen7b", 37, 29, kv=4900, layers=4, paged=True),
        # attention layers of the largest shape (240 query rows per KV head)
        _case("attn_b64", "attn", "qwen14b", 64, 48, kv=4000, layers=3, paged=False),
        # attention layers at low concurrency: few long sequences, the widest tree
        _case("attn_b8", "attn", "qwen7b", 8, 64, kv=10000, layers=4, paged=False),
        # verification of a small batch with a wide tree
        _case("verify_b16", "verify", "qwen7b", 16, 48, top_p=1.0, lazy=False),
        # verification as the experiments sample (nucleus 0.95), full concurrency
        _case("verify_nucleus_b256", "verify", "qwen1.5b", 256, 16, top_p=0.95, lazy=False),
        # verification from the target's hidden states, logits never stored
        _case("verify_fused_b32", "verify_fused", "qwen7b", 32, 32),
        # between two rounds: commit of the accepted paths, next hidden states, and the memory's feedback,
        # sketches and gate for one record per sequence and head
        _case("update_b128", "update", "qwen7b", 128, 32, kv=1500, layers=8),
    ]


def _tree_room(K, k):
    return min(64, sum(k ** i for i in range(K + 1)))


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_once(rng):
    op = rng.choice(["round", "propose", "propose", "attn", "attn", "verify", "verify", "verify_fused", "update"])
    model = rng.choice(["tiny", "qwen1.5b", "qwen7b", "qwen14b"] if op == "round" else ["qwen1.5b", "qwen7b", "qwen14b"])
    w = I.WORKLOADS[model]
    k = rng.choice([8, 8, 8, 8, 4, 2, 5]) if model != "tiny" else rng.choice([2, 3, 4])
    B = _log_int(rng, 1, 256)
    N = min(_log_int(rng, 4, 64), _tree_room(w.K, k))
    V = w.V if rng.random() < 0.6 else w.V - 8 * rng.randint(1, min(2000, w.V // 16))
    c = _case(None, op, model, B, N, k=k, V=V, T=rng.choice([1.0, 1.0, 1.0, 0.7, 1.3]))
    c["kv"] = _log_int(rng, 300, 10000) if model != "tiny" else _log_int(rng, 64, 1000)
    if op == "round":
        c.update(layers=_log_int(rng, 2, w.layers), clip=rng.choice([0.0, 0.1]), paged=rng.random() < 0.5)
    elif op == "propose":
        c.update(clip=rng.choice([0.0, 0.0, 0.1]), affine=rng.random() < 0.3, pre_head=rng.random() < 0.25)
    elif op == "attn":
        c.update(layers=rng.randint(2, 5), paged=rng.random() < 0.5)
    elif op == "verify":
        c.update(top_p=rng.choice([1.0, 0.95, 0.9]), lazy=rng.random() < 0.25)
    elif op == "update":
        c.update(layers=rng.randint(2, 8), kv=_log_int(rng, 300, 2000))
    return c


def _roof_s(c):
    w = work(c)
    return w["bytes"] / 6.4e12 + w["flops"] / 1.6e15


def draw(rng):
    """One more case of the same ranges: any piece of a round, any of the model shapes, 1 to 256 sequences, 4 to 64
    nodes, caches of 300 to 10000 tokens (median), ragged vocabularies, the options that a caller has."""
    most = 0.75 * max(_roof_s(c) for c in listed())
    while True:
        c = _draw_once(rng)
        if _roof_s(c) <= most and _state_bytes(c) <= 24e9:
            return c


# ------------------------------------------------------------------------------------------ sizes


def _lengths(c):
    """The cache lengths of a case: the quantiles of the workloads' log-normal law (the seed shuffles them)."""
    w, B = I.WORKLOADS[c["model"]], c["B"]
    most = w.kv_b if w.kv_kind == "lognormal" else 4 * c["kv"]
    z = np.array([NormalDist().inv_cdf((i + 0.5) / B) for i in range(B)])
    return np.rint(np.clip(c["kv"] * np.exp(0.7 * z), min(64, c["kv"]), max(most, c["kv"]))).astype(np.int32)


def _part_work(c, op):
    """Bytes and operations that one piece cannot do without: inputs read once, outputs written once."""
    w = I.WORKLOADS[c["model"]]
    B, N, K, k, d, V = c["B"], c["N"], w.K, c["k"], w.d, c["V"]
    if op == "propose":
        return (K * d * d * 2 + V * d * 2 + B * d * 2 + B * K * d * 4 + K * d * 2 + B * K * k * 8 + B * N * 13,
                2.0 * B * K * d * (d + V))
    if op == "attn":  # one layer
        t = int(_lengths(c).sum())
        return (t * w.Hkv * w.D * 4 + B * N * (2 * w.Hq + 2 * w.Hkv) * w.D * 2,
                4.0 * w.D * w.Hq * N * (t + B * (N + 1) / 2))
    if op == "verify":
        # statistics of every row; only the visited rows (about three of a sequence's) when the caller asks for those
        rows = min(N, 3) if c.get("lazy") else N
        return B * rows * V * 2 + B * N * 17 + B * K * k * 8 + B * (2 * K + 6) * 4, 4.0 * B * rows * V
    if op == "verify_fused":
        return V * d * 2 + B * N * d * 2 + B * N * 17 + B * K * k * 8, 2.0 * B * N * d * V
    # update: the records' logits rows, the support rows of W, the memory; the committed rows; hidden states
    R = B * K
    rows = B * (1 + K // 2) * w.Hkv * w.D * 2 * 2 * c["layers"]
    return (R * V * 2 + min(R * (SUPPORT + k), V) * d * 2 + R * d * 4 * 4 + 2 * rows + B * d * 4,
            4.0 * R * (SUPPORT + k) * d + 4.0 * R * RANK * d)


def work(c):
    if c["op"] == "round":
        parts = [_part_work(c, "propose")] + [_part_work(c, "attn")] * c["layers"] + [_part_work(c, "verify")]
    elif c["op"] == "attn":
        parts = [_part_work(c, "attn")] * c["layers"]
    else:
        parts = [_part_work(c, c["op"])]
    return {"bytes": float(sum(p[0] for p in parts)), "flops": float(sum(p[1] for p in parts))}


def _state_bytes(c):
    w, op = I.WORKLOADS[c["model"]], c["op"]
    weights = c["V"] * w.d * 2 + w.K * w.d * w.d * 2
    logits = c["B"] * c["N"] * c["V"] * 2
    cache = c["layers"] * _part_work(c, "attn")[0] * 1.2
    return {"round": weights + logits + cache, "propose": weights, "attn": cache, "verify": logits,
            "verify_fused": weights, "update": weights + logits + cache}[op] * 1.1


def tolerance(c):
    if c["op"] == "attn":
        return {"rel": 1e-2}  # bf16 outputs
    if c["op"] == "verify":
        # fp32 sums; a walk or a draw may turn where a uniform lies within rounding of its bound
        return {"rel": 1e-4, "differ": 5e-3}
    if c["op"] == "verify_fused":
        return {"rel": 2e-3, "differ": 1e-2}  # statistics of logits that are rounded to bf16
    if c["op"] == "update":
        return {"rel": 2e-4, "differ": 5e-3}  # fp32 sums with cancellation, then products of them
    # proposals round to bf16 twice before the projection: near ties of candidates may change places
    return {"rel": 1e-2, "differ": 1e-2}


# ------------------------------------------------------------------------------------------ inputs


def _randn(g, shape, std=1.0):
    x = torch.randn(shape, generator=g, device=DEV, dtype=BF16)
    return x.mul_(std) if std != 1.0 else x


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV, dtype=F32)


def _propose_state(c, g, st):
    w = I.WORKLOADS[c["model"]]
    B, N, K, k, d, V = c["B"], c["N"], w.K, c["k"], w.d, c["V"]
    pre = bool(c.get("pre_head"))
    st.update(A=_randn(g, (K, d, d), 0.02), bias=_randn(g, (K, d), 0.02), W=_randn(g, (V, d), 0.02),
              h=_randn(g, (B, d), 0.02), anchor=torch.randint(0, V, (B,), generator=g, device=DEV, dtype=I32),
              u_draw=_rand(g, B, N), gamma=None, beta=None)
    if c.get("affine"):
        st["gamma"], st["beta"] = 1.0 + _randn(g, (K, d), 0.1), _randn(g, (K, d), 0.1)
    # the gate is open for half of the rows
    ratio = torch.tensor((list(w.alpha_heads) + [0.003] * K)[:K], device=DEV)
    if pre:
        st["m"], st["alpha"] = torch.randn((B, d), generator=g, device=DEV), 0.02 * (_rand(g, B) < 0.5)
    else:
        st["m"], st["alpha"] = torch.randn((B, K, d), generator=g, device=DEV), (_rand(g, B, K) < 0.5) * ratio
    st["alpha"] = st["alpha"].to(F32).contiguous()
    st["propose_flags"] = S.REFLEX_PRE_HEAD if pre else 0
    st["ws_propose"] = torch.empty(S.propose_workspace_bytes(B, N, K, k, d, V, c["T"], flags=st["propose_flags"]),
                                   dtype=torch.uint8, device=DEV)
    st["prop"] = {"cand_id": torch.empty((B, K, k), dtype=I32, device=DEV),
                  "cand_logit": torch.empty((B, K, k), dtype=F32, device=DEV),
                  "tree_tok": torch.empty((B, N), dtype=I32, device=DEV),
                  "tree_cand": torch.empty((B, N), dtype=torch.uint8, device=DEV),
                  "slot_q": torch.empty((B, N), dtype=F32, device=DEV)}


def _propose(st):
    c = st["case"]
    return S.propose(st["h"], st["anchor"], st["A"], st["bias"], st["W"], st["m"], st["alpha"], st["parent"],
                     st["u_draw"], k=c["k"], temperature=c["T"], clip_c=c.get("clip", 0.0), ln_gamma=st["gamma"],
                     ln_beta=st["beta"], workspace=st["ws_propose"], out=st["prop"], flags=st["propose_flags"])


def _pages(L, spare, seed):
    """Page table of a pool: 128-token pages in a random order, room for `spare` more tokens per sequence."""
    own = (L.astype(np.int64) + spare + PAGE - 1) // PAGE
    indptr = np.zeros(len(L) + 1, np.int32)
    np.cumsum(own, out=indptr[1:])
    n_pages = int(indptr[-1]) + 3
    return I.rng(seed).permutation(n_pages)[: int(indptr[-1])].astype(np.int32), indptr, n_pages


def _attn_state(c, g, seed, st):
    w = I.WORKLOADS[c["model"]]
    B, N = c["B"], c["N"]
    L = I.rng(seed + 7).permutation(_lengths(c)).astype(np.int32)
    st["kv_len_host"] = L
    if c["paged"]:
        table, indptr, n_pages = _pages(L, w.K + 1, seed + 9)
        st["page_table"], st["page_indptr"] = torch.from_numpy(table).to(DEV), torch.from_numpy(indptr).to(DEV)
        st["kv_len"] = torch.from_numpy(L).to(DEV)
        shape = (n_pages, PAGE, w.Hkv, w.D)
        nbytes = S.tree_attn_paged_workspace_bytes(B, N, w.Hq, w.Hkv, w.D, L)
    else:
        ip = np.zeros(B + 1, np.int32)
        np.cumsum(L, out=ip[1:])
        st["kv_indptr_host"], st["kv_indptr"] = ip, torch.from_numpy(ip).to(DEV)
        shape = (int(ip[-1]), w.Hkv, w.D)
        nbytes = S.tree_attn_workspace_bytes(B, N, w.Hq, w.Hkv, w.D, ip)
    st["ws_attn"] = torch.empty(nbytes, dtype=torch.uint8, device=DEV)
    layers = range(c["layers"])
    st["Q"] = [_randn(g, (B, N, w.Hq, w.D)) for _ in layers]
    st["Kc"], st["Vc"] = [_randn(g, shape) for _ in layers], [_randn(g, shape) for _ in layers]
    st["Kt"] = [_randn(g, (B, N, w.Hkv, w.D)) for _ in layers]
    st["Vt"] = [_randn(g, (B, N, w.Hkv, w.D)) for _ in layers]
    st["O"] = [torch.empty((B, N, w.Hq, w.D), dtype=BF16, device=DEV) for _ in layers]


def _attn(st):
    # all layers of a round see the same lengths: the layers after the first keep the plan, and the caches were
    # written before the round began
    for i in range(st["case"]["layers"]):
        flags = S.ATTN_REUSE_PLAN | S.ATTN_CACHE_SETTLED if i else 0
        if st["case"]["paged"]:
            S.tree_attn_paged(st["Q"][i], st["Kc"][i], st["Vc"][i], st["page_table"], st["page_indptr"], st["kv_len"],
                              st["kv_len_host"], st["Kt"][i], st["Vt"][i], st["parent"], workspace=st["ws_attn"],
                              out=st["O"][i], flags=flags)
        else:
            S.tree_attn(st["Q"][i], st["Kc"][i], st["Vc"][i], st["kv_indptr"], st["kv_indptr_host"], st["Kt"][i],
                        st["Vt"][i], st["parent"], workspace=st["ws_attn"], out=st["O"][i], flags=flags)
    return st["O"]


def _candidates(c, g, rows):
    """k distinct token ids per row, with a peaked head's logits in descending order."""
    V, k = c["V"], c["k"]
    first = torch.randint(0, V, (rows, 1), generator=g, device=DEV)
    step = torch.randint(1, V // k, (rows, 1), generator=g, device=DEV)
    ids = ((first + step * torch.arange(k, device=DEV)) % V).to(I32)
    lg = torch.randn((rows, k), generator=g, device=DEV) * 1.5
    return ids, lg.sort(dim=1, descending=True).values.contiguous()


def _mode_tokens(c, g, parent, tree_tok):
    """Per node the target's favourite token: the first child's (45 %), the second child's (15 %) or any other."""
    B, N = tree_tok.shape
    mode = torch.randint(0, c["V"], (B, N), generator=g, device=DEV)
    pick = _rand(g, B, N)
    tok = tree_tok.long()
    kids = [[n for n in range(1, N) if parent[n] == u] for u in range(N)]
    for u in range(N):
        for i, (lo, hi) in enumerate(((0.0, 0.45), (0.45, 0.6))):
            if len(kids[u]) > i:
                hit = (pick[:, u] >= lo) & (pick[:, u] < hi)
                mode[:, u] = torch.where(hit, tok[:, kids[u][i]], mode[:, u])
    return mode


def _logits(c, g, mode):
    B, N = mode.shape
    lg = _randn(g, (B, N, c["V"]))
    at = mode.unsqueeze(-1)
    return lg.scatter_(2, at, (lg.gather(2, at).float() + 14.0).to(BF16))


def _verify_state(c, g, st):
    w = I.WORKLOADS[c["model"]]
    B, N, K, k, V = c["B"], c["N"], w.K, c["k"], c["V"]
    st["u_acc"], st["u_fin"] = _rand(g, B, N), _rand(g, B)
    size = S.verify_nucleus_workspace_bytes if c.get("top_p", 1.0) < 1.0 else S.verify_workspace_bytes
    st["ws_verify"] = torch.empty(size(B, N, K, k, V, c["T"]), dtype=torch.uint8, device=DEV)
    st["verify_flags"] = S.VERIFY_LAZY_STATS if c.get("lazy") else 0
    # (rows that a lazy verification does not visit keep what they hold)
    out = {n: torch.zeros(s, dtype=t, device=DEV) for n, s, t in (
        ("n_acc", (B,), I32), ("path_node", (B, K + 1), I32), ("out_tok", (B, K + 1), I32), ("term_node", (B,), I32),
        ("term_kind", (B,), I32), ("row_max", (B, N), F32), ("row_sum", (B, N), F32), ("min_margin", (B,), F32))}
    if c.get("top_p", 1.0) < 1.0:
        out["nucleus_thr"], out["nucleus_sum"] = torch.zeros((B, N), device=DEV), torch.zeros((B, N), device=DEV)
    st["ver"] = out


def _verify(st):
    c, p = st["case"], st["prop"]
    args = (st["logits"], st["parent"], p["tree_tok"], p["tree_cand"], p["cand_id"], p["cand_logit"], st["u_acc"],
            st["u_fin"])
    if c.get("top_p", 1.0) < 1.0:
        return S.verify_nucleus(*args, c["top_p"], temperature=c["T"], workspace=st["ws_verify"], out=st["ver"],
                                flags=st["verify_flags"])
    return S.verify(*args, temperature=c["T"], workspace=st["ws_verify"], out=st["ver"], flags=st["verify_flags"])


def _drawn_tree(c, g, st):
    """Candidates and a tree drawn from them, as a proposal leaves them."""
    w = I.WORKLOADS[c["model"]]
    B, N = c["B"], c["N"]
    ids, lg = _candidates(c, g, B * w.K)
    prop = {"cand_id": ids.view(B, w.K, c["k"]), "cand_logit": lg.view(B, w.K, c["k"])}
    anchor = torch.randint(0, c["V"], (B,), generator=g, device=DEV, dtype=I32)
    prop.update(S.tree_draw(st["parent"], anchor, prop["cand_id"], prop["cand_logit"], _rand(g, B, N), temperature=c["T"]))
    st["prop"] = prop


def _update_state(c, g, seed, st):
    w = I.WORKLOADS[c["model"]]
    B, N, K, k, d, V = c["B"], c["N"], w.K, c["k"], w.d, c["V"]
    parent, R, host = st["parent"], B * w.K, I.rng(seed + 11)
    depth = I.node_depths(parent)
    _drawn_tree(c, g, st)
    mode = _mode_tokens(c, g, parent, st["prop"]["tree_tok"])
    st["logits"] = _logits(c, g, mode)
    st["W"] = _randn(g, (V, d), 0.02)
    top, tot = [], []
    for rows in st["logits"].split(max(1, (1 << 27) // (N * V))):
        x = rows.float() / c["T"]
        top.append(rows.amax(-1).float())
        tot.append(torch.exp(torch.logsumexp(x, -1) - top[-1] / c["T"]))
    st["row_max"], st["row_sum"] = torch.cat(top).view(-1), torch.cat(tot).view(-1)
    # a record per (sequence, head): a node of the head's depth, the token that was emitted there
    levels = [np.flatnonzero(depth == min(h, int(depth.max()))) for h in range(K)]
    node = np.stack([host.choice(v, size=B) for v in levels], 1)
    row = torch.from_numpy((np.arange(B)[:, None] * N + node).reshape(-1).astype(np.int32)).to(DEV)
    st["rec_row"], st["y_star"] = row, mode.view(-1)[row.long()].to(I32)
    st["rec_cand"], st["rec_logit"] = (st["prop"][n].view(R, k) for n in ("cand_id", "cand_logit"))
    st["rho"], st["rec_mem"] = torch.full((R,), 0.9, device=DEV), torch.arange(R, device=DEV, dtype=I32)
    st["m"] = torch.randn((R, d), generator=g, device=DEV)
    st["ws_feedback"] = torch.empty(S.reflex_feedback_workspace_bytes(R, k, SUPPORT, d, V, c["T"]), dtype=torch.uint8, device=DEV)
    st["Pi"] = torch.randn((RANK, d), generator=g, device=DEV)
    s = torch.randn((R, RANK), generator=g, device=DEV)
    st["sketch"] = s / s.norm(dim=1, keepdim=True)
    st["slot"], st["horizon"] = torch.arange(R, device=DEV, dtype=I32), (torch.arange(R, device=DEV) % K).to(I32)
    st["n"], st["n_fb"] = torch.full((R,), 8, device=DEV, dtype=I32), torch.full((R,), 20, device=DEV, dtype=I32)
    st["mean"], st["M2"] = 0.3 * _rand(g, R), 0.5 + _rand(g, R)
    st["n_align"] = torch.tensor([min(1 << h, 8) for h in range(K)], device=DEV, dtype=I32)
    st["n_feed"] = torch.tensor([6, 16, 48, 48, 48, 48, 48, 48][:K], device=DEV, dtype=I32)
    hi = torch.tensor((list(w.alpha_heads) + [0.003] * K)[:K], device=DEV)
    st["alpha_lo"], st["alpha_hi"] = 0.5 * hi, hi
    # the accepted path of every sequence and the paged caches it is appended to
    last = host.integers(0, N, size=B)
    path, n_acc = np.full((B, K + 1), -1, np.int32), depth[last].astype(np.int32)
    for b in range(B):
        u = int(last[b])
        while u >= 0:
            path[b, depth[u]] = u
            u = int(parent[u])
    st["path_node"], st["n_acc"] = torch.from_numpy(path).to(DEV), torch.from_numpy(n_acc).to(DEV)
    st["term_node"] = torch.from_numpy(last.astype(np.int32)).to(DEV)
    st["hidden"] = _randn(g, (B, N, d))
    L = host.permutation(_lengths(c)).astype(np.int32)
    table, indptr, n_pages = _pages(L, K + 1, seed + 9)
    st["page_table"], st["page_indptr"] = torch.from_numpy(table).to(DEV), torch.from_numpy(indptr).to(DEV)
    st["kv_len"] = torch.from_numpy(L).to(DEV)
    st["kv_len_next"], st["status"] = torch.zeros_like(st["kv_len"]), torch.zeros(1, device=DEV, dtype=I32)
    st["Kp"], st["Vp"] = ([_randn(g, (n_pages, PAGE, w.Hkv, w.D)) for _ in range(c["layers"])] for _ in "KV")
    st["Kt"], st["Vt"] = ([_randn(g, (B, N, w.Hkv, w.D)) for _ in range(c["layers"])] for _ in "KV")


def _update(st):
    c = st["case"]
    S.commit_path_layers(st["Kt"], st["Vt"], st["path_node"], st["n_acc"], st["Kp"], st["Vp"], st["page_table"],
                         st["page_indptr"], st["kv_len"], kv_len_out=st["kv_len_next"], status=st["status"])
    h_next = S.gather_hidden(st["hidden"], st["term_node"])
    fb = S.reflex_feedback(st["logits"], st["rec_row"], st["row_max"], st["row_sum"], st["rec_cand"], st["rec_logit"],
                           st["y_star"], st["W"], st["rho"], st["rec_mem"], st["m"], k_support=SUPPORT,
                           temperature=c["T"], workspace=st["ws_feedback"], severity_min=SEVERITY_MIN, want_e=True)
    xi = S.reflex_sketch(fb["e"], st["Pi"])
    keep = (fb["severity"] >= SEVERITY_MIN).to(torch.uint8)
    gate = S.reflex_gate(st["sketch"], xi, st["slot"], keep, st["n"], st["mean"], st["M2"], st["n_fb"], st["m"],
                         st["horizon"], st["n_align"], st["n_feed"], st["alpha_lo"], st["alpha_hi"])
    s_next = S.reflex_sketch(st["m"], st["Pi"])
    return {"Kp": st["Kp"], "Vp": st["Vp"], "kv_len": st["kv_len_next"], "status": st["status"], "h": h_next,
            "feedback": fb, "xi": xi, "gate": gate, "sketch": s_next, "m": st["m"], "n": st["n"], "n_fb": st["n_fb"],
            "mean": st["mean"], "M2": st["M2"]}


def prepare(c, seed):
    op, seed = c["op"], int(seed)
    w = I.WORKLOADS[c["model"]]
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    st = {"case": c, "parent": I.best_first_topology(c["N"], w.K, c["k"])}
    if op in ("round", "propose"):
        _propose_state(c, g, st)
    if op in ("round", "attn"):
        _attn_state(c, g, seed, st)
    if op == "round":
        _verify_state(c, g, st)
        tok = _propose(st)["tree_tok"]
        st["logits"] = _logits(c, g, _mode_tokens(c, g, st["parent"], tok))
    elif op == "verify":
        _drawn_tree(c, g, st)
        _verify_state(c, g, st)
        st["logits"] = _logits(c, g, _mode_tokens(c, g, st["parent"], st["prop"]["tree_tok"]))
    elif op == "verify_fused":
        _drawn_tree(c, g, st)
        st["u_acc"], st["u_fin"] = _rand(g, c["B"], c["N"]), _rand(g, c["B"])
        st["W"] = _randn(g, (c["V"], w.d), 0.02)
        # hidden states that point along their mode token's row: its logit stands 14 above a background of about 1
        mode = _mode_tokens(c, g, st["parent"], st["prop"]["tree_tok"])
        rows = st["W"][mode.view(-1)].float()
        h = torch.randn((c["B"] * c["N"], w.d), generator=g, device=DEV) * (1.0 / (0.02 * math.sqrt(w.d)))
        h += rows * (14.0 / rows.square().sum(1, keepdim=True))
        st["hidden"] = h.to(BF16).view(c["B"], c["N"], w.d)
    elif op == "update":
        _update_state(c, g, seed, st)
    return st


def run(st):
    """One pass: a whole round (proposal, attention of every layer, verification), or one piece of it."""
    op = st["case"]["op"]
    if op == "round":
        return {"prop": _propose(st), "O": _attn(st), "ver": _verify(st)}
    if op == "propose":
        return _propose(st)
    if op == "attn":
        return _attn(st)
    if op == "verify":
        return _verify(st)
    if op == "verify_fused":
        p = st["prop"]
        return S.verify_fused(st["hidden"], st["W"], st["parent"], p["tree_tok"], p["tree_cand"], p["cand_id"],
                              p["cand_logit"], st["u_acc"], st["u_fin"], temperature=st["case"]["T"])
    return _update(st)
