"""Performance cases of the ReSS layer: the calls a user of this package makes, over the sizes
it is used at, each with its inputs, one pass of it, its work and its result in float64.

An operation is one of
  forward       ress_forward: selection and sparse attention of one layer, device buffers
  forward_host  ress_forward_host: the same from and to page-locked host buffers
  select        ress_score and ress_restore: the kept-block lists alone
  attn          ress_sparse_attn over kept-block lists the caller made itself
  out_proj      ress_out_proj: the residual update y = x + O W_o^T
  token_drift   ress_token_drift: what a change of the attention output leaves in the stream

Sizes are those of 3D-ViT global attention: every view brings 37 x 37 patch tokens and 5
special tokens, the special tokens of all views last (2 to 100 views), and generic ragged
lengths.  The random inputs follow the recipe of the package's synthetic layers: noise plus a
low-rank component shared by the tokens of a view and a positional ramp, rounded to bf16.
"""
import math

import torch

import paper_2609_35593_gb300 as ress

PATCHES, SPECIAL = 37 * 37, 5  # tokens of one view


def _views(n):
    return {"tokens": n * (PATCHES + SPECIAL), "special": n * SPECIAL, "views": n}


def listed():
    layer = {"op": "forward", "heads": 16, "d_model": 1024, "rank": 16, "cross": 0, "sparsity": 0.9,
             "rounds": 3, "q_block": 64}
    return [
        # the smallest layer that is used: a pair of images; launches and latency count
        {**layer, **_views(2), "name": "fwd_v2", "heads": 4, "d_model": 256, "rank": 8, "sparsity": 0.5,
         "rounds": 2},
        # a cropped sequence with odd sizes: ragged last block, three heads, one round
        {**layer, "name": "fwd_ragged", "tokens": 5003, "special": 37, "views": 4, "heads": 3,
         "d_model": 192, "rank": 4, "sparsity": 0.6, "rounds": 1},
        # an ordinary scene of few images
        {**layer, **_views(8), "name": "fwd_v8", "sparsity": 0.75},
        # the same layer for a program that keeps activations in host memory
        {**layer, **_views(8), "name": "fwd_host_v8", "op": "forward_host", "sparsity": 0.75},
        # the headline layer: 32 images at 90% block sparsity
        {**layer, **_views(32), "name": "fwd_v32"},
        # the headline layer on the grid of 128-token query blocks
        {**layer, **_views(32), "name": "fwd_v32_q128", "q_block": 128},
        # the long-view layer, the largest
        {**layer, **_views(100), "name": "fwd_v100", "cross": 4},
        # a low-sparsity point of the 64-view sweep: large budgets, many rounds, lists only
        {**layer, **_views(64), "name": "select_v64_s50", "op": "select", "sparsity": 0.5, "rounds": 4},
        # attention over a selection rule of the caller's own
        {**layer, **_views(12), "name": "attn_v12_s80", "op": "attn", "sparsity": 0.8, "rounds": 0},
        # the dense run of the attention that sparse runs are compared with
        {**layer, **_views(16), "name": "attn_v16_dense", "op": "attn", "sparsity": 0.0, "rounds": 0},
        # what follows the attention in the layer
        {**layer, **_views(32), "name": "out_proj_v32", "op": "out_proj"},
        # how far a sparse layer's output is from the dense one, in the residual stream
        {**layer, **_views(8), "name": "token_drift_v8", "op": "token_drift"},
    ]


def draw(rng):
    op = rng.choice(["forward"] * 6 + ["select"] * 2 + ["attn"] * 2 + ["out_proj", "token_drift", "forward_host"])
    case = {"op": op, "cross": 0, "rank": rng.choice([4, 8, 16]), "q_block": rng.choice([64, 64, 64, 128]),
            "sparsity": rng.choice([0.5, 0.6, 0.75, 0.8, 0.9, 0.9, 0.95]),
            "rounds": rng.choice([0, 1, 2, 3, 3, 4]), "heads": rng.choice([3, 4, 8, 12, 16, 16])}
    case["d_model"] = 64 * case["heads"]
    if op == "attn":
        case["sparsity"], case["rounds"] = rng.choice([0.0, 0.5, 0.8, 0.9]), 0
    # no dearer than the largest listed case: kept query-key pairs of all heads
    most = {"forward_host": 32 * 1374, "attn": 64 * 1374}.get(op, 100 * 1374)
    while True:
        if rng.random() < 0.5:  # whole views
            lo, hi = math.log(2), math.log(most / 1374)
            case.update(_views(round(math.exp(rng.uniform(lo, hi)))))
        else:  # any length
            n = int(math.exp(rng.uniform(math.log(2000), math.log(most))))
            case.update({"tokens": n, "special": rng.randrange(0, 200), "views": 1 + n // 1374})
        if _kept_pairs(case) <= 2.5e10 and case["tokens"] * case["heads"] <= 100 * 1374 * 16:
            return case


# ---- sizes ---------------------------------------------------------------------------------
def _grid(case):
    """Key blocks, candidate key blocks, query blocks, candidate query blocks, budget."""
    n, s, qb = case["tokens"], case["special"], case["q_block"]
    nb, nc, nq, nqc = -(-n // 64), (n - s) // 64, -(-n // qb), (n - s) // qb
    c = min(max(2, round((1.0 - case["sparsity"]) * nc)), nc)
    return nb, nc, nq, nqc, c


def _kept_pairs(case):
    nb, nc, nq, nqc, c = _grid(case)
    qb, n = case["q_block"], case["tokens"]
    return case["heads"] * (nqc * qb * ((c + nb - nc) * 64.0) + (n - nqc * qb) * float(n))


def work(case):
    n, h, dm, op = case["tokens"], case["heads"], case["d_model"], case["op"]
    nb, nc, nq, nqc, c = _grid(case)
    x = 2 * n * h * 64  # one of Q, K, V, O
    lists = 4 * (h * (nqc * (c + nb - nc) + (nq - nqc) * nb) + h * nq)
    # pooled logits, pooled output, drift norms and one gain product per round
    products = 2.0 * 64 * h * nqc * (3 * nb + case["rounds"] * nc)
    attention = 4.0 * 64 * _kept_pairs(case)
    if op in ("forward", "forward_host"):
        return {"bytes": 4 * x + lists + 4 * h * nq, "flops": products + attention}
    if op == "select":
        return {"bytes": 3 * x + lists + 4 * h * nq + h * nq * (nb / 8), "flops": products + 3 * n * h * 64}
    if op == "attn":
        return {"bytes": 4 * x + lists, "flops": attention}
    if op == "out_proj":
        return {"bytes": x + 2 * (dm * h * 64 + 2 * n * dm), "flops": 2.0 * n * h * 64 * dm}
    return {"bytes": 2 * x + 2 * dm * h * 64 + 4 * nb, "flops": 4.0 * n * h * 64 * dm}


# ---- inputs --------------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _qkv(case, g):
    n, s, h, v, r = case["tokens"], case["special"], case["heads"], case["views"], case["rank"]
    shared = torch.zeros(n, h * 64, device="cuda")
    U = _normal(g, v, r, h * 64)
    for t0, t1 in ((0, n - s), (n - s, n)):  # patch tokens of all views, then special tokens
        if t1 > t0:
            per = -(-(t1 - t0) // v)
            a = _normal(g, v, per, r)
            shared[t0:t1] = (torch.bmm(a, U) * (2.0 / math.sqrt(r))).reshape(v * per, h * 64)[:t1 - t0]
    if case["cross"]:
        shared += _normal(g, n, case["cross"]) @ _normal(g, case["cross"], h * 64) / math.sqrt(case["cross"])
    per = -(-(n - s) // v)
    ramp = torch.zeros(n, 1, device="cuda")
    ramp[:n - s, 0] = 2.0 * (torch.arange(n - s, device="cuda") % per) / max(1, per - 1) - 1.0
    out = []
    for _ in range(3):
        x = _normal(g, n, h * 64)
        x += shared
        x += ramp * _normal(g, 1, h * 64)
        out.append(x.to(torch.bfloat16).view(n, h, 64))
    return out


def _w_o(case, g):
    return (0.02 * _normal(g, case["d_model"], case["heads"] * 64)).to(torch.bfloat16)


def _caller_lists(case, Q, K):
    """Kept-block lists of a caller's own rule: the blocks whose mean key has the largest
    product with the query block's mean query, the blocks of special tokens always."""
    nb, nc, nq, nqc, c = _grid(case)
    h = case["heads"]
    rows = torch.arange(nb, device="cuda", dtype=torch.int32).repeat(h, nq, 1)
    if c >= nc:
        col = rows.reshape(-1)
        return torch.arange(0, h * nq * nb + 1, nb, device="cuda", dtype=torch.int32), col
    q, k = _block_means(Q.double(), case["q_block"]), _block_means(K.double(), 64)
    top = torch.sort(torch.einsum("hid,hjd->hij", q[:, :nqc], k[:, :nc]), dim=2, descending=True, stable=True)[1]
    kept = torch.sort(top[:, :, :c], dim=2)[0].int()
    kept = torch.cat([kept, rows[:, :nqc, nc:]], dim=2)
    col = torch.cat([torch.cat([kept[i].reshape(-1), rows[i, nqc:].reshape(-1)]) for i in range(h)])
    lengths = torch.full((h, nq), nb, device="cuda", dtype=torch.int64)
    lengths[:, :nqc] = kept.shape[2]
    ptr = torch.zeros(h * nq + 1, device="cuda", dtype=torch.int64)
    ptr[1:] = torch.cumsum(lengths.reshape(-1), 0)
    return ptr.int(), col.contiguous()


def _inputs(case, seed):
    g = _generator(seed)
    n, h, dm, op = case["tokens"], case["heads"], case["d_model"], case["op"]
    if op == "out_proj":
        return {"O": (0.7 * _normal(g, n, h, 64)).to(torch.bfloat16), "W_o": _w_o(case, g),
                "x": _normal(g, n, dm).to(torch.bfloat16)}
    if op == "token_drift":
        a = 0.7 * _normal(g, n, h, 64)
        b = a + 0.1 * _normal(g, n, h, 64)
        return {"O_a": a.to(torch.bfloat16), "O_b": b.to(torch.bfloat16), "W_o": _w_o(case, g)}
    Q, K, V = _qkv(case, g)
    return {"Q": Q, "K": K, "V": V, "W_o": _w_o(case, g)}


def prepare(case, seed):
    s = _inputs(case, seed)
    n, h, op = case["tokens"], case["heads"], case["op"]
    nb, nc, nq, nqc, c = _grid(case)
    d = ress.dims(n, h, case["special"], case["d_model"], case["q_block"])
    s.update(op=op, d=d, c_h=[c] * h, rounds=case["rounds"], rho=0.5)
    if op in ("out_proj", "token_drift", "attn"):
        s["ws"] = torch.zeros(ress.workspace_bytes(d), dtype=torch.uint8, device="cuda")
        if op == "out_proj":
            s["y"] = torch.empty_like(s["x"])
        elif op == "token_drift":
            s["drift"] = torch.empty(nb, dtype=torch.float32, device="cuda")
        else:
            s["row_ptr"], s["col_idx"] = _caller_lists(case, s["Q"], s["K"])
            s["O"] = torch.empty_like(s["Q"])
        return s
    s["buf"] = ress.Buffers(d, s["c_h"])
    ress.prepare_wo(d, s["W_o"], s["buf"].F)
    if op == "select":
        s["mask"] = torch.zeros(h * nq, -(-nb // 32), dtype=torch.int32, device="cuda")
    if op == "forward_host":
        for k in ("Q", "K", "V"):
            s[k + "_host"] = s[k].cpu().pin_memory()
        s["O_host"] = torch.empty(n, h, 64, dtype=torch.bfloat16).pin_memory()
    return s


# ---- one pass ------------------------------------------------------------------------------
def run(s):
    op, d = s["op"], s["d"]
    if op == "out_proj":
        ress.out_proj(d, s["O"], s["W_o"], s["x"], s["y"], s["ws"])
        return {"y": s["y"]}
    if op == "token_drift":
        ress.token_drift(d, s["O_a"], s["O_b"], s["W_o"], s["drift"], s["ws"])
        return {"drift": s["drift"]}
    if op == "attn":
        ress.sparse_attn(d, s["Q"], s["K"], s["V"], s["row_ptr"], s["col_idx"], s["O"], s["ws"])
        return {"O": s["O"]}
    b = s["buf"]
    lists = {"row_ptr": b.row_ptr, "col_idx": b.col_idx, "J_best": b.J_best}
    if op == "select":
        ress.score(d, s["Q"], s["K"], s["V"], b.F, s["c_h"], b.ws)
        ress.restore(d, s["c_h"], s["rounds"], s["rho"], b.ws, b.row_ptr, b.col_idx, b.J_best, s["mask"])
        return {**lists, "mask": s["mask"]}
    if op == "forward_host":
        ress.forward_host(d, s["Q_host"], s["K_host"], s["V_host"], s["O_host"], s["Q"], s["K"], s["V"], b.O,
                          b.F, s["c_h"], s["rounds"], s["rho"], b.ws, b.row_ptr, b.col_idx, b.J_best)
        torch.cuda.current_stream().synchronize()  # the output is read on the host
        return {**lists, "O": s["O_host"]}
    ress.forward(d, s["Q"], s["K"], s["V"], b.F, s["c_h"], s["rounds"], s["rho"], b.ws, b.row_ptr,
                 b.col_idx, b.O, b.J_best)
    return {**lists, "O": b.O}


# ---- the same in float64 -------------------------------------------------------------------
def _block_means(x, size):
    """[N, H, 64] float64 -> [H, blocks, 64]: the mean of each block's tokens."""
    n, h = x.shape[:2]
    blocks = -(-n // size)
    full = torch.zeros(blocks * size, h, 64, dtype=x.dtype, device=x.device)
    full[:n] = x
    count = torch.full((blocks,), float(size), dtype=x.dtype, device=x.device)
    count[-1] = n - (blocks - 1) * size
    return (full.view(blocks, size, h, 64).sum(1) / count[:, None, None]).transpose(0, 1).contiguous()


def _top(keys, member, m):
    """Mask of each row's m largest keys among the members, ties to the lower index."""
    order = torch.sort(keys.masked_fill(~member, -math.inf), dim=1, descending=True, stable=True)[1]
    out = torch.zeros_like(member)
    return out.scatter_(1, order[:, :m], True)


def _exact_selection(case, Q, K, V, W_o):
    """Drop sets [H, candidate rows, candidates] and their drift J [H, candidate rows]."""
    nb, nc, nq, nqc, c = _grid(case)
    eps, drops, drift = 1e-4, [], []
    q, k, v = (_block_means(x, s) for x, s in ((Q, case["q_block"]), (K, 64), (V, 64)))
    for h in range(case["heads"]):
        W = W_o[:, 64 * h:64 * h + 64].double()
        M = W.T @ W
        P = torch.softmax(q[h, :nqc] @ k[h].T / 8.0, dim=1)
        y = P @ v[h]
        yM, vM = y @ M, v[h] @ M
        qn = ((yM * y).sum(1)[:, None] + (vM * v[h]).sum(1)[None] - 2.0 * yM @ v[h].T).clamp_min(0.0)
        Pc, qc, vc = P[:, :nc], qn[:, :nc], v[h, :nc]
        everyone = torch.ones_like(Pc, dtype=torch.bool)
        D = ~_top(Pc * qc.sqrt() / (1.0 - Pc).clamp_min(eps), everyone, c)

        def state(D):
            PD = Pc * D
            g = PD.sum(1)[:, None] * y - PD @ vc
            kept = 1.0 - PD.sum(1)
            G = ((g @ M) * g).sum(1)
            return g, kept, G, G / kept.clamp_min(eps) ** 2

        g, kept, G, J = state(D)
        best, bestD = J.clone(), D.clone()
        for r in range(case["rounds"]):
            m = min(math.floor(0.5 * c / 2.0 ** (r + 1)), nc - c, c)
            if m <= 0:
                continue
            t = Pc * (((y @ M) * g).sum(1)[:, None] - g @ M @ vc.T)
            sign = torch.where(D, -1.0, 1.0).to(Pc.dtype)
            G2 = G[:, None] + 2.0 * sign * t + Pc * Pc * qc
            gain = J[:, None] - G2 / (kept[:, None] - sign * Pc).clamp_min(eps) ** 2
            D = (D & ~_top(gain, D, m)) | _top(gain, ~D, m)
            g, kept, G, J = state(D)
            better = J < best
            best = torch.where(better, J, best)
            bestD[better] = D[better]
        drops.append(bestD)
        drift.append(best)
    return torch.stack(drops), torch.stack(drift)


def _exact_rows(q, k, v, valid, idx):
    """Attention of query blocks q [R, size, 64] over the key blocks idx [R, L] of k, v
    [nb, 64, 64] (float64)."""
    out, step = torch.empty_like(q), max(1, int(2.5e7 // (idx.shape[1] * 64 * max(64, q.shape[1]))))
    for r in range(0, q.shape[0], step):
        i = idx[r:r + step]
        kk, vv = k[i].flatten(1, 2), v[i].flatten(1, 2)
        s = torch.bmm(q[r:r + step], kk.transpose(1, 2)) / 8.0
        s.masked_fill_(~valid[i].flatten(1)[:, None, :], -math.inf)
        out[r:r + step] = torch.bmm(torch.softmax(s, dim=2), vv)
    return out


def _exact_attention(case, Q, K, V, kept):
    """kept: [H, candidate rows, L] key blocks of each candidate query block."""
    nb, nc, nq, nqc, c = _grid(case)
    n, h, qb = case["tokens"], case["heads"], case["q_block"]

    def blocks(x, size, count):
        full = torch.zeros(count * size, 64, dtype=torch.float64, device="cuda")
        full[:n] = x
        return full.view(count, size, 64)

    out = torch.empty(n, h, 64, dtype=torch.float64, device="cuda")
    valid = (torch.arange(nb * 64, device="cuda") < n).view(nb, 64)
    everything = torch.arange(nb, device="cuda").repeat(max(1, nq - nqc), 1)
    for i in range(h):
        q, k, v = blocks(Q[:, i], qb, nq), blocks(K[:, i], 64, nb), blocks(V[:, i], 64, nb)
        parts = [_exact_rows(q[:nqc], k, v, valid, kept[i])] if nqc else []
        if nq > nqc:
            parts.append(_exact_rows(q[nqc:], k, v, valid, everything))
        out[:, i] = torch.cat(parts).reshape(-1, 64)[:n]
    return out


def exact(case, seed):
    s = _inputs(case, seed)
    n, h, dm, op = case["tokens"], case["heads"], case["d_model"], case["op"]
    nb, nc, nq, nqc, c = _grid(case)
    if op == "out_proj":
        return {"y": s["x"].double() + s["O"].view(n, h * 64).double() @ s["W_o"].double().T}
    if op == "token_drift":
        y = (s["O_a"].double() - s["O_b"].double()).view(n, h * 64) @ s["W_o"].double().T
        full = torch.zeros(nb * 64, dtype=torch.float64, device="cuda")
        full[:n] = (y * y).sum(1)
        return {"drift": full.view(nb, 64).sum(1)}
    Q, K, V = s["Q"].double(), s["K"].double(), s["V"].double()
    affordable = _kept_pairs(case) < 1e10  # else the attention takes too long in float64
    if op == "attn":
        if not affordable:
            return None
        col = _caller_lists(case, s["Q"], s["K"])[1].long()
        per = nqc * min(nb, c + nb - nc) + (nq - nqc) * nb
        kept = torch.stack([col[i * per:i * per + nqc * (c + nb - nc)].view(nqc, -1) for i in range(h)])
        return {"O": _exact_attention(case, Q, K, V, kept)}
    D, J = _exact_selection(case, Q, K, V, s["W_o"])
    J_best = torch.zeros(h, nq, dtype=torch.float64, device="cuda")
    J_best[:, :nqc] = J
    out = {"row_ptr": None, "col_idx": None, "J_best": J_best.reshape(-1)}
    if op == "select":
        return {**out, "mask": None}
    if not affordable:
        return {**out, "O": None}
    candidates = torch.nonzero(~D)[:, 2].view(h, nqc, c)  # every row keeps c of them
    always = torch.arange(nc, nb, device="cuda").expand(h, nqc, nb - nc)
    O = _exact_attention(case, Q, K, V, torch.cat([candidates, always], dim=2))
    return {**out, "O": O.cpu() if op == "forward_host" else O}
