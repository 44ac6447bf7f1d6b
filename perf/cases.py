"""The drafting path's calls as user programs make them: inputs, one pass, its work and its accuracy.

A case is one call (or the one short sequence of calls that belongs together) on the GPU:

  step    Drafter.draft: both stages, the tree and its mask from device tensors (a serving engine)
  host    tf_draft_tree_host: the same step between page-locked host buffers, on the current stream
  lists   tf_stage1_marginals: log-softmax and top-K1 of every depth's hidden state
  rows    tf_lmhead_partials and tf_lmhead_merge: the LM head on rows that the caller has
  approx  tf_ar_approx: the AR-approximator (SwiGLU, linear or two previous tokens)
  tree    tf_build_tree_mask: tree selection, mask and position ids from candidate lists
  walk    tf_accept_walk: the verifier's acceptance walk over a drafted tree

Tensors are Gaussian with the path's shapes (weights of standard deviation 0.02); hidden states are
scaled so that the marginals go from peaked (first depth) to flat (last depth), as a block drafter's
do. `exact` restates each call in 64 bits with torch and a heap, apart from the package.
"""
import heapq
import math

import torch

from paper_2606_03819_gb300 import Dims, Drafter
from paper_2606_03819_gb300 import binding as B

POOL = 2048          # tokens that the candidate lists of one depth are drawn from (tree, walk)


def _case(kind, **kw):
    c = dict(kind=kind, batch=1, d=4096, V=151936, I=4096, gamma=16, M=16, K2=64, B=64, dtype="bf16", mode="ar",
             approx="swiglu")
    c.update(kw)
    return c


def listed():
    return [
        # smallest whole step, all in fp32: latency and launches
        dict(_case("step", d=128, V=2048, I=512, gamma=4, M=4, K2=12, B=12, dtype="f32"), name="step_f32_tiny"),
        # a whole step of a small model kept in fp32
        dict(_case("step", d=1024, V=32768, I=3072, gamma=8, M=8, K2=32, B=32, dtype="f32"), name="step_f32_small"),
        # one sequence's marginals at the 8B verifier's sizes: the LM head is streamed for 16 rows
        dict(_case("lists"), name="lists_b1"),
        # LM head and top-k of rows that are no multiple of a tile, ragged vocabulary, between one sequence and a batch
        dict(_case("rows", batch=3, d=3584, V=152064 - 191, M=11, gamma=13, K2=48, B=48), name="rows_ragged"),
        # Eq. 1 of one sequence: M = 16, and M = 8 with the verifier's own intermediate width
        dict(_case("approx"), name="approx_m16"),
        dict(_case("approx", M=8, K2=32, B=32, I=12288), name="approx_m8_wide_i"),
        # Eq. 1 of a batch of eight at d = 5120: a dense contraction
        dict(_case("approx", batch=8, d=5120, I=5120), name="approx_batch8"),
        # tree selection: the usual budget in a batch, and a large budget with exact lists
        dict(_case("tree", batch=8), name="tree_b64"),
        dict(_case("tree", K2=512, B=512), name="tree_b512"),
        # the verifier's walk over a batch of drafted trees
        dict(_case("walk", batch=32), name="walk_b64"),
        # the whole step of one sequence, host memory to host memory
        dict(_case("host"), name="host_step"),
        # the whole step of 32 sequences
        dict(_case("step", batch=32, M=8, K2=32, B=32), name="step_batch32"),
    ]


def _rows(c):
    """Stage-2 rows of one sequence."""
    if c["approx"] == "swiglu_2prev" and c["mode"] == "ar":
        return 1 if c["gamma"] == 1 else 1 + c["M"] + c["M"] ** 2 * (c["gamma"] - 2)
    return 1 + c["M"] * (c["gamma"] - 1)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the ranges above: sequences 1..32, hidden sizes 512..5120, vocabularies 32000..152064, block sizes
    3..16, branching 2..32, budgets 8..1023; fp32 at a small model's sizes."""
    kind = rng.choice(["step", "step", "host", "lists", "rows", "approx", "approx", "tree", "tree", "walk"])
    f32 = kind in ("step", "lists", "rows") and rng.random() < 0.25
    while True:
        c = _case(kind, batch=_log_int(rng, 1, 32), d=64 * rng.randint(8, 80), V=rng.randint(32000, 152064),
                  I=64 * _log_int(rng, 16, 192), gamma=rng.randint(3, 16), M=_log_int(rng, 2, 32))
        c["B"] = _log_int(rng, 8, 1023 if kind in ("tree", "walk") else 128)
        c["K2"] = min(c["B"], 512)
        if rng.random() < 0.15:
            c["K2"] = max(4, c["K2"] // 2)            # shorter lists than the budget
        if kind in ("step", "host", "tree") and rng.random() < 0.2:
            c["mode"] = rng.choice(["marginal", "marginal_mary"])
        if kind in ("step", "approx", "tree") and c["mode"] == "ar":
            c["approx"] = rng.choice(["swiglu"] * 4 + ["linear", "swiglu_2prev"])
        if f32:
            c.update(dtype="f32", d=4 * rng.randint(32, 320), V=rng.randint(2000, 33000), I=_log_int(rng, 256, 4096))
        w = work(c)
        rows = c["batch"] * _rows(c)
        limit = 1.2e10 if f32 else 4.5e12             # the largest listed case is 5.1e12
        if w["flops"] <= limit and rows * max(c["K2"], 64) <= 1 << 20 and rows <= 4096:
            return c


def _dims(c):
    return Dims(c["batch"], c["d"], c["V"], c["I"], c["gamma"], c["M"], c["K2"], c["B"], 1.0, 1e-6, c["dtype"], c["mode"],
                c["approx"])


def _randn(g, shape, std, dtype):
    return torch.randn(shape, generator=g, device="cuda").mul_(std).to(dtype)


def _hidden(g, c, dtype):
    # logits of h = s N(0, 1) against N(0, 0.02^2) rows have deviation 0.02 s sqrt(d); a softmax over V Gaussian logits
    # of deviation sqrt(2 (ln V - H)) has an entropy of about H nats: 2 at the first depth, 4 at the last
    h = torch.randn((c["batch"], c["gamma"], c["d"]), generator=g, device="cuda")
    for i in range(c["gamma"]):
        nats = 2.0 + 2.0 * i / max(1, c["gamma"] - 1)
        h[:, i] *= math.sqrt(2.0 * (math.log(c["V"]) - nats)) / (0.02 * math.sqrt(c["d"]))
    return h.to(dtype)


def _model(g, c, D):
    dt = D.torch_dtype
    d, V, I = c["d"], c["V"], c["I"]
    w = dict(lm_head=_randn(g, (V, d), 0.02, dt))
    if c["kind"] not in ("lists", "rows") and c["mode"] == "ar":
        w.update(embed=_randn(g, (V, d), 0.02, dt), norm_h=1 + _randn(g, (d,), 0.05, dt), norm_e=1 + _randn(g, (d,), 0.05, dt))
        if c["approx"] == "linear":
            w.update(w_lin=_randn(g, (d, 2 * d), 0.02, dt))
        else:
            w.update(w_gate=_randn(g, (I, D.k_in), 0.02, dt), w_up=_randn(g, (I, D.k_in), 0.02, dt), w_down=_randn(g, (d, I), 0.02, dt))
    return w


def _tokens(g, V, shape):
    return torch.randint(0, V, shape, generator=g, device="cuda", dtype=torch.int32)


def _candidates(g, c, D):
    """Candidate lists as the two stages leave them: per depth a pool of tokens with Gaussian logits, and child rows whose
    logits scatter about their depth's, so that favourites of a row are often stage-1 candidates."""
    b, gm = c["batch"], c["gamma"]
    step = c["V"] // POOL                                                           # one token of each run of `step`
    ids = torch.randint(0, step, (b * gm, POOL), generator=g, device="cuda") + step * torch.arange(POOL, device="cuda")
    z = 3.0 * torch.randn(ids.shape, generator=g, device="cuda")
    lp, at = torch.log_softmax(z, -1).topk(D.K1)
    top_ids = ids.gather(1, at).int().view(b, gm, D.K1)
    top_logp = lp.view(b, gm, D.K1).contiguous()
    if c["mode"] != "ar":
        return top_ids.contiguous(), top_logp, None, None
    R, M = D.R, c["M"]
    r = torch.arange(R, device="cuda")
    if c["approx"] == "swiglu_2prev":
        depth = torch.where(r == 0, 0, torch.where(r <= M, 1, 2 + (r - 1 - M) // (M * M)))
    else:
        depth = torch.where(r == 0, 0, 1 + (r - 1) // M)
    child_ids = torch.empty((b, R, c["K2"]), dtype=torch.int32, device="cuda")
    child_logp = torch.empty((b, R, c["K2"]), dtype=torch.float32, device="cuda")
    for s in range(b):
        zz = z.view(b, gm, -1)[s][depth] + 1.5 * torch.randn((R, ids.shape[1]), generator=g, device="cuda")
        lp, at = torch.log_softmax(zz, -1).topk(c["K2"])
        child_ids[s] = ids.view(b, gm, -1)[s][depth].gather(1, at).int()
        child_logp[s] = lp
    return top_ids.contiguous(), top_logp, child_ids, child_logp


def _tree_buffers(c):
    b, n = c["batch"], c["B"] + 1
    i32 = dict(dtype=torch.int32, device="cuda")
    return dict(node_tok=torch.empty((b, n), **i32), node_parent=torch.empty((b, n), **i32), node_depth=torch.empty((b, n), **i32),
                node_score=torch.empty((b, n), dtype=torch.float32, device="cuda"),
                mask=torch.empty((b, n, n), dtype=torch.uint8, device="cuda"), pos_ids=torch.empty((b, n), **i32),
                dev_status=torch.empty((b,), **i32))


def _inputs(case, seed):
    """The call's inputs (and model) as device tensors."""
    c = case
    D = _dims(c)
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = dict(case=c, dims=D)
    two = c["approx"] == "swiglu_2prev" and c["mode"] == "ar"
    s["root_tok"] = _tokens(g, c["V"], (c["batch"], 2) if two else (c["batch"],))
    s["root_pos"] = 1000 + _tokens(g, 30000, (c["batch"],))
    if c["kind"] in ("tree", "walk"):
        s["top_ids"], s["top_logp"], s["child_ids"], s["child_logp"] = _candidates(g, c, D)
        s["coin"] = torch.rand((c["batch"], c["B"] + 1), generator=g, device="cuda")
        return s
    s["w"] = _model(g, c, D)
    if c["kind"] == "rows":
        n = c["batch"] * D.R
        x = torch.randn((n, c["d"]), generator=g, device="cuda")
        nats = 2.0 + 2.0 * torch.rand((n, 1), generator=g, device="cuda")
        s["x"] = (x * (2.0 * (math.log(c["V"]) - nats)).sqrt() / (0.02 * math.sqrt(c["d"]))).to(D.torch_dtype)
        return s
    s["hidden"] = _hidden(g, c, D.torch_dtype)
    if c["kind"] == "approx":      # candidates of every depth, as stage 1 leaves them: distinct within a depth
        step = c["V"] // D.K1
        at = torch.randint(0, step, (c["batch"], c["gamma"], D.K1), generator=g, device="cuda", dtype=torch.int32)
        s["top_ids"] = at + step * torch.arange(D.K1, device="cuda", dtype=torch.int32)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    c, D = s["case"], s["dims"]
    b, gm = c["batch"], c["gamma"]
    i32, f32 = dict(dtype=torch.int32, device="cuda"), dict(dtype=torch.float32, device="cuda")
    kind = c["kind"]
    if kind == "step":
        s["drafter"] = Drafter(D, s["w"])
    elif kind == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        s["ws"] = B.alloc_workspace(D)
        s["hidden"], s["root_tok"], s["root_pos"] = pin(s["hidden"]), pin(s["root_tok"]), pin(s["root_pos"])
        s["out"] = {k: torch.empty(v.shape, dtype=v.dtype, pin_memory=True) for k, v in _tree_buffers(c).items()}
    elif kind == "lists":
        s["ws"] = B.alloc_workspace(D)
        s["top_ids"], s["top_logp"] = torch.empty((b, gm, D.K1), **i32), torch.empty((b, gm, D.K1), **f32)
    elif kind == "rows":
        s["ws"] = B.alloc_workspace(D)
        s["ids"], s["logp"] = torch.empty((b * D.R, c["K2"]), **i32), torch.empty((b * D.R, c["K2"]), **f32)
    elif kind == "approx":
        s["ws"] = B.alloc_workspace(D)
        s["h_prime"] = torch.empty((b, D.R, c["d"]), dtype=D.torch_dtype, device="cuda")
    else:
        s["out"] = _tree_buffers(c)
        if kind == "walk":      # a drafted tree; the verifier agrees with a child of a node four times in five
            _build(s)
            o = s["out"]
            n = c["B"] + 1
            child = torch.zeros((b, n), dtype=torch.long, device="cuda")
            child.scatter_reduce_(1, o["node_parent"].long().clamp(min=0), torch.arange(n, device="cuda").expand(b, n), "amax")
            s["verifier"] = torch.where(s["coin"] < 0.8, o["node_tok"].gather(1, child), o["node_tok"].roll(1, 1)).contiguous()
            s["accept"] = dict(accept_len=torch.empty((b,), **i32), accept_path=torch.empty((b, gm + 1), **i32),
                               next_tok=torch.empty((b,), **i32))
    return s


def _build(s):
    o = s["out"]
    B.tf_build_tree_mask(s["dims"], s["root_tok"], s["root_pos"], s["top_ids"], s["top_logp"], s["child_ids"], s["child_logp"],
                         o["node_tok"], o["node_parent"], o["node_depth"], o["node_score"], o["mask"], o["pos_ids"],
                         o["dev_status"])


def run(state):
    s = state
    D, kind = s["dims"], s["case"]["kind"]
    if kind == "step":
        out = s["drafter"].draft(s["hidden"], s["root_tok"], s["root_pos"])
        return {k: v for k, v in out.items() if v is not None}
    if kind == "host":
        o = s["out"]
        B.tf_draft_tree_host(D, s["w"], s["hidden"], s["root_tok"], s["root_pos"], o["node_tok"], o["node_parent"],
                             o["node_depth"], o["node_score"], o["mask"], o["pos_ids"], o["dev_status"], s["ws"])
        return o
    if kind == "lists":
        B.tf_stage1_marginals(D, s["w"], s["hidden"], s["top_ids"], s["top_logp"], s["ws"])
        return {"ids": s["top_ids"], "logp": s["top_logp"]}
    if kind == "rows":
        n = s["x"].shape[0]
        B.tf_lmhead_partials(D, s["w"]["lm_head"], s["x"], n, s["ws"])
        B.tf_lmhead_merge(D, s["w"]["lm_head"], s["x"], n, s["case"]["K2"], s["ids"], s["logp"], s["ws"])
        return {"ids": s["ids"], "logp": s["logp"]}
    if kind == "approx":
        B.tf_ar_approx(D, s["w"], s["hidden"], s["root_tok"], s["top_ids"], s["h_prime"], s["ws"])
        return {"h_prime": s["h_prime"]}
    if kind == "tree":
        _build(s)
        return s["out"]
    a = s["accept"]
    B.tf_accept_walk(D, s["out"]["node_tok"], s["out"]["node_parent"], s["verifier"], a["accept_len"], a["accept_path"],
                     a["next_tok"])
    return a


def work(case):
    """Bytes and operations of one pass. A step reads W_lm twice: stage 2 needs stage 1's candidates, and W_lm is ten
    times the L2."""
    c = case
    kind, b, gm, d, V, I, M, K2, n = (c[k] for k in ("kind", "batch", "gamma", "d", "V", "I", "M", "K2", "B"))
    e = 4 if c["dtype"] == "f32" else 2
    K1, R, ar = max(M, K2), _rows(c), c["mode"] == "ar"
    n += 1
    tree_out = b * (n * n + 5 * n * 4)
    if kind == "walk":
        return {"bytes": b * (3 * n * 4 + (gm + 3) * 4), "flops": 0}
    if kind == "tree":
        # a tree can take at most B + 1 entries of the lists
        return {"bytes": tree_out + b * (min((R if ar else gm) * (K2 if ar else K1), n * 8) * 8 + gm * M * 4), "flops": 0}
    if kind == "rows":
        return {"bytes": V * d * e + b * R * (d * e + K2 * 8), "flops": 2 * b * R * V * d}
    lists = {"bytes": V * d * e + b * gm * (d * e + K1 * 8), "flops": 2 * b * gm * V * d}
    if kind == "lists":
        return lists
    two = c["approx"] == "swiglu_2prev" and ar
    k_in = (3 if two else 2) * d
    mlp = d * 2 * d if c["approx"] == "linear" else 2 * I * k_in + d * I
    tokens = b * (gm - 1) * M + b * (2 if two else 1)
    approx = {"bytes": (mlp + 2 * d + tokens * d + b * gm * d + b * R * d) * e, "flops": 2 * b * R * mlp}
    if kind == "approx":
        return approx
    total = {"bytes": lists["bytes"] + tree_out, "flops": lists["flops"]}
    if ar:
        total["bytes"] += approx["bytes"] - b * (gm + R) * d * e + V * d * e + b * R * K2 * 8
        total["flops"] += approx["flops"] + 2 * b * R * V * d
    return total


def tolerance(case):
    kind, f32 = case["kind"], case["dtype"] == "f32"
    if kind in ("tree", "walk"):
        return "exact"             # copies, comparisons and one fp32 addition per node
    if kind in ("lists", "rows") or f32 or (kind in ("step", "host") and case["mode"] != "ar"):
        # fp32 sums of d products: order of the sums moves log-probabilities by a few 1e-6 of their size; near ties swap
        return {"rel": 1e-5, "max": 2e-4, "differ": 0.005}
    if kind == "approx":
        return {"rel": 1e-2, "max": 0.1}           # h' and two intermediates are rounded to bf16
    # the same roundings, seen through the LM head (child log-probabilities are 2e-2 off 64 bits): near ties of a list
    # swap, and trees follow
    return {"rel": 0.03, "max": 0.5, "differ": 0.01}


# ---- 64-bit restatement -------------------------------------------------------------------------


def _lists64(W, x, k):
    """log-softmax of W x and its k best entries (values, ids), best first; x [n, d]."""
    x = x.double()
    best = torch.empty((x.shape[0], 0), dtype=torch.double, device="cuda")
    ids = torch.empty((x.shape[0], 0), dtype=torch.long, device="cuda")
    lse = torch.full((x.shape[0],), -math.inf, dtype=torch.double, device="cuda")
    for v in range(0, W.shape[0], 16384):
        z = x @ W[v:v + 16384].double().t()
        lse = torch.logaddexp(lse, z.logsumexp(1))
        t, at = z.topk(min(k, z.shape[1]), dim=1)
        best, ids = torch.cat([best, t], 1), torch.cat([ids, at + v], 1)
        best, at = best.topk(min(k, best.shape[1]), dim=1)
        ids = ids.gather(1, at)
    return best - lse[:, None], ids


def _approx64(c, D, w, hidden, root, top_ids):
    """h' [b, R, d] of Eq. 1."""
    b, gm, M, R = c["batch"], c["gamma"], c["M"], D.R
    r = torch.arange(R, device="cuda")
    norm = lambda t, wt: t / (t.square().mean(-1, keepdim=True) + 1e-6).sqrt() * wt.double()  # noqa: E731
    out = torch.empty((b, R, c["d"]), dtype=torch.double, device="cuda")
    gate, up, down, lin = (w[k].double() if k in w else None for k in ("w_gate", "w_up", "w_down", "w_lin"))
    for s in range(b):
        top = top_ids[s].long()
        if c["approx"] == "swiglu_2prev":
            x_t, x_p = root[s, 0].long(), root[s, 1].long()
            q = (r - 1 - M).clamp(min=0)
            depth = torch.where(r == 0, 0, torch.where(r <= M, 1, 2 + q // (M * M)))
            deep1 = top[(depth - 1).clamp(min=0), q % (M * M) // M]
            deep2 = top[(depth - 2).clamp(min=0), q % M]
            first = top[0, (r - 1).clamp(0, M - 1)]
            prev = [torch.where(r == 0, x_t, torch.where(r <= M, first, deep1)),
                    torch.where(r == 0, x_p, torch.where(r <= M, x_t, deep2))]
        else:
            depth = torch.where(r == 0, 0, 1 + (r - 1) // M)
            prev = [torch.where(r == 0, root[s].long(), top[(depth - 1).clamp(min=0), (r - 1).clamp(min=0) % M])]
        h = hidden[s].double()[depth]
        x = torch.cat([norm(h, w["norm_h"])] + [norm(w["embed"][p].double(), w["norm_e"]) for p in prev], 1)
        if lin is not None:
            out[s] = h + x @ lin.t()
        else:
            out[s] = h + (torch.nn.functional.silu(x @ gate.t()) * (x @ up.t())) @ down.t()
    return out


def _scores64(c, top_ids, top_lp, child_ids, child_lp):
    """Scores of the B + 1 nodes of every sequence's tree in pop order (-inf where there is no such node)."""
    ar, two = c["mode"] == "ar", c["approx"] == "swiglu_2prev"
    M, gm = c["M"], c["gamma"]
    ids = (child_ids if ar else top_ids).tolist()
    lps = (child_lp if ar else top_lp).double().tolist()
    cand = top_ids[:, :, :M].tolist()
    out = []
    for s in range(c["batch"]):
        K = min(c["K2"], len(ids[s][0]))
        place = [{t: m for m, t in reversed(list(enumerate(cand[s][i])))} for i in range(gm)]
        score, mary = [0.0], [-1]
        heap = [(-lps[s][0][0], 1, 0, 0, 0)]      # -score, depth, parent, list, rank
        while heap and len(score) <= c["B"]:
            neg, depth, par, row, rank = heapq.heappop(heap)
            node, tok = len(score), ids[s][row][rank]
            score.append(-neg)
            m = place[depth - 1].get(tok, -1)
            mary.append(m)
            if rank + 1 < K:
                heapq.heappush(heap, (-(score[par] + lps[s][row][rank + 1]), depth, par, row, rank + 1))
            if depth < gm and (m >= 0 or c["mode"] == "marginal"):
                if not ar:
                    child = depth
                elif not two:
                    child = 1 + (depth - 1) * M + m
                else:
                    child = 1 + m if depth == 1 else 1 + M + (depth - 2) * M * M + m * M + mary[par]
                heapq.heappush(heap, (neg - lps[s][child][0], depth + 1, node, child, 0))
        out.append(score + [-math.inf] * (c["B"] + 1 - len(score)))
    return torch.tensor(out, dtype=torch.double)


def exact(case, seed):
    s = _inputs(case, seed)
    c, D, kind = s["case"], s["dims"], s["case"]["kind"]
    if kind == "walk":
        return None
    if kind == "tree":
        return {"node_score": _scores64(c, s["top_ids"], s["top_logp"], s["child_ids"], s["child_logp"])}
    W = s["w"]["lm_head"]
    if kind == "rows":
        return {"ids": None, "logp": _lists64(W, s["x"], c["K2"])[0]}
    if kind == "approx":
        return {"h_prime": _approx64(c, D, s["w"], s["hidden"], s["root_tok"], s["top_ids"])}
    top_lp, top_ids = _lists64(W, s["hidden"].view(-1, c["d"]), D.K1)
    top_lp, top_ids = top_lp.view(c["batch"], c["gamma"], -1), top_ids.view(c["batch"], c["gamma"], -1)
    if kind == "lists":
        return {"ids": None, "logp": top_lp}
    out = {"top_logp": top_lp}
    child_lp = child_ids = None
    if c["mode"] == "ar":
        h = _approx64(c, D, s["w"], s["hidden"], s["root_tok"], top_ids)
        child_lp, child_ids = _lists64(W, h.view(-1, c["d"]), c["K2"])
        child_lp, child_ids = child_lp.view(c["batch"], D.R, -1), child_ids.view(c["batch"], D.R, -1)
        out["child_logp"] = child_lp
    out["node_score"] = _scores64(c, top_ids, top_lp, child_ids, child_lp)
    return {"node_score": out["node_score"]} if kind == "host" else out
