"""The calls whose speed this library is measured by, over the range they are used in.

Every case goes through the package's public entry points the way a decoding loop does: the
tensors, the SpecStep (or the workspace and output tensors) are made once, a pass makes the
calls.  Cases with ``graph`` set replay the calls from a CUDA graph, which is how a loop of many
short dependent launches is run; the others call them one by one.

  step    one whole speculative step: selection with the carried window LSE, gamma drafter
          passes, the verify block.
  select  the KV-budget selection alone (token or chunk level, with the carried window LSE or
          computing it), e.g. a drafter that is re-sparsified between steps or after prefill.
  drafts  gamma drafter passes over a view that persists (the paper's loop sparsifies once).
  verify  the verifier's block over the full cache.
  lse     the window's softmax normalisers (SpecStep.window_lse), what carry mode starts from.
  settle  the end of a step: the drafter's and the verifier's arg max tokens, acceptance, and
          the cache update (window slide, view append).

Sizes: contexts of 1K to 16K (the evaluation's 1K/4K/8K/16K), 32K and 128K (the verifier is a
128K-context model), budgets 256 to 2048 and larger views for long contexts, gamma 5 and the
paper's longest, 20, GQA groups 1 (multi-head), 4 and 8, head_dim 64 and 128.
"""

from __future__ import annotations

import math

import torch

import paper_2606_00144_gb300 as bd

BF = torch.bfloat16
N_SINK = 4
WINDOW = 32
VOCAB = 128256            # Llama-3's vocabulary, the layer shape of the workloads
UNIT_ROWS = 8 * 8 * 16384 * 128   # batch * h_kv * t_ctx * head_dim of the largest cases


def _case(kind, batch, heads, t_ctx, budget=512, gamma=5, chunk=1, self_mode=False, ragged=0.0, graph=False, **kw):
    h_q, h_kv, d = heads
    return dict(kind=kind, batch=batch, h_q=h_q, h_kv=h_kv, d=d, t_ctx=t_ctx, budget=budget, gamma=gamma, chunk=chunk,
                self_mode=self_mode, ragged=ragged, graph=graph, **kw)


TINY, GQA4, GQA8, MHA = (8, 2, 64), (32, 8, 128), (32, 4, 128), (32, 32, 128)


def listed():
    return [
        # the smallest step there is: eight dependent launches of a few microseconds
        dict(_case("step", 1, TINY, 1024, 256, graph=True), name="step_1k_tiny"),
        # the headline: a serving batch at 16K context, a view re-selected every step
        dict(_case("step", 8, GQA4, 16384, 512, graph=True), name="step_16k_b8"),
        # selection straight after prefill, when no window LSE has been carried yet
        dict(_case("select", 8, GQA4, 16384, 1024, self_mode=True), name="select_self_16k_b8"),
        # one long document: token-level selection over 128K positions
        dict(_case("select", 1, GQA4, 131072, 2048), name="select_128k_b1"),
        # the paper's chunk policy on a batch of documents of unequal, odd lengths
        dict(_case("select", 3, GQA4, 36001, 1024, chunk=8, ragged=0.6), name="select_chunk8_ragged"),
        # five drafter passes at the largest budget the paper trains for
        dict(_case("drafts", 8, GQA4, 16384, 2048, graph=True), name="drafts_16k_b8"),
        # one long document, a view of a quarter of it, the paper's longest draft
        dict(_case("drafts", 1, GQA8, 32768, 8192, gamma=20, graph=True), name="drafts_32k_b1"),
        # a multi-head verifier (Llama-2's 32 KV heads), sequences of unequal lengths
        dict(_case("verify", 4, MHA, 4099, ragged=0.4), name="verify_mha_ragged_b4"),
        # a single user's request: one sequence, the paper's longest draft
        dict(_case("verify", 1, GQA4, 4096, gamma=20), name="verify_4k_b1_gamma20"),
        # a serving batch with the paper's longest draft: 8 x 21 query rows per KV head
        dict(_case("verify", 4, GQA8, 16384, gamma=20), name="verify_16k_b4_gamma20"),
        # the carried LSE's first values, for a whole batch
        dict(_case("lse", 8, GQA4, 16384), name="lse_16k_b8"),
        # tokens from logits, acceptance, cache update for a serving batch
        dict(_case("settle", 8, GQA4, 16384, 512, graph=True, vocab=VOCAB), name="settle_b8"),
    ]


def draw(rng):
    """One more case of the same ranges: sizes spread over their logarithm, odd ones among them."""
    kind = rng.choice(["step", "select", "select", "drafts", "verify", "verify", "lse", "settle"])

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    heads = rng.choice([TINY, GQA4, GQA4, GQA8, MHA])
    t_hi = {"step": 16384, "settle": 16384, "verify": 32768, "lse": 32768, "drafts": 32768, "select": 131072}[kind]
    t = log(1024, min(t_hi, UNIT_ROWS // (heads[1] * heads[2])))
    batch = min(8, log(1, max(1, UNIT_ROWS // (heads[1] * heads[2] * t))))
    budget = min(log(256, 8192 if kind == "drafts" else 2048), t // 2)
    gamma = rng.choice([1, 3, 5, 5, 8, 12, 20])
    ragged = rng.choice([0.0, 0.0, 0.5]) if kind in ("select", "verify", "step") and batch > 1 else 0.0
    c = _case(kind, batch, heads, t, budget, gamma, ragged=ragged, graph=kind in ("step", "drafts", "settle"))
    if kind == "select":
        c["chunk"] = rng.choice([1, 1, 8])
        c["self_mode"] = rng.random() < 0.3 and heads[0] // heads[1] * WINDOW <= 128
    if kind == "lse":
        c["h_q"] = min(c["h_q"], c["h_kv"] * 4)          # at most 128 window rows per KV head
    if kind == "settle":
        c["vocab"] = log(32000, VOCAB)
    return c


# ------------------------------------------------------------------------------------ shapes


def _lens(c):
    """Context length of every sequence: t_ctx, or spread evenly over [(1 - ragged) t_ctx, t_ctx]."""
    b, t = c["batch"], c["t_ctx"]
    if not c["ragged"]:
        return [t] * b
    return [max(WINDOW + 1, t - int(i * c["ragged"] * t / max(1, b - 1))) for i in range(b)]


def _recent(c):
    return c["budget"] // 4


def _n_mid(c, t):
    return max(0, t - N_SINK - _recent(c))


def work(c):
    b, hq, hkv, d, g, lens = c["batch"], c["h_q"], c["h_kv"], c["d"], c["gamma"], _lens(c)
    row, G = 2 * d, c["h_q"] // c["h_kv"]
    # a phase's inputs once each: the verify's queries depend on the drafts', the drafts' on the
    # selection, so a step reads K in the selection and again in the verify block
    sel_rows = sum(t if c["self_mode"] else _n_mid(c, t) for t in lens) * hkv
    sel = dict(bytes=sel_rows * row + b * hq * WINDOW * (row + (0 if c["self_mode"] else 4)) + b * hkv * (c["budget"] + 1) * 4,
               flops=2 * d * G * WINDOW * sel_rows)
    view = sum(min(c["budget"], t) + g for t in lens) * hkv
    dr = dict(bytes=view * 2 * row + b * hkv * c["budget"] * 4 + g * b * hq * (2 * row + 4),
              flops=4 * d * G * view * g)
    ver_rows = sum(t + g + 1 for t in lens) * hkv
    ver = dict(bytes=ver_rows * 2 * row + b * hq * (g + 1) * (2 * row + 4), flops=4 * d * G * (g + 1) * ver_rows)
    k = c["kind"]
    if k == "select":
        return sel
    if k == "drafts":
        return dr
    if k == "verify":
        return ver
    if k == "lse":
        return dict(bytes=sum(lens) * hkv * row + b * hq * WINDOW * (row + 4), flops=2 * d * G * WINDOW * sum(lens) * hkv)
    if k == "settle":
        return dict(bytes=b * (2 * g + 1) * c["vocab"] * 2 + 2 * b * hq * WINDOW * row, flops=b * (2 * g + 1) * c["vocab"])
    return {m: sel[m] + dr[m] + ver[m] for m in ("bytes", "flops")}


def tolerance(c):
    k = c["kind"]
    if k == "lse":
        return {"rel": 2e-7, "max": 2e-6}                 # fp32 sums over a prefix of the context: 4e-8 from 64 bits
    if k == "settle":
        return "exact"                                    # tokens, counts and copied rows
    if k == "select":
        return {"rel": 0.0, "differ": 0.01}               # positions; scores tied within fp32 rounding
    # bf16 outputs: one rounding is 1.7e-3 of the result (2-norm) and 2^-8 of a value at most
    return {"rel": 7e-3, "max": 0.02, "differ": 0.01}


# ------------------------------------------------------------------------------------ inputs


def _window_lse(k, qw, lens):
    """Normalisers of the window rows over their causal prefixes, fp32 (what a previous step carried)."""
    b, hkv, _, d = k.shape
    hq = qw.shape[1]
    G = hq // hkv
    out = torch.empty(b, hq, WINDOW, device=k.device)
    for i, t in enumerate(lens):
        for g in range(hkv):
            q = qw[i, g * G:(g + 1) * G].reshape(G * WINDOW, d).float()
            s = (q @ k[i, g, :t].float().T) / math.sqrt(d)
            pos = t - WINDOW + torch.arange(WINDOW, device=k.device).repeat(G)
            s.masked_fill_(torch.arange(t, device=k.device)[None, :] > pos[:, None], -math.inf)
            out[i, g * G:(g + 1) * G] = torch.logsumexp(s, 1).view(G, WINDOW)
    return out


class _State:
    pass


def prepare(c, seed):
    """The caches (i.i.d. rows with a share of heavy hitters along the window's direction, as in the
    package's workloads), the queries, the carried LSE, and the SpecStep that a loop keeps."""
    dev = "cuda"
    g = torch.Generator(device=dev).manual_seed(seed)
    b, hq, hkv, d, t, gamma = c["batch"], c["h_q"], c["h_kv"], c["d"], c["t_ctx"], c["gamma"]
    G, kind, lens = hq // hkv, c["kind"], _lens(c)
    s = _State()
    s.case, s.lens = dict(c), lens
    rnd = lambda *shape: torch.randn(*shape, generator=g, device=dev, dtype=torch.float32).to(BF)  # noqa: E731
    s.qw = rnd(b, hq, WINDOW, d)
    if kind != "settle":
        s.k = torch.empty(b, hkv, t + gamma + 1, d, dtype=BF, device=dev)
        for i in range(b):
            kk = torch.randn(hkv, t + gamma + 1, d, generator=g, device=dev)
            for h in range(hkv):
                u = s.qw[i, h * G:(h + 1) * G].float().sum(dim=(0, 1))
                pos = torch.randint(0, lens[i], (max(1, lens[i] // 100),), generator=g, device=dev)
                kk[h, pos] += 3.0 * u / u.norm()
            s.k[i] = kk
    if kind in ("step", "drafts", "verify"):
        s.v = rnd(b, hkv, t + gamma + 1, d)
    s.qd = rnd(gamma, b, hq, d) if kind in ("step", "drafts") else None
    s.qv = rnd(b, hq, gamma + 1, d) if kind in ("step", "verify", "settle") else None
    dlens = torch.tensor(lens, dtype=torch.int32, device=dev) if c["ragged"] else None
    s.step = bd.SpecStep(b, hq, hkv, d, t, t + gamma + 1, c["budget"], N_SINK, _recent(c), WINDOW, gamma, c["chunk"],
                         dev, dlens)
    s.dlens = dlens
    s.lse = None
    if kind == "step" or (kind == "select" and not c["self_mode"]):
        s.lse = _window_lse(s.k, s.qw, lens)
    if kind == "drafts":                                 # a view left by an earlier selection
        for i in range(b):
            for h in range(hkv):
                keep = torch.randperm(lens[i], generator=g, device=dev)[:c["budget"]].sort().values
                s.step.idx[i, h] = keep.int()
        s.step.count.fill_(c["budget"])
    keep = []
    if kind == "settle":
        v = c["vocab"]
        s.ld = (2 * torch.randn(gamma, b, v, generator=g, device=dev)).to(BF)     # drafter logits, pass-major
        s.lv = (2 * torch.randn(b, gamma + 1, v, generator=g, device=dev)).to(BF)
        agree = torch.randint(0, gamma + 1, (b,), generator=g, device=dev).tolist()
        for i, a in enumerate(agree):                    # the verifier agrees with the first a drafts
            s.lv[i, :a] = s.ld[:a, i]
        s.lse_v = torch.randn(b, hq, gamma + 1, generator=g, device=dev)
        s.lse_w = torch.randn(b, hq, WINDOW, generator=g, device=dev)
        cap = c["budget"] + gamma + 1
        s.idx = torch.arange(cap, device=dev, dtype=torch.int32).repeat(b, hkv, 1)
        s.count = torch.full((b, hkv), c["budget"], dtype=torch.int32, device=dev)
        i32 = dict(dtype=torch.int32, device=dev)
        s.td, s.tv = torch.empty(gamma, b, **i32), torch.empty(b, gamma + 1, **i32)
        s.n_acc, s.emit, s.adv = torch.empty(b, **i32), torch.empty(b, gamma + 1, **i32), torch.empty(b, **i32)
        keep = [s.qw, s.lse_w, s.idx, s.count]           # updated in place
    s.graph = None
    if c["graph"]:
        saved = [x.clone() for x in keep]
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _calls(s)
            for x, y in zip(keep, saved):
                x.copy_(y)
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            s.out = _calls(s)
        s.graph = graph
    return s


# ------------------------------------------------------------------------------------ a pass


def _calls(s):
    c, st = s.case, s.step
    kind, gamma, b = c["kind"], c["gamma"], c["batch"]
    if kind == "step":
        st.run(s.k, s.v, s.qw, s.qd, s.qv, s.lse)
        return {"idx": st.idx, "count": st.count, "draft_o": st.draft_o, "draft_lse": st.draft_lse,
                "verify_o": st.verify_o, "verify_lse": st.verify_lse}
    if kind == "select":
        st.select(s.k, s.qw, s.lse)
        return {"idx": st.idx, "count": st.count}
    if kind == "drafts":
        for j in range(gamma):
            st.draft(j, s.qd[j], s.k, s.v, view_ready=j > 0)
        return {"draft_o": st.draft_o, "draft_lse": st.draft_lse}
    if kind == "verify":
        st.verify(s.qv, s.k, s.v)
        return {"verify_o": st.verify_o, "verify_lse": st.verify_lse}
    if kind == "lse":
        return {"lse": st.window_lse(s.k, s.qw)}
    bd.bd_argmax(s.ld.view(gamma * b, c["vocab"]), s.td)
    bd.bd_argmax(s.lv.view(b * (gamma + 1), c["vocab"]), s.tv)
    bd.bd_accept(s.td, s.tv, s.n_acc, s.emit)
    bd.bd_advance(st.shape, WINDOW, gamma + 1, s.n_acc, s.qv, s.lse_v, s.qw, s.lse_w, s.idx, s.count, s.adv)
    return {"td": s.td, "tv": s.tv, "n_accept": s.n_acc, "emit": s.emit, "advance": s.adv, "q_win": s.qw,
            "lse_win": s.lse_w, "idx": s.idx, "count": s.count}


def run(s):
    if s.graph is not None:
        s.graph.replay()
        return s.out
    return _calls(s)


# ------------------------------------------------------------------------------------ in 64 bits


def _attend(q, k, v, limit, d):
    """q [n, d] over keys k [t, d]; key j is seen by query i when j <= limit[i]."""
    x = (q @ k.T) / math.sqrt(d)
    x.masked_fill_(torch.arange(k.shape[0], device=k.device)[None, :] > limit[:, None], -math.inf)
    return (torch.softmax(x, 1) @ v if v is not None else None), torch.logsumexp(x, 1)


def _top(score, t, c):
    """Kept positions of one unit from its middle positions' scores (chunk = 1 or s), ascending."""
    B, R, S, s = c["budget"], _recent(c), N_SINK, c["chunk"]
    lo, hi = S, t - R
    dev = score.device
    if s == 1:
        mid = lo + torch.sort(score, descending=True, stable=True).indices[:B - S - R]
    else:
        pos = torch.arange(lo, hi, device=dev) // s
        first = lo // s
        tot = torch.zeros(int(pos[-1]) - first + 1, dtype=score.dtype, device=dev).index_add_(0, pos - first, score)
        top = torch.sort(tot, descending=True, stable=True).indices[:(B - S - R) // s]
        mid = lo + torch.nonzero(torch.isin(pos - first, top)).flatten()
    out = torch.cat([torch.arange(S, device=dev), mid.sort().values, torch.arange(hi, t, device=dev)])
    return out


def exact(c, seed):
    s = prepare(dict(c, graph=False), seed)
    b, hq, hkv, d, gamma, lens, kind = c["batch"], c["h_q"], c["h_kv"], c["d"], c["gamma"], s.lens, c["kind"]
    G, dev, f8 = hq // hkv, "cuda", torch.float64
    if kind == "settle":
        td, tv = s.ld.float().argmax(-1), s.lv.float().argmax(-1)
        n_acc = torch.stack([(td[:, i] == tv[i, :gamma]).long().cumprod(0).sum() for i in range(b)])
        emit = torch.full((b, gamma + 1), -1, dtype=torch.int64, device=dev)
        for i in range(b):
            emit[i, :n_acc[i] + 1] = tv[i, :n_acc[i] + 1]
        a = int(n_acc.min()) + 1
        idx, count = s.idx.clone(), s.count + a
        idx[:, :, c["budget"]:c["budget"] + a] = c["t_ctx"] + torch.arange(a, device=dev, dtype=torch.int32)
        return {"td": td, "tv": tv, "n_accept": n_acc, "emit": emit, "advance": torch.full((b,), a, device=dev),
                "q_win": torch.cat([s.qw, s.qv], 2)[:, :, a:a + WINDOW].double(),
                "lse_win": torch.cat([s.lse_w, s.lse_v], 2)[:, :, a:a + WINDOW].double(), "idx": idx, "count": count}
    out = {}
    if kind in ("step", "select"):
        out["idx"] = torch.full((b, hkv, c["budget"]), -1, dtype=torch.int64, device=dev)
        out["count"] = torch.zeros(b, hkv, dtype=torch.int64, device=dev)
    if kind in ("step", "drafts"):
        out["draft_o"] = torch.empty(gamma, b, hq, d, dtype=f8, device=dev)
        out["draft_lse"] = torch.empty(gamma, b, hq, dtype=f8, device=dev)
    if kind in ("step", "verify"):
        out["verify_o"] = torch.empty(b, hq, gamma + 1, d, dtype=f8, device=dev)
        out["verify_lse"] = torch.empty(b, hq, gamma + 1, dtype=f8, device=dev)
    if kind == "lse":
        out["lse"] = torch.empty(b, hq, WINDOW, dtype=f8, device=dev)
    for i in range(b):
        t = lens[i]
        for h in range(hkv):
            hs = slice(h * G, (h + 1) * G)
            k = s.k[i, h, :t + gamma + 1].double()
            v = s.v[i, h, :t + gamma + 1].double() if kind in ("step", "drafts", "verify") else None
            wpos = (t - WINDOW + torch.arange(WINDOW, device=dev)).repeat(G)
            if kind in ("step", "select", "lse"):
                q = s.qw[i, hs].reshape(G * WINDOW, d).double()
                x = (q @ k[:t].T) / math.sqrt(d)
                x.masked_fill_(torch.arange(t, device=dev)[None, :] > wpos[:, None], -math.inf)
                lse = torch.logsumexp(x, 1)
                if kind == "lse":
                    out["lse"][i, hs] = lse.view(G, WINDOW)
                    continue
                if s.lse is not None:
                    lse = s.lse[i, hs].reshape(-1).double()
                if c["budget"] >= t:
                    keep = torch.arange(t, device=dev)
                else:
                    score = torch.exp(x - lse[:, None]).sum(0)[N_SINK:t - _recent(c)]
                    keep = _top(score, t, c)
                out["idx"][i, h, :keep.numel()] = keep
                out["count"][i, h] = keep.numel()
            elif kind == "drafts":
                keep = s.step.idx[i, h].long()
            if kind in ("step", "drafts"):
                for j in range(gamma):
                    rows = torch.cat([keep, t + torch.arange(j + 1, device=dev)])
                    lim = torch.full((G,), rows.numel(), device=dev)
                    o, l = _attend(s.qd[j, i, hs].double(), k[rows], v[rows], lim, d)
                    out["draft_o"][j, i, hs], out["draft_lse"][j, i, hs] = o, l
            if kind in ("step", "verify"):
                q = s.qv[i, hs].reshape(G * (gamma + 1), d).double()
                lim = (t + torch.arange(gamma + 1, device=dev)).repeat(G)
                o, l = _attend(q, k, v, lim, d)
                out["verify_o"][i, hs] = o.view(G, gamma + 1, d)
                out["verify_lse"][i, hs] = l.view(G, gamma + 1)
    return out
