"""The work this library is used for, as cases that can be timed and compared.

A speculative-decoding server calls the library once per verify step: the QKV projection of the
verify block (once per layer), the attention of the k+1 verify positions against the KV cache
(once per layer), and the LM head with the accept test, the correction draw and the KV commit
(once per step).  Each case is one such call, or the three in sequence, through the package's
public entry points, at the sizes of the verifier families of workloads.py.

Inputs come from the seed alone.  Lengths are a fixed spread over the case's range, dealt to the
sequences in an order the seed picks, so every seed of a case asks for the same work.
"""
import math

import torch

import paper_2608_13076_gb300 as spade

DEV = "cuda"
ROPE_THETA = 500000.0
SMS = 152  # streaming multiprocessors of a GB300: bounds the one-launch LM head's sizes below

# Sizes of the verifier families: heads, head dim, hidden size, vocabulary.
TINY = dict(Hq=8, Hkv=8, D=64, H=512, V=1024)
LLAMA2_7B = dict(Hq=32, Hkv=32, D=128, H=4096, V=32000)
LLAMA3_8B = dict(Hq=32, Hkv=8, D=128, H=4096, V=128256)
LONG_70B = dict(Hq=64, Hkv=8, D=128, H=8192, V=32000)
GQA_40_8 = dict(Hq=40, Hkv=8, D=128, H=5120, V=152064)


def _case(name, op, family, B, ctx, k, mode="greedy", page=0, temperature=False, top_p=1.0):
    """ctx, k: inclusive ranges over the batch; page: slots per page of a paged cache (0: dense);
    temperature: one per sequence; top_p: nucleus mass of the sampled sequences (1: all of p)."""
    return dict(name=name, op=op, B=B, ctx_lo=ctx[0], ctx_hi=ctx[1], k_lo=k[0], k_hi=k[1], mode=mode, page=page,
                temperature=temperature, top_p=top_p, **family)


def listed():
    return [
        # One short sequence on a small model: latency, launches and host work are all there is.
        _case("attention_tiny", "attention", TINY, 1, (256, 256), (4, 4)),
        # An ordinary serving batch with grouped-query heads.
        _case("attention_8b", "attention", LLAMA3_8B, 8, (4096, 4096), (8, 8)),
        # Few very long contexts: each KV head's keys are split over many SMs.
        _case("attention_70b_long", "attention", LONG_70B, 4, (32768, 32768), (4, 4)),
        # A large batch of very different lengths, as paged caches exist for.
        _case("attention_ragged_paged", "attention", GQA_40_8, 64, (128, 8192), (1, 10), page=64),
        # The projection for a single sequence: six rows against the whole weight.
        _case("qkv_7b_single", "qkv", LLAMA2_7B, 1, (2048, 2048), (5, 5)),
        _case("qkv_8b", "qkv", LLAMA3_8B, 8, (4096, 4096), (8, 8)),
        # More than 400 rows, into a paged cache.
        _case("qkv_ragged_paged", "qkv", GQA_40_8, 64, (128, 8192), (1, 10), page=64),
        # One interactive user, greedy decoding.
        _case("accept_7b_greedy", "accept", LLAMA2_7B, 1, (2048, 2048), (5, 5)),
        # Rejection sampling over a large vocabulary.
        _case("accept_8b", "accept", LLAMA3_8B, 8, (4096, 4096), (8, 8), mode="stochastic"),
        # The same with the sampling options that chat services set.
        _case("accept_8b_top_p", "accept", LLAMA3_8B, 8, (4096, 4096), (8, 8), mode="stochastic", temperature=True,
              top_p=0.9),
        # Greedy and sampling users in one large batch: more rows than stay on chip at once.
        _case("accept_ragged", "accept", GQA_40_8, 64, (128, 8192), (1, 10), mode="mixed"),
        # A whole verify step (projection, attention, accept and commit) of the small model.
        _case("step_tiny", "step", TINY, 1, (256, 256), (4, 4), mode="stochastic"),
    ]


# ---- drawn cases ---------------------------------------------------------------------------------
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lengths(rng, B, ctx_max, k_max):
    """Ranges of context and draft lengths: one length for all, or a spread."""
    ctx_hi = _log_int(rng, 1, ctx_max)
    k_hi = rng.randint(0, k_max)
    if rng.random() < 0.5:
        return (ctx_hi, ctx_hi), (k_hi, k_hi)
    return (rng.randint(0, ctx_hi), ctx_hi), (rng.randint(0, k_hi), k_hi)


def draw(rng):
    """One more case of the listed ranges; none costs more than the largest listed one."""
    op = rng.choice(["attention", "qkv", "accept", "step"])
    while True:
        D = rng.choice([64, 128, 128])
        Hkv = rng.choice([1, 2, 4, 8, 8, 16, 32])
        Hq = Hkv * rng.choice([1, 1, 2, 4, 4, 5, 7, 8])
        B = _log_int(rng, 1, 64)
        # Hidden sizes are multiples of 8; half of them not of 64.
        H = 8 * _log_int(rng, 32, 1024) if rng.random() < 0.5 else 64 * _log_int(rng, 4, 128)
        V = _log_int(rng, 1000, 152064)
        ctx, k = _lengths(rng, B, 32768, 12)
        mode = rng.choice(["greedy", "stochastic", "mixed"])
        temperature = mode != "greedy" and rng.random() < 0.4
        top_p = rng.choice([0.8, 0.9, 0.95]) if mode != "greedy" and rng.random() < 0.3 else 1.0
        page = rng.choice([0, 0, 64, 128, 256])
        c = _case("", op, dict(Hq=Hq, Hkv=Hkv, D=D, H=H, V=V), B, ctx, k, mode, page, temperature, top_p)
        del c["name"]
        if op == "accept":
            c["page"] = 0  # the head alone uses no cache
        if op in ("attention", "qkv"):
            c["mode"] = "greedy"
        if op != "accept":
            c["temperature"], c["top_p"] = False, 1.0  # steps commit through the plain fused call
        R = _rows(c)
        if R > 416 or Hq > 64 or (Hq + 2 * Hkv) * D % 128:
            continue
        if c["top_p"] < 1.0:
            # Top-p needs the logits of every row resident on chip.
            tiles = -(-(-(-V // SMS)) // 128)
            if R > 128 or tiles * (-(-R // 8) * 8) + 16 > 512:
                continue
        cap = _capacity(c)
        if B * Hkv * cap * D * 4 > 2.2e9:  # the cache of the listed ragged batch
            continue
        w = work(c)
        if w["bytes"] > 1.7e9 or w["flops"] > 6.0e11:
            continue
        return c


# ---- sizes ---------------------------------------------------------------------------------------
def _spread(lo, hi, n):
    return [lo] * n if n == 1 or lo == hi else [lo + (hi - lo) * i // (n - 1) for i in range(n)]


def _rows(c):
    return sum(_spread(c["k_lo"], c["k_hi"], c["B"])) + c["B"]


def _capacity(c):
    cap = c["ctx_hi"] + c["k_hi"] + 1
    return -(-cap // c["page"]) * c["page"] if c["page"] else cap


def work(case):
    """Every weight, cache row in use and input read once, every output written once."""
    c = case
    B, Hq, Hkv, D, H, V = (c[n] for n in ("B", "Hq", "Hkv", "D", "H", "V"))
    ctx, k = _spread(c["ctx_lo"], c["ctx_hi"], B), _spread(c["k_lo"], c["k_hi"], B)
    R = sum(k) + B
    by = fl = 0
    if c["op"] in ("attention", "step"):
        by += 2 * Hkv * D * 2 * sum(a + b + 1 for a, b in zip(ctx, k)) + 2 * R * Hq * D * 2 + R * Hq * 4
        fl += 4 * Hq * D * sum((b + 1) * (a + 1) + b * (b + 1) // 2 for a, b in zip(ctx, k))
    if c["op"] in ("qkv", "step"):
        N = (Hq + 2 * Hkv) * D
        by += N * H * 2 + R * H * 2 + R * N * 2
        fl += 2 * R * N * H
    if c["op"] in ("accept", "step"):
        sampled = {"greedy": 0, "stochastic": B, "mixed": B // 2}[c["mode"]]
        by += V * H * 2 + R * H * 2 + (sampled * V * 4 if c["k_hi"] else 0)
        fl += 2 * R * H * V
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """About four times the measured distance from the 64-bit result: 2.2e-3 for the attention (P
    and the outputs are bf16), 1.7e-3 for the projection (outputs rounded once to bf16), 2.5e-5 for
    the LM head's fp32 row statistics (largest in the sums of exponentials of logits near 20).
    Decisions and tokens are whole numbers."""
    if case["op"] == "attention":
        return {"rel": 1e-2, "max": 0.1}
    if case["op"] == "qkv":
        return {"rel": 7e-3, "max": 3e-2}
    if case["op"] == "accept":
        return {"rel": 1e-4, "max": 1e-3, "differ": 0.005}
    return {"rel": 1e-2, "max": 0.1, "differ": 0.005}


# ---- inputs --------------------------------------------------------------------------------------
def _randn(gen, *shape, std=1.0):
    x = torch.randn(shape, generator=gen, device=DEV, dtype=torch.bfloat16)
    return x.mul_(std) if std != 1.0 else x


def _inputs(c, seed):
    """The tensors a program has before the call."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    host = torch.Generator().manual_seed(int(seed))
    B, Hq, Hkv, D, H, V = (c[n] for n in ("B", "Hq", "Hkv", "D", "H", "V"))
    ctx = torch.tensor(_spread(c["ctx_lo"], c["ctx_hi"], B), dtype=torch.int32)[torch.randperm(B, generator=host)]
    k = torch.tensor(_spread(c["k_lo"], c["k_hi"], B), dtype=torch.int32)[torch.randperm(B, generator=host)]
    cu = torch.zeros(B + 1, dtype=torch.int32)
    cu[1:] = torch.cumsum(k + 1, 0)
    s = dict(case=c, op=c["op"], paged=c["page"] > 0, B=B, R=int(cu[-1]), max_k=c["k_hi"], ctx_list=ctx.tolist(),
             k_list=k.tolist(), cu_list=cu.tolist(), ctx_lens=ctx.to(DEV), n_draft=k.to(DEV), cu_q=cu.to(DEV))
    R = s["R"]
    if c["op"] in ("attention", "qkv", "step"):
        _caches(s, gen, host)
    if c["op"] == "attention":
        # Some heads attend broadly, others to a few keys.
        q = torch.randn((R, Hq, D), generator=gen, device=DEV)
        sharp = torch.exp(torch.rand((1, Hq, 1), generator=gen, device=DEV) * math.log(8.0)) * 0.5
        s["q"] = (q * sharp).to(torch.bfloat16)
    if c["op"] in ("qkv", "step"):
        s["x"] = _randn(gen, R, H)
        s["w_qkv"] = _randn(gen, (Hq + 2 * Hkv) * D, H, std=1.0 / math.sqrt(H))
    if c["op"] in ("accept", "step"):
        _drafts(s, gen, host)
    return s


def _caches(s, gen, host):
    """Dense caches [B, Hkv, cap, D], or pools of pages in a shuffled order and their table.  The
    projection only writes its block's slots, so its cache starts empty."""
    c = s["case"]
    B, Hkv, D, cap, page = c["B"], c["Hkv"], c["D"], _capacity(c), c["page"]
    if page:
        n = cap // page
        shape = (B * n + 2, Hkv, page, D)
        table = torch.randperm(B * n + 2, generator=host)[:B * n].reshape(B, n)
        s["table"] = table.to(torch.int32).to(DEV)
    else:
        shape = (B, Hkv, cap, D)
    for name in ("k_cache", "v_cache"):
        s[name] = torch.zeros(shape, dtype=torch.bfloat16, device=DEV) if c["op"] == "qkv" else _randn(gen, *shape)


def _drafts(s, gen, host):
    """Hidden rows, LM head weight, and a draft model's tokens and distributions.  Its logits are
    the verifier's with noise; rows are between flat and peaked, as language-model logits are."""
    c = s["case"]
    B, R, H, V = c["B"], s["R"], c["H"], c["V"]
    spread = torch.exp(torch.rand((R, 1), generator=gen, device=DEV) * math.log(2.5)) * 2.0  # logit std 2 .. 5
    s["hidden"] = (torch.randn((R, H), generator=gen, device=DEV) * spread).to(torch.bfloat16)
    s["w_lm"] = _randn(gen, V, H, std=1.0 / math.sqrt(H))
    sampled = {"greedy": [0] * B, "stochastic": [1] * B, "mixed": [b % 2 for b in range(B)]}[c["mode"]]
    s["mode_list"] = sampled
    s["mode"] = torch.tensor(sampled, dtype=torch.int32, device=DEV)
    s["temperature"] = torch.rand(B, generator=gen, device=DEV) * 0.6 + 0.6 if c["temperature"] else None
    s["top_p"] = torch.full((B,), c["top_p"], device=DEV) if c["top_p"] < 1.0 else None
    s["uniforms"] = torch.rand(R, generator=gen, device=DEV)
    logits = _logits(s["hidden"], s["w_lm"], torch.float32)
    s["draft_rows"] = [s["cu_list"][b] + i for b in range(B) for i in range(s["k_list"][b])]
    n = len(s["draft_rows"])
    rows = torch.tensor(s["draft_rows"], dtype=torch.long, device=DEV)
    noisy = logits[rows]
    noisy += 0.8 * torch.randn(noisy.shape, generator=gen, device=DEV)
    q = torch.softmax(noisy, -1)
    del noisy
    tokens = torch.zeros(n, dtype=torch.int64, device=DEV)
    if n:
        drawn = torch.multinomial(q, 1, generator=gen).flatten()
        best = logits[rows].argmax(-1)
        miss = torch.rand(n, generator=gen, device=DEV) < 0.3
        guess = torch.where(miss, drawn, best)
        is_sampled = torch.tensor([sampled[b] for b in range(B) for _ in range(s["k_list"][b])], device=DEV) == 1
        tokens = torch.where(is_sampled, drawn, guess)
    s["draft_tokens"] = tokens.to(torch.int32)
    s["draft_probs"] = q.contiguous() if any(sampled) and n else None
    # Uniforms that decide nothing by rounding: acceptance thresholds keep their side by 2e-3, and
    # a sampling uniform moves to the middle of the interval of the token it picks.
    _verify(s, logits.double(), settle=True)


def _logits(hidden, w, dtype, rows_of_w=16384):
    out = torch.empty((hidden.shape[0], w.shape[0]), dtype=dtype, device=DEV)
    h = hidden.to(dtype)
    for v in range(0, w.shape[0], rows_of_w):
        out[:, v:v + rows_of_w] = h @ w[v:v + rows_of_w].to(dtype).t()
    return out


def _verify(s, logits, settle=False):
    """Algorithm 1's verification on given 64-bit logits, in plain torch: accepted lengths, next
    tokens and the row statistics.  `settle` moves s["uniforms"] off the edges of the decisions."""
    c = s["case"]
    B, R = c["B"], s["R"]
    if s["temperature"] is not None:
        per_row = torch.repeat_interleave(s["temperature"].double(), torch.tensor([k + 1 for k in s["k_list"]], device=DEV))
        logits = logits / per_row[:, None]
    top, arg = logits.max(-1)
    sums = torch.exp(logits - top[:, None]).sum(-1)
    n = len(s["draft_rows"])
    rows = torch.tensor(s["draft_rows"], dtype=torch.long, device=DEV)
    tokens = s["draft_tokens"].long()
    l_draft = logits[rows, tokens]
    sampled_row = torch.tensor([s["mode_list"][b] for b in range(B) for _ in range(s["k_list"][b])], device=DEV) == 1
    u = s["uniforms"]
    whole = torch.exp(l_draft - top[rows]) / sums[rows]
    if s["draft_probs"] is not None:
        qd = s["draft_probs"][torch.arange(n, device=DEV), tokens].double()
        plain = torch.where(sampled_row, u[rows].double() * qd < whole, tokens == arg[rows])
    else:
        plain = tokens == arg[rows]
    ok = plain
    floor = torch.full((R,), -math.inf, dtype=torch.float64, device=DEV)  # lowest logit of the nucleus
    mass = sums.clone()
    if s["top_p"] is not None:
        for b in range(B):
            if not s["mode_list"][b]:
                continue
            r = slice(s["cu_list"][b], s["cu_list"][b + 1])
            by = logits[r].sort(-1, descending=True).values
            cum = torch.cumsum(torch.exp(by - top[r, None]), -1)
            at = (cum < s["top_p"][b].double() * sums[r, None]).sum(-1).clamp(max=by.shape[1] - 1)
            floor[r] = by.gather(1, at[:, None])[:, 0]
            mass[r] = torch.where(logits[r] >= floor[r, None], torch.exp(logits[r] - top[r, None]), 0.0).sum(-1)
    if s["draft_probs"] is not None:
        pd = torch.where(l_draft >= floor[rows], torch.exp(l_draft - top[rows]) / mass[rows], 0.0)
        edge = pd / qd
        if settle and n:
            ud = u[rows].double()
            moved = torch.where(ud < edge, edge - 2e-3, edge + 2e-3).clamp(0.0, 1.0 - 2.0 ** -24)
            for e in (edge, whole / qd):  # the plain test is reported too
                near = sampled_row & ((ud - e).abs() < 1e-3)
                ud = torch.where(near, moved, ud)
            u[rows] = ud.float()
        ok = torch.where(sampled_row, u[rows].double() < edge, plain)
    accepted, following = [], []
    ok_list, first = ok.tolist(), 0
    for b in range(B):
        k = s["k_list"][b]
        a = 0
        while a < k and ok_list[first + a]:
            a += 1
        r = s["cu_list"][b] + a
        accepted.append(a)
        if s["mode_list"][b]:
            p = torch.where(logits[r] >= floor[r], torch.exp(logits[r] - top[r]) / mass[r], 0.0)
            if a < k:
                p = (p - s["draft_probs"][first + a].double()).clamp_(min=0.0)
            cum = torch.cumsum(p, 0)
            last = s["cu_list"][b] + k
            x = torch.searchsorted(cum, u[last].double() * cum[-1], right=True).clamp_(max=p.numel() - 1)
            if settle:
                u[last] = ((cum[x] - 0.5 * p[x]) / cum[-1]).clamp(0.0, 1.0 - 2.0 ** -24).float()
            following.append(x.reshape(()))
        else:
            following.append(arg[r])
        first += k
    bit = torch.zeros(R, dtype=torch.int64, device=DEV)
    bit[rows] = plain.long()
    drafted = torch.zeros(R, dtype=torch.float64, device=DEV)
    drafted[rows] = l_draft
    return dict(accepted=torch.tensor(accepted, device=DEV), next=torch.stack(following), row_max=top, row_sum=sums,
                row_arg_accept=torch.stack([arg, bit], 1), draft_logit=drafted)


def prepare(case, seed):
    """Inputs, and what a program allocates once for its shapes: outputs, workspaces, status word."""
    s = _inputs(case, seed)
    c = s["case"]
    B, R, Hq, Hkv, D, H, V = c["B"], s["R"], c["Hq"], c["Hkv"], c["D"], c["H"], c["V"]
    s["status"] = spade.status_tensor(DEV)
    cap = _capacity(c)
    if s["op"] in ("qkv", "step"):
        s["q"] = torch.empty((R, Hq, D), dtype=torch.bfloat16, device=DEV)
        s["qkv_ws"] = spade.qkv_workspace(R, Hq, Hkv, D, device=DEV)
    if s["op"] in ("attention", "step"):
        s["out"] = torch.empty((R, Hq, D), dtype=torch.bfloat16, device=DEV)
        s["lse"] = torch.empty((R, Hq), dtype=torch.float32, device=DEV)
        s["attn_ws"] = spade.attn_workspace(B, Hq, Hkv, D, cap, s["max_k"], device=DEV)
    if s["op"] in ("accept", "step"):
        s["accepted"] = torch.empty(B, dtype=torch.int32, device=DEV)
        s["next"] = torch.empty(B, dtype=torch.int32, device=DEV)
        ws = s["accept_ws"] = spade.accept_workspace(B, R, H, V, device=DEV)
        # Views of the row statistics that the call leaves in its workspace: maximum, sum of
        # exponentials, argmax and accept bit of each row, and the logits of the draft tokens.
        at, drafts, _ = spade.spade_accept_stats_layout(B, R, H, V)
        stats = ws[at:at + 16 * R]
        s["row_max"], s["row_sum"] = (stats.view(torch.float32).view(R, 4)[:, i] for i in (0, 1))
        s["row_arg_accept"] = stats.view(torch.int32).view(R, 4)[:, 2:]
        s["draft_logit"] = ws[drafts:drafts + 4 * R].view(torch.float32)
    if s["op"] == "step":
        s["ctx_now"] = s["ctx_lens"].clone()
    return s


def _qkv(s, ctx):
    c = s["case"]
    if s["paged"]:
        spade.spade_verify_qkv_rope_paged(s["x"], s["w_qkv"], s["table"], ctx, s["n_draft"], s["cu_q"], s["q"],
                                          s["k_cache"], s["v_cache"], Hq=c["Hq"], rope_theta=ROPE_THETA,
                                          max_k=s["max_k"], workspace=s["qkv_ws"], status=s["status"])
    else:
        spade.spade_verify_qkv_rope(s["x"], s["w_qkv"], ctx, s["n_draft"], s["cu_q"], s["q"], s["k_cache"],
                                    s["v_cache"], Hq=c["Hq"], Hkv=c["Hkv"], rope_theta=ROPE_THETA, max_k=s["max_k"],
                                    workspace=s["qkv_ws"], status=s["status"])


def _attention(s, ctx):
    if s["paged"]:
        spade.spade_verify_attention_paged(s["q"], s["k_cache"], s["v_cache"], s["table"], ctx, s["n_draft"],
                                           s["cu_q"], s["out"], s["lse"], max_k=s["max_k"], workspace=s["attn_ws"],
                                           status=s["status"])
    else:
        spade.spade_verify_attention(s["q"], s["k_cache"], s["v_cache"], ctx, s["n_draft"], s["cu_q"], s["out"],
                                     s["lse"], max_k=s["max_k"], workspace=s["attn_ws"], status=s["status"])


def _accept_args(s):
    return (s["hidden"], s["w_lm"], s["draft_tokens"], s["draft_probs"], s["uniforms"], s["mode"], s["cu_q"],
            s["n_draft"], s["accepted"], s["next"])


def _said(s, names):
    return {n: s[n] for n in names}


_HEAD = ("accepted", "next", "row_max", "row_sum", "row_arg_accept", "draft_logit", "status")


def run(state):
    s = state
    op = s["op"]
    if op == "attention":
        _attention(s, s["ctx_lens"])
        return _said(s, ("out", "lse", "status"))
    if op == "qkv":
        _qkv(s, s["ctx_lens"])
        return _said(s, ("q", "k_cache", "v_cache", "status"))
    if op == "accept":
        if s["temperature"] is not None or s["top_p"] is not None:
            spade.spade_verify_accept_sampling(*_accept_args(s), workspace=s["accept_ws"], status=s["status"],
                                               temperature=s["temperature"], top_p=s["top_p"])
        else:
            spade.spade_verify_accept(*_accept_args(s), workspace=s["accept_ws"], status=s["status"])
        return _said(s, _HEAD)
    # One verify step: the scheduler's context lengths come first, the commit advances them.
    s["ctx_now"].copy_(s["ctx_lens"])
    _qkv(s, s["ctx_now"])
    _attention(s, s["ctx_now"])
    if s["paged"]:
        spade.spade_verify_accept_commit_paged(*_accept_args(s), s["k_cache"], s["v_cache"], s["table"], s["ctx_now"],
                                               workspace=s["accept_ws"], status=s["status"])
    else:
        spade.spade_verify_accept_commit(*_accept_args(s), s["k_cache"], s["v_cache"], s["ctx_now"],
                                         workspace=s["accept_ws"], status=s["status"])
    return _said(s, ("q", "out", "lse", "k_cache", "v_cache", "ctx_now") + _HEAD)


# ---- 64-bit results ------------------------------------------------------------------------------
def _slots(s, b, lo, hi):
    """Index of slots [lo, hi) of sequence b in a cache: (leading index, slot index), each [hi - lo]."""
    at = torch.arange(lo, hi, device=DEV)
    if s["paged"]:
        page = s["case"]["page"]
        return s["table"][b].long()[at // page], at % page
    return torch.full_like(at, b), at


def _exact_qkv(s):
    """Queries, and the caches with the block's keys and values in their slots."""
    c = s["case"]
    Hq, Hkv, D = c["Hq"], c["Hkv"], c["D"]
    y = s["x"].double() @ s["w_qkv"].double().t()
    y = y.view(s["R"], Hq + 2 * Hkv, D)
    pos = torch.cat([torch.arange(x, x + k + 1, device=DEV) for x, k in zip(s["ctx_list"], s["k_list"])]).double()
    freq = ROPE_THETA ** (-2.0 * torch.arange(D // 2, device=DEV).double() / D)
    angle = pos[:, None, None] * freq
    cos, sin = torch.cos(angle), torch.sin(angle)
    a, b = y[:, :Hq + Hkv, :D // 2], y[:, :Hq + Hkv, D // 2:]
    turned = torch.cat([a * cos - b * sin, b * cos + a * sin], -1)
    keys, values = s["k_cache"].double(), s["v_cache"].double()
    for i in range(c["B"]):
        r = slice(s["cu_list"][i], s["cu_list"][i + 1])
        lead, at = _slots(s, i, s["ctx_list"][i], s["ctx_list"][i] + s["k_list"][i] + 1)
        keys[lead, :, at] = turned[r, Hq:]
        values[lead, :, at] = y[r, Hq + Hkv:]
    return turned[:, :Hq], keys, values


def _exact_attention(s, q, keys, values):
    c = s["case"]
    Hq, Hkv, D = c["Hq"], c["Hkv"], c["D"]
    G = Hq // Hkv
    out = torch.empty((s["R"], Hq, D), dtype=torch.float64, device=DEV)
    lse = torch.empty((s["R"], Hq), dtype=torch.float64, device=DEV)
    for b in range(c["B"]):
        ctx, k = s["ctx_list"][b], s["k_list"][b]
        r = slice(s["cu_list"][b], s["cu_list"][b + 1])
        lead, at = _slots(s, b, 0, ctx + k + 1)
        kb, vb = (t[lead, :, at].double().transpose(0, 1) for t in (keys, values))  # [Hkv, L, D]
        qb = q[r].double().view(k + 1, Hkv, G, D).permute(1, 2, 0, 3)                # [Hkv, G, k + 1, D]
        score = qb.reshape(Hkv, G * (k + 1), D) @ kb.transpose(1, 2) / math.sqrt(D)
        score = score.view(Hkv, G, k + 1, -1)
        seen = torch.arange(ctx + k + 1, device=DEV)[None, :] <= ctx + torch.arange(k + 1, device=DEV)[:, None]
        score = score.masked_fill(~seen, -math.inf)
        lse[r] = torch.logsumexp(score, -1).permute(2, 0, 1).reshape(k + 1, Hq)
        o = torch.softmax(score, -1).view(Hkv, G * (k + 1), -1) @ vb
        out[r] = o.view(Hkv, G, k + 1, D).permute(2, 0, 1, 3).reshape(k + 1, Hq, D)
    return out, lse


def exact(case, seed):
    s = _inputs(case, seed)
    c = s["case"]
    said = {"status": torch.zeros(1, dtype=torch.int64)}
    if s["op"] == "attention":
        said["out"], said["lse"] = _exact_attention(s, s["q"], s["k_cache"], s["v_cache"])
        return said
    if s["op"] in ("qkv", "step"):
        said["q"], said["k_cache"], said["v_cache"] = _exact_qkv(s)
    if s["op"] == "step":
        said["out"], said["lse"] = _exact_attention(s, said["q"], said["k_cache"], said["v_cache"])
    if s["op"] in ("accept", "step"):
        said.update(_verify(s, _logits(s["hidden"], s["w_lm"], torch.float64)))
    if s["op"] == "step":
        said["ctx_now"] = s["ctx_lens"] + said["accepted"].to(torch.int32) + 1
        for b, a in enumerate(said["accepted"].tolist()):  # rejected drafts' slots are cleared
            lead, at = _slots(s, b, s["ctx_list"][b] + a + 1, s["ctx_list"][b] + s["k_list"][b] + 1)
            for name in ("k_cache", "v_cache"):
                said[name][lead, :, at] = 0.0
    return said
