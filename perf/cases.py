"""The work a serving program has this package do, as cases that can be timed and compared.

A case is one call of a public entry point on inputs already on the GPU:

  step    the fuse-and-verify step of one speculation round, FuseVerify (a
          workspace and the output tensors kept between rounds, as a serving
          loop keeps them);
  draft   the drafter's draw, draft_tokens (one drafted position of every
          sequence, or every position of a round at once);
  xvocab  the step for a drafter and a verifier with different vocabularies,
          fuse_verify_xvocab.

The logits are shaped like a trained model's next-token distributions: for
each row a heavy-tailed profile over the vocabulary in random order (one or a
few tokens hold most of the mass), the verifier and the drafter half a nat
apart on every token, and the drafter on the compressed context differing
from the one on the full context on a fraction of the tokens.  Drafts are
drawn from the drafter, greedily or by sampling, as the mode has it.
"""
from __future__ import annotations

import math

import torch

from paper_2608_26004_gb300 import asymspec as A

TORCH_DTYPE = {"fp32": torch.float32, "bf16": torch.bfloat16}
ABI_DTYPE = {"fp32": A.FP32, "bf16": A.BF16}
MODE = {"greedy": A.MODE_GREEDY, "stochastic": A.MODE_STOCHASTIC}
GATE = {"jsd": A.DIV_JSD, "none": A.DIV_NONE, "kl": A.DIV_KL, "lambda": A.DIV_LAMBDA}
GAMMA, BETA, LAMBDA = 0.5, 1.0, 0.1
PROFILE = 2.5    # logit = -PROFILE ln(rank): the most likely token holds about 0.7 of a row
DRAFTER = 0.5    # standard deviation between the verifier's and the drafter's logits
SHIFT = 3.0      # standard deviation of a token's shift between the two contexts
LARGEST = 3 * 256 * 5 * 151936 * 4  # logit bytes of the largest listed step


def _step(name, B, K, V, dtype, mode, gate="jsd", fuse_bonus=False, outputs="tokens", shifted=0.05):
    return dict(name=name, kind="step", B=B, K=K, V=V, dtype=dtype, mode=mode, gate=gate,
                fuse_bonus=fuse_bonus, outputs=outputs, shifted=shifted)


def _draft(name, rows, V, dtype, mode):
    return dict(name=name, kind="draft", rows=rows, V=V, dtype=dtype, mode=mode)


def _xvocab(name, B, K, S, V_d, V_v, dtype, mode, shifted=0.05):
    return dict(name=name, kind="xvocab", B=B, K=K, S=S, V_d=V_d, V_v=V_v, dtype=dtype,
                mode=mode, shifted=shifted)


def listed():
    return [
        # one interactive sequence, a small vocabulary, fp32 logits: launches and latency
        _step("step-1x4-fp32-greedy", 1, 4, 32000, "fp32", "greedy"),
        # a lightly loaded server, sampling
        _step("step-8x5-bf16-stochastic", 8, 5, 151936, "bf16", "stochastic"),
        # a loaded server, the paper's greedy decoding
        _step("step-64x7-bf16-greedy", 64, 7, 128256, "bf16", "greedy"),
        # the same, sampling: the benchmark's workload
        _step("step-64x7-bf16-stochastic", 64, 7, 128256, "bf16", "stochastic"),
        # long drafts under the KL gate of the ablation, contexts far apart
        _step("step-32x8-bf16-stochastic-kl", 32, 8, 151936, "bf16", "stochastic", gate="kl",
              shifted=0.2),
        # the largest batch, fp32 logits
        _step("step-256x4-fp32-stochastic", 256, 4, 151936, "fp32", "stochastic"),
        # a vocabulary that no vector divides (added tokens): rows at odd addresses
        _step("step-32x4-odd-bf16-greedy", 32, 4, 100003, "bf16", "greedy", fuse_bonus=True),
        # an evaluation run that records every row's statistics and fused log-probabilities
        _step("step-8x5-bf16-greedy-recorded", 8, 5, 151936, "bf16", "greedy", outputs="all"),
        # the drafter's draw, one position of every sequence: K times a round
        _draft("draft-64-bf16-stochastic", 64, 128256, "bf16", "stochastic"),
        # every position at once (a round replayed)
        _draft("draft-512-bf16-stochastic", 512, 128256, "bf16", "stochastic"),
        # one sequence drafting greedily in fp32
        _draft("draft-1-fp32-greedy", 1, 32000, "fp32", "greedy"),
        # drafter and verifier of different families sharing most of their tokens
        _xvocab("xvocab-64x7-bf16-stochastic", 64, 7, 109568, 151936, 128256, "bf16", "stochastic"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocabulary(rng, lo=32000, hi=151936):
    """Two in three padded to a multiple of 64, the others as they come (every other one odd)."""
    v = _log_uniform(rng, lo, hi)
    return min(hi, max(lo, (v + 32) // 64 * 64)) if rng.random() < 2 / 3 else v


def draw(rng):
    kind = rng.choices(("step", "draft", "xvocab"), (7, 2, 1))[0]
    dtype = rng.choices(("bf16", "fp32"), (2, 1))[0]
    mode = rng.choice(("greedy", "stochastic"))
    elt = 2 if dtype == "bf16" else 4
    if kind == "draft":
        c = _draft("", _log_uniform(rng, 1, 512), _vocabulary(rng), dtype, mode)
    elif kind == "xvocab":
        V_d, V_v = _vocabulary(rng, 64000), _vocabulary(rng, 64000)
        S = int(min(V_d, V_v) * rng.uniform(0.6, 0.95))
        S = S // 64 * 64 if rng.random() < 0.5 else S
        c = _xvocab("", _log_uniform(rng, 1, 64), rng.randint(1, 8), S, V_d, V_v, dtype, mode,
                    rng.choice((0.02, 0.05, 0.1, 0.2)))
    else:
        outputs = rng.choices(("tokens", "all"), (6, 1))[0]
        V, K = _vocabulary(rng), rng.randint(1, 8)
        most = min(256, LARGEST // (3 * (K + 1) * V * elt), 64 if outputs == "all" else 256)
        gate = rng.choices(("jsd", "kl", "none", "lambda"), (7, 1, 1, 1))[0]
        c = _step("", _log_uniform(rng, 1, most), K, V, dtype, mode, gate,
                  mode == "greedy" and rng.random() < 0.25, outputs, rng.choice((0.02, 0.05, 0.1, 0.2)))
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs

def _profile(rows, V, gen):
    """[rows, V] fp32 logits: -PROFILE ln(rank) for ranks in random order."""
    u = torch.rand(rows, V, generator=gen, device="cuda")
    return u.mul_(V).add_(1.0).log_().mul_(-PROFILE)


def _normal_like(x, gen):
    return torch.randn(x.shape, generator=gen, device="cuda")


def _drafter_pair(z, shifted, gen):
    """The drafter on the full and on the compressed context, from the verifier's profile."""
    a = z + DRAFTER * _normal_like(z, gen)
    hit = torch.rand(z.shape, generator=gen, device="cuda") < shifted
    return a, a + hit * (SHIFT * _normal_like(z, gen))


def _drafts(a, mode, gen):
    """(token, probability) of each row of the drafter's logits, int32 and fp32."""
    x = a.float()
    g = x
    if mode == "stochastic":  # one draw of softmax(a)
        e = torch.rand(x.shape, generator=gen, device="cuda").clamp_(1e-30)
        g = x - e.log_().neg_().log_()
    d = g.argmax(-1, keepdim=True)
    p = (x.gather(-1, d) - x.logsumexp(-1, keepdim=True)).exp().clamp_(1e-30, 1.0)
    return d[..., 0].int(), p[..., 0]


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = TORCH_DTYPE[case["dtype"]]
    if case["kind"] == "draft":
        return dict(logits=_profile(case["rows"], case["V"], gen).to(dt),
                    unif=torch.rand(case["rows"], generator=gen, device="cuda"))
    B, K1 = case["B"], case["K"] + 1
    x = {}
    if case["kind"] == "xvocab":
        S, V_d, V_v = case["S"], case["V_d"], case["V_v"]
        # the shared tokens keep the drafter's order; the verifier numbers them its own way
        x["map_d"] = torch.randperm(V_d, generator=gen, device="cuda")[:S].sort().values.int()
        x["map_v"] = torch.randperm(V_v, generator=gen, device="cuda")[:S].int()
        z = _profile(B * K1, V_d, gen)
        t = _profile(B * K1, V_v, gen)
        t[:, x["map_v"].long()] = z[:, x["map_d"].long()]
        a, b = _drafter_pair(z, case["shifted"], gen)
        a, b, t = a.to(dt), b.to(dt), t.to(dt)
        d, p = _drafts(a[:, x["map_d"].long()], case["mode"], gen)
    else:
        z = _profile(B * K1, case["V"], gen)
        a, b = _drafter_pair(z, case["shifted"], gen)
        a, b, t = a.to(dt), b.to(dt), z.to(dt)
        d, p = _drafts(a, case["mode"], gen)
    x.update(a=a.view(B, K1, -1), b=b.view(B, K1, -1), t=t.view(B, K1, -1),
             tokens=d.view(B, K1)[:, :-1].contiguous(), probs=p.view(B, K1)[:, :-1].contiguous(),
             unif=torch.rand(B, K1, generator=gen, device="cuda"))
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    state = dict(case=case, x=x)
    if case["kind"] == "draft":
        rows = case["rows"]
        state["out"] = (torch.empty(rows, dtype=torch.int32, device="cuda"),
                        torch.empty(rows, dtype=torch.float32, device="cuda"))
        return state
    B, K = case["B"], case["K"]
    # accepted length and next token of every sequence in one tensor, read back in one copy
    state["result"] = torch.empty(2, B, dtype=torch.int32, device="cuda")
    state["error"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    if case["kind"] == "xvocab":
        n = A.xvocab_workspace_bytes(B, K, case["S"], case["V_d"], case["V_v"],
                                     ABI_DTYPE[case["dtype"]])
        state["workspace"] = torch.zeros(n, dtype=torch.uint8, device="cuda")
        state["gate"] = A.gate_params(GAMMA, BETA, LAMBDA, MODE[case["mode"]], A.DIV_JSD)
        return state
    out = dict(accept_len=state["result"][0], next_token=state["result"][1],
               error_word=state["error"])
    if case["outputs"] == "all":
        V = case["V"]
        out["row_stats"] = torch.empty(B, K + 1, 8, device="cuda")
        out["row_tokens"] = torch.empty(B, K + 1, 2, dtype=torch.int32, device="cuda")
        out["fused_logprobs"] = torch.empty(B, K + 1, V, device="cuda")
    state["out"] = out
    state["step"] = A.FuseVerify(B, K, V_max=case["V"])
    return state


# ---------------------------------------------------------------- one pass

def run(state):
    case, x = state["case"], state["x"]
    if case["kind"] == "draft":
        return A.draft_tokens(x["logits"], x["unif"], mode=MODE[case["mode"]], out=state["out"])
    if case["kind"] == "xvocab":
        r, ws = state["result"], state["workspace"]
        st = A.fuse_verify_xvocab(
            x["a"].data_ptr(), x["b"].data_ptr(), case["V_d"], x["t"].data_ptr(), case["V_v"],
            x["map_d"].data_ptr(), x["map_v"].data_ptr(), case["S"], x["tokens"].data_ptr(),
            x["probs"].data_ptr(), x["unif"].data_ptr(), case["B"], case["K"],
            ABI_DTYPE[case["dtype"]], state["gate"], r[0].data_ptr(), r[1].data_ptr(), 0,
            ws.data_ptr(), ws.numel(), state["error"].data_ptr(),
            torch.cuda.current_stream().cuda_stream)
        if st != A.OK:
            raise A.AsymSpecError(st, "asymspec_fuse_verify_xvocab")
        return [r, state["error"]]
    stochastic, record = case["mode"] == "stochastic", case["outputs"] == "all"
    out = state["step"](
        x["a"], x["b"], x["t"], x["tokens"], x["probs"] if stochastic else None,
        x["unif"] if stochastic else None, gamma=GAMMA, beta=BETA, lam=LAMBDA,
        mode=MODE[case["mode"]], divergence=GATE[case["gate"]], fuse_bonus=case["fuse_bonus"],
        row_stats=record, row_tokens=record, fused_logprobs=record, out=state["out"])
    if record:
        return [state["result"], out["error_word"], out["row_tokens"], out["row_stats"],
                out["fused_logprobs"]]
    return [state["result"], out["error_word"]]


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    elt = 2 if case["dtype"] == "bf16" else 4
    if case["kind"] == "draft":
        n = case["rows"] * case["V"]
        return {"bytes": n * elt + 12 * case["rows"], "flops": 3 * n}
    B, K = case["B"], case["K"]
    rows, stochastic = B * (K + 1), case["mode"] == "stochastic"
    # the bonus row of a greedy step emits argmax t and needs no other logits
    bonus_t_only = not stochastic and not case.get("fuse_bonus") and case.get("outputs") != "all"
    abrows = rows - B if bonus_t_only else rows
    small = 8 * B + 4 * B * K + (4 * B * K + 4 * rows if stochastic else 0)
    if case["kind"] == "xvocab":
        S = case["S"]
        # the pairs' logits (spread over whole rows: nearly every sector holds some), and the maps
        return {"bytes": (2 * abrows * case["V_d"] + rows * case["V_v"]) * elt + 8 * S + small,
                "flops": 12 * S * (abrows + rows)}
    V = case["V"]
    more = rows * (32 + 8 + 4 * V) if case["outputs"] == "all" else 0
    return {"bytes": (2 * abrows + rows) * V * elt + small + more, "flops": 12 * V * (abrows + rows)}


def tolerance(case):
    # whole values: the last digits of a sum decide a draw that falls on the boundary of two
    # tokens, an argmax of two equal scores or an acceptance at its threshold; floating outputs
    # are 32-bit sums and logarithms
    if case["kind"] == "draft":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
    if case["kind"] == "step" and case["outputs"] == "all":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
    return {"rel": 0.0, "differ": 0.01}


# ---------------------------------------------------------------- the same in 64 bits

def _draw(mass, u):
    """Smallest index whose cumulative mass exceeds u times the total, for each row."""
    c = mass.cumsum(-1)
    tau = u[:, None] * c[:, -1:]
    return (c <= tau).sum(-1).clamp_(max=mass.shape[-1] - 1)


def _exact_step(case, a, b, t, x, record):
    """Sequences [B, K+1, V] in 64 bits: (accepted length, emitted index, rows' records)."""
    B, K1, V = a.shape
    K, stochastic = K1 - 1, case["mode"] == "stochastic"
    gate = case.get("gate", "jsd")
    lens, nexts, stats, toks, lps = [], [], [], [], []
    lng = math.log(GAMMA)
    for i in range(B):
        ai, bi, ti = a[i].double(), b[i].double(), t[i].double()
        s = ti + BETA * (ai - bi)
        L = [v.logsumexp(-1) for v in (ai, bi, ti, s)]
        la, lb = ai - L[0][:, None], bi - L[1][:, None]
        p, q = la.exp(), lb.exp()
        d = x["tokens"][i].long()
        k = torch.arange(K, device=a.device)
        D = torch.zeros(K1, dtype=torch.float64, device=a.device)
        if gate == "jsd":
            lm = ((p + q) / 2).log()
            D = 0.5 * (torch.xlogy(p, p) - p * lm + torch.xlogy(q, q) - q * lm).nan_to_num(0.0).sum(-1)
        elif gate == "kl":
            D = (p * (la - lb)).sum(-1)
        elif gate == "lambda":
            D[:K] = LAMBDA * (la[k, d] - lb[k, d])
        lngeff = lng - D
        margin = torch.full((K1,), math.nan, dtype=torch.float64, device=a.device)
        mass = margin.clone()
        emit = s.argmax(-1)
        if stochastic:
            lq = s - L[3][:, None]
            ratio = lq[k, d].exp() / x["probs"][i].double() / lngeff[:K].exp()
            u = x["unif"][i].double()
            accept = ratio > u[:K]
            margin[:K] = u[:K] - ratio
            m = lq.exp()
            m[:K] = (m[:K] - p[:K]).clamp_(min=0.0)
            mass = m.sum(-1)
            empty = mass == 0
            m[empty] = lq[empty].exp()
            emit = _draw(m, u[K].expand(K1))
        else:
            lr = (ti[k, d] - L[2][:K]) - lb[k, d]
            accept = lr > lngeff[:K]
            margin[:K] = 1 - (lr - lngeff[:K]).exp()
            if not case.get("fuse_bonus"):
                emit[K] = ti[K].argmax()
        n = int(accept.long().cumprod(0).sum())
        lens.append(n)
        nexts.append(int(emit[n]))
        if record:
            stats.append(torch.stack(L + [D, lngeff.exp(), margin, mass], -1))
            toks.append(torch.stack([s.argmax(-1), emit], -1).int())
            lps.append(s - L[3][:, None])
    both = torch.tensor([lens, nexts], dtype=torch.int32)
    return both, (torch.stack(toks), torch.stack(stats), torch.stack(lps)) if record else None


def exact(case, seed):
    x = _inputs(case, seed)
    if case["kind"] == "draft":
        tokens, probs = [], []
        for r in range(case["rows"]):
            p = x["logits"][r].double().softmax(-1)
            if case["mode"] == "greedy":
                d = x["logits"][r].float().argmax()
            else:
                d = _draw(p[None], x["unif"][r:r + 1].double())[0]
            tokens.append(int(d))
            probs.append(float(p[d]))
        return torch.tensor(tokens, dtype=torch.int32), torch.tensor(probs, dtype=torch.float64)
    error = torch.zeros(1, dtype=torch.int32)
    if case["kind"] == "xvocab":
        md, mv = x["map_d"].long(), x["map_v"].long()
        both, _ = _exact_step(case, x["a"][..., md], x["b"][..., md], x["t"][..., mv], x, False)
        both[1] = x["map_v"].cpu()[both[1].long()]
        return [both, error]
    record = case["outputs"] == "all"
    both, more = _exact_step(case, x["a"], x["b"], x["t"], x, record)
    return [both, error, *more] if record else [both, error]
