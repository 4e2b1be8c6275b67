"""The work that a user of this library has it do, as cases that can be timed and compared.

A speculative-decoding loop calls three things per step: the draft-token draw while it drafts, the verify step, and,
after a verify step that stopped short, the distribution modification.  The verify step is by far the largest and the
listed cases follow its range: one prompt, a small batch, the batches of a server, one and many drafts, float32 and
bfloat16 logits, vocabularies of 32k to 152k entries, rows that start on 16-byte boundaries and rows that do not.  The
remaining cases are the draw and the modification, the position-wise verifier that the block verifier is compared
with, and one rank's share of the step when the output layer is split over the vocabulary.  ``draw`` gives further
cases of the same kinds and ranges.

Inputs come from ``workloads`` (language-model-like rows, draft tokens drawn from the draft rows, uniforms), so what is
decided, and how many of the rows need the exact form of Eq. 2, is what these inputs give.
"""
from __future__ import annotations

import math

import torch

from paper_2604_25925_b200 import binding, sharded, workloads

DEVICE = "cuda"
LARGEST_BYTES = 64 * 8 * 17 * 151936 * 4     # logits of the largest listed case


def _case(name, kind, B, K, gamma, V, dtype="fp32", temperature=1.0, alpha=0.85, ranks=1):
    return {"name": name, "kind": kind, "B": B, "K": K, "gamma": gamma, "V": V, "dtype": dtype,
            "temperature": temperature, "alpha": alpha, "ranks": ranks}


def listed():
    return [
        # one prompt, three drafts of twelve tokens: an interactive session, where only latency counts
        _case("verify_one_prompt", "verify", 1, 3, 12, 32256, temperature=0.4),
        # a handful of prompts on a 32k vocabulary
        _case("verify_b8", "verify", 8, 4, 4, 32000),
        # a serving batch with bfloat16 logits and a 128k vocabulary
        _case("verify_b32_bf16", "verify", 32, 4, 5, 128256, dtype="bf16", temperature=0.7, alpha=0.7),
        # a serving batch whose vocabulary is odd: rows start at any multiple of the element size
        _case("verify_b16_odd_vocab_bf16", "verify", 16, 4, 4, 50257, dtype="bf16", temperature=0.8, alpha=0.8),
        # many prompts, many drafts, 32k vocabulary
        _case("verify_b256_k8", "verify", 256, 8, 4, 32000, alpha=0.8),
        # the largest step: 5.3 GB of logits
        _case("verify_b64_largest", "verify", 64, 8, 8, 151936, alpha=0.9),
        # one draft per prompt: single-draft greedy block verification
        _case("gbv_b256", "gbv", 256, 1, 4, 32000, alpha=0.8),
        # the position-wise verifier the paper compares with, on its operating point as a batch
        _case("kseq_b64", "kseq", 64, 3, 12, 32256, temperature=0.4),
        # drafting: one token per prompt and draft from the draft model's logits; one prompt, and a serving batch
        _case("draw_one_prompt", "draw", 1, 3, 1, 32256, temperature=0.4),
        _case("draw_b32_bf16", "draw", 32, 4, 1, 128256, dtype="bf16", temperature=0.7, alpha=0.7),
        # one position of the distribution modification for a serving batch
        _case("modify_b64", "modify", 64, 8, 1, 151936, alpha=0.9),
        # one rank's share of the step with the output layer split over eight ranks
        _case("sharded_rank_of_8", "shard", 32, 8, 8, 151936, alpha=0.9, ranks=8),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["verify"] * 6 + ["gbv", "kseq", "draw", "draw", "modify", "shard"])
    dtype = rng.choice(["fp32", "bf16"])
    V = _log_uniform(rng, 8000, 160000)
    if rng.random() < 0.7:
        V = V // 64 * 64                      # padded vocabularies are the rule, odd ones occur
    B = _log_uniform(rng, 1, 256)
    K = rng.choice([1, 2, 3, 4, 4, 5, 6, 8, 8])
    gamma = rng.randint(1, 12)
    ranks = 1
    if kind == "gbv":
        K = 1
    elif kind in ("draw", "modify"):
        gamma = 1
    elif kind == "kseq":
        B, K, V = min(B, 128), rng.randint(2, 4), min(V, 50000)
    elif kind == "shard":
        ranks, B, V = rng.choice([2, 4, 8]), min(B, 64), max(V, 30000) // 64 * 64
    size = 2 if dtype == "bf16" else 4
    budget = LARGEST_BYTES // (4 if kind == "shard" else 2)
    B = max(1, min(B, budget // (K * (2 * gamma + 1) * V * size)))
    return {"kind": kind, "B": B, "K": K, "gamma": gamma, "V": V, "dtype": dtype,
            "temperature": rng.choice([0.4, 0.6, 0.7, 0.8, 1.0]), "alpha": rng.choice([0.5, 0.7, 0.8, 0.85, 0.9, 0.95]),
            "ranks": ranks}


def _config(case, seed, **other):
    f = {k: case[k] for k in ("B", "K", "gamma", "V", "dtype", "temperature", "alpha")}
    f.update(other)
    return workloads.VerifyConfig("case", seed=1 + seed, **f)


class _PeersOf:
    """The exchange of one rank whose peers' parts have arrived: rank r's own part goes into its place.  Stands where a
    process group's collectives stand, so that what is timed is this rank's own work."""

    def __init__(self, rank, stats_all, sums_all):
        self.rank = rank
        self.parts = [stats_all, sums_all]
        self.turn = 0

    def all_gather(self, t):
        part = self.parts[self.turn]
        self.turn = 1 - self.turn
        part[self.rank].copy_(t)
        return part

    def all_reduce_max(self, t):
        return t


def _verify_out(B, K, gamma):
    i32 = dict(dtype=torch.int32, device=DEVICE)
    f64 = dict(dtype=torch.float64, device=DEVICE)
    return binding.VerifyOutput(torch.empty(B, **i32), torch.empty(B, **i32), torch.empty((B, gamma + 1), **i32),
                                torch.empty((B, K, gamma), **f64), torch.empty((B, K, gamma), **f64), torch.empty(B, **i32))


def prepare(case, seed):
    """Logits, draft tokens and uniforms on the device, and what a decode loop keeps besides: the output buffers."""
    kind, B, K, gamma, V, T = (case[k] for k in ("kind", "B", "K", "gamma", "V", "temperature"))
    st = {"kind": kind, "T": float(T), "K": K}
    if kind in ("draw", "modify"):
        # rows of one position; the verify inputs of a one-draft batch hold such rows
        n = B * K if kind == "draw" else B
        inp = workloads.make_inputs(_config(case, seed, B=n, K=1, gamma=1), device=DEVICE)
        st["draft"] = inp.draft_logits[:, 0, 0].contiguous()
        st["u"] = inp.uniforms[:, 0].contiguous()
        if kind == "modify":
            st["target"] = inp.target_logits[:, 0, 0].contiguous()
            g = torch.Generator().manual_seed(seed)
            la = -6.0 * torch.rand(B, generator=g, dtype=torch.float64)
            st["log_a"] = la.to(DEVICE)
            st["log_b"] = (la + 0.8 * torch.randn(B, generator=g, dtype=torch.float64)).to(DEVICE)
        return st
    inp = workloads.make_inputs(_config(case, seed), device=DEVICE)
    if kind == "gbv":
        st.update(target=inp.target_logits[:, 0].contiguous(), draft=inp.draft_logits[:, 0].contiguous(),
                  tokens=inp.draft_tokens[:, 0].contiguous(), u=inp.uniforms)
        return st
    st.update(target=inp.target_logits, draft=inp.draft_logits, tokens=inp.draft_tokens, u=inp.uniforms)
    if kind == "verify":
        st["out"] = _verify_out(B, K, gamma)
    if kind == "shard":
        # every rank's records and sums, as the exchanges deliver them; the state keeps one rank's range
        bounds = sharded.shard_bounds(V, case["ranks"])
        rank = case["ranks"] // 2
        code = binding.DTYPE_BF16 if case["dtype"] == "bf16" else binding.DTYPE_F32
        shards = [(inp.target_logits[..., lo:hi].contiguous(), inp.draft_logits[..., lo:hi].contiguous(), lo)
                  for lo, hi in bounds]
        stats = torch.stack([binding.sgbv_shard_stats(q, p, inp.draft_tokens, lo, V, T) for q, p, lo in shards])
        sums = torch.stack([binding.sgbv_shard_sums(q, p, T, stats, torch.empty(
            binding.sgbv_shard_workspace_bytes(B, K, gamma, q.shape[-1], code), dtype=torch.uint8, device=DEVICE))
            for q, p, _ in shards])
        st["target"], st["draft"], st["v_begin"] = shards[rank]
        st["V"] = V
        st["exchange"] = _PeersOf(rank, stats, sums)
    return st


def run(st):
    kind, T = st["kind"], st["T"]
    if kind == "verify":
        o = binding.sgbv_verify_ex(st["target"], st["draft"], st["tokens"], st["u"], T, out=st["out"])
        return [o.accept_len, o.draft_idx, o.tokens, o.h, o.resmass, o.status]
    if kind == "gbv":
        o = binding.sgbv_verify_gbv(st["target"], st["draft"], st["tokens"], st["u"], T)
        return [o.accept_len, o.tokens, o.accept_prob, o.status]
    if kind == "kseq":
        o = binding.sgbv_verify_kseq(st["target"], st["draft"], st["tokens"], st["u"], T)
        return [o.accept_len, o.tokens, o.rho, o.accept_prob, o.status]
    if kind == "draw":
        return list(binding.sgbv_draw_tokens(st["draft"], st["u"], T))
    if kind == "modify":
        o = binding.sgbv_modify(st["target"], st["draft"], st["log_a"], st["log_b"], st["u"], st["K"], T)
        return [o.token, o.log_a, o.log_b, o.resmass, o.status]
    o = sharded.verify(st["target"], st["draft"], st["tokens"], st["u"], T, st["v_begin"], st["V"], st["exchange"])
    return [o.accept_len, o.draft_idx, o.tokens, o.h, o.resmass, o.status]


def work(case):
    """Every logit the method needs, once (the target rows behind the blocks are read for accepted blocks only and are
    left out), and the small tensors.  Per pair of logits: two exponentials, the sums, and Eq. 4's term."""
    kind, B, K, gamma, V = (case[k] for k in ("kind", "B", "K", "gamma", "V"))
    size = 2 if case["dtype"] == "bf16" else 4
    small = B * K * gamma * (4 + 4 + 16) + B * (gamma + 4) * 4
    pairs = B * K * gamma * V
    if kind == "draw":
        return {"bytes": B * K * (V * size + 24), "flops": 5 * B * K * V}
    if kind == "modify":
        return {"bytes": 2 * B * V * size + 48 * B, "flops": (10 + K) * B * V}
    if kind == "kseq":
        # two positions are reached on average (block efficiency 1.6 to 2.3), each a pair of rows, a dozen evaluations
        # of beta(rho)
        return {"bytes": 4 * B * V * size + small, "flops": 2 * B * V * (10 + 12 * 3)}
    if kind == "shard":
        # the statistics of all rows have to leave before the sums can start: the target rows behind the blocks are
        # part of the first sweep, and each row pair of the shard is read once
        return {"bytes": (2 * pairs + B * K * V) // case["ranks"] * size + small, "flops": (10 + K) * pairs // case["ranks"]}
    return {"bytes": 2 * pairs * size + small, "flops": (10 + K) * pairs}


def tolerance(case):
    """Vocabulary sums in float32, weights in float64: against the float64 oracle the listed cases (the large ones on 32
    batch rows) differ by up to 2e-7 in the 2-norm and 6e-7 in the largest value, and two implementations by twice that.
    Decisions are whole numbers and agree unless a uniform falls on a threshold or on the edge of a cell of the inverse
    CDF."""
    return {"rel": 2e-6, "max": 1e-5, "differ": 0.01}


def _f32(T):
    """The temperature as the library takes it, a float32, in 64 bits."""
    return float(torch.tensor(T, dtype=torch.float32))


def _g(u, K):
    """1 - (1 - u)^K without cancellation, u clamped to [0, 1]."""
    return -torch.expm1(K * torch.log1p(-u.clamp(0.0, 1.0)))


def _exact_block(zq, zp, tok, T, K_exp):
    """h (Eq. 2, Eq. 3) and residual masses of one batch row: zq [K,gamma+1,V], zp [K,gamma,V], tok [K,gamma]."""
    gamma = zp.shape[1]
    lq = torch.log_softmax(zq[:, :gamma].double() / T, -1)
    lp = torch.log_softmax(zp.double() / T, -1)
    at = tok.long().unsqueeze(-1)
    zero = torch.zeros_like(lq[:, :1, 0])
    la = torch.cat([zero, lq.gather(-1, at)[..., 0].cumsum(-1)], -1)        # [K,gamma+1]
    lb = torch.cat([zero, lp.gather(-1, at)[..., 0].cumsum(-1)], -1)
    c = (lb - la)[:, :gamma].exp()
    q = lq.exp_()
    t = torch.where(q > 0, c.unsqueeze(-1) * lp.exp_() / q, 1.0)
    R = (q * (1.0 - t).clamp(min=0.0) ** K_exp).sum(-1)                     # [K,gamma]
    a, b = la.exp(), lb.exp()
    gb_a = _g(b, K_exp) / a
    num = (R - (1.0 - c).clamp(min=0.0) ** K_exp).clamp(min=0.0)
    den = num + (gb_a[:, :gamma] - _g(c, K_exp)).clamp(min=0.0)
    sub = torch.where(den > 1e-12 * (gb_a[:, :gamma] + 1.0), num / den, 1.0)  # 0/0: accepted
    c_end = (lb - la)[:, gamma].exp()
    full = (a[:, gamma] * _g(c_end, K_exp) / _g(b[:, gamma], K_exp)).unsqueeze(-1)
    return torch.cat([sub[:, 1:], full], -1).clamp(0.0, 1.0), a[:, :gamma] * R


def _exact_kseq(st):
    """rho per position and the acceptance probabilities of the tried tokens, NaN where nothing was tried."""
    T, K = _f32(st["T"]), st["K"]
    B, _, g1, _ = st["target"].shape
    gamma = g1 - 1
    rho_out = torch.full((B, gamma), math.nan, dtype=torch.float64)
    acc_out = torch.full((B, K, gamma), math.nan, dtype=torch.float64)
    tok, u = st["tokens"].cpu(), st["u"].cpu()
    for b in range(B):
        kept = list(range(K))
        for i in range(gamma):
            lq = torch.log_softmax(st["target"][b, kept[0], i].double() / T, -1)
            lp = torch.log_softmax(st["draft"][b, kept[0], i].double() / T, -1)
            q, p, n = lq.exp(), lp.exp(), len(kept)
            rho = torch.ones((), dtype=torch.float64, device=DEVICE)
            if n > 1:
                lo, hi = rho.clone(), rho * n
                for _ in range(52):
                    mid = 0.5 * (lo + hi)
                    beta = torch.minimum(p, q / mid).sum()
                    up = _g(beta, n) - mid * beta > 0
                    lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
                rho = 0.5 * (lo + hi)
            rho = float(rho)
            rho_out[b, i] = rho
            hit = None
            for k in kept:
                x = int(tok[b, k, i])
                acc_out[b, k, i] = min(1.0, math.exp(float(lq[x] - lp[x])) / rho)
                if float(u[b, k * gamma + i]) < float(acc_out[b, k, i]):
                    hit = x
                    break
            if hit is None:
                break
            kept = [k for k in kept if int(tok[b, k, i]) == hit]
    return rho_out, acc_out


def exact(case, seed):
    """The weights, masses and acceptance probabilities in 64 bits.  Tokens are drawn by inverse CDF, where an entry's
    cell can be narrower than the rounding of any 32-bit sum, so what follows from the drawn token (its log-probability)
    has no value of its own here."""
    kind, K = case["kind"], case["K"]
    if kind == "draw":
        return None
    st = prepare(case, seed)
    T = _f32(st["T"])
    if kind == "kseq":
        if case["B"] * case["gamma"] > 1600:
            return None                       # tens of seconds
        rho, acc = _exact_kseq(st)
        return [None, None, rho, acc, None]
    if kind == "modify":
        q = torch.softmax(st["target"].double() / T, -1)
        p = torch.softmax(st["draft"].double() / T, -1)
        c = (st["log_b"] - st["log_a"]).exp().unsqueeze(-1)
        t = torch.where(q > 0, c * p / q, 1.0)
        return [None, None, None, (q * (1.0 - t).clamp(min=0.0) ** K).sum(-1), None]
    if kind == "shard":                       # the state holds one rank's range: the whole rows again
        del st
        inp = workloads.make_inputs(_config(case, seed), device=DEVICE)
        zq, zp, tok = inp.target_logits, inp.draft_logits, inp.draft_tokens
    else:
        zq, zp, tok = st["target"], st["draft"], st["tokens"]
    if kind == "gbv":
        zq, zp, tok = zq.unsqueeze(1), zp.unsqueeze(1), tok.unsqueeze(1)
    rows = [_exact_block(zq[b], zp[b], tok[b], T, K) for b in range(case["B"])]
    h, S = (torch.stack([r[n] for r in rows]) for n in (0, 1))
    if kind == "gbv":
        return [None, None, h, None]
    return [None, None, None, h, S, None]
