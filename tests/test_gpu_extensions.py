"""GPU parity of the entry points beyond the verify step: Algorithm 2's draw (``sgbv_modify``) and the
comparison verifiers, against the oracle's functions on the same seeded inputs."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_25925_b200 import binding, sharded, workloads

pytestmark = pytest.mark.gpu


def _position_rows(cfg, device="cuda"):
    """[B,V] target and draft logits of one position: the position-0 rows of a seeded verify input set."""
    inp = workloads.make_inputs(cfg, device=device)
    return inp.target_logits[:, 0, 0].contiguous(), inp.draft_logits[:, 0, 0].contiguous()


@pytest.mark.parametrize("B,K,V,dtype,T", [(5, 3, 4099, "fp32", 0.8), (7, 1, 32000, "fp32", 1.0), (40, 4, 32000, "bf16", 0.7),
                                          (3, 8, 151936, "fp32", 1.0), (2, 2, 17, "fp32", 1.0), (200, 3, 9000, "bf16", 0.4)])
def test_modify_matches_the_oracle(B, K, V, dtype, T):
    cfg = workloads.VerifyConfig("mod", B=B, K=1, gamma=1, V=V, dtype=dtype, temperature=T, alpha=0.8, seed=900 + V % 97)
    zq, zp = _position_rows(cfg)
    g = torch.Generator().manual_seed(B * 131 + K)
    la = (-6.0 * torch.rand(B, generator=g, dtype=torch.float64)).cuda()
    lb = (la.cpu() + 0.8 * torch.randn(B, generator=g, dtype=torch.float64)).cuda()
    la[0], lb[0] = 0.0, 0.0                                    # an empty carried sequence: c = 1
    u = torch.rand(B, generator=g, dtype=torch.float32).cuda()
    out = binding.sgbv_modify(zq, zp, la, lb, u, K, T)
    torch.cuda.synchronize()
    ref = oracle.modify(zq.float().cpu().numpy(), zp.float().cpu().numpy(), la.cpu().numpy(), lb.cpu().numpy(),
                        u.cpu().numpy(), K, T)
    tok, st = out.token.cpu().numpy(), out.status.cpu().numpy()
    R = out.resmass.cpu().numpy()
    np.testing.assert_allclose(R, ref.R, rtol=1e-5, atol=1e-9)
    assert (st == ref.status).all()
    near = ref.margin < 1e-6                                    # draws within 1e-6 of a CDF edge may differ: counted
    assert near.sum() <= max(2, B // 3)
    assert (tok[~near] == ref.token[~near]).all()
    same = tok == ref.token
    np.testing.assert_allclose(out.log_a.cpu().numpy()[same], ref.loga[same], rtol=0, atol=2e-5)
    np.testing.assert_allclose(out.log_b.cpu().numpy()[same], ref.logb[same], rtol=0, atol=2e-5)


def test_modify_flags_and_degenerate_rows():
    cfg = workloads.VerifyConfig("modf", B=4, K=1, gamma=1, V=700, alpha=0.8, seed=77)
    zq, zp = _position_rows(cfg)
    zq, zp = zq.clone(), zp.clone()
    zp[1] = zq[1]                          # p == q and b >= a: no residual mass, the draw comes from q
    zq[2, 5] = float("nan")
    zq[3, 9] = float("-inf")               # allowed
    la = torch.tensor([-1.0, -2.0, -1.0, -1.0], dtype=torch.float64).cuda()
    lb = torch.tensor([-1.5, -1.0, -1.0, -0.5], dtype=torch.float64).cuda()
    u = torch.tensor([0.2, 0.5, 0.5, 0.9], dtype=torch.float32).cuda()
    out = binding.sgbv_modify(zq, zp, la, lb, u, 2, 1.0)
    torch.cuda.synchronize()
    ref = oracle.modify(zq.cpu().numpy(), zp.cpu().numpy(), la.cpu().numpy(), lb.cpu().numpy(), u.cpu().numpy(), 2, 1.0)
    st = out.status.cpu().numpy()
    assert (st == ref.status).all()
    assert st[1] & binding.STATUS_DEGENERATE_RESIDUAL and st[2] & binding.STATUS_NONFINITE_LOGIT
    assert out.token[2].item() == -1 and (out.token.cpu().numpy()[[0, 1, 3]] == ref.token[[0, 1, 3]]).all()


@pytest.mark.parametrize("entry", ["modify", "verify", "sharded"])
def test_a_residual_of_nothing_but_rounding_still_gives_a_token(entry):
    """Rows of two entries in cells of their own, the draft's logits the target's plus 0.1 rounded to float32: q and p differ by
    rounding, and what one kernel sees of max(q - p, 0) in a cell need not be there when the cell is worked out again.
    Whatever is drawn is one of the two entries, and flagged if it came from q."""
    B, V = 1 << 16, 512
    g = torch.Generator().manual_seed(1)
    q = torch.full((B, V), float("-inf"))
    q[:, 3] = torch.randn(B, generator=g)
    q[:, 300] = q[:, 3] - 3 * torch.rand(B, generator=g)
    p, u = (q + 0.1).cuda(), torch.rand(B, 2, generator=g).cuda()
    q = q.cuda()
    zero = torch.zeros(B, dtype=torch.float64, device="cuda")
    if entry == "modify":
        out = binding.sgbv_modify(q, p, zero, zero, u[:, 1].contiguous(), 1, 1.0)
        drawn, status = out.token, out.status
    else:
        target, draft = torch.stack([q, q], 1).view(B, 1, 2, V), p.view(B, 1, 1, V)
        u[:, 0] = 1.0 - 2.0 ** -24                            # rejects whatever is not certain
        tok = torch.where(q[:, 3:4] < -5.0, 3, 300).int().view(B, 1, 1)
        tok[::2] = 3
        if entry == "verify":
            out = binding.sgbv_verify_ex(target, draft, tok, u, 1.0)
        else:
            parts = [(target[..., lo:lo + 256].contiguous(), draft[..., lo:lo + 256].contiguous(), lo) for lo in (0, 256)]
            out = sharded.verify_all_ranks_on_one_device(parts, tok, u, 1.0, V)[0]
        rejected = out.accept_len == 0
        assert rejected.sum() > 100
        drawn, status = out.tokens[rejected, 0], out.status[rejected]
    assert ((drawn == 3) | (drawn == 300)).all(), int((drawn < 0).sum())
    assert ((status & ~binding.STATUS_DEGENERATE_RESIDUAL) == 0).all()


@pytest.mark.parametrize("V,dtype,shift", [(701, "fp32", 0), (40001, "bf16", 1), (40000, "fp32", 3), (151937, "bf16", 0)])
def test_modify_flags_on_rows_that_start_anywhere(V, dtype, shift):
    """Among them NaN and +inf in the first and the last entry of a tensor, which no copy brings."""
    B = 7
    cfg = workloads.VerifyConfig("modany", B=B, K=1, gamma=1, V=V, dtype=dtype, alpha=0.8, seed=V)
    zq, zp = _position_rows(cfg)

    def moved(t):
        return torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)[shift:].view(t.shape).copy_(t)
    zq, zp = moved(zq), moved(zp)
    zq[0, 0] = float("nan")
    zp[1, V // 2] = float("inf")
    zp[2] = zq[2]                          # p == q and b >= a: no residual mass, the draw comes from q
    zq[3, V // 2:] = float("-inf")         # a masked half
    zq[4] = float("-inf")                  # no finite entry
    zp[B - 1, V - 1] = float("inf")
    g = torch.Generator().manual_seed(V)
    la = -2.0 * torch.rand(B, dtype=torch.float64, generator=g)
    lb = la - 0.4
    lb[2] = la[2] + 0.5
    u = torch.rand(B, generator=g)
    out = binding.sgbv_modify(zq, zp, la.cuda(), lb.cuda(), u.cuda(), 3, 0.9)
    ref = oracle.modify(zq.float().cpu().numpy(), zp.float().cpu().numpy(), la.numpy(), lb.numpy(), u.numpy(), 3, 0.9)
    assert binding.last_main_kernel() == "fused_chain_kernel"
    st, tok = out.status.cpu().numpy(), out.token.cpu().numpy()
    bad = binding.STATUS_NONFINITE_LOGIT
    assert st.tolist() == [bad, bad, binding.STATUS_DEGENERATE_RESIDUAL, 0, bad, 0, bad] and (st == ref.status).all()
    assert (tok[[0, 1, 4, 6]] == -1).all() and out.log_a[[0, 1, 4, 6]].isnan().all()
    for b in (2, 3, 5):
        assert tok[b] == ref.token[b] or ref.margin[b] < 1e-6
    np.testing.assert_allclose(out.resmass.cpu().numpy()[[3, 5]], ref.R[[3, 5]], rtol=1e-5, atol=1e-9)


def test_modify_over_several_positions_follows_the_oracle_chain():
    """A few positions in a row, the carried logs fed back (in place), as a decode loop would do."""
    B, V, K, T = 6, 12000, 3, 0.9
    g = torch.Generator().manual_seed(5)
    la = torch.zeros(B, dtype=torch.float64).cuda() - 0.7
    lb = torch.zeros(B, dtype=torch.float64).cuda() - 1.1
    rla, rlb = la.cpu().numpy().copy(), lb.cpu().numpy().copy()
    for pos in range(4):
        cfg = workloads.VerifyConfig("modp", B=B, K=1, gamma=1, V=V, temperature=T, alpha=0.85, seed=300 + pos)
        zq, zp = _position_rows(cfg)
        u = torch.rand(B, generator=g, dtype=torch.float32).cuda()
        out = binding.sgbv_modify(zq, zp, la, lb, u, K, T)
        torch.cuda.synchronize()
        ref = oracle.modify(zq.cpu().numpy(), zp.cpu().numpy(), rla, rlb, u.cpu().numpy(), K, T)
        ok = ref.margin >= 1e-6
        assert (out.token.cpu().numpy()[ok] == ref.token[ok]).all()
        # carry on from the oracle's state where the draws agree (they all do unless a uniform sits on an edge)
        la, lb = out.log_a, out.log_b
        rla, rlb = ref.loga, ref.logb
        np.testing.assert_allclose(la.cpu().numpy()[ok], rla[ok], atol=5e-5)
        la = torch.from_numpy(rla).cuda()
        lb = torch.from_numpy(rlb).cuda()


def _kseq_compare(inp, T):
    out = binding.sgbv_verify_kseq(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, T)
    torch.cuda.synchronize()
    ref = oracle.kseq_verify(inp.target_logits.float().cpu().numpy(), inp.draft_logits.float().cpu().numpy(),
                             inp.draft_tokens.cpu().numpy(), inp.uniforms.cpu().numpy(), T)
    tau, tokens, st = out.accept_len.cpu().numpy(), out.tokens.cpu().numpy(), out.status.cpu().numpy()
    rho, acc = out.rho.cpu().numpy(), out.accept_prob.cpu().numpy()
    B = tau.shape[0]
    near = (ref.margin_accept < 1e-6) | (ref.margin_sample < 1e-6)     # a uniform on a threshold: counted, excused
    assert near.sum() <= max(2, B // 3)
    ok = ~near
    assert (st[ok] == ref.status[ok]).all()
    assert (tau[ok] == ref.tau[ok]).all() and (tokens[ok] == ref.tokens[ok]).all()
    # rho and the acceptance probabilities of what both sides tried
    both = ok[:, None] & ~np.isnan(ref.rho) & ~np.isnan(rho)
    np.testing.assert_allclose(rho[both], ref.rho[both], rtol=1e-5)
    assert (np.isnan(rho[ok]) == np.isnan(ref.rho[ok])).all()
    both = ok[:, None, None] & ~np.isnan(ref.acc) & ~np.isnan(acc)
    np.testing.assert_allclose(acc[both], ref.acc[both], rtol=1e-5, atol=1e-9)
    return out, ref


@pytest.mark.parametrize("B,K,gamma,V,dtype,T,alpha", [(6, 3, 4, 4099, "fp32", 0.8, 0.8), (8, 4, 4, 32000, "fp32", 1.0, 0.85),
                                                      (5, 1, 5, 9000, "fp32", 0.9, 0.9), (4, 8, 3, 32000, "bf16", 0.7, 0.7),
                                                      (2, 2, 2, 151936, "fp32", 1.0, 0.9), (3, 5, 2, 17, "fp32", 1.0, 0.5)])
def test_kseq_matches_the_oracle(B, K, gamma, V, dtype, T, alpha):
    cfg = workloads.VerifyConfig("ks", B=B, K=K, gamma=gamma, V=V, dtype=dtype, temperature=T, alpha=alpha, seed=640 + K)
    inp = workloads.make_inputs(cfg, device="cuda")
    _kseq_compare(inp, T)
    assert binding.last_main_kernel() == "kseq_kernel"


@pytest.mark.parametrize("B,K,gamma,V,dtype,T,alpha,shift", [
    (1, 4, 6, 50257, "bf16", 0.6, 0.95, 0),     # eight CTAs per row, rows that start anywhere
    (40, 2, 3, 8191, "fp32", 0.9, 0.8, 1),      # four, off a 16-byte boundary
    (80, 3, 2, 9000, "fp32", 0.5, 0.9, 0),      # two
    (150, 2, 2, 3000, "bf16", 1.0, 0.7, 0),     # one
    (1, 3, 2, 221000, "bf16", 1.0, 0.9, 0),     # more tiles than the shared memory of eight CTAs holds
    (3, 64, 2, 2048, "fp32", 0.4, 0.99, 0),     # the most drafts
])
def test_kseq_shared_out_over_the_ctas_of_a_row(B, K, gamma, V, dtype, T, alpha, shift):
    """Rows held by clusters of one to eight CTAs, ragged and unaligned rows, and rows too long for shared memory.  Then
    with equal models: rho = 1, an n-fold root there, so that a rounding error e in the sums would move it by e^(1/n) (the
    float64 oracle itself is 2e-5 off at n = 3, hence no comparison with it); every token is accepted."""
    cfg = workloads.VerifyConfig("kc", B=B, K=K, gamma=gamma, V=V, dtype=dtype, temperature=T, alpha=alpha, seed=77 + V % 83)
    inp = workloads.make_inputs(cfg, device="cuda")

    def moved(t):
        v = torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)[shift:].view(t.shape)
        return v.copy_(t)
    inp = workloads.VerifyInputs(cfg, moved(inp.target_logits), moved(inp.draft_logits), inp.draft_tokens, inp.uniforms)
    out, ref = _kseq_compare(inp, T)
    again = binding.sgbv_verify_kseq(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, T)
    assert torch.equal(out.tokens, again.tokens) and torch.equal(out.rho.nan_to_num(-1), again.rho.nan_to_num(-1))
    equal = inp.target_logits[:, :, :gamma].contiguous()
    same = binding.sgbv_verify_kseq(inp.target_logits, equal, inp.draft_tokens, inp.uniforms, T)
    np.testing.assert_allclose(same.rho.cpu().numpy(), 1.0, atol=1e-6)
    assert (same.accept_len == gamma).all() and ((same.tokens >= 0) & (same.tokens < V)).all() and (same.status == 0).all()


@pytest.mark.parametrize("K,V,eps", [(2, 32256, 1e-4), (3, 32256, 1e-5), (4, 128256, 1e-3), (8, 32256, 1e-3), (8, 50257, 1e-2), (64, 8192, 0.1)])
def test_kseq_rho_of_rows_close_to_one_another(K, V, eps):
    """Draft logits = target logits + eps noise: both sides of the equation of rho are 1 up to eps there, and rho lies near the
    largest q / p.  Reference: the equation in the form that does not cancel, E = (1 - beta)^n with E = sum max(q - rho p, 0) and
    1 - beta = (E + rho - 1) / rho, bisected in float64.  1e-5, as for all rho: the exponentials of logits 20 below the
    maximum carry 20 * 2^-24 of relative error, 1.2e-6 each."""
    g = torch.Generator(device="cuda").manual_seed(K)
    B = 3
    target = (3.0 * torch.randn((B, 1, 2, V), device="cuda", generator=g)).expand(B, K, 2, V).contiguous()
    draft = (target[:, :1, :1] + eps * torch.randn((B, 1, 1, V), device="cuda", generator=g)).expand(B, K, 1, V).contiguous()
    tok = torch.zeros((B, K, 1), dtype=torch.int32, device="cuda")
    u = torch.full((B, K + 1), 0.5, device="cuda")
    rho = binding.sgbv_verify_kseq(target, draft, tok, u, 1.0).rho[:, 0]
    q, p = torch.softmax(target[:, 0, 0].double(), -1), torch.softmax(draft[:, 0, 0].double(), -1)
    lo, hi = torch.ones(B, 1, dtype=torch.float64, device="cuda"), torch.full((B, 1), float(K), dtype=torch.float64, device="cuda")
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        E = (q - mid * p).clamp(min=0.0).sum(-1, keepdim=True)
        up = E > ((E + mid - 1.0) / mid) ** K
        lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
    np.testing.assert_allclose(rho.cpu().numpy(), (0.5 * (lo + hi))[:, 0].cpu().numpy(), rtol=1e-5)


@pytest.mark.parametrize("B,K,V", [(2, 1, 300), (2, 3, 9000), (1, 2, 50257), (160, 1, 9000)])
def test_kseq_residual_of_entries_far_below_the_maximum(B, K, V):
    """Equal rows (four ones each: exact normalisers) but for an entry at 2^-130 that the draft excludes and, at 2^-128, the
    drafted token that the target excludes: the token is rejected, and all that is left of q - rho p is the first of them."""
    zq = torch.full((B, K, 2, V), float("-inf"))
    zq[..., 10:14] = 0.0
    zp = zq[:, :, :1].clone()
    zq[:, :, 0, V - 3] = -130.0 * float(np.log(2.0))
    zp[:, :, 0, 20] = -128.0 * float(np.log(2.0))
    tok = torch.full((B, K, 1), 20, dtype=torch.int32)
    u = torch.full((B, K + 1), 0.5)
    out = binding.sgbv_verify_kseq(zq.cuda(), zp.cuda(), tok.cuda(), u.cuda(), 1.0)
    ref = oracle.kseq_verify(zq.numpy(), zp.numpy(), tok.numpy(), u.numpy(), 1.0)
    assert (ref.tokens[:, 0] == V - 3).all() and (ref.status == 0).all()
    assert (out.tokens[:, 0].cpu().numpy() == ref.tokens[:, 0]).all() and (out.status == 0).all() and (out.accept_len == 0).all()


@pytest.mark.parametrize("B,V,dtype,shift", [
    (600, 777, "fp32", 0),       # one CTA per prompt, a few tiles
    (150, 32000, "bf16", 0),     # one, pieces of 16 bytes
    (100, 32001, "fp32", 0),     # two, rows that start anywhere
    (60, 40000, "bf16", 1),      # four, off a 16-byte boundary
    (20, 151936, "fp32", 0),     # eight
    (50, 221001, "bf16", 0),     # four, more tiles than have a place in shared memory
])
def test_one_draft_on_rows_that_are_not_held(B, V, dtype, shift):
    """Token-level verification of batches: parity, then a NaN in the target row of the first position, +inf in the draft row,
    nothing finite in a row, a token out of range, and equal rows with a token that the target excludes, so that nothing is left
    of q - p and the draw comes from q."""
    cfg = workloads.VerifyConfig("one", B=B, K=1, gamma=3, V=V, dtype=dtype, temperature=0.8, alpha=0.85, seed=V)
    inp = workloads.make_inputs(cfg, device="cuda")

    def moved(t):
        v = torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)[shift:].view(t.shape)
        return v.copy_(t)
    zq, zp, tok, u = moved(inp.target_logits), moved(inp.draft_logits), inp.draft_tokens.clone(), inp.uniforms
    good, _ = _kseq_compare(workloads.VerifyInputs(cfg, zq, zp, tok, u), cfg.temperature)
    zq[1, 0, 0, V - 1] = float("nan")
    zp[2, 0, 0, V // 2] = float("inf")
    zq[3, 0, 0] = float("-inf")
    tok[4, 0, 2] = V
    zp[5, 0, 0] = zq[5, 0, 0] = 0.0
    zq[5, 0, 0, 7] = float("-inf")
    zp[5, 0, 0, 7] = -100.0                        # e^-125: beside V ones it adds nothing to the normaliser
    zp[5, 0, 0, 8] = float("-inf")                 # (as many ones in both rows)
    zq[5, 0, 0, 8] = float("-inf")
    tok[5, 0, 0] = 7
    out = binding.sgbv_verify_kseq(zq, zp, tok, u, cfg.temperature)
    st = out.status.cpu().numpy()
    bad, rng = binding.STATUS_NONFINITE_LOGIT, binding.STATUS_TOKEN_RANGE
    assert st[1] == bad and st[2] == bad and st[3] == bad and st[4] == rng and st[5] == binding.STATUS_DEGENERATE_RESIDUAL
    assert (out.accept_len[1:5] == -1).all() and (out.tokens[1:5] == -1).all() and out.accept_len[5].item() == 0
    assert 0 <= out.tokens[5, 0].item() < V and out.tokens[5, 0].item() not in (7, 8)
    same = [0] + list(range(6, B))
    assert torch.equal(out.tokens[same], good.tokens[same]) and (st[same] == good.status.cpu().numpy()[same]).all()


@pytest.mark.parametrize("V,dtype", [(9000, "fp32"), (50257, "bf16")])
def test_kseq_flags_with_several_ctas_per_row(V, dtype):
    """Every way out of the walk by clusters of four (V = 9000) and eight CTAs: a token out of range, NaN in the first and second
    position, a row without a finite entry, a bonus row with +inf, a residual without mass.  The other rows keep their bits."""
    B, K, gamma = 8, 2, 2
    cfg = workloads.VerifyConfig("kfl", B=B, K=K, gamma=gamma, V=V, dtype=dtype, temperature=0.8, alpha=0.85, seed=V)
    inp = workloads.make_inputs(cfg, device="cuda")
    zq, zp, tok, u = inp.target_logits.clone(), inp.draft_logits.clone(), inp.draft_tokens.clone(), inp.uniforms.clone()
    good, _ = _kseq_compare(inp, cfg.temperature)
    tok[1, 1, 1] = V
    zq[2, :, 0, V - 1] = float("nan")
    zp[3, :, :, :] = zq[3, :, :gamma]                # all accepted up to the NaN of the second position
    zp[3, :, 1, V // 3] = float("nan")
    zq[4, :, 0] = float("-inf")
    zp[5] = zq[5, :, :gamma]                         # all accepted, then a bonus row that cannot be drawn from
    zq[5, :, gamma, 0] = float("inf")
    zp[6, :, 0] = zq[6, :, 0] = 0.0                  # equal rows but for a token that the target excludes
    zq[6, :, 0, 7] = zq[6, :, 0, 8] = zp[6, :, 0, 8] = float("-inf")
    zp[6, :, 0, 7] = -100.0                          # e^-125: beside V ones it adds nothing to the normaliser
    tok[6, :, 0] = 7
    out = binding.sgbv_verify_kseq(zq, zp, tok, u, cfg.temperature)
    st = out.status.cpu().numpy()
    bad, rng = binding.STATUS_NONFINITE_LOGIT, binding.STATUS_TOKEN_RANGE
    assert st.tolist() == [good.status[0].item(), rng, bad, bad, bad, bad, binding.STATUS_DEGENERATE_RESIDUAL, good.status[7].item()]
    assert (out.accept_len[1:6] == -1).all() and (out.tokens[1:6] == -1).all() and out.accept_len[6].item() == 0
    assert 0 <= out.tokens[6, 0].item() < V and out.tokens[6, 0].item() not in (7, 8)
    for b in (0, 7):
        assert torch.equal(out.tokens[b], good.tokens[b])
        assert torch.equal(out.accept_prob[b].nan_to_num(-1), good.accept_prob[b].nan_to_num(-1))


def test_kseq_flags():
    cfg = workloads.VerifyConfig("ksf", B=4, K=2, gamma=2, V=300, alpha=0.8, seed=9)
    inp = workloads.make_inputs(cfg, device="cuda")
    zq, tok = inp.target_logits.clone(), inp.draft_tokens.clone()
    tok[1, 0, 1] = 300
    zq[2, :, 0, 17] = float("nan")
    mod = workloads.VerifyInputs(cfg, zq, inp.draft_logits, tok, inp.uniforms)
    out, ref = _kseq_compare(mod, 1.0)
    st = out.status.cpu().numpy()
    assert st[1] & binding.STATUS_TOKEN_RANGE and st[2] & binding.STATUS_NONFINITE_LOGIT and st[0] == 0
    assert (out.accept_len.cpu().numpy()[1:3] == -1).all()


def test_single_draft_entry_points():
    """Token-level speculative sampling = K-SEQ with one draft; single-draft greedy block verification = the block
    verifier with K = 1 (whose parity with an independent GBV is covered by the verify-step tests)."""
    cfg = workloads.VerifyConfig("sd", B=7, K=1, gamma=5, V=12000, temperature=0.8, alpha=0.85, seed=12)
    inp = workloads.make_inputs(cfg, device="cuda")
    zq, zp, tok = inp.target_logits[:, 0].contiguous(), inp.draft_logits[:, 0].contiguous(), inp.draft_tokens[:, 0].contiguous()
    sd = binding.sgbv_verify_token(zq, zp, tok, inp.uniforms, cfg.temperature)
    ks = binding.sgbv_verify_kseq(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, cfg.temperature)
    gb = binding.sgbv_verify_gbv(zq, zp, tok, inp.uniforms, cfg.temperature)
    ex = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, cfg.temperature)
    torch.cuda.synchronize()
    assert torch.equal(sd.accept_len, ks.accept_len) and torch.equal(sd.tokens, ks.tokens)
    assert torch.equal(gb.accept_len, ex.accept_len) and torch.equal(gb.tokens, ex.tokens)
    assert torch.equal(gb.accept_prob[:, 0], ex.h[:, 0])
    ref = oracle.kseq_verify(inp.target_logits.cpu().numpy(), inp.draft_logits.cpu().numpy(), inp.draft_tokens.cpu().numpy(),
                             inp.uniforms.cpu().numpy(), cfg.temperature)
    ok = (ref.margin_accept >= 1e-6) & (ref.margin_sample >= 1e-6)
    assert (sd.accept_len.cpu().numpy()[ok] == ref.tau[ok]).all()


@pytest.mark.parametrize("N,V,dtype,T", [(9, 4099, "fp32", 0.8), (64, 32000, "fp32", 1.0), (33, 128256, "bf16", 0.7),
                                        (3, 17, "fp32", 1.0), (300, 9000, "bf16", 0.4)])
def test_draft_token_draw_matches_the_oracle(N, V, dtype, T):
    cfg = workloads.VerifyConfig("dr", B=N, K=1, gamma=1, V=V, dtype=dtype, temperature=T, alpha=0.8, seed=40 + V % 89)
    _, zp = _position_rows(cfg)
    g = torch.Generator().manual_seed(N)
    u = torch.rand(N, generator=g, dtype=torch.float32).cuda()
    tok, lp, st = binding.sgbv_draw_tokens(zp, u, T)
    torch.cuda.synchronize()
    rtok, rlp, margin = oracle.draw_tokens(zp.float().cpu().numpy(), u.cpu().numpy(), T)
    near = margin < 1e-6
    assert near.sum() <= max(2, N // 3) and (st.cpu().numpy() == 0).all()
    tok = tok.cpu().numpy()
    assert (tok[~near] == rtok[~near]).all()
    same = tok == rtok
    np.testing.assert_allclose(lp.cpu().numpy()[same], rlp[same], atol=2e-5)
    assert binding.last_main_kernel() == "draw_rows_kernel"
    # the draws feed the verify step as draft tokens: in range, and a flagged row for a NaN logit
    assert ((tok >= 0) & (tok < V)).all()
    zbad = zp.clone()
    zbad[0, 3] = float("nan")
    tok2, _, st2 = binding.sgbv_draw_tokens(zbad, u, T)
    assert tok2[0].item() == -1 and st2[0].item() & binding.STATUS_NONFINITE_LOGIT


@pytest.mark.parametrize("N,V,dtype", [(1, 40000, "fp32"), (37, 8192, "bf16"), (74, 16385, "fp32"), (75, 20011, "bf16"),
                                       (149, 270000, "bf16"), (2, 2048, "fp32")])
def test_draws_shared_out_over_the_ctas_of_a_row(N, V, dtype):
    """Few rows are drawn by clusters of 2 to 8 CTAs, many by one CTA each (with more tiles than shared memory holds for
    the longest): finite entries in one CTA's share only, the smallest and largest uniforms, a row that starts off a
    16-byte boundary, NaN, +inf and no finite entry at all.  Tokens as the oracle's unless a uniform is within 1e-6 of an
    edge of the drawn cell; log-probabilities to 2e-5 (float32 sums)."""
    g = torch.Generator().manual_seed(N * V)
    z = (2.0 * torch.randn(N, V, generator=g)).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    u = torch.rand(N, generator=g)
    u[0] = 0.0
    u[N - 1] = 1.0 - 2.0 ** -24
    last = z[N // 2, -200:].clone()
    z[N // 2] = float("-inf")              # all the mass at the end of the row
    z[N // 2, -200:] = last
    if N > 2:
        first = z[1, :5].clone()
        z[1] = float("-inf")               # ... at its start
        z[1, :5] = first
    buf = torch.empty(N * V + 1, dtype=z.dtype, device="cuda")
    for view in (buf[:-1].view(N, V), buf[1:].view(N, V)):
        view.copy_(z)
        tok, lp, st = (t.cpu().numpy() for t in binding.sgbv_draw_tokens(view, u.cuda(), 0.9))
        rtok, rlp, margin = oracle.draw_tokens(z.float().numpy(), u.numpy(), 0.9)
        assert (st == 0).all()
        near = margin < 1e-6
        assert (tok[~near] == rtok[~near]).all() and ((tok >= 0) & (tok < V)).all()
        same = tok == rtok
        np.testing.assert_allclose(lp[same], rlp[same], atol=2e-5)
    for value, at in ((float("nan"), V - 1), (float("inf"), 0), (float("-inf"), slice(None))):
        bad = z.clone()
        bad[N - 1, at] = value
        tok, lp, st = (t.cpu().numpy() for t in binding.sgbv_draw_tokens(bad.cuda(), u.cuda(), 0.9))
        assert tok[N - 1] == -1 and np.isnan(lp[N - 1]) and st[N - 1] == binding.STATUS_NONFINITE_LOGIT
        assert (st[:N - 1] == 0).all()
