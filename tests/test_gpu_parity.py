"""GPU parity: the CUDA path (through the C ABI) against the float64 oracle on the same seeded
inputs.  Rules are those of ``oracle/compare.py``: decisions bit-exact except rows within 1e-6 of
a threshold (counted), weights and residual masses within 1e-5 relative."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
from oracle.compare import compare
from paper_2604_25925_b200 import binding, workloads
from treemodel import chi_square, gbv_single_draft, np_softmax

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _to_np32(t):
    return t.detach().to("cpu", torch.float32).numpy()


def run_both(inp, rows=None, host_inp=None):
    """GPU on the whole batch; oracle on the batch rows `rows` (all if None). Returns the report."""
    cfg = inp.cfg
    out = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms,
                                 cfg.temperature)
    torch.cuda.synchronize()
    sel = slice(None) if rows is None else torch.as_tensor(rows, device=inp.target_logits.device)
    ref = oracle.verify(_to_np32(inp.target_logits[sel]), _to_np32(inp.draft_logits[sel]),
                        inp.draft_tokens[sel].cpu().numpy(), inp.uniforms[sel].cpu().numpy(), cfg.temperature)
    rep = compare(ref, out.accept_len[sel].cpu().numpy(), out.draft_idx[sel].cpu().numpy(),
                  out.tokens[sel].cpu().numpy(), out.h[sel].cpu().numpy(), out.resmass[sel].cpu().numpy(),
                  out.status[sel].cpu().numpy())
    print(cfg.name, rep.summary())
    for d in rep.detail:
        print("   ", d)
    return rep, out, ref


def assert_parity(rep):
    assert rep.decision_mismatches == 0, rep.detail
    assert rep.status_mismatches == 0, rep.detail
    assert rep.h_violations == 0, rep.detail
    assert rep.S_violations == 0, rep.detail
    # cells of Eq. 4 narrower than 2e-6 are always within 1e-6 of an edge, so on flat rows a fair
    # share of draws is excused by the rule; they are counted, and must still mostly agree
    assert rep.threshold_exceptions <= max(2, rep.rows // 3)
    assert rep.exceptions_matching >= rep.threshold_exceptions // 2


def test_config1_parity_and_20000_trials():
    cfg = workloads.CONFIGS["c1"]
    inp = workloads.make_inputs(cfg).to("cuda")
    rep, _, _ = run_both(inp)
    assert_parity(rep)
    # 20,000 trials on fixed logits/tokens with fresh uniforms: exact parity row by row and the
    # empirical law of (tau, f, y) against the exhaustively enumerated law
    n = 20000
    big = workloads.VerifyInputs(
        workloads.with_batch(cfg, n),
        inp.target_logits.expand(n, -1, -1, -1).contiguous(), inp.draft_logits.expand(n, -1, -1, -1).contiguous(),
        inp.draft_tokens.expand(n, -1, -1).contiguous(),
        workloads.make_uniforms(n, cfg.K, cfg.gamma, seed=cfg.seed + 1, device="cuda"))
    rep, out, ref = run_both(big)
    assert_parity(rep)
    from test_oracle_montecarlo import _chi2_critical, _exact_law_fixed_drafts
    law = _exact_law_fixed_drafts(_to_np32(inp.target_logits)[0], _to_np32(inp.draft_logits)[0],
                                  inp.draft_tokens.cpu().numpy()[0], cfg.temperature, cfg.K)
    tau = out.accept_len.cpu().numpy()
    f = out.draft_idx.cpu().numpy()
    tokens = out.tokens.cpu().numpy()
    counts = {}
    for t, ff, row in zip(tau, f, tokens):
        key = (int(t), int(ff), int(row[t]))
        counts[key] = counts.get(key, 0) + 1
    stat, dof = chi_square(counts, law)
    assert stat < _chi2_critical(dof), (stat, dof)
    assert abs(rep.block_efficiency_got - rep.block_efficiency_ref) < 1e-3


def test_config2_parity_full():
    inp = workloads.make_inputs(workloads.CONFIGS["c2"], device="cuda")
    rep, _, _ = run_both(inp)
    assert_parity(rep)


def test_config3_bf16_parity_full():
    inp = workloads.make_inputs(workloads.CONFIGS["c3"], device="cuda")
    assert inp.target_logits.dtype == torch.bfloat16
    rep, _, _ = run_both(inp)
    assert_parity(rep)


def test_config4_parity_sampled_rows():
    """Full-size launch (the configuration the benchmark times); the oracle recomputes a sample of
    whole batch rows, which are independent units."""
    inp = workloads.make_inputs(workloads.CONFIGS["c4"], device="cuda")
    rep, out, _ = run_both(inp, rows=[0, 7, 21, 38, 50, 63])
    assert_parity(rep)
    # properties that hold at any size, on all rows
    tau = out.accept_len.cpu().numpy()
    f = out.draft_idx.cpu().numpy()
    tokens = out.tokens.cpu().numpy()
    tok = inp.draft_tokens.cpu().numpy()
    cfg = inp.cfg
    assert ((tau >= 0) & (tau <= cfg.gamma)).all()
    assert ((f == -1) == (tau == 0)).all()
    for b in range(cfg.B):
        assert list(tokens[b, :tau[b]]) == list(tok[b, f[b], :tau[b]])
        assert 0 <= tokens[b, tau[b]] < cfg.V and (tokens[b, tau[b] + 1:] == -1).all()
    h = out.h.cpu().numpy()
    assert ((h >= 0) & (h <= 1)).all()


@pytest.mark.parametrize("K", [1, 2, 4, 8])
def test_config5_sweep_parity_sampled_rows(K):
    rows = list(range(0, 256, 16))
    for cfg in [c for c in workloads.sweep_c5() if c.K == K]:
        inp = workloads.make_inputs(cfg, device="cuda")
        rep, out, ref = run_both(inp, rows=rows)
        assert_parity(rep)
        if K == 1:   # K = 1 must reproduce single-draft GBV
            zq, zp = _to_np32(inp.target_logits), _to_np32(inp.draft_logits)
            tok, u = inp.draft_tokens.cpu().numpy(), inp.uniforms.cpu().numpy()
            for b in rows[:4]:
                q_rows = [np_softmax(zq[b, 0, i], cfg.temperature) for i in range(cfg.gamma + 1)]
                p_rows = [np_softmax(zp[b, 0, i], cfg.temperature) for i in range(cfg.gamma)]
                alpha, tau, y = gbv_single_draft(q_rows, p_rows, tok[b, 0], u[b, :cfg.gamma], float(u[b, cfg.gamma]))
                np.testing.assert_allclose(out.h[b, 0].cpu().numpy(), alpha, rtol=1e-5, atol=1e-9)
                if min(abs(u[b, j] - alpha[j]) for j in range(cfg.gamma)) > 1e-6:
                    assert int(out.accept_len[b]) == tau


@pytest.mark.parametrize("name", ["paper_l12", "paper_l8", "paper_l24"])
def test_paper_operating_points(name):
    """K = 3 drafts of 12, 8 or 24 tokens at T = 0.4 over a 32k vocabulary (the paper's Table 2 settings and
    the longest draft of its sweep over L),
    as a batch of 6 prompts so that several chains share the machine."""
    cfg = workloads.with_batch(workloads.CONFIGS[name], 6)
    inp = workloads.make_inputs(cfg, device="cuda")
    rep, _, _ = run_both(inp)
    assert_parity(rep)


@pytest.mark.parametrize("K,dtype", [(5, "fp32"), (6, "bf16"), (7, "fp32"), (16, "fp32")])
def test_draft_counts_without_a_specialised_kernel(K, dtype):
    """K outside {1,2,3,4,8} takes the run-time-K code of the fused kernel (rows are 16-byte aligned)."""
    cfg = workloads.VerifyConfig(f"k{K}", B=3, K=K, gamma=3, V=8192, dtype=dtype, temperature=0.8, alpha=0.85,
                                 seed=500 + K)
    inp = workloads.make_inputs(cfg, device="cuda")
    rep, _, _ = run_both(inp)
    assert_parity(rep)
    assert binding.last_main_kernel() == "fused_chain_kernel"


@pytest.mark.parametrize("B,K,gamma,V,dtype", [(50, 3, 4, 2048, "fp32"), (75, 2, 7, 4096, "bf16"), (149, 1, 5, 1024, "fp32"),
                                              (33, 4, 6, 40000, "fp32")])
def test_chains_cut_between_clusters(B, K, gamma, V, dtype):
    """The chain walk gives every cluster an equal share of the rows, so with a chain count that is no multiple of the
    clusters most chains begin on one cluster and end on another (the ratio c is handed over through global memory).
    Every batch row is compared."""
    cfg = workloads.VerifyConfig(f"cut_{B}_{K}_{gamma}", B=B, K=K, gamma=gamma, V=V, dtype=dtype, temperature=0.9,
                                 alpha=0.85, seed=700 + B)
    inp = workloads.make_inputs(cfg, device="cuda")
    rep, _, _ = run_both(inp)
    assert_parity(rep)
    assert binding.last_main_kernel() == "fused_chain_kernel"
    binding.set_option("walk", 1)            # and with the chain walk forced where the row walk would be chosen
    try:
        small = workloads.VerifyConfig("cut_small", B=7, K=3, gamma=5, V=3000, dtype=dtype, temperature=0.8, seed=701)
        rep, _, _ = run_both(workloads.make_inputs(small, device="cuda"))
        assert_parity(rep)
    finally:
        binding.set_option("walk", 0)


EDGE_SHAPES = [
    # B, K, gamma, V
    (3, 1, 1, 1), (2, 2, 3, 7), (5, 3, 2, 1000), (2, 2, 2, 1025), (2, 4, 3, 32001), (1, 1, 1, 5000),
    (4, 8, 1, 333), (1, 64, 2, 50), (2, 2, 64, 40), (1, 5, 7, 4099),
]


@pytest.mark.parametrize("B,K,gamma,V", EDGE_SHAPES)
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_edge_shapes(B, K, gamma, V, dtype):
    cfg = workloads.VerifyConfig(f"edge_{B}_{K}_{gamma}_{V}_{dtype}", B=B, K=K, gamma=gamma, V=V, dtype=dtype,
                                 temperature=0.9, alpha=0.8, boost=4.0, seed=4242 + V)
    inp = workloads.make_inputs(cfg, device="cuda")
    rep, _, _ = run_both(inp)
    assert_parity(rep)


@pytest.mark.parametrize("T", [0.05, 0.2, 3.0, 25.0])
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_temperature_extremes(T, dtype):
    """Very low temperatures turn rows into near point masses (exponentials underflow to zero away from the
    maximum, residual masses become tiny); very high ones flatten them (every CDF cell is narrow)."""
    cfg = workloads.VerifyConfig(f"temp_{T}_{dtype}", B=4, K=3, gamma=4, V=12288, dtype=dtype, temperature=T,
                                 alpha=0.9, seed=int(1000 * T) + 77)
    inp = workloads.make_inputs(cfg, device="cuda")
    rep, _, _ = run_both(inp)
    assert_parity(rep)


def test_vocabulary_beyond_the_fused_kernel_capacity():
    """Rows longer than 8 CTAs x 32,768 entries (the tensor memory of the largest cluster) take the generic
    two-sweep kernels, aligned or not."""
    cfg = workloads.VerifyConfig("bigv", B=2, K=2, gamma=2, V=8 * 32768 + 4096, alpha=0.85, seed=606)
    inp = workloads.make_inputs(cfg, device="cuda")
    rep, _, _ = run_both(inp)
    assert_parity(rep)
    assert binding.last_main_kernel() == "otreduce_kernel"


@pytest.mark.parametrize("V,dtype", [(8 * 32768, "fp32"), (8 * 32768 - 8, "bf16"), (5 * 32768 + 264, "fp32")])
def test_vocabulary_at_the_fused_kernel_capacity(V, dtype):
    """The longest rows the fused kernel takes (clusters of 8 with every tensor-memory column in use), and a
    row that needs a cluster of 6."""
    cfg = workloads.VerifyConfig("capv", B=2, K=2, gamma=2, V=V, dtype=dtype, alpha=0.85, seed=607)
    inp = workloads.make_inputs(cfg, device="cuda")
    rep, _, _ = run_both(inp)
    assert_parity(rep)
    assert binding.last_main_kernel() == "fused_chain_kernel"


def test_more_than_2_to_the_31_logits_per_tensor():
    """Element offsets beyond 32 bits: 2.8e9 bf16 logits in the target tensor (5.6 GB), 2.5e9 in the draft tensor.
    The oracle recomputes sampled batch rows from both ends of the tensors."""
    cfg = workloads.VerifyConfig("huge", B=256, K=8, gamma=8, V=151936, dtype="bf16", temperature=0.9, alpha=0.9,
                                 seed=808)
    assert cfg.B * cfg.K * (cfg.gamma + 1) * cfg.V > 2 ** 31
    inp = workloads.make_inputs(cfg, device="cuda")
    rep, out, _ = run_both(inp, rows=[0, 131, 255])
    assert_parity(rep)
    tau = out.accept_len.cpu().numpy()
    assert ((tau >= 0) & (tau <= cfg.gamma)).all() and (out.status.cpu().numpy() == 0).all()
    del inp, out
    torch.cuda.empty_cache()


def _slice_fits(V, cluster):
    """A CTA of the fused kernel holds at most 128 cells of 256 entries of a row in tensor memory."""
    cells = -(-V // 256)
    return -(-cells // cluster) <= 128


@pytest.mark.parametrize("option", [("path", 1), ("path", 2), ("cluster", 1), ("cluster", 2), ("cluster", 3),
                                    ("cluster", 4), ("cluster", 5), ("cluster", 7), ("cluster", 8),
                                    ("max_clusters", 3), ("walk", 1), ("walk", 2), ("aux", 1), ("aux", 2)])
def test_every_kernel_path_and_launch_shape_matches(option):
    """The generic two-sweep kernels and the fused kernel at every cluster size / walk /
    persistent-grid size must all agree with the oracle (automatic choice is covered elsewhere)."""
    cfgs = [workloads.VerifyConfig("paths_a", B=5, K=3, gamma=3, V=20480, temperature=0.8, alpha=0.8, seed=21),
            workloads.VerifyConfig("paths_b", B=3, K=2, gamma=2, V=33000, dtype="bf16", temperature=1.1, alpha=0.7,
                                   seed=22),
            workloads.VerifyConfig("paths_c", B=2, K=2, gamma=5, V=1000, alpha=0.9, seed=23),
            workloads.VerifyConfig("paths_d", B=40, K=2, gamma=3, V=9000, temperature=0.9, alpha=0.85, seed=24)]
    binding.set_option(*option)
    try:
        for cfg in cfgs:
            if option[0] == "cluster" and not _slice_fits(cfg.V, option[1]):
                continue   # forced cluster size whose slices do not fit the tensor memory
            if option == ("walk", 2) and cfg.B * cfg.K * cfg.gamma > 256:
                continue   # the row walk has one ratio word per row, 256 in all
            inp = workloads.make_inputs(cfg, device="cuda")
            rep, _, _ = run_both(inp)
            assert_parity(rep)
    finally:
        binding.set_option(option[0], 0)


@pytest.mark.parametrize("K,dtype,alpha,T", [(1, "fp32", 0.8, 1.0), (2, "bf16", 0.9, 0.7), (8, "fp32", 0.9, 1.0),
                                             (3, "fp32", 0.9995, 1.0), (5, "fp32", 0.99, 0.4), (8, "bf16", 0.9999, 1.0)])
def test_extra_sums_in_kernels_of_their_own(K, dtype, alpha, T):
    """Chain walk with the two extra sums of Eq. 2 (rows with c < 1) left to the kernels behind the fused kernel, which
    only do the rows whose plain numerator would cancel: ordinary drafts (few such rows), drafts nearly equal to the
    target (nearly all rows with c < 1 qualify), and a draft count without a specialised kernel; and the same inputs
    with the sums worked out in the fused kernel must give the same weights."""
    cfg = workloads.VerifyConfig(f"aux_{K}_{dtype}_{alpha}", B=24, K=K, gamma=5, V=40192, dtype=dtype, temperature=T,
                                 alpha=alpha, seed=300 + K)
    inp = workloads.make_inputs(cfg, device="cuda")
    res = {}
    for aux in (2, 1):
        binding.set_option("walk", 1)
        binding.set_option("aux", aux)
        try:
            rep, out, _ = run_both(inp)
            assert_parity(rep)
            res[aux] = out.h.cpu().numpy()
            assert binding.last_launch_count() == (4 if aux == 2 else 2)
        finally:
            binding.set_option("walk", 0)
            binding.set_option("aux", 0)
    np.testing.assert_allclose(res[2], res[1], rtol=2e-5, atol=1e-9)


@pytest.mark.parametrize("B,K,gamma,V,dtype,launches", [
    (16, 8, 4, 98304, "bf16", 2), (64, 6, 2, 50304, "bf16", 2), (64, 7, 1, 100352, "bf16", 2), (16, 8, 4, 98304, "fp32", 2),
    (43, 8, 8, 98304, "bf16", 4), (43, 4, 8, 98304, "fp32", 4),     # 1.08e9 bytes: just above 2^30
    (42, 8, 8, 98304, "bf16", 2), (42, 4, 8, 98304, "fp32", 2),     # 1.06e9
    (86, 1, 16, 98304, "fp32", 2),                                  # one draft: in the kernel at any size
])
def test_where_the_extra_sums_are_worked_out(B, K, gamma, V, dtype, launches):
    """Kernels of their own (two more launches) for the extra sums of rows with c < 1: from 1 GB of logits on and not below, at any
    type and number of drafts but one."""
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    target = torch.zeros(B, K, gamma + 1, V, dtype=dt, device="cuda")
    draft = torch.zeros(B, K, gamma, V, dtype=dt, device="cuda")
    binding.sgbv_verify_ex(target, draft, torch.zeros(B, K, gamma, dtype=torch.int32, device="cuda"),
                           torch.full((B, K * gamma + 1), 0.5, device="cuda"), 1.0)
    torch.cuda.synchronize()
    assert binding.last_main_kernel() == "fused_chain_kernel" and binding.last_launch_count() == launches


def _far_rows(B, V, K, dtype, kind):
    cfg = workloads.VerifyConfig(f"far_{V}_{kind}", B=B, K=K, gamma=4, V=V, dtype=dtype, temperature=0.8, alpha=0.9, seed=V + K)
    inp = workloads.make_inputs(cfg, device="cuda")
    x = torch.arange(V, device="cuda")
    for t in (inp.target_logits, inp.draft_logits):
        if kind == "ramp":
            t += (5.0 * (x // 256)).to(t.dtype)
        elif kind == "far":
            t += 1.0e6
        else:
            for b, value in enumerate((float("-inf"), -1e9, torch.finfo(t.dtype).min)):
                t[b::3, :, :, (x < V // 3 * (b + 1) // 2) & (x % 97 != 5)] = value
    if kind == "ramp":
        inp.draft_tokens.copy_(V - 1 - inp.draft_tokens % min(V, 150))
    elif kind == "masked":
        inp.draft_tokens.copy_((inp.draft_tokens % (V // 97)) * 97 + 5)
    return inp


@pytest.mark.parametrize("V,K,dtype,kind", [
    (200, 4, "fp32", "ramp"), (31 * 256, 1, "fp32", "ramp"), (31 * 256 + 1, 3, "bf16", "masked"), (32 * 256 + 8, 8, "bf16", "ramp"),
    (124 * 256, 4, "fp32", "masked"), (124 * 256 + 4, 2, "fp32", "ramp"), (125 * 256, 1, "bf16", "masked"), (128 * 256, 8, "fp32", "far"),
    (33025, 3, "fp32", "masked"), (33032, 5, "bf16", "ramp"), (70000, 8, "fp32", "ramp"), (50257, 4, "bf16", "masked"),
])
def test_logits_far_from_the_first_ones_of_a_row(V, K, dtype, kind):
    """Rows whose first entries say little about the rest: rising from cell to cell, masked up to some place (-inf, -1e9 or the type's
    lowest value) but for an entry here and there, or a million from 0.  Two clusters walk all rows, so that every cell of a warp takes
    every place it can have, at the sizes where the cells per warp change.  Both tensors get the same offsets, and the
    draft tokens are entries that they leave likely."""
    inp = _far_rows(3, V, K, dtype, kind)
    binding.set_option("walk", 1)
    binding.set_option("max_clusters", 2)
    try:
        rep, _, _ = run_both(inp)
        assert binding.last_main_kernel() == "fused_chain_kernel"
    finally:
        binding.set_option("walk", 0)
        binding.set_option("max_clusters", 0)
    assert rep.decision_mismatches == 0 and rep.status_mismatches == 0, rep.detail
    assert rep.h_violations == 0 and rep.S_violations == 0, rep.detail


@pytest.mark.parametrize("walk,aux", [(2, 0), (1, 1), (1, 2)])
@pytest.mark.parametrize("V,K,dtype,kind", [
    (31 * 256, 4, "fp32", "ramp"), (33 * 256, 1, "bf16", "masked"), (64 * 256 + 4, 2, "fp32", "ramp"), (128 * 256, 3, "fp32", "masked"),
    (125 * 256, 8, "bf16", "ramp"), (97 * 256 + 8, 5, "bf16", "masked"), (40001, 4, "fp32", "masked"), (70001, 8, "fp32", "ramp"),
])
def test_references_that_move_in_both_walks_and_with_the_extra_sums(V, K, dtype, kind, walk, aux):
    """The same kinds of rows in the row walk, where the combining warp has its share of the cells, and in the chain walk with the
    extra sums of rows with c < 1 in the kernel and behind it."""
    inp = _far_rows(6, V, K, dtype, kind)
    options = {"walk": walk, "aux": aux, "cluster": 1 if V <= 128 * 256 else 0}
    for name, value in options.items():
        binding.set_option(name, value)
    try:
        rep, _, _ = run_both(inp)
        assert binding.last_main_kernel() == "fused_chain_kernel"
        assert binding.last_launch_count() == (4 if aux == 2 else 2)
    finally:
        for name in options:
            binding.set_option(name, 0)
    assert_parity(rep)


@pytest.mark.parametrize("V,base,T,walk", [(124 * 256, 6e5, 0.01, 1), (124 * 256, 1e8, 1.0, 1), (128 * 256, -1e8, 1.0, 1), (124 * 256, 6e5, 0.01, 2),
                                           (124 * 256 + 1, 6e5, 0.01, 1), (124 * 256, 0.0, 1e38, 1)])
def test_references_move_by_differences_that_a_sum_rounds_away(V, base, T, walk):
    """Rows of two neighbouring float32 numbers, so large that one step between them is more than the references' rise while their
    sum with it rounds to the next number: every warp's first cell holds the lower one, the cells behind it the upper one, which is
    2^9 to 2^12 times as likely.  (At a temperature near the largest float32 the rise itself is infinite.)  Against the two-sweep
    path, at twice the tolerance against the oracle: every draft token is likely under both rows."""
    cfg = workloads.VerifyConfig("steps", B=3, K=2, gamma=3, V=V, temperature=T, alpha=0.9, seed=3)
    inp = workloads.make_inputs(cfg, device="cuda")
    x = torch.arange(V, device="cuda")
    low = torch.tensor(base, device="cuda")
    high = torch.nextafter(low, low + 1e9)
    first = x % 1024 < 256
    inp.target_logits.copy_(torch.where(first, low, high))
    inp.draft_logits.copy_(torch.where(first | (x % 3 == 0), low, high))
    if T > 1e30:  # masked first cells
        inp.target_logits[..., first] = float("-inf")
        inp.draft_logits[..., first] = float("-inf")
    inp.draft_tokens.copy_(256 + 1024 * (inp.draft_tokens % 30) + inp.draft_tokens % 256 * 3)
    inp.draft_tokens.add_((inp.draft_tokens % 3 == 0).int())
    outs = []
    for options in ({"walk": walk, "cluster": 1}, {"path": 1}):
        for name, value in options.items():
            binding.set_option(name, value)
        try:
            outs.append(binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, T))
            torch.cuda.synchronize()
            assert binding.last_main_kernel() == ("otreduce_kernel" if "path" in options else "fused_chain_kernel")
        finally:
            for name in options:
                binding.set_option(name, 0)
    a, b = outs
    assert (a.status == 0).all() and torch.equal(a.status, b.status)
    torch.testing.assert_close(a.h, b.h, rtol=2e-5, atol=2e-9)
    torch.testing.assert_close(a.resmass, b.resmass, rtol=2e-5, atol=0)


@pytest.mark.parametrize("V", [31 * 256, 31 * 256 + 1])
def test_factors_between_units_far_apart(V):
    """One entry D nats above all others, which the draft covers: the residual mass lies in warps whose references are 21 to 65 powers
    of two below the row's.  A float32 exponent of that size is rounded by up to 2^-19 (2.6e-6 of the factor); ex2.approx itself and
    the float32 scalars of a row are good to 2^-22 each (2.4e-7): 6e-7 for the mass, whose terms carry three of them (what q - c p
    cancels comes on top, and makes up to 1.7e-6 of it with other draws).  scale is the float32 that the kernels are given."""
    B, K = 48, 4
    g = torch.Generator().manual_seed(7)
    zq = torch.randn(B, V, generator=g)
    zp = zq + 0.7 * torch.randn(B, V, generator=g)
    zq[:, 5] = zp[:, 5] = torch.linspace(15.0, 45.0, B) + 0.01 * torch.randn(B, generator=g)
    binding.set_option("path", 2)
    binding.set_option("cluster", 1)
    try:
        target = torch.stack([zq, zq], 1).view(B, 1, 2, V).expand(B, K, 2, V).contiguous().cuda()
        draft = zp.view(B, 1, 1, V).expand(B, K, 1, V).contiguous().cuda()
        out = binding.sgbv_verify_ex(target, draft, torch.full((B, K, 1), 5, dtype=torch.int32, device="cuda"),
                                     torch.full((B, K + 1), 0.5, device="cuda"), 1.0)
    finally:
        binding.set_option("path", 0)
        binding.set_option("cluster", 0)
    scale = np.float64(np.float32(1.4426950408889634))
    q, p = (np.exp2((z.numpy().astype(np.float64) - z.numpy().max(1, keepdims=True)) * scale) for z in (zq, zp))
    q, p = q / q.sum(1, keepdims=True), p / p.sum(1, keepdims=True)
    want = (q * np.maximum(1.0 - p / q, 0.0) ** K).sum(1)
    np.testing.assert_allclose(out.resmass[:, 0, 0].cpu().numpy(), want, rtol=6e-7)


def _all_but_excluded(T=0.05):
    """Draft blocks whose first token has a target log-probability from -700 to -760 and a draft probability near 1: a = q(x^i) goes
    through the smallest normal float64 number, the denormal ones (where c = p/q overflows) and 0.  Other rows are flat."""
    cfg = workloads.VerifyConfig("excluded", B=31, K=2, gamma=3, V=3000, temperature=T, alpha=0.9, seed=5)
    inp = workloads.make_inputs(cfg, device="cuda")
    for t in (inp.target_logits, inp.draft_logits):
        t.mul_(0.1).clamp_(-0.5, 0.5)
    first = inp.draft_tokens[:, :, :1].long()
    b = torch.arange(cfg.B, device="cuda", dtype=torch.float32)
    inp.target_logits[:, :, 0].scatter_(2, first, (-34.5 - 0.1 * b).view(-1, 1, 1).expand(-1, cfg.K, 1))
    inp.draft_logits[:, :, 0].scatter_(2, first, 3.0)
    inp.uniforms.fill_(0.5)
    return inp


def test_a_block_that_the_target_all_but_excludes_is_not_accepted():
    inp = _all_but_excluded()
    rep, out, ref = run_both(inp)
    assert_parity(rep)
    assert (ref.tau == 0).all() and out.h[:, :, 0].max() < 1e-290


_IN_A_PROCESS_OF_ITS_OWN = """
import sys, torch
sys.path.insert(0, {root!r})
from paper_2604_25925_b200 import binding, sharded, workloads
inp = workloads.make_inputs(workloads.VerifyConfig("window", B=2, K={K}, gamma={gamma}, V={V}, seed=1), device="cuda")
if {ranks} > 1:
    parts = [(inp.target_logits[..., lo:hi].contiguous(), inp.draft_logits[..., lo:hi].contiguous(), lo)
             for lo, hi in sharded.shard_bounds({V}, {ranks})]
    out = sharded.verify_all_ranks_on_one_device(parts, inp.draft_tokens, inp.uniforms, 1.0, {V})[0]
else:
    out = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, 1.0)
torch.cuda.synchronize()
assert (out.status == 0).all()
"""


@pytest.mark.parametrize("K,gamma,V,ranks", [(17, 58, 256, 1), (41, 23, 256, 1), (16, 63, 600, 2), (35, 28, 600, 2), (40, 24, 600, 2)])
def test_shared_memory_just_below_what_a_kernel_gets_without_asking(K, gamma, V, ranks):
    """Draft counts and lengths for which the finishing kernel's or the sharded decision's dynamic shared memory is below 48 KB and
    the sum with what the kernel declares itself above.  In a process of its own: one larger call asks for all later ones."""
    code = _IN_A_PROCESS_OF_ITS_OWN.format(root=ROOT, K=K, gamma=gamma, V=V, ranks=ranks)
    run = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr[-1500:]


def test_unaligned_views_and_repeated_calls_are_deterministic():
    cfg = workloads.VerifyConfig("unaligned", B=3, K=2, gamma=3, V=4099, alpha=0.8, seed=99)
    inp = workloads.make_inputs(cfg, device="cuda")
    # place the logits one element past a 16-byte boundary
    def shifted(t):
        buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
        v = buf[1:].view(t.shape)
        v.copy_(t)
        return v
    sh = workloads.VerifyInputs(cfg, shifted(inp.target_logits), shifted(inp.draft_logits), inp.draft_tokens,
                                inp.uniforms)
    assert sh.target_logits.data_ptr() % 16 != 0
    rep, out1, _ = run_both(sh)
    assert_parity(rep)
    out2 = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms,
                                  cfg.temperature)
    out3 = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms,
                                  cfg.temperature)
    torch.cuda.synchronize()
    for a, b in ((out2, out3), (out1, out2)):
        assert torch.equal(a.accept_len, b.accept_len) and torch.equal(a.tokens, b.tokens)
        assert torch.equal(a.h, b.h) and torch.equal(a.resmass, b.resmass)


@pytest.mark.parametrize("B,K,gamma,V,dtype,walk", [
    (2, 2, 3, 32003, "bf16", 0),      # row walk
    (40, 3, 4, 8191, "fp32", 0),      # chain walk, chains cut between clusters
    (20, 8, 4, 33025, "bf16", 1),     # clusters of two, a last cell of one entry
    (3, 1, 2, 131071, "fp32", 1),     # one draft, four CTAs
    (2, 5, 2, 1023, "bf16", 1),       # a draft count without a specialised kernel
    (4, 2, 3, 777, "bf16", 0),        # a few cells
])
def test_rows_that_start_anywhere(B, K, gamma, V, dtype, walk):
    """The fused kernel on rows that do not start on 16-byte boundaries, with the two tensors off theirs by different
    amounts and each ending where its allocation ends: parity with the oracle, and the same bits wherever the tensors lie."""
    cfg = workloads.VerifyConfig(f"any_{V}", B=B, K=K, gamma=gamma, V=V, dtype=dtype, temperature=0.8, alpha=0.85, seed=V)
    inp = workloads.make_inputs(cfg, device="cuda")

    def moved(t, shift):
        return torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)[shift:].view(t.shape).copy_(t)
    binding.set_option("walk", walk)
    try:
        outs = []
        for sq, sp in ((0, 0), (1, 3), (3, 2)):
            rep, out, _ = run_both(workloads.VerifyInputs(cfg, moved(inp.target_logits, sq), moved(inp.draft_logits, sp),
                                                          inp.draft_tokens, inp.uniforms))
            assert binding.last_main_kernel() == "fused_chain_kernel"
            assert_parity(rep)
            outs.append(out)
    finally:
        binding.set_option("walk", 0)
    for o in outs[1:]:
        assert torch.equal(o.tokens, outs[0].tokens) and torch.equal(o.status, outs[0].status)
        assert torch.equal(o.h, outs[0].h) and torch.equal(o.resmass, outs[0].resmass)


@pytest.mark.parametrize("V,dtype,d,T", [(20001, "fp32", 9.375, 1.0), (70001, "fp32", 10.75, 0.9), (70001, "bf16", 10.75, 1.0),
                                        (151937, "fp32", 11.5, 0.7)])
def test_normalisers_of_rows_that_start_anywhere_are_combined_in_float64(V, dtype, d, T):
    """One target entry at 0 that only one warp sees, the others' maxima d below it, all of their exponentials 1 in their own
    units: the residual mass is 1 / Z with Z = 1 + n 2^(-d scale), and all that can be inexact in it are the factors between the
    warps' and the CTAs' units.  scale is the float32 that the kernels are given; 1e-13 covers a dozen float64 roundings."""
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    zq = torch.full((V,), -d)
    zp = torch.zeros(V)
    for cell in (0, 32, 64, 96):            # the first CTA's first warp
        zq[cell * 256:(cell + 1) * 256] = float("-inf")
        zp[cell * 256:(cell + 1) * 256] = float("-inf")
    n = int(torch.isfinite(zq).sum())
    zq[5] = 0.0
    target = torch.stack([zq, zq]).to(dt).view(1, 1, 2, V).cuda()
    draft = zp.to(dt).view(1, 1, 1, V).cuda()
    binding.set_option("path", 2)
    try:
        out = binding.sgbv_verify_ex(target, draft, torch.full((1, 1, 1), V - 1, dtype=torch.int32, device="cuda"),
                                     torch.full((1, 2), 0.5, device="cuda"), T)
    finally:
        binding.set_option("path", 0)
    scale = np.float64(np.float32(np.float64(np.float32(1.4426950408889634)) / np.float64(np.float32(T))))
    want = 1.0 / (1.0 + n * np.exp2(-np.float64(d) * scale))
    np.testing.assert_allclose(out.resmass.item(), want, rtol=1e-13)


@pytest.mark.parametrize("B,K,gamma,V,dtype,kernel", [
    (256, 4, 4, 777, "bf16", "otreduce_kernel"),      # 4096 rows of 4 cells
    (512, 1, 4, 6143, "fp32", "otreduce_kernel"),     # 2048 of 24: the longest rows that many of them take two sweeps for
    (512, 1, 4, 6145, "fp32", "fused_chain_kernel"),  # 25
    (56, 4, 4, 3071, "bf16", "otreduce_kernel"),      # 896 of 12
    (55, 4, 4, 3071, "bf16", "fused_chain_kernel"),   # 880
    (56, 4, 4, 3073, "bf16", "fused_chain_kernel"),   # 896 of 13
    (64, 8, 1, 777, "fp32", "otreduce_kernel"),       # one position: 512 rows
    (40, 8, 1, 777, "fp32", "fused_chain_kernel"),    # 320
    (64, 6, 4, 2303, "fp32", "otreduce_kernel"),      # a draft count without a kernel of its own: 9 cells at most
    (64, 6, 4, 2305, "fp32", "fused_chain_kernel"),
    (256, 4, 4, 776, "bf16", "fused_chain_kernel"),   # rows on the boundaries never do
])
def test_many_short_rows_that_start_anywhere_take_two_sweeps(B, K, gamma, V, dtype, kernel):
    """Both sides of the rule, each with parity and against the other path (twice the tolerance).  Residual masses: where the
    draft covers nearly all of the target, S / a = sum of max(q - c p, 0)^K q^(1-K) is a small remainder of terms that each carry
    the float32 rounding of q and c p, 4 of 2^-24 in all, so that S is good to 2.4e-7 a and no better."""
    cfg = workloads.VerifyConfig(f"short_{B}_{V}", B=B, K=K, gamma=gamma, V=V, dtype=dtype, temperature=0.8, alpha=0.85, seed=V)
    inp = workloads.make_inputs(cfg, device="cuda")
    _, out, ref = run_both(inp)
    assert binding.last_main_kernel() == kernel
    assert_parity(compare(ref, *(t.cpu().numpy() for t in (out.accept_len, out.draft_idx, out.tokens, out.h, out.resmass,
                                                           out.status)), S_atol_rel_a=2.4e-7))
    binding.set_option("path", 1 if kernel == "fused_chain_kernel" else 2)
    try:
        other = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, cfg.temperature)
        assert binding.last_main_kernel() != kernel
    finally:
        binding.set_option("path", 0)
    torch.testing.assert_close(out.h, other.h, rtol=2e-5, atol=2e-9)
    torch.testing.assert_close(out.resmass, other.resmass, rtol=2e-5, atol=5e-7)   # a <= 1


@pytest.mark.parametrize("walk", [1, 2])
@pytest.mark.parametrize("cells,K,dtype", [(1, 4, "fp32"), (31, 2, "bf16"), (32, 4, "bf16"), (32, 1, "fp32"), (33, 3, "fp32"), (62, 8, "bf16"), (63, 4, "fp32"),
                                           (64, 4, "bf16"), (65, 2, "fp32"), (95, 4, "bf16"), (96, 4, "fp32"), (97, 3, "bf16"), (126, 8, "fp32"), (127, 5, "bf16"),
                                           (128, 4, "fp32")])
def test_cells_of_a_slice_among_its_warps_on_rows_that_start_anywhere(cells, K, dtype, walk):
    """One CTA per row and slices around the multiples of 32 cells, where the number of cells per warp changes and whether the combining
    warp has any."""
    cfg = workloads.VerifyConfig(f"cells_{cells}", B=3, K=K, gamma=3, V=256 * cells - 3, dtype=dtype, alpha=0.85, seed=cells)
    inp = workloads.make_inputs(cfg, device="cuda")
    options = {"walk": walk, "cluster": 1, "max_clusters": 2 if walk == 1 else 0}
    for name, value in options.items():
        binding.set_option(name, value)
    try:
        rep, _, _ = run_both(inp)
        assert binding.last_main_kernel() == "fused_chain_kernel"
    finally:
        for name in options:
            binding.set_option(name, 0)
    assert_parity(rep)


@pytest.mark.parametrize("shift", [0, 1, 7])
@pytest.mark.parametrize("V,dtype,walk", [(1, "fp32", 1), (2, "bf16", 1), (3, "bf16", 2), (7, "bf16", 1), (9, "fp32", 1), (15, "fp32", 2), (17, "fp32", 1),
                                          (31, "bf16", 1), (33, "bf16", 2), (257, "bf16", 1), (511, "fp32", 1)])
def test_short_rows_near_the_ends_of_the_tensors(V, dtype, walk, shift):
    """Rows of which several lie within the 64 bytes at either end of a tensor that copies must not leave, at several remainders: to the bit
    what the same rows give in the middle of a larger batch, where all of them are copied."""
    cfg = workloads.VerifyConfig("short", B=3, K=2, gamma=3, V=V, dtype=dtype, alpha=0.8, seed=V + shift)
    inp = workloads.make_inputs(cfg, device="cuda")

    def moved(t):
        return torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)[shift:].view(t.shape).copy_(t)

    def padded(t):
        return torch.cat([t[:1]] * 8 + [t] + [t[:1]] * 8)
    outs = []
    for place in (moved, padded):
        logits = [place(t) for t in (inp.target_logits, inp.draft_logits)]
        rest = [padded(t) if place is padded else t for t in (inp.draft_tokens, inp.uniforms)]
        binding.set_option("path", 2)
        binding.set_option("walk", walk)
        try:
            outs.append(binding.sgbv_verify_ex(*logits, *rest, cfg.temperature))
        finally:
            binding.set_option("path", 0)
            binding.set_option("walk", 0)
    a, b = outs
    assert (a.status & binding.STATUS_NONFINITE_LOGIT == 0).all()
    for name in ("accept_len", "draft_idx", "tokens", "h", "resmass", "status"):
        assert torch.equal(getattr(a, name), getattr(b, name)[8:11]), name


@pytest.mark.parametrize("V,dtype,walk,shift", [(8191, "fp32", 1, 0), (8191, "bf16", 2, 1), (40001, "bf16", 1, 3), (40001, "fp32", 2, 1),
                                               (151937, "bf16", 1, 0)])
def test_flagged_and_masked_rows_that_start_anywhere(V, dtype, walk, shift):
    """NaN, +inf and missing rows where rows start anywhere, among them the entries at the two ends of the tensors, which no copy
    brings; masked halves; equal rows; a token out of range.  The ordinary rows keep their bits."""
    B = 9
    cfg = workloads.VerifyConfig("anyflags", B=B, K=2, gamma=2, V=V, dtype=dtype, alpha=0.85, seed=V)
    inp = workloads.make_inputs(cfg, device="cuda")

    def moved(t):
        return torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)[shift:].view(t.shape).copy_(t)
    zq, zp = moved(inp.target_logits), moved(inp.draft_logits)
    tok, u = inp.draft_tokens.clone(), inp.uniforms.clone()
    ninf = float("-inf")
    tok[5] %= V // 2
    tok[6] = V // 2 + tok[6] % (V - V // 2)
    zq[5, :, :, V // 2:] = zp[5, :, :, V // 2:] = ninf       # masked: the second half, and the first
    zq[6, :, :, :V // 2] = zp[6, :, :, :V // 2] = ninf
    zp[7] = zq[7, :, :2]                                     # p == q: no residual mass
    u[7, :4] = 0.999
    binding.set_option("walk", walk)
    binding.set_option("path", 2)
    try:
        rep, good, _ = run_both(workloads.VerifyInputs(cfg, zq, zp, tok, u))
        assert_parity(rep)
        zq[0, 0, 0, 0] = float("nan")                        # the first entry of the target tensor
        zp[B - 1, 1, 1, V - 1] = float("nan")                # the last one of the draft tensor
        zq[1, 1, 0, V // 2] = float("inf")
        zp[2, 0, 1] = ninf                                   # a row without a finite entry
        zq[3, 0, 1, V - 1] = float("nan")
        tok[4, 1, 1] = V
        out = binding.sgbv_verify_ex(zq, zp, tok, u, cfg.temperature)
    finally:
        binding.set_option("walk", 0)
        binding.set_option("path", 0)
    st = out.status.cpu().numpy()
    assert (st[[0, 1, 2, 3, 8]] == binding.STATUS_NONFINITE_LOGIT).all() and st[4] == binding.STATUS_TOKEN_RANGE
    bad = [0, 1, 2, 3, 4, 8]
    assert (out.tokens[bad] == -1).all() and (out.accept_len[bad] == -1).all() and out.h[bad].isnan().all()
    for b in (5, 6, 7):
        assert torch.equal(out.tokens[b], good.tokens[b]) and torch.equal(out.h[b], good.h[b]) and out.status[b] == good.status[b]
    assert st[7] & binding.STATUS_DEGENERATE_RESIDUAL


@pytest.mark.parametrize("K,dtype,alpha", [(2, "bf16", 0.9), (8, "fp32", 0.95), (5, "bf16", 0.99), (3, "fp32", 0.9995)])
def test_extra_sums_in_kernels_of_their_own_on_rows_that_start_anywhere(K, dtype, alpha):
    """As the test on aligned rows, for an odd vocabulary; and the plain entry point, which takes no weights: the rows' totals
    then lie where the weights go."""
    cfg = workloads.VerifyConfig(f"auxany_{K}", B=20, K=K, gamma=4, V=20225, dtype=dtype, temperature=0.8, alpha=alpha, seed=K)
    inp = workloads.make_inputs(cfg, device="cuda")
    res = {}
    for aux in (2, 1):
        binding.set_option("walk", 1)
        binding.set_option("aux", aux)
        try:
            rep, res[aux], _ = run_both(inp)
            assert_parity(rep)
            for _ in range(2):
                plain = binding.sgbv_verify(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, cfg.temperature)
                assert binding.last_launch_count() == (4 if aux == 2 else 2)
                assert torch.equal(plain.tokens, res[aux].tokens) and torch.equal(plain.accept_len, res[aux].accept_len)
                assert torch.equal(plain.draft_idx, res[aux].draft_idx)
        finally:
            binding.set_option("walk", 0)
            binding.set_option("aux", 0)
    np.testing.assert_allclose(res[2].h.cpu().numpy(), res[1].h.cpu().numpy(), rtol=2e-5, atol=1e-9)


@pytest.mark.parametrize("V,dtype,shift", [(8 * 32768 + 1, "fp32", 0), (8 * 32768 + 4099, "bf16", 0), (8 * 32768 + 8, "bf16", 1)])
def test_vocabulary_beyond_the_fused_kernel_capacity_on_rows_that_start_anywhere(V, dtype, shift):
    cfg = workloads.VerifyConfig("biganyv", B=2, K=2, gamma=2, V=V, dtype=dtype, alpha=0.85, seed=608)
    inp = workloads.make_inputs(cfg, device="cuda")

    def moved(t):
        return torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)[shift:].view(t.shape).copy_(t)
    rep, _, _ = run_both(workloads.VerifyInputs(cfg, moved(inp.target_logits), moved(inp.draft_logits), inp.draft_tokens, inp.uniforms))
    assert_parity(rep)
    assert binding.last_main_kernel() == "otreduce_kernel"


def test_degenerate_and_flagged_rows():
    cfg = workloads.VerifyConfig("flags", B=6, K=2, gamma=2, V=300, alpha=0.8, seed=7)
    inp = workloads.make_inputs(cfg, device="cuda")
    zq, zp = inp.target_logits.clone(), inp.draft_logits.clone()
    tok, u = inp.draft_tokens.clone(), inp.uniforms.clone()
    zp[1] = zq[1, :, :2]                 # row 1: p == q everywhere -> zero residual mass
    u[1, :4] = 0.999
    tok[2, 1, 0] = 300                   # row 2: token out of range
    zq[3, 0, 1, 17] = float("nan")       # row 3: NaN logit
    zp[4, 1, 0, 5] = float("inf")        # row 4: +inf logit
    zq[5, :, :, 11] = float("-inf")      # row 5: -inf is allowed (probability 0)
    zp[5, :, :, 12] = float("-inf")
    mod = workloads.VerifyInputs(cfg, zq, zp, tok, u)
    rep, out, ref = run_both(mod)
    assert_parity(rep)
    st = out.status.cpu().numpy()
    assert st[1] & binding.STATUS_DEGENERATE_RESIDUAL
    assert st[2] & binding.STATUS_TOKEN_RANGE and st[3] & binding.STATUS_NONFINITE_LOGIT
    assert st[4] & binding.STATUS_NONFINITE_LOGIT and st[0] == 0 and (st[5] & 3) == 0
    assert (out.tokens[2:5].cpu().numpy() == -1).all() and (out.accept_len[2:5].cpu().numpy() == -1).all()


def test_repeated_calls_on_the_library_scratch_match_calls_on_a_fresh_workspace():
    """The row walk's "not published yet" words are cleared by a memset on a caller's workspace, but on the
    library's own scratch they are put back by the finishing kernel for the next call of the same layout.
    Sequences of calls (same shape repeated, another shape in between) must give what a fresh workspace gives."""
    row_cfg = workloads.with_batch(workloads.CONFIGS["paper_l8"], 2)
    other_cfg = workloads.VerifyConfig("other", B=16, K=4, gamma=4, V=8192, alpha=0.85, seed=31)
    sets = [workloads.make_inputs(row_cfg, device="cuda", set_index=i) for i in range(4)]
    other = workloads.make_inputs(other_cfg, device="cuda")

    def fresh(inp):
        ws = torch.empty(binding.workspace_bytes(inp.cfg.B, inp.cfg.K, inp.cfg.gamma, inp.cfg.V) + 256,
                         dtype=torch.uint8, device="cuda")
        ws.fill_(0x5a)
        off = (-ws.data_ptr()) % 256
        return binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms,
                                      inp.cfg.temperature, workspace=ws[off:off + ws.numel() - 256])

    order = [sets[0], sets[1], sets[1], other, sets[2], sets[3], other, other, sets[0]]
    for inp in order:
        got = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms,
                                     inp.cfg.temperature)
        want = fresh(inp)
        torch.cuda.synchronize()
        assert torch.equal(got.accept_len, want.accept_len) and torch.equal(got.draft_idx, want.draft_idx)
        assert torch.equal(got.tokens, want.tokens) and torch.equal(got.status, want.status)
        assert torch.equal(got.h, want.h) and torch.equal(got.resmass, want.resmass)
    rep, _, _ = run_both(sets[2])
    assert_parity(rep)


@pytest.mark.parametrize("name", ["c2", "paper_l8"])
def test_calls_replayed_from_a_cuda_graph_give_the_eager_results(name):
    """After a warm-up call per shape a call only enqueues kernels (the chain walk of c2, the row walk of the
    one-prompt shape): a captured sequence of calls, replayed, must reproduce the eager outputs."""
    cfg = workloads.CONFIGS[name]
    sets = [workloads.make_inputs(cfg, device="cuda", set_index=i) for i in range(3)]
    eager = [binding.sgbv_verify(i.target_logits, i.draft_logits, i.draft_tokens, i.uniforms, cfg.temperature)
             for i in sets]
    torch.cuda.synchronize()
    outs = [binding.VerifyOutput(torch.full_like(e.accept_len, -7), torch.full_like(e.draft_idx, -7),
                                 torch.full_like(e.tokens, -7)) for e in eager]
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            for i, o in zip(sets, outs):
                binding.sgbv_verify(i.target_logits, i.draft_logits, i.draft_tokens, i.uniforms, cfg.temperature,
                                    out=o)
    for _ in range(2):
        for o in outs:
            o.accept_len.fill_(-7), o.draft_idx.fill_(-7), o.tokens.fill_(-7)
        graph.replay()
        torch.cuda.synchronize()
        for e, o in zip(eager, outs):
            assert torch.equal(e.accept_len, o.accept_len) and torch.equal(e.draft_idx, o.draft_idx)
            assert torch.equal(e.tokens, o.tokens)


def _full_out(cfg):
    dev = "cuda"
    return binding.VerifyOutput(torch.full((cfg.B,), -7, dtype=torch.int32, device=dev),
                                torch.full((cfg.B,), -7, dtype=torch.int32, device=dev),
                                torch.full((cfg.B, cfg.gamma + 1), -7, dtype=torch.int32, device=dev),
                                torch.zeros((cfg.B, cfg.K, cfg.gamma), dtype=torch.float64, device=dev),
                                torch.zeros((cfg.B, cfg.K, cfg.gamma), dtype=torch.float64, device=dev),
                                torch.full((cfg.B,), -7, dtype=torch.int32, device=dev))


def _fresh_workspace_result(inp):
    ws = torch.empty(binding.workspace_bytes(inp.cfg.B, inp.cfg.K, inp.cfg.gamma, inp.cfg.V) + 256,
                     dtype=torch.uint8, device="cuda")
    ws.fill_(0x5a)
    off = (-ws.data_ptr()) % 256
    out = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms,
                                 inp.cfg.temperature, workspace=ws[off:off + ws.numel() - 256])
    torch.cuda.synchronize()
    return out


def _assert_identical(got, want):
    assert torch.equal(got.accept_len, want.accept_len) and torch.equal(got.draft_idx, want.draft_idx)
    assert torch.equal(got.tokens, want.tokens) and torch.equal(got.status, want.status)
    assert torch.equal(got.h, want.h) and torch.equal(got.resmass, want.resmass)


def _capture_call(inp, out):
    """A CUDA graph holding one verify call on the library's own scratch (warmed up first, so nothing allocates)."""
    args = (inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, inp.cfg.temperature)
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            binding.sgbv_verify_ex(*args, out=out)
    return graph


def test_graph_replays_and_eager_calls_of_other_shapes_in_any_order():
    """The row walk relies on words of the scratch that hold a "not published yet" pattern when a call starts.
    That must hold whatever ran before on the library's scratch: captures that never ran, replays of graphs of
    other shapes, eager calls in between.  Every result equals the one computed on a fresh caller workspace."""
    row_a = workloads.make_inputs(workloads.with_batch(workloads.CONFIGS["paper_l8"], 2), device="cuda")
    row_b = workloads.make_inputs(workloads.VerifyConfig("rowb", B=3, K=2, gamma=5, V=12288, temperature=0.7,
                                                         alpha=0.8, seed=41), device="cuda")
    c2 = workloads.make_inputs(workloads.CONFIGS["c2"], device="cuda")
    big = workloads.make_inputs(workloads.VerifyConfig("bigger", B=64, K=4, gamma=4, V=32000, alpha=0.85, seed=42),
                                device="cuda")
    want = {id(x): _fresh_workspace_result(x) for x in (row_a, row_b, c2, big)}

    def eager(inp):
        out = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms,
                                     inp.cfg.temperature)
        torch.cuda.synchronize()
        assert_row_walk = inp is row_a or inp is row_b
        assert binding.last_main_kernel() == "fused_chain_kernel"
        _assert_identical(out, want[id(inp)])
        return assert_row_walk

    for inp in (big, row_a, row_b, c2):   # warm-up: the scratch has its final size from here on
        eager(inp)
    # (i) capture the row walk, run another shape eagerly, replay
    out_a = _full_out(row_a.cfg)
    graph_a = _capture_call(row_a, out_a)
    eager(c2)
    graph_a.replay()
    torch.cuda.synchronize()
    _assert_identical(out_a, want[id(row_a)])
    # (ii) a large shape eagerly, a capture that is not replayed, then the captured shape eagerly
    eager(big)
    out_b = _full_out(row_b.cfg)
    graph_b = _capture_call(row_b, out_b)
    eager(row_b)
    eager(row_a)
    # (iii) graphs of two row-walk shapes replayed alternately, eager calls in between
    for _ in range(3):
        graph_a.replay()
        graph_b.replay()
        torch.cuda.synchronize()
        _assert_identical(out_a, want[id(row_a)])
        _assert_identical(out_b, want[id(row_b)])
        eager(c2)
        graph_b.replay()
        graph_a.replay()
        torch.cuda.synchronize()
        _assert_identical(out_a, want[id(row_a)])
        _assert_identical(out_b, want[id(row_b)])


def test_a_bounded_wait_that_runs_out_flags_every_row_and_the_next_call_is_correct():
    """Failure detection without a fault: in the row walk a row waits (bounded) for the ratios that the rows
    before it publish.  With the first row of every chain withholding its ratio and the limit of that poll
    shortened, the poll expires; the kernel runs to its end, every batch row comes back flagged TIMEOUT with
    -1 outputs, and the next ordinary call on the same scratch is correct."""
    cfg = workloads.with_batch(workloads.CONFIGS["paper_l8"], 2)
    inp = workloads.make_inputs(cfg, device="cuda")
    args = (inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, cfg.temperature)
    binding.set_option("withhold", 1)
    binding.set_option("poll_us", 300)
    try:
        out = binding.sgbv_verify_ex(*args)
        torch.cuda.synchronize()
    finally:
        binding.set_option("withhold", 0)
        binding.set_option("poll_us", 0)
    assert binding.last_main_kernel() == "fused_chain_kernel"
    st = out.status.cpu().numpy()
    assert ((st & binding.STATUS_TIMEOUT) != 0).all()
    assert (out.accept_len.cpu().numpy() == -1).all() and (out.draft_idx.cpu().numpy() == -1).all()
    assert (out.tokens.cpu().numpy() == -1).all()
    rep, again, _ = run_both(inp)
    assert_parity(rep)
    assert (again.status.cpu().numpy() & binding.STATUS_TIMEOUT == 0).all()


def test_plain_bf16_and_host_entry_points_agree_with_extended():
    for name in ("c2",):
        cfg = workloads.CONFIGS[name]
        inp = workloads.make_inputs(cfg, device="cuda")
        ex = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms,
                                    cfg.temperature)
        plain = binding.sgbv_verify(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms,
                                    cfg.temperature)
        ws = torch.empty(binding.workspace_bytes(cfg.B, cfg.K, cfg.gamma, cfg.V) + 256, dtype=torch.uint8,
                         device="cuda")
        off = (-ws.data_ptr()) % 256
        ex2 = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms,
                                     cfg.temperature, workspace=ws[off:off + ws.numel() - 256])
        host = binding.sgbv_verify_host(inp.target_logits.cpu().pin_memory(), inp.draft_logits.cpu().pin_memory(),
                                        inp.draft_tokens.cpu().pin_memory(), inp.uniforms.cpu().pin_memory(),
                                        cfg.temperature)
        torch.cuda.synchronize()
        for o in (plain, ex2):
            assert torch.equal(o.accept_len, ex.accept_len) and torch.equal(o.tokens, ex.tokens)
            assert torch.equal(o.draft_idx, ex.draft_idx)
        assert torch.equal(host.accept_len, ex.accept_len.cpu()) and torch.equal(host.tokens, ex.tokens.cpu())
        assert binding.last_launch_count() > 0
    small = workloads.VerifyConfig("bf", B=2, K=2, gamma=2, V=2048, dtype="bf16", seed=5)
    inp = workloads.make_inputs(small, device="cuda")
    a = binding.sgbv_verify(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, 1.0)
    b = binding.sgbv_verify_ex(inp.target_logits, inp.draft_logits, inp.draft_tokens, inp.uniforms, 1.0)
    torch.cuda.synchronize()
    assert torch.equal(a.tokens, b.tokens)
