"""GPU parity: the CUDA path, called through the C ABI, against the float64 oracle on the same seeded inputs.

Bar: token ids, accept/reject decisions, commit sources, gate bits, commit steps, per-step row counts and the
App. D/E counters bit-exact; logits within max-abs 3e-2 + 2e-2 relative (the stated bf16 bound) -- and, because
the kernels keep activations fp32-faithful, within 2e-3 absolute in practice, which is also asserted.
"""
import numpy as np
import pytest
import torch

import workloads as W
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


# ---- the weight-streaming GEMM against its definition -----------------------------------------------
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("M,N,K", [(1, 128, 256), (4, 768, 256), (7, 1408, 256), (8, 256, 704), (5, 2000, 768),
                                   (3, 2048, 2048), (8, 4000, 768), (16, 768, 768), (29, 512, 2000), (64, 256, 256),
                                   (2, 11264, 2048), (6, 2048, 5632), (4, 256, 688)])
def test_linear_matches_definition(dtype, M, N, K):
    import paper_2609_17184_b200 as ls
    rng = np.random.default_rng(N * 7 + K + M)
    Wn = (rng.standard_normal((N, K)) * 0.05).astype(np.float32)
    if dtype == "bf16":
        Wn = W.bf16_round(Wn)
    x = rng.standard_normal((M, K)).astype(np.float32) * rng.uniform(0.1, 3.0, (M, 1)).astype(np.float32)
    Wt = torch.from_numpy(Wn).cuda().to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    xt = torch.from_numpy(x).cuda()
    y = ls.linear(Wt, xt).cpu().numpy()
    ref = x.astype(np.float64) @ Wn.astype(np.float64).T
    scale = np.abs(x).astype(np.float64) @ np.abs(Wn).astype(np.float64).T
    assert (np.abs(y - ref) <= 2e-6 * scale + 1e-30).all(), np.abs(y - ref).max()
    # batch invariance: a row's bits do not depend on which other rows share the call
    y1 = ls.linear(Wt, xt[:1].contiguous()).cpu().numpy()
    assert np.array_equal(y1[0].view(np.uint32), y[0].view(np.uint32))
    # reproducible bit for bit
    assert np.array_equal(ls.linear(Wt, xt).cpu().numpy().view(np.uint32), y.view(np.uint32))


@pytest.mark.parametrize("M,N,K", [(1, 128, 64), (4, 768, 256), (7, 1408, 256), (8, 256, 704), (5, 2000, 768),
                                   (3, 2048, 2048), (16, 768, 768), (29, 512, 1984), (64, 256, 256), (33, 2000, 768),
                                   (2, 11264, 2048), (6, 2048, 5632), (64, 11264, 2048)])
def test_linear_tc_matches_definition(M, N, K):
    """The tcgen05 / TMA operator against the definition of the product (exact three-plane split of x, fp32
    accumulation in tensor memory): ragged row blocks, several k-splits, every column-tile width."""
    import paper_2609_17184_b200 as ls
    rng = np.random.default_rng(N * 7 + K + M)
    Wn = W.bf16_round((rng.standard_normal((N, K)) * 0.05).astype(np.float32))
    x = rng.standard_normal((M, K)).astype(np.float32) * rng.uniform(0.1, 3.0, (M, 1)).astype(np.float32)
    Wt = torch.from_numpy(Wn).cuda().to(torch.bfloat16)
    xt = torch.from_numpy(x).cuda()
    y = ls.linear_tc(Wt, xt).cpu().numpy()
    ref = x.astype(np.float64) @ Wn.astype(np.float64).T
    scale = np.abs(x).astype(np.float64) @ np.abs(Wn).astype(np.float64).T
    assert (np.abs(y - ref) <= 2e-6 * scale + 1e-30).all(), np.abs(y - ref).max()
    # reproducible bit for bit, and a row does not depend on the rows beside it in the same column tile
    assert np.array_equal(ls.linear_tc(Wt, xt).cpu().numpy().view(np.uint32), y.view(np.uint32))
    if M <= 16:
        y1 = ls.linear_tc(Wt, xt[:1].contiguous()).cpu().numpy()
        assert np.array_equal(y1[0].view(np.uint32), y[0].view(np.uint32))
    # agrees with the mma.sync kernel of the decode pass to rounding
    y2 = ls.linear(Wt, xt).cpu().numpy()
    assert (np.abs(y - y2) <= 4e-6 * scale + 1e-30).all()


@pytest.mark.parametrize("M,N,K", [(1, 16, 8), (3, 16, 40), (8, 9488, 520), (9, 12304, 1032), (16, 304, 72), (17, 304, 72), (40, 2064, 1000)])
def test_linear_reads_row_major_weights_at_the_edges(M, N, K):
    """Weights read in place (one launch up to 16 rows, the cluster GEMM beyond): rows that end inside a 32-wide k-block,
    odd tile counts, one and two tiles per warp; an x that is not 16-byte aligned gives the same bits."""
    import paper_2609_17184_b200 as ls
    rng = np.random.default_rng(N + K + M)
    Wn = W.bf16_round((rng.standard_normal((N, K)) * 0.05).astype(np.float32))
    x = rng.standard_normal((M, K)).astype(np.float32)
    Wt, buf = torch.from_numpy(Wn).cuda().to(torch.bfloat16), torch.zeros(M * K + 1, device="cuda")
    y = ls.linear(Wt, torch.from_numpy(x).cuda()).cpu().numpy()
    ref = x.astype(np.float64) @ Wn.astype(np.float64).T
    scale = np.abs(x).astype(np.float64) @ np.abs(Wn).astype(np.float64).T
    assert (np.abs(y - ref) <= 2e-6 * scale + 1e-30).all()
    xo = buf[1:].view(M, K)
    xo.copy_(torch.from_numpy(x))
    assert np.array_equal(ls.linear(Wt, xo).cpu().numpy().view(np.uint32), y.view(np.uint32))


@pytest.mark.parametrize("M,N,K,dtype,shift", [(16, 304, 72, "bf16", 1), (17, 304, 72, "bf16", 0), (64, 4096, 1000, "bf16", 0), (9, 272, 264, "fp32", 0)])
def test_linear_stays_within_its_scratch(M, N, K, dtype, shift):
    """The calls that split x in a launch of their own, with exactly the scratch that is asked for and a guard behind it."""
    import paper_2609_17184_b200 as ls
    rng = np.random.default_rng(M)
    Wn = W.bf16_round((rng.standard_normal((N, K)) * 0.05).astype(np.float32))
    x = rng.standard_normal((M, K)).astype(np.float32)
    xt = torch.zeros(M * K + shift, device="cuda")[shift:].view(M, K)
    xt.copy_(torch.from_numpy(x))
    need = ls.linear_scratch_bytes(M, N, K)
    buf = torch.full((need + 65536,), 77, dtype=torch.uint8, device="cuda")
    y = ls.linear(torch.from_numpy(Wn).cuda().to(torch.bfloat16 if dtype == "bf16" else torch.float32), xt, buf[:need]).cpu().numpy()
    scale = np.abs(x).astype(np.float64) @ np.abs(Wn).astype(np.float64).T
    assert (np.abs(y - x.astype(np.float64) @ Wn.astype(np.float64).T) <= 2e-6 * scale + 1e-30).all()
    assert (buf[need:] == 77).all()


def test_linear_tc_rejects_unsupported_shapes():
    import paper_2609_17184_b200 as ls
    assert ls.lib.loopspec_linear_tc_scratch_bytes(4, 256, 256) > 0
    for M, N, K in [(0, 256, 256), (65, 256, 256), (4, 252, 256), (4, 256, 200), (4, 256, 32)]:
        assert ls.lib.loopspec_linear_tc_scratch_bytes(M, N, K) == 0
    Wt = torch.zeros(256, 200, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(ls.LoopSpecError):
        ls.linear_tc(Wt, torch.zeros(4, 200, device="cuda"))


# ---- end-to-end parity -------------------------------------------------------------------------------
GREEDY_CASES = [
    ("tiny", 16, 64, 1, 0, True),            # the small greedy workload (16-token prompt, 64 tokens, d1 = 1, no second proposal)
    ("tiny", 16, 40, 1, 2, True),
    ("tiny", 9, 30, 2, 0, True),
    ("tiny_bf16", 16, 64, 1, 2, True),
    ("tiny_bf16", 16, 48, 1, 3, True),
    ("tiny_bf16", 16, 48, 1, 2, False),      # gate forced open: 7 rows
    ("tiny_bf16", 5, 40, 2, 0, True),
    ("small_bf16", 70, 48, 1, 2, True),      # context spans two attention chunks, ragged GEMM tails
    ("small_bf16", 130, 24, 1, 0, True),
]


@pytest.mark.parametrize("name,n_prompt,n_decode,d1,d2,gate", GREEDY_CASES)
def test_greedy_decode_matches_oracle(name, n_prompt, n_decode, d1, d2, gate):
    ref = U.oracle_run(name, n_prompt, n_decode, d1, d2, gate=gate)
    ctx = U.make_ctx(name, d1, d2, gate=gate, max_ctx=n_prompt + n_decode + 8)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    np.testing.assert_allclose(ctx.debug_logits(0, 0), ref["dec"].first_logits, atol=2e-3, rtol=0)
    out = ctx.decode(n_decode)
    assert out[0].tolist() == ref["tokens"], (U.first_diff(out[0].tolist(), ref["tokens"]), U.min_margin(ref["dec"]))
    err = U.assert_same_run(ctx, ref, n_decode)
    assert err < 2e-3
    st, so = ctx.stats(), ref["dec"].stats
    for k in ("steps", "n_decode", "n_accept1", "n_accept2", "n_restart", "gate_evals", "gate_opens", "rows_total",
              "rows_max", "readout_rows_total"):
        assert st[k] == so[k], (k, st[k], so[k])
    assert abs(st["gamma"] - so["gamma"]) < 1e-12
    assert ctx.row_trace().tolist() == ref["dec"].rows_per_step
    ctx.close()


@pytest.mark.parametrize("name,n_prompt,n_decode,d1,d2", [("tiny", 16, 64, 1, 0), ("tiny_bf16", 16, 64, 1, 2),
                                                           ("small_bf16", 70, 40, 1, 2)])
def test_greedy_loopspec_equals_vanilla_on_gpu(name, n_prompt, n_decode, d1, d2):
    """Losslessness on the device: same tokens from the pipelined path and from all-R decoding (same kernels)."""
    prompt = W.make_prompt(W.CONFIGS[name].vocab, n_prompt)
    a = U.make_ctx(name, d1, d2, max_ctx=n_prompt + 2 * n_decode + 8)
    fa = a.prefill(prompt)
    van = a.vanilla_decode(n_decode)[0].tolist()
    ref = U.oracle_run(name, n_prompt, n_decode, d1, d2, vanilla=True)
    assert fa == ref["first"] and van == ref["tokens"]
    np.testing.assert_allclose(a.debug_logits(0, 0), ref["dec"].verify_logits[-1], atol=2e-3, rtol=0)
    # continue with the pipelined path from the vanilla state, and compare with a fresh pipelined run
    cont = a.decode(n_decode)[0].tolist()
    b = U.make_ctx(name, d1, d2, max_ctx=n_prompt + 2 * n_decode + 8)
    b.prefill(prompt)
    both = b.decode(2 * n_decode)[0].tolist()
    assert both[:n_decode] == van and both[n_decode:] == cont
    a.close(), b.close()


SAMPLED_CASES = [
    ("tiny_bf16", 16, 64, 1, 2, 1.0, True, True),
    ("tiny_bf16", 16, 64, 1, 2, 0.7, True, True),
    ("tiny_bf16", 16, 48, 1, 3, 1.0, True, True),
    ("tiny_bf16", 16, 48, 1, 2, 1.0, False, True),     # ungated
    ("tiny_bf16", 16, 48, 1, 2, 1.0, True, False),     # non-residual second proposal
    ("tiny", 16, 48, 1, 2, 1.0, True, True),
    ("tiny", 16, 48, 2, 0, 1.3, True, True),
    ("small_bf16", 70, 40, 1, 2, 1.0, True, True),
]


@pytest.mark.parametrize("name,n_prompt,n_decode,d1,d2,T,gate,residual", SAMPLED_CASES)
def test_sampled_decode_matches_oracle(name, n_prompt, n_decode, d1, d2, T, gate, residual):
    """Rejection-sampling verification: same draws, same accept/reject decisions, same resampled tokens."""
    ref = U.oracle_run(name, n_prompt, n_decode, d1, d2, T=T, seed=2, gate=gate, residual_q2=residual)
    ctx = U.make_ctx(name, d1, d2, T=T, seed=2, gate=gate, residual_q2=residual, max_ctx=n_prompt + n_decode + 8)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(n_decode)
    U.assert_same_run(ctx, ref, n_decode)
    st, so = ctx.stats(), ref["dec"].stats
    for k in ("steps", "n_accept1", "n_accept2", "n_restart", "gate_evals", "gate_opens", "rows_total"):
        assert st[k] == so[k], (k, st[k], so[k])
    srcs = {c["source"] for c in ref["dec"].commits}
    assert len(srcs) >= 2          # the case exercises acceptance and rejection
    ctx.close()


DEEP_LOOP_CASES = [
    # name, d1, d2, T          (R = 8 / 16; up to ~50 rows in one pass, close to the branch bound of 54)
    ("tiny_r8", 1, 2, 0.0), ("tiny_r8", 1, 2, 1.0), ("tiny_r8", 1, 4, 0.0), ("tiny_r8", 2, 6, 1.0), ("tiny_r8", 4, 0, 1.0),
    ("tiny_r16", 2, 4, 0.0), ("tiny_r16", 2, 8, 1.0), ("tiny_r16", 4, 12, 1.0),
]


@pytest.mark.parametrize("name,d1,d2,T", DEEP_LOOP_CASES)
def test_deeper_loops_match_oracle(name, d1, d2, T):
    """More pipeline levels and wider passes than R = 4 gives (Sec. 4.3: the branch bound grows quickly with R / d1)."""
    n_prompt, n_decode = 16, 40
    ref = U.oracle_run(name, n_prompt, n_decode, d1, d2, T=T, seed=2)
    ctx = U.make_ctx(name, d1, d2, T=T, seed=2, max_ctx=n_prompt + n_decode + 24)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(n_decode)
    U.assert_same_run(ctx, ref, n_decode)
    st, so = ctx.stats(), ref["dec"].stats
    for k in ("steps", "n_accept1", "n_accept2", "n_restart", "gate_evals", "gate_opens", "rows_total"):
        assert st[k] == so[k], (k, st[k], so[k])
    if (d1, d2) == (1, 2) or (name, d1, d2) == ("tiny_r16", 2, 4):
        assert so["rows_max"] > 32           # the widest kernels (more than 32 rows) really run
    ctx.close()


MASKED_CASES = [
    # name, n_prompt, n_decode, d1, d2, T, gate, residual, top_k, top_p
    ("tiny", 16, 64, 1, 2, 0.0, False, True, 0, 1.0),         # greedy, ungated: the runner-up whenever the drafts agree
    ("tiny_bf16", 16, 64, 1, 2, 0.0, False, True, 0, 1.0),
    ("tiny_bf16", 16, 48, 1, 2, 0.0, True, True, 0, 1.0),     # greedy, gated: the mask never bites
    ("tiny_bf16", 16, 64, 1, 2, 1.0, False, True, 0, 1.0),
    ("tiny_bf16", 16, 64, 1, 2, 1.0, False, False, 0, 1.0),   # masked p_{d2} itself
    ("tiny_bf16", 16, 48, 1, 3, 0.8, True, True, 0, 1.0),
    ("tiny_bf16", 16, 48, 1, 2, 1.0, False, True, 0, 0.7),    # with a nucleus
    ("tiny", 16, 48, 1, 2, 1.0, False, False, 0, 0.6),
    ("small_bf16", 40, 32, 1, 2, 1.0, False, True, 0, 1.0),
    ("tiny_bf16", 16, 48, 1, 2, 1.0, False, True, 2, 1.0),  # two-token nuclei: the residual can sit on the first candidate alone
    ("tiny_bf16", 16, 48, 1, 2, 1.0, False, True, 1, 1.0),  # one-token nuclei: no second proposal where the drafts agree
    ("tiny", 16, 48, 1, 2, 1.0, False, True, 2, 1.0),
]


@pytest.mark.parametrize("name,n_prompt,n_decode,d1,d2,T,gate,residual,top_k,top_p", MASKED_CASES)
def test_masked_second_proposal_matches_oracle(name, n_prompt, n_decode, d1, d2, T, gate, residual, top_k, top_p):
    """The variant of the second-proposal ablation (Sec. 6): the first candidate is masked out of the second
    proposal; draws, decisions and tokens as the oracle's."""
    kw = dict(T=T, seed=4, gate=gate, residual_q2=residual, top_k=top_k, top_p=top_p, mask_first=True)
    ref = U.oracle_run(name, n_prompt, n_decode, d1, d2, **kw)
    ctx = U.make_ctx(name, d1, d2, max_ctx=n_prompt + n_decode + 8, **kw)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(n_decode)
    U.assert_same_run(ctx, ref, n_decode)
    st, so = ctx.stats(), ref["dec"].stats
    for k in ("steps", "n_accept1", "n_accept2", "n_restart", "gate_evals", "gate_opens", "rows_total"):
        assert st[k] == so[k], (k, st[k], so[k])
    if name == "tiny" and T == 0.0:   # the two drafts agree here, so the mask really picks runners-up
        assert sum(e["kind"] == "draft2" for e in ref["dec"].log) > 10
    if T == 0.0:
        assert ref["tokens"] == U.oracle_run(name, n_prompt, n_decode, 0, 0, vanilla=True)["tokens"]
    ctx.close()


FILTERED_CASES = [
    # name, n_prompt, n_decode, d1, d2, T, top_k, top_p
    ("tiny_bf16", 16, 48, 1, 2, 1.0, 0, 0.7),       # the paper's sampling setting: T = 1, top-p 0.7
    ("tiny_bf16", 9, 40, 1, 3, 0.8, 20, 1.0),       # top-k alone
    ("tiny", 16, 40, 2, 0, 1.2, 50, 0.9),           # both, fp32 weights, single proposal
    ("small_bf16", 40, 32, 1, 2, 1.0, 0, 0.7),
]


@pytest.mark.parametrize("name,n_prompt,n_decode,d1,d2,T,top_k,top_p", FILTERED_CASES)
def test_filtered_sampling_matches_oracle(name, n_prompt, n_decode, d1, d2, T, top_k, top_p):
    """top-k / top-p inside C (Sec. 3.1) at every readout depth: same nuclei, same draws, same decisions."""
    ref = U.oracle_run(name, n_prompt, n_decode, d1, d2, T=T, seed=2, top_k=top_k, top_p=top_p)
    ctx = U.make_ctx(name, d1, d2, T=T, seed=2, max_ctx=n_prompt + n_decode + 8, top_k=top_k, top_p=top_p)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(n_decode)
    got = [c["token"] for c in ctx.commits(0)]
    assert got == ref["tokens"], (U.first_diff(got, ref["tokens"]), U.min_margin(ref["dec"]))
    for g, o in zip(ctx.commits(0), ref["dec"].commits):
        assert tuple(g[k] for k in U.COMMIT_KEYS) == tuple(o[k] for k in U.COMMIT_KEYS)
    st, so = ctx.stats(), ref["dec"].stats
    for k in ("steps", "n_accept1", "n_accept2", "n_restart", "gate_evals", "gate_opens", "rows_total"):
        assert st[k] == so[k], (k, st[k], so[k])
    # the filters change the stream (else the case tests nothing)
    plain = U.oracle_run(name, n_prompt, n_decode, d1, d2, T=T, seed=2)
    assert plain["tokens"] != ref["tokens"]
    # vanilla decoding draws from the same filtered target
    refv = U.oracle_run(name, n_prompt, 16, d1, d2, T=T, seed=2, top_k=top_k, top_p=top_p, vanilla=True)
    assert ctx.prefill(refv["prompt"]) == refv["first"]
    assert ctx.vanilla_decode(16)[0].tolist() == refv["tokens"]
    ctx.close()


# runs of the seed sweep whose closest decision in the oracle is below the 1e-5 threshold (found by running the oracle
# alone): greedy tiny_bf16 with (d1, d2) = (1, 2), seed 4, a gate score 1.9e-6 from its threshold at position 37
NEAR_TIES = {("tiny_bf16", 1, 2, 0.0, 0, 1.0): {4}}


@pytest.mark.parametrize("name,n_prompt,n_decode,d1,d2,T,top_k,top_p", [
    ("tiny_bf16", 11, 40, 1, 2, 0.0, 0, 1.0), ("tiny_bf16", 16, 40, 1, 2, 1.0, 0, 1.0), ("tiny_bf16", 9, 40, 2, 0, 0.9, 0, 0.7),
    ("tiny", 16, 40, 1, 3, 1.1, 30, 0.9), ("small_bf16", 33, 24, 1, 2, 1.0, 0, 1.0)])
def test_parity_holds_across_seeds(name, n_prompt, n_decode, d1, d2, T, top_k, top_p):
    """Not one lucky seed: eight prompt / sampling seeds per setting, tokens and counters equal to the oracle's.

    A run whose closest decision in the oracle has a margin below 1e-5 cannot be compared decision by decision: fp32
    logits (error ~3e-5 here) do not resolve it, and either outcome is a correct execution of the step.  Such runs
    are listed by name in NEAR_TIES (the list is checked, so none is passed over silently) and still run on the
    device: the tokens before the tied position must agree, and under greedy decoding the whole stream must, because
    the output of a lossless scheme does not depend on what a gate or a proposal decided."""
    seen = set()
    for seed in range(1, 9):
        ref = U.oracle_run(name, n_prompt, n_decode, d1, d2, T=T, seed=seed, prompt_seed=seed + 10, top_k=top_k, top_p=top_p)
        decisions = sorted((e["margin"], e["kind"], e.get("pos", -1)) for e in ref["dec"].log if e["kind"] != "filter")
        ctx = U.make_ctx(name, d1, d2, T=T, seed=seed, max_ctx=n_prompt + n_decode + 8, top_k=top_k, top_p=top_p)
        assert ctx.prefill(ref["prompt"]) == ref["first"], seed
        out = ctx.decode(n_decode)[0].tolist()
        if decisions[0][0] < 1e-5:
            seen.add(seed)
            tie_pos = min(pos for m, _, pos in decisions if m < 1e-5)
            keep = n_decode if T == 0.0 else max(0, tie_pos - n_prompt - 2)
            assert out[:keep] == ref["tokens"][:keep], (seed, U.first_diff(out, ref["tokens"]), decisions[:3])
            ctx.close()
            continue
        assert out == ref["tokens"], (seed, U.first_diff(out, ref["tokens"]), decisions[:3])
        st, so = ctx.stats(), ref["dec"].stats
        for k in ("steps", "n_accept1", "n_accept2", "n_restart", "gate_evals", "gate_opens", "rows_total"):
            assert st[k] == so[k], (seed, k, st[k], so[k])
        ctx.close()
    assert seen == NEAR_TIES.get((name, d1, d2, T, top_k, top_p), set()), seen


@pytest.mark.parametrize("name,gate,top_p", [("tiny_bf16", True, 1.0), ("tiny_bf16", False, 1.0), ("small_bf16", False, 0.8)])
def test_measured_tv_profile_matches_oracle_and_feeds_the_depth_picker(name, gate, top_p):
    """measure_tv records TV(p_d1, p_R) and TV(p_d2, p_R) at every verification (Sec. 4.1); the means equal the
    oracle's, and the fitted envelope gives an admissible depth pair."""
    import paper_2609_17184_b200 as ls
    R = W.CONFIGS[name].R
    prof = {}
    for d2 in (2, 3):
        ref = U.oracle_run(name, 24, 40, 1, d2, T=1.0, seed=3, gate=gate, top_p=top_p)
        ctx = U.make_ctx(name, 1, d2, T=1.0, seed=3, gate=gate, max_ctx=80, top_p=top_p, measure_tv=True)
        assert ctx.prefill(ref["prompt"]) == ref["first"]
        assert ctx.decode(40)[0].tolist() == ref["tokens"]      # measuring does not change the stream
        st = ctx.stats()
        tvs = ref["dec"].tv_log
        t1 = [a for a, _ in tvs]
        t2 = [b for _, b in tvs if b is not None]
        assert st["tv_n1"] == len(t1) == 40 and st["tv_n2"] == len(t2)
        # fp32 against fp64 probabilities; with a nucleus, which of the near-equal tokens sit at its edge may differ
        tol = 2e-5 if top_p >= 1.0 else 2e-4
        assert abs(st["tv_d1"] - np.mean(t1)) < tol
        if t2:
            assert abs(st["tv_d2"] - np.mean(t2)) < tol
            prof[d2] = st["tv_d2"]
        prof[1] = st["tv_d1"]
        ctx.close()
    assert sorted(prof) == [1, 2, 3]
    alpha, beta = ls.fit_envelope([prof[r] for r in range(1, R)])
    d1s, d2s, d1, d2 = ls.pick_depths(alpha, beta, R)
    assert alpha > 0 and beta > 0 and 1 <= d1 < d2 < R and d2 % d1 == 0 and R % d1 == 0
    # not measuring leaves the fields at zero
    ctx = U.make_ctx(name, 1, 2, T=1.0, seed=3, max_ctx=80)
    ctx.prefill(ref["prompt"]); ctx.decode(8)
    assert ctx.stats()["tv_n1"] == 0 and ctx.stats()["tv_d1"] == 0.0
    ctx.close()


def test_filters_off_values_and_unsupported_vocab():
    """top_k = 0 with top_p = 0 or 1 is the plain softmax: bit-identical to a context built without the fields."""
    ref = U.oracle_run("tiny_bf16", 16, 24, 1, 2, T=1.0, seed=2)
    for top_p in (0.0, 1.0):
        ctx = U.make_ctx("tiny_bf16", 1, 2, T=1.0, seed=2, max_ctx=64, top_k=0, top_p=top_p)
        assert ctx.prefill(ref["prompt"]) == ref["first"]
        assert ctx.decode(24)[0].tolist() == ref["tokens"]
        ctx.close()
    with pytest.raises(Exception) as e:
        U.make_ctx("tiny_bf16", 1, 2, T=1.0, top_k=-1)
    assert "EINVAL" in str(e.value)


def test_sampled_vanilla_matches_oracle():
    ref = U.oracle_run("tiny_bf16", 16, 40, 1, 0, T=1.0, seed=5, vanilla=True)
    ctx = U.make_ctx("tiny_bf16", 1, 0, T=1.0, seed=5, max_ctx=80)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    assert ctx.vanilla_decode(40)[0].tolist() == ref["tokens"]
    ctx.close()


def test_step_verify_calls_equal_decode():
    """loopspec_decode produces exactly the tokens of alternating loopspec_step / loopspec_verify."""
    name, n_prompt, n = "tiny_bf16", 16, 32
    ref = U.oracle_run(name, n_prompt, n, 1, 2, T=1.0, seed=2)
    ctx = U.make_ctx(name, 1, 2, T=1.0, seed=2, max_ctx=80)
    ctx.prefill(ref["prompt"])
    toks, rows, commits = [], [], []
    while len(toks) < n:
        n_rows, need = ctx.step()
        rows.append(n_rows)
        if need:
            for c in ctx.verify():
                toks.append(c["token"])
                commits.append(c)
    assert toks == ref["tokens"]
    assert rows == ref["dec"].rows_per_step[: len(rows)]
    for g, o in zip(commits, ref["dec"].commits):
        assert tuple(g[k] for k in U.COMMIT_KEYS) == tuple(o[k] for k in U.COMMIT_KEYS)
    with pytest.raises(Exception) as e:
        ctx.verify()
    assert "ESTATE" in str(e.value)
    ctx.close()


def test_batch_of_sequences_equals_each_alone():
    """Independent sequences share the passes; each must decode exactly as it does alone (and as the oracle)."""
    name, n_prompt, n = "tiny_bf16", 12, 32
    S = 3
    refs = [U.oracle_run(name, n_prompt + 3 * s, n, 1, 2, T=0.9, seed=7, seq=s) for s in range(S)]
    ctx = U.make_ctx(name, 1, 2, T=0.9, seed=7, max_seqs=S, max_ctx=96)
    for s in range(S):
        assert ctx.prefill(refs[s]["prompt"], seq=s) == refs[s]["first"]
    out = ctx.decode(n)
    for s in range(S):
        assert out[s].tolist() == refs[s]["tokens"], s
        got = ctx.commits(s)
        assert [c["source"] for c in got] == [c["source"] for c in refs[s]["dec"].commits]
    ctx.close()


@pytest.mark.parametrize("name,T", [("tiny_bf16", 0.9), ("tiny_gqa", 0.0)])
def test_batch_of_mid_length_contexts_streams_runs_of_chunks(name, T):
    """Several sequences with contexts of 9 to 17 attention chunks: in a context that holds more than one sequence the
    attention work items are runs of chunks from 8 chunks on (the streaming kernel); each sequence must still decode exactly
    as the oracle decodes it alone, whatever the other rows of the pass are."""
    S, n = 3, 20
    lens = [600, 830, 1050]
    refs = [U.oracle_run(name, lens[s], n, 1, 2, T=T, seed=9, seq=s) for s in range(S)]
    ctx = U.make_ctx(name, 1, 2, T=T, seed=9, max_seqs=S, max_ctx=1100, max_prefill_rows=64)
    assert ctx.decode_paths()[1] == 1
    for s in range(S):
        assert ctx.prefill(refs[s]["prompt"], seq=s) == refs[s]["first"]
    out = ctx.decode(n)
    for s in range(S):
        assert out[s].tolist() == refs[s]["tokens"], (s, U.min_margin(refs[s]["dec"]))
        got = ctx.commits(s)
        assert [(c["source"], c["gate_open"]) for c in got] == [(c["source"], c["gate_open"]) for c in refs[s]["dec"].commits]
    ctx.close()


@pytest.mark.parametrize("name,S,lens", [("tiny_bf16", 2, [15, 113]), ("tiny_bf16", 3, [62, 127, 176]), ("small_bf16", 2, [31, 111]),
                                          ("tiny_gqa", 4, [1, 16, 240, 255])])
def test_attention_of_several_sequences_at_the_edges_of_tiles_and_runs(name, S, lens):
    """One warp per run of chunks: contexts of a single key, that grow over the edge of a 16-key tile, of a chunk and of a run
    (2 to 4 chunks, as many as the context has sequences) while speculative keys follow the committed ones; head sizes 64 and 128,
    one and four query heads per kv head."""
    n = 20
    refs = [U.oracle_run(name, lens[s], n, 1, 2, seed=4, seq=s) for s in range(S)]
    ctx = U.make_ctx(name, 1, 2, seed=4, max_seqs=S, max_ctx=300)
    for s in range(S):
        assert ctx.prefill(refs[s]["prompt"], seq=s) == refs[s]["first"]
    out = ctx.decode(n)
    for s in range(S):
        assert out[s].tolist() == refs[s]["tokens"], (s, U.min_margin(refs[s]["dec"]))
    ctx.close()


@pytest.mark.parametrize("S,lens", [(3, [185, 1, 505]), (4, [311, 180, 500, 319]), (5, [250, 100, 375, 20, 383])])
def test_attention_runs_change_length_while_a_batch_decodes(S, lens):
    """Contexts that grow over the edges of the rule that cuts attention runs while they decode: of a batch of three or four, past 3, 5 and
    8 chunks; of a larger one, past 4 and 6 (five sequences are passes of up to 35 rows)."""
    n = 20
    refs = [U.oracle_run("tiny_bf16", lens[s], n, 1, 2, seed=4, seq=s) for s in range(S)]
    ctx = U.make_ctx("tiny_bf16", 1, 2, seed=4, max_seqs=S, max_ctx=560)
    for s in range(S):
        assert ctx.prefill(refs[s]["prompt"], seq=s) == refs[s]["first"]
    out = ctx.decode(n)
    for s in range(S):
        assert out[s].tolist() == refs[s]["tokens"], (s, U.min_margin(refs[s]["dec"]))
    ctx.close()


def test_prefill_chunking_does_not_change_results():
    name = "tiny_bf16"
    ref = U.oracle_run(name, 37, 16, 1, 2)
    outs = []
    for rows in (5, 8, 32, 64):
        ctx = U.make_ctx(name, 1, 2, max_ctx=80, max_prefill_rows=rows)
        assert ctx.prefill(ref["prompt"]) == ref["first"]
        outs.append(ctx.debug_logits(0, 0).copy())
        assert ctx.decode(16)[0].tolist() == ref["tokens"]
        ctx.close()
    for o in outs[1:]:
        assert np.array_equal(o.view(np.uint32), outs[0].view(np.uint32))   # bit-identical across chunkings


def test_norm_gains_are_applied():
    ref = U.oracle_run("tiny_bf16", 16, 24, 1, 2, wseed=3, gain_jitter=0.2)
    ctx = U.make_ctx("tiny_bf16", 1, 2, max_ctx=64, wseed=3, gain_jitter=0.2)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    assert ctx.decode(24)[0].tolist() == ref["tokens"]
    U.assert_same_run(ctx, ref, 24)
    ctx.close()


def test_error_paths_leave_the_context_usable():
    import paper_2609_17184_b200 as ls
    ctx = U.make_ctx("tiny_bf16", 1, 2, max_ctx=64)
    for call in (ctx.step, lambda: ctx.decode(4), lambda: ctx.vanilla_decode(4)):
        with pytest.raises(ls.LoopSpecError) as e:
            call()
        assert e.value.status == "ESTATE"
    with pytest.raises(ls.LoopSpecError) as e:
        ctx.prefill(np.arange(100) % 512)
    assert e.value.status == "ECAPACITY"
    with pytest.raises(ls.LoopSpecError) as e:
        ctx.prefill([1, 2, 9999])
    assert e.value.status == "EINVAL"
    prompt = W.make_prompt(512, 16)
    ctx.prefill(prompt)
    with pytest.raises(ls.LoopSpecError) as e:
        ctx.decode(1000)
    assert e.value.status == "ECAPACITY"
    # fewer tokens than max_ctx, but prompt + tokens + the speculative chain would leave the KV pool: refused on the
    # host, before any pass is launched (17 committed ids + 50 + R/d1 + 2 > 64), and nothing has been disturbed
    for call in (lambda: ctx.decode(50), lambda: ctx.vanilla_decode(50)):
        with pytest.raises(ls.LoopSpecError) as e:
            call()
        assert e.value.status == "ECAPACITY"
    assert ctx.stats()["steps"] == 0
    ref = U.oracle_run("tiny_bf16", 16, 8, 1, 2)
    assert ctx.decode(8)[0].tolist() == ref["tokens"]
    assert ctx.decode(64 - 17 - 8 - 4 - 2).shape[1] == 33       # exactly up to the limit is accepted
    with pytest.raises(ls.LoopSpecError) as e:
        ctx.decode(1)
    assert e.value.status == "ECAPACITY"
    with pytest.raises(ls.LoopSpecError) as e:
        U.make_ctx("tiny_bf16", 3, 0)
    assert e.value.status == "EINVAL"
    ctx.close()


@pytest.mark.parametrize("name,d1,d2,T,gate", [
    ("tiny_raven_r4", 1, 2, 0.0, True), ("tiny_raven_r4", 1, 2, 1.0, True), ("tiny_raven_r4", 1, 3, 0.8, False),
    ("tiny_raven_r4", 2, 0, 1.0, True), ("tiny_raven", 2, 8, 0.0, True), ("tiny_raven", 2, 8, 1.0, True),
    ("tiny_raven", 4, 8, 1.0, False), ("tiny_raven", 2, 4, 0.7, True)])
def test_raven_layout_matches_oracle(name, d1, d2, T, gate):
    """Raven-style layout (Sec. 3.1: P and C hold transformer blocks; App. B: prelude cache, one coda cache per readout
    depth): prelude pass for the rows entering their first recurrence, adapter on [state; prelude output], recurrent
    blocks, coda pass on copies of the reading-out rows' states - tokens, decisions, counters and the stored proposal
    logits as the oracle's; greedy LoopSpec equals vanilla decoding on the device."""
    n_prompt, n_decode = 40, 24
    ref = U.oracle_run(name, n_prompt, n_decode, d1, d2, T=T, seed=5, gate=gate)
    ctx = U.make_ctx(name, d1, d2, T=T, seed=5, gate=gate, max_ctx=n_prompt + n_decode + 24, max_prefill_rows=16)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    z0 = ref["dec"].first_logits      # 16 recurrences deep: the stated bf16 tolerance, not the tighter bound of the shallow models
    assert (np.abs(ctx.debug_logits(0, 0) - z0) <= 3e-2 + 2e-2 * np.abs(z0)).all()
    ctx.decode(n_decode)
    U.assert_same_run(ctx, ref, n_decode)
    st, ost = ctx.stats(), ref["dec"].stats
    for k in ("steps", "n_accept1", "n_accept2", "n_restart", "gate_evals", "gate_opens", "rows_total", "rows_max", "readout_rows_total"):
        assert st[k] == ost[k], k
    assert ctx.row_trace().tolist() == ref["dec"].rows_per_step
    van = U.oracle_run(name, n_prompt, n_decode, d1, d2, T=T, seed=5, vanilla=True)
    ctx.prefill(van["prompt"])
    assert ctx.vanilla_decode(n_decode)[0].tolist() == van["tokens"]
    if T == 0.0:
        assert van["tokens"] == ref["tokens"]
    ctx.close()


@pytest.mark.parametrize("name,d1,d2,T,gate", [("tiny_r32", 2, 8, 1.0, False), ("tiny_raven_r32", 2, 8, 1.0, True),
                                                ("tiny_r32", 2, 10, 1.0, True), ("tiny_r32", 4, 8, 0.0, True)])
def test_thirty_two_recurrences_with_hundreds_of_rows_per_pass(name, d1, d2, T, gate):
    """The Raven family's loop count, R = 32, with the paper's depth pairs (2, 8) and (2, 10) (Sec. 4.3 "Gating Mechanism":
    up to B = 249 branches; appendix on the effective batch size: observed peaks of 176-239 rows): passes of up to 249 rows
    (GEMMs in groups of 64 token columns), chains of up to 16 uncommitted positions - tokens, decisions, row counts per
    pass and counters as the oracle's."""
    import paper_2609_17184_b200 as ls
    n_prompt, n_decode = 24, 16
    ref = U.oracle_run(name, n_prompt, n_decode, d1, d2, T=T, seed=5, gate=gate)
    ctx = U.make_ctx(name, d1, d2, T=T, seed=5, gate=gate, max_ctx=n_prompt + n_decode + 40, max_prefill_rows=16)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(n_decode)
    U.assert_same_run(ctx, ref, n_decode)
    st, ost = ctx.stats(), ref["dec"].stats
    for k in ("steps", "n_accept1", "n_accept2", "n_restart", "gate_evals", "gate_opens", "rows_total", "rows_max", "readout_rows_total"):
        assert st[k] == ost[k], k
    assert ctx.row_trace().tolist() == ref["dec"].rows_per_step
    assert st["rows_max"] <= ls.max_branches(32, d1, d2)
    if (d1, d2, gate) == (2, 8, False):
        assert st["rows_max"] == 249 == ls.max_branches(32, 2, 8)     # the bound of Sec. 4.3 is reached
    ctx.close()


def test_a_bounded_device_wait_that_runs_out_is_reported_and_survived():
    """Failure detection without a fault: a ring tile of the readout GEMM is never requested, so the MMA issuer's wait
    for it runs out after ~0.1 ms; the kernel raises its flag, carries on and ends; the call returns ETIMEOUT; after the
    injection is switched off and the sequence prefilled again the context decodes exactly like the oracle."""
    import time
    import paper_2609_17184_b200 as ls
    ref = U.oracle_run("tiny_bf16", 16, 12, 1, 2)
    ctx = U.make_ctx("tiny_bf16", 1, 2, max_ctx=64)
    ctx.prefill(ref["prompt"])
    ctx.debug_drop_tile(0, wait_us=100)
    t0 = time.time()
    with pytest.raises(ls.LoopSpecError) as e:
        for _ in range(4):          # the first readout happens in the first pass (d1 = 1)
            ctx.step()
    assert e.value.status == "ETIMEOUT", e.value
    assert time.time() - t0 < 5.0    # bounded: nothing spun for long
    with pytest.raises(ls.LoopSpecError) as e:       # the captured decode loop reports it too
        ctx.prefill(ref["prompt"])
        ctx.decode(4)
    assert e.value.status == "ETIMEOUT"
    ctx.debug_drop_tile(-1)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    assert ctx.decode(12)[0].tolist() == ref["tokens"]
    U.assert_same_run(ctx, ref, 12)
    ctx.close()


@pytest.mark.parametrize("unit", [0, 1, 3])
def test_a_bounded_wait_of_the_wide_decode_gemms_that_runs_out_is_reported_and_survived(unit):
    """The same for the layers' GEMMs of a context of several sequences (tcgen05 path): no lane of an issuing warp leaves its loop
    alone - the others would wait for it - and an accumulator that is not complete is not stored."""
    import time
    import paper_2609_17184_b200 as ls
    refs = [U.oracle_run("tiny_bf16", 16 + s, 12, 1, 2, seq=s) for s in range(4)]
    ctx = U.make_ctx("tiny_bf16", 1, 2, max_seqs=4, max_ctx=64)
    assert ctx.decode_paths()[0] == 1
    prefill = lambda: [ctx.prefill(refs[s]["prompt"], seq=s) for s in range(4)]
    prefill()
    ctx.decode(12)                   # (every partial sum has been written once: what a dropped tile leaves behind is finite)
    prefill()
    ctx.debug_drop_tile(unit, wait_us=100)
    t0 = time.time()
    with pytest.raises(ls.LoopSpecError) as e:
        ctx.step()
    assert e.value.status == "ETIMEOUT", e.value
    assert time.time() - t0 < 5.0
    ctx.debug_drop_tile(-1)
    assert prefill() == [r["first"] for r in refs]
    out = ctx.decode(12)
    for s in range(4):
        assert out[s].tolist() == refs[s]["tokens"], U.min_margin(refs[s]["dec"])
    ctx.close()


def test_depths_from_the_closed_form_are_used_when_none_are_given():
    """d1 = d2 = 0 at init: the library picks the admissible pair minimising Theorem 2's bound, like the oracle."""
    from oracle import depths as dp
    alpha, beta = 1.0, 0.3
    R = W.CONFIGS["tiny_bf16"].R
    d1, d2 = dp.snap_depths(float(np.float32(alpha)), float(np.float32(beta)), R)
    ref = U.oracle_run("tiny_bf16", 16, 40, d1, d2, T=1.0, seed=2)
    ctx = U.make_ctx("tiny_bf16", 0, 0, T=1.0, seed=2, max_ctx=64, alpha=alpha, beta=beta)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(40)
    U.assert_same_run(ctx, ref, 40)
    assert ctx.stats()["steps"] == ref["dec"].stats["steps"]
    ctx.close()


@pytest.mark.parametrize("name,T,rows", [("tiny_bf16", 0.0, 64), ("tiny_bf16", 1.0, 16), ("small_bf16", 1.0, 64), ("tiny_gqa", 0.0, 32)])
@pytest.mark.parametrize("skinny", [False, True])
def test_prefill_paths_match_oracle(name, T, rows, skinny):
    """The two ways a prefill pass can run its layer GEMMs: the wide tcgen05 kernel + fused-epilogue kernel (default where
    the shapes allow), or the kernels of the decode passes (`prefill_skinny`).  Their K splits differ, so each is compared
    with the oracle, not bit for bit with the other."""
    ref = U.oracle_run(name, 150, 24, 1, 2, T=T, seed=9)
    ctx = U.make_ctx(name, 1, 2, T=T, seed=9, max_ctx=200, max_prefill_rows=rows, prefill_skinny=skinny)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(24)
    U.assert_same_run(ctx, ref, 24)
    ctx.close()


@pytest.mark.parametrize("name", ["tiny_gqa", "tiny_gqa_f32"])
@pytest.mark.parametrize("T", [0.0, 1.0])
def test_grouped_query_attention(name, T):
    """Four query heads per KV head (the Raven-style head layout), head sizes 64 and 128, bf16 and fp32 weights; a
    context of several attention chunks."""
    ref = U.oracle_run(name, 150, 32, 1, 2, T=T, seed=6)
    ctx = U.make_ctx(name, 1, 2, T=T, seed=6, max_ctx=200, max_prefill_rows=64)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(32)
    U.assert_same_run(ctx, ref, 32)
    ctx.close()


@pytest.mark.parametrize("name,T,skinny", [("tiny_bf16", 0.0, False), ("tiny_bf16", 1.0, False), ("tiny_gqa", 1.0, False),
                                           ("tiny_gqa_f32", 0.0, False), ("tiny_bf16", 1.0, True), ("tiny_gqa", 0.0, True)])
def test_context_beyond_2560_uses_runs_of_attention_chunks(name, T, skinny):
    """A 2700-token prompt: more than 40 chunks per row, so attention work items are runs of several chunks folded with
    the running-softmax rescaling (every decode row; with `prefill_skinny` also the prompt's rows, whose passes write
    the last positions they attend to - otherwise the prompt runs the prefill attention kernel)."""
    ref = U.oracle_run(name, 2700, 16, 1, 2, T=T, seed=3)
    ctx = U.make_ctx(name, 1, 2, T=T, seed=3, max_ctx=2740, max_prefill_rows=64, prefill_skinny=skinny)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(16)
    U.assert_same_run(ctx, ref, 16)
    ctx.close()


def test_longer_context_spans_many_attention_chunks():
    """A 300-token prompt: five 64-position attention chunks plus the speculative slots, prefill in 64-row passes."""
    ref = U.oracle_run("tiny_bf16", 300, 24, 1, 2, T=1.0, seed=4)
    ctx = U.make_ctx("tiny_bf16", 1, 2, T=1.0, seed=4, max_ctx=340, max_prefill_rows=64)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(24)
    U.assert_same_run(ctx, ref, 24)
    ctx.close()


def test_contexts_of_different_widths_coexist():
    """A kernel's shared-memory limit belongs to the process: a context (or a stand-alone call) that needs less of it must
    not lower the limit under one that was created before."""
    import paper_2609_17184_b200 as ls
    ref = U.oracle_run("tiny_bf16", 20, 12, 1, 2, T=1.0, seed=2)
    a = U.make_ctx("tiny_bf16", 1, 2, T=1.0, seed=2, max_ctx=64, max_prefill_rows=32)
    b = U.make_ctx("tiny_bf16", 1, 2, T=1.0, seed=2, max_ctx=64, max_prefill_rows=64)
    ls.linear_tc(torch.zeros(128, 64, dtype=torch.bfloat16, device="cuda"), torch.zeros(1, 64, device="cuda"))
    for ctx in (a, b):
        assert ctx.prefill(ref["prompt"]) == ref["first"]
        assert ctx.decode(12)[0].tolist() == ref["tokens"]
        ctx.close()


@pytest.mark.parametrize("name,n_prompt,T", [("tiny_bf16", 64, 0.0), ("tiny_bf16", 65, 1.0), ("tiny_bf16", 128, 0.0), ("tiny_bf16", 129, 1.0),
                                             ("tiny_bf16", 1025, 0.0), ("tiny_gqa", 300, 1.0), ("small_bf16", 97, 1.0),
                                             ("small_bf16", 260, 0.0), ("tiny_raven_r4", 161, 1.0)])
def test_wide_prompt_passes_match_oracle(name, n_prompt, T):
    """Prompts without a bound on the pass (the default) run the wide kernels from 65 tokens on: the edges of a 128-token
    tile, two passes, ragged feature and row blocks, grouped-query heads, both layouts."""
    ref = U.oracle_run(name, n_prompt, 12, 1, 2, T=T, seed=9)
    ctx = U.make_ctx(name, 1, 2, T=T, seed=9, max_ctx=n_prompt + 40)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    np.testing.assert_allclose(ctx.debug_logits(0, 0), ref["dec"].first_logits, atol=2e-3, rtol=0)
    ctx.decode(12)
    U.assert_same_run(ctx, ref, 12)
    ctx.close()


@pytest.mark.parametrize("n_prompt", [96, 97, 160, 192, 224, 257])
def test_prompt_tiles_of_every_width_match_oracle(n_prompt):
    """The token tiles of a wide pass are 128, 96 or 64 columns (whichever fills the pairs of CTAs evenly) with a narrower one for the
    leftover tokens: prompts at the edges of the widths, against the oracle's logits."""
    ref = U.oracle_run("small_bf16", n_prompt, 6, 1, 2, seed=3)
    ctx = U.make_ctx("small_bf16", 1, 2, seed=3, max_ctx=320)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    assert ctx.decode(6)[0].tolist() == ref["tokens"], U.min_margin(ref["dec"])
    U.assert_same_run(ctx, ref, 6)
    ctx.close()


def _prompt_error(shape, n_prompt, **kw):
    """Relative error (2-norm) of a prompt's logits against the float64 oracle, of a model without attention (its keys and values are
    zero, so no rounding to bf16 hides the GEMMs' own error)."""
    import paper_2609_17184_b200 as ls
    from oracle.loopspec import Decoder
    from oracle.model import LoopedLM
    w = W.make_weights(shape, seed=3, out_scale=1.0)
    for k in w:
        if k.endswith("wqkv"):
            w[k][:] = 0
    prompt = W.make_prompt(shape.vocab, n_prompt, seed=1)
    ref = Decoder(LoopedLM(shape, w), temperature=0.0, seed=0)
    ref.prefill(prompt, 4)
    gw = ls.upload_weights(shape, w)
    out = []
    for rows in (0, 64):  # the wide passes, passes of up to 64 rows
        ctx = ls.LoopSpec(shape, gw, d1=1, d2=0, max_ctx=n_prompt + 16, max_prefill_rows=rows)
        ctx.prefill(prompt)
        z = ctx.debug_logits(0, 0).astype(np.float64)
        out.append(np.linalg.norm(z - ref.first_logits) / np.linalg.norm(ref.first_logits))
        ctx.close()
    return out


@pytest.mark.parametrize("hidden,ffn,n_prompt", [(2048, 5632, 70), (2048, 5632, 130), (768, 2000, 97)])
def test_wide_prompt_passes_are_as_exact_as_narrow_ones(hidden, ffn, n_prompt):
    """The tensor cores truncate their fp32 accumulators after every 16 values of k, so a GEMM's error grows with the length of its
    accumulation chains: the wide passes may not have longer ones than the passes of up to 64 rows.  A chain of c steps of a random
    walk loses about 2/3 c 2^-24: 1.3e-6 at the 32 steps allowed at most (whole k-ranges: 2.7e-6 at these widths)."""
    shape = W.CONFIGS["ouro_1p4b"].with_(vocab=512, hidden=hidden, n_q_heads=hidden // 128, n_kv_heads=hidden // 128, ffn=ffn, n_recurrent=1, R=2)
    wide, narrow = _prompt_error(shape, n_prompt)
    assert wide < 1.3e-6 and wide < 1.25 * narrow, (wide, narrow)
