"""Which kernel a lone sequence's decode attention runs: one CTA per chunk, or one warp per run of chunks.  By the context capacity
beyond 2560 positions; within it by the committed length alone - pipelined passes change over where R / d1 rows of n_kv_heads chunks per
64 positions exceed six (four query heads per key head: ten) per SM.  Both sides of either line against the oracle; and a job's bits
depend neither on how much larger than the job its context is nor on how calls cut it."""
import numpy as np
import pytest

from tests import gpu_util as U
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_ctx", [1000, 1001, 2561])
@pytest.mark.parametrize("name,n_prompt,T", [("tiny_bf16", 3, 0.0), ("tiny_bf16", 60, 1.0), ("tiny_gqa", 65, 0.0), ("tiny", 150, 1.0)])
def test_both_sides_of_the_line_match_the_oracle(name, n_prompt, T, max_ctx):
    ref = U.oracle_run(name, n_prompt, 10, 1, 2, T=T, seed=5)
    ctx = U.make_ctx(name, 1, 2, T=T, seed=5, max_seqs=1, max_ctx=max_ctx)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(10)
    U.assert_same_run(ctx, ref, 10)
    van = U.oracle_run(name, n_prompt, 10, 1, 2, T=T, seed=5, vanilla=True)
    assert ctx.prefill(ref["prompt"]) == van["first"]
    assert ctx.vanilla_decode(10)[0].tolist() == van["tokens"]
    ctx.close()


def same_bits(a, b):
    return np.array_equal(a.view(np.uint32), b.view(np.uint32))


@pytest.mark.parametrize("name,n_prompt", [("tiny_bf16", 40), ("tiny_bf16", 150), ("small_bf16", 130), ("tiny_gqa", 65), ("tiny", 100)])
def test_a_job_has_the_same_bits_in_every_capacity(name, n_prompt):
    prompt = W.make_prompt(W.CONFIGS[name].vocab, n_prompt, seed=7)
    want = {}
    for max_ctx in (256, 1000, 1001, 2048, 2560):
        ctx = U.make_ctx(name, 1, 2, max_seqs=1, max_ctx=max_ctx)
        assert ctx.decode_paths()[1] == 0, max_ctx
        for run in (ctx.decode, ctx.vanilla_decode):
            ctx.prefill(prompt)
            got = run(12)[0].tolist(), ctx.debug_logits(0, 0)
            ids, z = want.setdefault(run.__name__, got)
            assert got[0] == ids and same_bits(got[1], z), (max_ctx, run.__name__, np.abs(got[1] - z).max())
        ctx.close()


# model, query / kv heads, (d1, d2), committed positions up to which pipelined passes run a CTA per chunk
LINES = [("tiny_r16", 4, 4, 1, 0, 832), ("tiny_r32", 4, 4, 2, 0, 832), ("tiny_r8", 4, 4, 1, 2, 1728), ("tiny_r8", 32, 8, 1, 0, 1472),
         ("small_bf16", 6, 6, 1, 2, 2368)]


@pytest.mark.parametrize("name,nq,nkv,d1,d2,line", LINES)
def test_a_job_over_the_line_has_the_same_bits_however_it_is_cut(name, nq, nkv, d1, d2, line):
    import paper_2609_17184_b200 as ls
    shape = W.CONFIGS[name].with_(n_q_heads=nq, n_kv_heads=nkv)
    w = ls.upload_weights(shape, W.make_weights(shape))
    N = 14
    prompt = W.make_prompt(shape.vocab, line - 6, seed=7)  # one id is committed with the prompt: the sixth token is the first beyond

    def by_steps(ctx):
        n = 0
        while n < N:
            if ctx.step()[1]:
                n += len(ctx.verify())

    cuts = [lambda c: c.decode(N), lambda c: [c.decode(k) for k in (5, 1, 1, 7)], lambda c: [c.decode(k) for k in (2, 12)], by_steps]
    want = None
    for max_ctx, cut in [(line + 40, cuts[0]), (2560, cuts[0]), (2560, cuts[1]), (line + 40, cuts[2]), (2560, cuts[3])]:
        ctx = ls.LoopSpec(shape, w, d1=d1, d2=d2, max_ctx=max_ctx)
        ctx.prefill(prompt)
        cut(ctx)
        got = [c["token"] for c in ctx.commits(0)], ctx.debug_logits(0, 0)
        want = want or got
        assert got[0] == want[0] and same_bits(got[1], want[1]), (max_ctx, np.abs(got[1] - want[1]).max())
        ctx.close()


@pytest.mark.parametrize("name,n_prompt,d1,d2,T,max_ctx", [("tiny_r16", 828, 1, 0, 0.0, 900), ("tiny_r8", 1722, 1, 2, 1.0, 2048), ("tiny_r8", 1740, 1, 0, 0.0, 1800),
                                                           ("tiny_bf16", 2400, 1, 2, 0.0, 2560), ("tiny_bf16", 2400, 1, 2, 0.0, 2561)])
def test_long_lone_sequences_match_the_oracle(name, n_prompt, d1, d2, T, max_ctx):
    """13 to 41 chunks, on the near side of a line, across it and beyond it."""
    ref = U.oracle_run(name, n_prompt, 10, d1, d2, T=T, seed=5)
    ctx = U.make_ctx(name, d1, d2, T=T, seed=5, max_seqs=1, max_ctx=max_ctx)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(10)
    U.assert_same_run(ctx, ref, 10)
    ctx.close()
