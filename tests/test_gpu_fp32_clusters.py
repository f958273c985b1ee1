"""The fp32 GEMM's hand-over inside a cluster: every rank waits for the bytes of the columns it finishes, counted by the stores of the
others.  Sizes at which that can go wrong: launches without a cluster (a single k-block; more row blocks than the device holds pairs of
CTAs, the last case of them in two rounds per CTA - a cluster of several CTAs only ever has one), ranks that finish no column, one, and
several, k-ranges that end inside a block.  And the waits themselves: too short, and for sums that never come."""
import numpy as np
import pytest
import torch

from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 16, 8), (3, 19072, 24), (2, 48000, 40), (1, 128, 2048), (7, 128, 2048), (8, 304, 72), (9, 304, 1032), (64, 256, 688)])
def test_fp32_linear_inside_clusters(M, N, K):
    import paper_2609_17184_b200 as ls
    rng = np.random.default_rng(N + K + M)
    w = (rng.standard_normal((N, K)) * 0.05).astype(np.float32)
    x = rng.standard_normal((M, K)).astype(np.float32)
    wt, xt = torch.from_numpy(w).cuda(), torch.from_numpy(x).cuda()
    y = ls.linear(wt, xt).cpu().numpy()
    # A lane adds eight products of every k-block of its rank one after the other, two more additions fold the four lanes of a row, the
    # cluster's ranks are added in order: every product goes through at most `chain` roundings of 2^-24.  That is 4.4e-6 of the sum of
    # magnitudes at K = 2048, should all of them point the same way; 2e-6 is asked for in any case.
    kb = (K + 31) // 32
    cs = 1
    while 2 * cs <= min(8, kb) and 2 * cs * ((N + 127) // 128) <= 296:
        cs *= 2
    chain = 8 * -(-kb // cs) + 2 + cs - 1
    scale = np.abs(x).astype(np.float64) @ np.abs(w).astype(np.float64).T
    assert (np.abs(y - x.astype(np.float64) @ w.astype(np.float64).T) <= min(2e-6, chain * 2.0 ** -24) * scale + 1e-30).all()
    for _ in range(3):  # bit for bit, and whatever shares the call
        assert np.array_equal(ls.linear(wt, xt).cpu().numpy().view(np.uint32), y.view(np.uint32))
    assert np.array_equal(ls.linear(wt, xt[:1].contiguous()).cpu().numpy()[0].view(np.uint32), y[0].view(np.uint32))


def test_a_hand_over_that_never_comes_is_reported_and_survived():
    """The waits for a cluster's partial sums count on four bytes that nobody sends: they run out, twice, the kernel raises its flag and
    ends, the call returns ETIMEOUT; afterwards the context works like before."""
    import time
    import paper_2609_17184_b200 as ls
    ref = U.oracle_run("tiny", 16, 12, 1, 2)
    ctx = U.make_ctx("tiny", 1, 2, max_ctx=64)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    for call in (ctx.step, lambda: ctx.prefill(ref["prompt"]), lambda: ctx.decode(4), lambda: ctx.vanilla_decode(4)):
        ctx.debug_drop_tile(-1)
        ctx.prefill(ref["prompt"])
        ctx.debug_drop_tile(0, wait_us=20)
        t0 = time.time()
        with pytest.raises(ls.LoopSpecError) as e:
            call()
        assert e.value.status == "ETIMEOUT", e.value
        assert time.time() - t0 < 5.0
    ctx.debug_drop_tile(-1)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(12)
    U.assert_same_run(ctx, ref, 12)
    ctx.close()


@pytest.mark.parametrize("name", ["tiny", "tiny_gqa_f32"])
def test_a_bound_shorter_than_a_hand_over_costs_time_and_nothing_else(name):
    """Whoever has waited for a microsecond in vain stays until every sum has been sent and finishes with them."""
    ref = U.oracle_run(name, 16, 12, 1, 2)
    ctx = U.make_ctx(name, 1, 2, max_ctx=64)
    want = None
    for short in (False, True):
        if short:
            ctx.debug_drop_tile(1, wait_us=1)
        assert ctx.prefill(ref["prompt"]) == ref["first"]
        ctx.decode(12)
        U.assert_same_run(ctx, ref, 12)
        z = ctx.debug_logits(0, 0).view(np.uint32)
        assert want is None or np.array_equal(z, want)
        want = z
    ctx.close()
