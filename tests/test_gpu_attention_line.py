"""A lone sequence's decode attention changes kernels with the context capacity: one CTA per chunk up to the line, one warp per chunk
beyond it, while vanilla passes (one row) stay with the former up to one chunk per item.  Both sides of the line against the oracle, at
contexts of one chunk, a chunk and one position, and several."""
import pytest

from tests import gpu_util as U

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
