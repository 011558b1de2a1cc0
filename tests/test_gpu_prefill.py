"""Prompt lengths around the limits of the prefill's paths: 32 rows (small-M kernels), one row more (dense kernels), the
edges of their token blocks and chunks; query heads per KV head 1 and 2."""
import numpy as np
import pytest

import oracle
from paper_2605_13319_b200 import synth
from harness import logit_rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_kv_heads,max_rows", [(4, 32), (2, 17), (2, 96)])
@pytest.mark.parametrize("n", [31, 33, 47, 64, 65, 129, 257])
def test_prefill_lengths(n, n_kv_heads, max_rows):
    from paper_2605_13319_b200 import binding
    shape = synth.TINY.scaled(name=f"tiny-kv{n_kv_heads}", n_kv_heads=n_kv_heads)
    w = synth.make_weights(shape, 3)
    prefix = synth.make_prefix(shape, n + 40, 3)
    orc = oracle.Oracle(shape, w, n + 48)
    ctx = binding.Context(shape, w, n_pages=(n + 48) // 16 + 1, max_seq=n + 48, max_rows=max_rows, max_draft=16, poison=True)
    req = ctx.req_open()
    # a prompt, then a second piece on top of it: the chunk's keys are partly cached, partly its own
    for part in (prefix[:n], prefix[n:n + 40]):
        want = orc.prefill(part, want_last_logits=True)
        got = ctx.prefill(req, part, want_last_logits=True)
        assert logit_rel_err(got[None], np.reshape(want, (1, -1))).max() < 1e-3     # as the verify passes: crossed K/V roundings
        # the last chunk's logits stay readable: (length - 1) % min(max_rows, 32) + 1 rows, the prompt's last one at the end
        rows = (len(part) - 1) % min(max_rows, 32) + 1
        assert np.array_equal(ctx.debug_get_logits(rows)[-1], got)
    for layer in range(shape.n_layers):
        kg, vg = ctx.debug_read_kv(req, layer, 0, n + 40)
        for bits, want in ((kg, [orc.get_kv(layer, p)[0] for p in range(n + 40)]), (vg, [orc.get_kv(layer, p)[1] for p in range(n + 40)])):
            got, want = synth.bf16_to_f32(bits), np.stack(want)
            # one bf16 step where a rounding boundary was crossed (2^-7 of the value at most), 2e-4 accumulated below it
            assert np.all(np.abs(got - want) <= 2.0 ** -7 * np.maximum(np.abs(got), np.abs(want)) + 2e-4 * np.abs(want).max())
    ctx.close()


def test_prefill_wide():
    """Widths of the 7b shape, where the projections of a long chunk run with blocks of up to 256 tokens: a chunk of 1024 rows
    and one of 750 on top of it, rows of every layer's K and V and the last logits against the CPU checker."""
    from paper_2605_13319_b200 import binding
    shape = synth.TINY.scaled(name="wide", d_model=4096, n_q_heads=32, n_kv_heads=32, head_dim=128, d_ffn=5504, vocab=512)
    w = synth.make_weights(shape, 8)
    n = 1024 + 750
    prefix = synth.make_prefix(shape, n, 8)
    orc = oracle.Oracle(shape, w, n)
    ctx = binding.Context(shape, w, n_pages=n // 16 + 1, max_seq=n, poison=True)
    req = ctx.req_open()
    for part in (prefix[:1024], prefix[1024:]):
        want = orc.prefill(part, want_last_logits=True)
        got = ctx.prefill(req, part, want_last_logits=True)
        assert logit_rel_err(got[None], np.reshape(want, (1, -1))).max() < 1e-3
    for layer in range(shape.n_layers):
        kg, vg = ctx.debug_read_kv(req, layer, 0, n)
        for i, bits in enumerate((kg, vg)):
            got, want = synth.bf16_to_f32(bits), np.stack([orc.get_kv(layer, p)[i] for p in range(n)])
            # The bounds of the full-size test.  Layer 0 sees identical inputs: an element differs by one bf16 step where a
            # rounding boundary was crossed (2^-7 of the value at most; here 4 elements in 10,000).  Such a step in a large
            # element of K moves a score by 2^-7 |q| |k|, a few percent, and where that key has most of a row's weight, the
            # row's whole attention output by as much: in layer 1 single rows are off by two steps, so an element is held
            # to 2e-2 of the largest and the mean to twice what prompts of 32-row passes show (1.6e-4; here 1.1e-4).
            diff, slack, l1 = np.abs(got - want), *((2e-5, 1e-4) if layer == 0 else (2e-2, 3.2e-4))
            assert np.all(diff <= 2.0 ** -7 * np.maximum(np.abs(got), np.abs(want)) + slack * np.abs(want).max()), (layer, i)
            assert diff.sum() < l1 * np.abs(want).sum(), (layer, i)
    ctx.close()


def test_prefill_chunks_agree():
    """Two chunks of the longest kind (1024 rows at most, cut in equal parts) against the same prompt fed in two calls."""
    from paper_2605_13319_b200 import binding
    shape, n = synth.TINY, 1031
    w = synth.make_weights(shape, 4)
    prefix = synth.make_prefix(shape, n, 4)
    ctx = binding.Context(shape, w, n_pages=2 * (n // 16 + 1), max_seq=n, max_requests=2, poison=True)
    a, b = ctx.req_open(), ctx.req_open()
    la = ctx.prefill(a, prefix, want_last_logits=True)
    ctx.prefill(b, prefix[:300])
    lb = ctx.prefill(b, prefix[300:], want_last_logits=True)
    assert logit_rel_err(la[None], lb[None]).max() < 1e-3
    ctx.close()
