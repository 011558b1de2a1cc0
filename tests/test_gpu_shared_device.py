"""Passes of up to 32 rows of a context that shares its device run on a kernel per projection and the attention kernel of larger
passes: the checks of test_gpu_verify.py against the CPU checker, on those; and the attention kernel's merge in a larger pass."""
import numpy as np
import pytest

from paper_2605_13319_b200 import binding, synth
from test_gpu_stack import T, _context
from test_gpu_verify import (test_attention_scores_of_wide_range, test_draft_lengths_across_token_tile_counts, test_merge_without_waiting,
                             test_multi_round_verify_rollback_lockstep, test_page_sizes_other_than_16)  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def shared(monkeypatch):
    """Every context is told that it shares its device, and has launched more than the three kernels of a whole-device pass."""
    create, verify = binding.Context.__init__, binding.Context.verify

    def shared_create(self, *a, **kw):
        create(self, *a, **kw)
        self.share_device()

    def counted_verify(self, *a, **kw):
        self.profile_read()
        out = verify(self, *a, **kw)
        assert self.profile_read()["kernel_launches"] > 3
        return out
    monkeypatch.setattr(binding.Context, "__init__", shared_create)
    monkeypatch.setattr(binding.Context, "verify", counted_verify)


@pytest.mark.parametrize("n_kv_heads,lens,ks", [(4, [4090, 300, 1000], [16, 16, 12]), (2, [4090, 700], [16, 16]), (1, [2000, 90, 3000, 40], [8, 8, 8, 8])])
def test_merge_without_waiting_in_a_large_pass(n_kv_heads, lens, ks):
    """More than 32 rows: the same bits whether or not the splits' CTAs see each other finish."""
    ctx, items, rows = _context(T.scaled(n_kv_heads=n_kv_heads), lens, ks)
    assert rows > 32
    want = None
    for polls in (128, 0, 0, 1, 3, 8, 128):
        ctx.debug_merge_polls(polls)
        ctx.verify(items, flags=binding.Q_HOST)
        got = ctx.debug_get_logits(rows)
        want = got if want is None else want
        assert np.isfinite(got).all() and np.array_equal(got, want), polls
        ctx.kv_rollback([it["req"] for it in items], [0] * len(items))
        for it, P in zip(items, lens):
            ctx.debug_set_len(it["req"], P)
    ctx.close()
