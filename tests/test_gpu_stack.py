"""The layer-stack kernel (passes of up to 32 rows) against the kernels per projection, which run the same pass while GEMM
launches are timed: logits and the new K/V rows, at the sizes where its plans change."""
import numpy as np
import pytest

from paper_2605_13319_b200 import synth
from harness import logit_rel_err

pytestmark = pytest.mark.gpu

# Both sum fp32 in different orders; what differs beyond 2^-20 is that K and V are stored as bf16, where a value at a rounding
# boundary goes either way (2^-8 of itself) and later layers see that: up to 4e-4 of a row's largest logit in these shapes.
TOL = 2e-3

T = synth.TINY
CASES = {
    # one request: shape, prefix lengths, drafts per request, page size
    "one key": (T, [1], [1], 16),
    "head 128": (T.scaled(d_model=512, n_q_heads=4, n_kv_heads=4, head_dim=128), [130], [8], 16),
    "four heads share, 72 rows": (T.scaled(n_q_heads=8, n_kv_heads=2, head_dim=64, d_model=512), [700], [17], 16),
    "eight heads share one, 72 rows": (T.scaled(n_q_heads=8, n_kv_heads=1, head_dim=128, d_model=1024), [5000], [8], 16),
    "32 rows": (T, [257], [31], 16),
    "25 rows, pages of 8": (T, [255], [24], 8),
    "pages of 256": (T, [600], [6], 256),
    "ranges of several tiles": (T.scaled(d_model=2048, n_q_heads=16, n_kv_heads=16, head_dim=128), [2500], [8], 16),
    "ragged widths": (T.scaled(d_model=272, d_ffn=176, vocab=1040), [33], [3], 16),
    "narrow": (T.scaled(d_model=48, n_q_heads=1, n_kv_heads=1, d_ffn=32, vocab=48), [90], [2], 16),
    "wide, whole row blocks": (T.scaled(d_model=1024, d_ffn=4096, vocab=32000), [64], [5], 16),
    "16 requests of two rows": (T, [3, 17, 400, 129, 5, 6, 7, 900, 1, 64, 65, 66, 31, 32, 33, 250], [1] * 16, 16),
    "more heads than SMs": (T.scaled(d_model=1024, n_q_heads=16, n_kv_heads=16), [130, 170, 400, 110, 190, 260, 164, 500, 133, 148, 300, 129], [1, 2] * 6, 16),
    "three requests": (T.scaled(n_kv_heads=2), [40, 1200, 300], [16, 2, 9], 16),
    # CTAs that hold a whole row block and finish rows of one they share, where the epilogue reads memory: a CTA takes eight
    # k16 steps at least, more than one row block's 6 (or 5) of these
    "whole and shared row blocks of QKV": (T.scaled(d_model=96), [40], [8], 16),
    "whole and shared row blocks of QKV, 32 rows": (T.scaled(d_model=80, n_q_heads=8, n_kv_heads=4), [300], [31], 16),
    "whole and shared row blocks of down": (T.scaled(d_ffn=96), [40], [1], 16),
    "whole and shared row blocks of down, 32 rows": (T.scaled(d_model=1024, d_ffn=80), [300], [31], 16),
    # heads whose keys are one CTA's: finished from tensor memory
    "a head of one's own, 72 rows": (T.scaled(n_q_heads=8, n_kv_heads=1, head_dim=128, d_model=1024), [40], [8], 16),
    "heads of one's own, 25 rows": (T.scaled(d_model=512, n_q_heads=4, n_kv_heads=4, head_dim=128), [20], [24], 16),
    "heads of one's own, 7 and 21 rows": (T.scaled(n_q_heads=6, n_kv_heads=2), [30, 5], [6, 20], 8),
}


def _run(ctx, items, lens, rows, layers):
    from paper_2605_13319_b200 import binding
    got = ctx.verify(items, flags=binding.Q_HOST)
    logits = ctx.debug_get_logits(rows)
    ctx.kv_rollback([it["req"] for it in items], [len(it["tokens"]) - 1 for it in items])
    kv = []
    for it, P in zip(items, lens):
        for l in layers:
            kv += [synth.bf16_to_f32(x) for x in ctx.debug_read_kv(it["req"], l, P, len(it["tokens"]))]
        ctx.debug_set_len(it["req"], P)
    return got, logits, kv


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("growing", [False, True])
def test_against_the_kernels_per_projection(name, growing):
    """`growing`: keys grow along the prefix, so that scores exceed a segment's first one by far and sums are rescaled."""
    from paper_2605_13319_b200 import binding
    shape, lens, ks, page = CASES[name]
    if growing and max(lens) < 200:
        pytest.skip("nothing to rescale")
    w = synth.make_weights(shape, 11)
    rows = sum(ks) + len(ks)
    ctx = binding.Context(shape, w, n_pages=sum((P + 40) // page + 1 for P in lens), max_requests=len(lens), max_rows=rows, max_seq=max(lens) + 40,
                          max_draft=max(ks), page_size=page, poison=True)
    items = []
    for i, (P, k) in enumerate(zip(lens, ks)):
        req = ctx.req_open()
        for l in range(shape.n_layers):
            kb, vb = synth.make_synthetic_kv(shape, P, 11 + i, l)
            if growing:
                ramp = np.linspace(0.0, 60.0, P, dtype=np.float32)[:, None]
                kb = synth.f32_to_bf16(synth.bf16_to_f32(kb).reshape(P, -1) * ramp).reshape(kb.shape)
            ctx.debug_write_kv(req, l, 0, kb, vb)
        items.append(dict(req=req, tokens=synth.tokens_i32(k + 1, 11, 900 + i, shape.vocab), u=synth.make_accept_uniforms(k, 11, i),
                          q=np.full((k, shape.vocab), 1.0 / shape.vocab, np.float32)))
    layers = range(shape.n_layers)
    ctx.profile_enable(True)
    _, want, want_kv = _run(ctx, items, lens, rows, layers)
    launches = ctx.profile_read()["kernel_launches"]
    ctx.profile_enable(False)
    for _ in range(2):                                         # the second on what the first left in the exchange words
        _, got, got_kv = _run(ctx, items, lens, rows, layers)
        assert ctx.profile_read()["kernel_launches"] == 3 < launches
        assert np.isfinite(got).all()
        # scores of a few hundred carry errors of 2^-17 of themselves, and probabilities as much in relative terms
        assert logit_rel_err(got, want).max() < (2e-2 if growing else TOL)
        for a, b in zip(got_kv, want_kv):
            assert np.all(np.abs(a - b) <= 2.0 ** -7 * np.abs(b) + (2e-2 if growing else 2e-3) * np.abs(b).max())
    ctx.close()


def _context(shape, lens, ks, page=16, seed=11, stream=None):
    """A context with these prefixes cached, the items of a pass over them, and the number of its rows."""
    from paper_2605_13319_b200 import binding
    rows = sum(ks) + len(ks)
    ctx = binding.Context(shape, synth.make_weights(shape, seed), n_pages=sum((P + 40) // page + 1 for P in lens), max_requests=len(lens),
                          max_rows=rows, max_seq=max(lens) + 40, max_draft=max(ks), page_size=page, poison=True, stream=stream)
    items = []
    for i, (P, k) in enumerate(zip(lens, ks)):
        req = ctx.req_open()
        for l in range(shape.n_layers):
            ctx.debug_write_kv(req, l, 0, *synth.make_synthetic_kv(shape, P, seed + i, l))
        items.append(dict(req=req, tokens=synth.tokens_i32(k + 1, seed, 900 + i, shape.vocab), u=synth.make_accept_uniforms(k, seed, i),
                          q=np.full((k, shape.vocab), 1.0 / shape.vocab, np.float32)))
    return ctx, items, rows


def _close(got, want, got_kv, want_kv, tol=TOL):
    assert np.isfinite(got).all()
    assert logit_rel_err(got, want).max() < tol
    for a, b in zip(got_kv, want_kv):
        assert np.all(np.abs(a - b) <= 2.0 ** -7 * np.abs(b) + tol * np.abs(b).max())


@pytest.mark.parametrize("name, some", [("32 rows", (2, 3, 13, 40)), ("ragged widths", (1, 2, 3, 7)), ("three requests", (10, 26, 27, 40)),
                                        ("wide, whole row blocks", (2, 3, 13, 40))])
def test_fewer_ctas(name, some):
    """As on a device of fewer SMs: fewer CTAs than rows, several whole row blocks to a CTA, and whole and shared ones."""
    shape, lens, ks, page = CASES[name]
    ctx, items, rows = _context(shape, lens, ks, page)
    layers = range(shape.n_layers)
    ctx.profile_enable(True)
    _, want, want_kv = _run(ctx, items, lens, rows, layers)
    ctx.profile_enable(False)
    for ctas in (*some, 0):
        ctx.debug_stack_ctas(ctas)
        ctx.profile_read()
        _, got, got_kv = _run(ctx, items, lens, rows, layers)
        assert ctx.profile_read()["kernel_launches"] == 3, ctas
        _close(got, want, got_kv, want_kv)
    ctx.close()


def _part_of_the_device(sms):
    """A stream that has `sms` SMs of device 0 to itself (a green context's); skips where that cannot be had."""
    import torch
    driver = pytest.importorskip("cuda.bindings.driver")

    def ok(r):
        if r[0] != driver.CUresult.CUDA_SUCCESS:
            pytest.skip(f"no green context: {r[0]}")
        return r[1]
    torch.zeros(1, device="cuda")
    dev = ok(driver.cuDeviceGet(0))
    whole = ok(driver.cuDeviceGetDevResource(dev, driver.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    part = ok(driver.cuDevSmResourceSplitByCount(1, whole, 0, sms))[0]
    green = ok(driver.cuGreenCtxCreate(ok(driver.cuDevResourceGenerateDesc([part], 1)), dev,
                                       driver.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    stream = ok(driver.cuGreenCtxStreamCreate(green, driver.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))
    return torch.cuda.ExternalStream(int(stream))


def test_stream_of_fewer_sms():
    """The kernel wants as many SMs as the device has; on a stream that has fewer its launch is refused, and the pass, and every
    later one, runs on the kernels per projection."""
    shape, lens, ks = T, [100], [8]
    results = []
    for stream in (None, _part_of_the_device(64)):
        ctx, items, rows = _context(shape, lens, ks, stream=stream)
        ctx.profile_read()
        results += [(_run(ctx, items, lens, rows, range(shape.n_layers)), ctx.profile_read()["kernel_launches"]) for _ in range(2)]
        ctx.close()
    (want, n), _, (first, n1), (second, n2) = results
    assert n == 3 < n1 == n2
    for got in (first, second):
        _close(got[1], want[1], got[2], want[2])
    assert first[0] == second[0] and np.array_equal(first[1], second[1])


def test_shared_device():
    """A pass of a context that shares its device is done while another stream's kernel still holds an SM; and agrees with the
    one that takes them all."""
    import torch
    from paper_2605_13319_b200 import binding
    shape, lens, ks = T, [100], [8]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    (ctx, items, rows), (other, _, _) = (_context(shape, lens, ks, stream=s) for s in streams)
    layers = range(shape.n_layers)
    _, want, want_kv = _run(ctx, items, lens, rows, layers)
    ctx.share_device()
    _run(ctx, items, lens, rows, layers)
    held = torch.cuda.Event()
    other.debug_wait_timeout(100000)                           # one warp for 100 ms
    held.record(streams[1])
    got, logits, kv = _run(ctx, items, lens, rows, layers)
    assert not held.query()                                    # it is still there
    _close(logits, want, kv, want_kv)
    with pytest.raises(binding.PipesdError):
        other.ctx_sync()
    ctx.share_device(False)
    ctx.profile_read()
    _, again, _ = _run(ctx, items, lens, rows, layers)
    assert ctx.profile_read()["kernel_launches"] == 3 and np.array_equal(again, want)
    ctx.close()
    other.close()


@pytest.mark.parametrize("long, fits", [(2174, True), (2175, False)])
def test_long_request_beside_a_short_one(long, fits):
    """A CTA's table holds 16 parts of key ranges.  At 32 KV heads, beside a request of two 16-key units per head, ranges of 30 units
    have at most 16 of them, ranges of 31 may have 17: such a pass runs on the kernels per projection."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("ranges are other ones")
    shape, lens, ks = T.scaled(n_q_heads=32, n_kv_heads=32), [30, long], [1, 1]
    ctx, items, rows = _context(shape, lens, ks)
    layers = range(shape.n_layers)
    ctx.profile_enable(True)
    _, want, want_kv = _run(ctx, items, lens, rows, layers)
    ctx.profile_enable(False)
    _, got, got_kv = _run(ctx, items, lens, rows, layers)
    assert (ctx.profile_read()["kernel_launches"] == 3) == fits
    assert np.array_equal(got, want) != fits
    _close(got, want, got_kv, want_kv)
    ctx.close()


@pytest.mark.parametrize("keys, one", [(60, False), (398, True), (700, True)])
def test_many_short_requests(keys, one):
    """256 (request, KV head) pairs of a small model: below 400 keys each (the pass's own two among them) a kernel per projection."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count > 196:
        pytest.skip("no more pairs than the device has SMs for")
    shape, lens, ks = T.scaled(d_model=512, n_q_heads=16, n_kv_heads=16), [keys] * 16, [1] * 16
    ctx, items, rows = _context(shape, lens, ks)
    layers = range(shape.n_layers)
    ctx.profile_enable(True)
    _, want, want_kv = _run(ctx, items, lens, rows, layers)
    ctx.profile_enable(False)
    _, got, got_kv = _run(ctx, items, lens, rows, layers)
    assert (ctx.profile_read()["kernel_launches"] == 3) == one
    _close(got, want, got_kv, want_kv)
    ctx.close()


@pytest.mark.parametrize("name", ["one key", "ranges of several tiles", "three requests", "whole and shared row blocks of down"])
def test_waits_that_run_out(name):
    """So few looks at what other CTAs write that roles give up: the pass ends, the error is reported, and the next pass of the
    context is what it was before, bit for bit.  At one look nobody gets past the first phase; at more of them each gives up
    somewhere else, or nowhere."""
    from paper_2605_13319_b200 import binding
    shape, lens, ks, page = CASES[name]
    ctx, items, rows = _context(shape, lens, ks, page)
    reqs, layers = [it["req"] for it in items], range(shape.n_layers)
    want, logits, kv = _run(ctx, items, lens, rows, layers)
    for looks in (1, 4, 16, 1):
        ctx.debug_stack_looks(looks)
        failed = None
        try:
            got = ctx.verify(items, flags=binding.Q_HOST)
        except binding.PipesdError as e:
            failed = e
        if failed is None:
            assert looks > 1 and got == want and np.array_equal(ctx.debug_get_logits(rows), logits), looks
        else:
            assert failed.code == binding.E_CUDA and "timed out" in str(failed)
        ctx.kv_rollback(reqs, [0] * len(reqs))
        for req, P in zip(reqs, lens):
            ctx.debug_set_len(req, P)
        ctx.debug_stack_looks(0)
        again = _run(ctx, items, lens, rows, layers)
        assert again[0] == want and np.array_equal(again[1], logits), looks
        assert all(np.array_equal(a, b) for a, b in zip(again[2], kv)), looks
    with pytest.raises(binding.PipesdError):
        ctx.debug_stack_looks(-1)
    ctx.close()


def test_pass_behind_a_wait_that_ran_out():
    """A pass enqueued behind a wait that ran out, before the host has seen that, leaves at once: what it would have written stays
    as it was."""
    from paper_2605_13319_b200 import binding
    shape, n = T, 20
    ctx, items, rows = _context(shape, [100], [8])
    want, logits, kv = _run(ctx, items, [100], rows, range(shape.n_layers))
    ctx.close()
    ctx = binding.Context(shape, synth.make_weights(shape, 11), n_pages=20, max_requests=2, max_rows=32, max_seq=140, max_draft=8, poison=True)
    (req, other), tokens = (ctx.req_open(), ctx.req_open()), synth.tokens_i32(n, 11, 77, shape.vocab)
    there = [synth.make_synthetic_kv(shape, n, 5, l) for l in range(shape.n_layers)]
    for l in range(shape.n_layers):
        ctx.debug_write_kv(req, l, 0, *synth.make_synthetic_kv(shape, 100, 11, l))
        ctx.debug_write_kv(other, l, 0, *there[l])
    ctx.debug_set_len(other, 0)
    ctx.debug_wait_timeout(1000)
    ctx.prefill(other, tokens)                                 # into the same page
    with pytest.raises(binding.PipesdError):
        ctx.ctx_sync()
    for l in range(shape.n_layers):
        for a, b in zip(ctx.debug_read_kv(other, l, 0, n), there[l]):
            assert np.array_equal(np.asarray(a).ravel(), np.asarray(b).ravel())
    items[0]["req"] = req
    again = _run(ctx, items, [100], rows, range(shape.n_layers))
    assert again[0] == want and np.array_equal(again[1], logits) and all(np.array_equal(a, b) for a, b in zip(again[2], kv))
    ctx.debug_set_len(other, 0)
    ctx.prefill(other, tokens)
    ctx.ctx_sync()
    assert not np.array_equal(np.asarray(ctx.debug_read_kv(other, 0, 0, n)[0]).ravel(), np.asarray(there[0][0]).ravel())
    ctx.close()
