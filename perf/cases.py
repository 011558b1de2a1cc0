"""Timed workloads of the verify library: what a cloud server of speculative decoding has it do all day.

Two kinds of pass, through the C ABI (include/pipesd.h) as a server calls it:

  verify    one round for the requests of a batch: pipesd_verify, pipesd_ctx_sync, the rows' logits (servers hand
            log-probabilities on), pipesd_kv_rollback -- or, with "commit": "device", a verify that commits on the
            device and a chained verify of proactively sent drafts behind it, one sync for both;
  prefill   pipesd_prefill of one prompt with the logits of its last position.

After a pass the requests are put back to their starting lengths (host bookkeeping), so that a pass can be repeated.
The shapes are the repository's (paper_2605_13319_b200/synth: tiny, 1b, 7b, 8b), prefix and draft lengths those of its
benchmark and tests; weights and caches are random with the scales those use.  The final norm's gain is 8 instead of
1: next-token distributions are then about as peaked as a trained model's (most of the mass on a few tokens).
"""
import ctypes
import math

import numpy as np
import torch

from paper_2605_13319_b200 import binding, synth

STD = 0.02           # of every weight matrix
FINAL_GAIN = 8.0
PAGE = 16


def _verify(name, shape, n_req, prefix, k, *, mode="stochastic", q="device", commit="host", max_rows=32, mix=0):
    return dict(name=name, op="verify", shape=shape, n_req=n_req, prefix_lo=prefix[0], prefix_hi=prefix[1], k_lo=k[0],
                k_hi=k[1], mode=mode, q=q, commit=commit, max_rows=max_rows, mix=mix)


def _prefill(name, shape, n, *, max_rows=32):
    return dict(name=name, op="prefill", shape=shape, n=n, max_rows=max_rows)


def listed():
    return [
        # a toy target: nothing but latency and launches
        _verify("tiny-k4", "tiny", 1, (64, 64), (4, 4)),
        # a 1B-class target for one edge device, q resident on the device
        _verify("1b-k8", "1b", 1, (512, 512), (8, 8)),
        # the same with proactive transmission: two short drafts in flight, committed on the device
        _verify("1b-chain-k5", "1b", 1, (777, 777), (5, 5), commit="device"),
        # the headline: 7B target, 8 drafts; q arrives from the network in (pinned) host memory
        _verify("7b-k8", "7b", 1, (2048, 2048), (8, 8), q="host"),
        # long drafts (17 rows)
        _verify("7b-k16", "7b", 1, (2048, 2048), (16, 16)),
        # grouped-query attention, long context, 128k vocabulary
        _verify("8b-k16", "8b", 1, (8192, 8192), (16, 16)),
        # a handful of edge devices behind one small cloud model, greedy matching
        _verify("1b-batch5", "1b", 5, (100, 1500), (1, 16), mode="greedy", max_rows=96, mix=3),
        # multi-edge serving: ragged prefixes and drafts
        _verify("7b-batch16", "7b", 16, (256, 4096), (1, 16), q="host", max_rows=272, mix=1),
        _verify("8b-batch32", "8b", 32, (256, 4096), (1, 16), max_rows=544, mix=2),
        # prompts: a short odd one, the headline's prefix, and one on a server sized for batches
        _prefill("1b-prompt200", "1b", 203),
        _prefill("7b-prompt2048", "7b", 2048),
        _prefill("8b-prompt1500", "8b", 1500, max_rows=544),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    shape = rng.choice(["tiny", "1b", "7b", "8b"])
    top = {"tiny": 1024, "1b": 2048, "7b": 4096, "8b": 8192}[shape]
    kind = rng.choice(["single", "single", "batch", "prompt"])
    if kind == "prompt":
        n = _log_int(rng, 20, min(top, 1900))
        c = _prefill("", shape, n, max_rows=rng.choice([32, 32, 272, 544]))
    elif kind == "single":
        k, P = rng.randint(1, 16), _log_int(rng, 30, top)
        c = _verify("", shape, 1, (P, P), (k, k), mode=rng.choice(["stochastic", "stochastic", "greedy"]),
                    q=rng.choice(["device", "host"]), commit=rng.choice(["host", "host", "host", "device"]))
    else:
        n, hi = rng.randint(2, 12), _log_int(rng, 200, min(top, 4096))
        k_hi = rng.randint(2, 16)
        c = _verify("", shape, n, (max(20, hi // 16), hi), (1, k_hi), mode=rng.choice(["stochastic", "stochastic", "greedy"]),
                    q=rng.choice(["device", "host"]), max_rows=max(32, n * (k_hi + 1)), mix=rng.randint(0, 1 << 20))
    del c["name"]
    return c


def _requests(case):
    """Prefix and draft lengths of the case's requests."""
    lens, ks, _ = synth.ragged_requests(case["mix"], case["n_req"], case["prefix_lo"], case["prefix_hi"], case["k_lo"], case["k_hi"])
    return [int(x) for x in lens], [int(x) for x in ks]


# --------------------------------------------------------------------------- the server's side: model and caches
class Model:
    """A target model behind a context of the library, with random weights made on the GPU."""

    def __init__(self, shape, gen, n_pages, max_requests, max_rows, max_seq):
        self.lib, self.handle = binding.lib(), ctypes.c_void_p()
        dev = torch.device("cuda", 0)
        s = shape
        cfg = binding.ModelCfg(s.n_layers, s.d_model, s.n_q_heads, s.n_kv_heads, s.head_dim, s.d_ffn, s.vocab, s.rms_eps,
                               s.rope_base, PAGE, n_pages, max_requests, 16, max_rows, max_seq, 0, 0)
        size = binding.Sizes()
        self.check(self.lib.pipesd_query_sizes(ctypes.byref(cfg), ctypes.byref(size)))
        self.weights = torch.empty(size.weights_bytes, dtype=torch.uint8, device=dev)
        self.kv = torch.zeros(size.kv_bytes // 2, dtype=torch.bfloat16, device=dev)
        self.workspace = torch.zeros(size.workspace_bytes, dtype=torch.uint8, device=dev)
        keep = []

        def matrix(n, k):
            keep.append(torch.empty((n, k), dtype=torch.bfloat16, device=dev).normal_(0.0, STD, generator=gen))
            return keep[-1].data_ptr()

        def gain(v):
            keep.append(torch.full((s.d_model,), v, device=dev))
            return keep[-1].data_ptr()

        layers = (binding.LayerWeights * s.n_layers)()
        for l in layers:
            l.wq, l.wk, l.wv = matrix(s.q_dim, s.d_model), matrix(s.kv_dim, s.d_model), matrix(s.kv_dim, s.d_model)
            l.wo = matrix(s.d_model, s.q_dim)
            l.wg, l.wu, l.wd = matrix(s.d_ffn, s.d_model), matrix(s.d_ffn, s.d_model), matrix(s.d_model, s.d_ffn)
            l.attn_norm, l.ffn_norm = gain(1.0), gain(1.0)
        w = binding.Weights(matrix(s.vocab, s.d_model), matrix(s.vocab, s.d_model), gain(FINAL_GAIN), layers)
        mem = binding.Mem(self.weights.data_ptr(), size.weights_bytes, self.kv.data_ptr(), size.kv_bytes,
                          self.workspace.data_ptr(), size.workspace_bytes)
        stream = ctypes.c_void_p(torch.cuda.current_stream(dev).cuda_stream)
        self.check(self.lib.pipesd_ctx_create(ctypes.byref(cfg), ctypes.byref(w), ctypes.byref(mem), stream,
                                              ctypes.byref(self.handle)))
        self.check(self.lib.pipesd_ctx_sync(self.handle))     # the caller's weights may go now

    def check(self, rc):
        if rc != binding.OK:
            raise binding.PipesdError(rc, "perf case", self.lib.pipesd_last_error(self.handle).decode() if self.handle else "")

    def open(self):
        req = ctypes.c_int32()
        self.check(self.lib.pipesd_req_open(self.handle, ctypes.byref(req)))
        return req.value

    def __del__(self):
        if self.handle:
            self.lib.pipesd_ctx_destroy(self.handle)


def _write_prefix(model, shape, gen, reqs, lens):
    """Cached prefixes: random K and V rows (std 0.02 sqrt(d), what a prefill of these weights leaves behind).  One block
    of rows serves all: a request and layer take it from a row of their own."""
    rows = max(lens) + shape.n_layers + 8 * len(reqs)
    block = torch.empty((2, rows, shape.kv_dim), dtype=torch.bfloat16, pin_memory=True)
    block.copy_(torch.empty(block.shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, STD * math.sqrt(shape.d_model), generator=gen))
    for i, (req, P) in enumerate(zip(reqs, lens)):
        for layer in range(shape.n_layers):
            at = layer + 8 * i
            model.check(model.lib.pipesd_debug_write_kv(model.handle, req, layer, 0, P, block[0, at].data_ptr(), block[1, at].data_ptr()))


class Round:
    """The items of one pipesd_verify call and the arrays they point into."""

    def __init__(self, case, shape, reqs, ks, gen):
        greedy, n, V = case["mode"] == "greedy", len(reqs), shape.vocab
        self.items, self.results = (binding.VerifyItem * n)(), (binding.VerifyResult * n)()
        self.flags = 0
        rows = sum(ks) + n
        self.tokens = torch.randint(V, (rows,), dtype=torch.int32, device="cuda", generator=gen).cpu()
        self.u = (torch.randint(1 << 24, (rows,), device="cuda", generator=gen).float() * 2.0 ** -24).cpu()
        self.q = None
        if not greedy:
            # the edge model's distributions, as peaked as the target's; the drafts are drawn from them
            self.q = torch.empty((sum(ks), V), device="cuda").normal_(0.0, FINAL_GAIN * STD * math.sqrt(shape.d_model), generator=gen)
            self.q = torch.softmax(self.q, 1)
            drafts = torch.multinomial(self.q, 1, generator=gen)[:, 0].to(torch.int32).cpu()
            if case["q"] == "host":
                self.flags |= binding.Q_HOST
                self.q = torch.empty(self.q.shape, pin_memory=True).copy_(self.q)
        row = qrow = 0
        for i, (req, k) in enumerate(zip(reqs, ks)):
            if not greedy:
                self.tokens[row + 1:row + 1 + k] = drafts[qrow:qrow + k]
            self.items[i] = binding.VerifyItem(req, k, binding.MODE_GREEDY if greedy else binding.MODE_STOCHASTIC, 0,
                                               self.tokens[row:].data_ptr(), None if greedy else self.q[qrow:].data_ptr(),
                                               self.u[row:].data_ptr())
            row += k + 1
            qrow += k
        # results as the server reads them: (n_accepted, next_token, status, -) per request
        self.table = np.frombuffer(self.results, np.int32).reshape(n, 4)


class State:
    pass


def prepare(case, seed):
    shape = synth.SHAPES[case["shape"]]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    st = State()
    st.op, st.shape = case["op"], shape
    if case["op"] == "prefill":
        n = case["n"]
        st.model = Model(shape, gen, (n + PAGE - 1) // PAGE, 1, case["max_rows"], n)
        st.req, st.n = st.model.open(), n
        st.prompt = torch.randint(shape.vocab, (n,), dtype=torch.int32, device="cuda", generator=gen).cpu()
        st.logits = torch.zeros(shape.vocab, pin_memory=True)
        return st
    lens, ks = _requests(case)
    spare = 2 * (max(ks) + 1)                              # a pass and a chained one behind it
    st.model = Model(shape, gen, sum((P + spare) // PAGE + 1 for P in lens), len(lens), case["max_rows"], max(lens) + spare)
    st.reqs = [st.model.open() for _ in lens]
    st.reqs_np = np.array(st.reqs, np.int32)
    st.lens, st.rows = lens, sum(ks) + len(ks)
    _write_prefix(st.model, shape, gen, st.reqs, lens)
    st.rounds = [Round(case, shape, st.reqs, ks, gen)]
    st.rounds[0].flags |= binding.AUTOCOMMIT if case["commit"] == "device" else 0
    if case["commit"] == "device":
        st.rounds.append(Round(case, shape, st.reqs, ks, gen))
        st.rounds[1].flags |= binding.CHAIN
    st.device_commit = case["commit"] == "device"
    st.logits = torch.zeros((st.rows, shape.vocab), pin_memory=True)
    return st


def run(st):
    lib, h, check = st.model.lib, st.model.handle, st.model.check
    if st.op == "prefill":
        check(lib.pipesd_prefill(h, st.req, st.prompt.data_ptr(), st.n, st.logits.data_ptr()))
        check(lib.pipesd_debug_set_len(h, st.req, 0))
        return {"logits": st.logits, "kv": st.model.kv}
    for r in st.rounds:
        check(lib.pipesd_verify(h, len(st.reqs), r.items, r.results, r.flags))
    check(lib.pipesd_ctx_sync(h))
    check(lib.pipesd_debug_get_logits(h, st.logits.data_ptr(), st.rows))
    tables = [r.table.copy() for r in st.rounds]
    if not st.device_commit:
        accepted, token = (np.ascontiguousarray(tables[0][:, c]) for c in (0, 1))
        check(lib.pipesd_kv_rollback(h, len(st.reqs), st.reqs_np.ctypes.data, accepted.ctypes.data, token.ctypes.data))
    for req, P in zip(st.reqs, st.lens):
        check(lib.pipesd_debug_set_len(h, req, P))
    out = {"results": tables, "logits": st.logits}
    if len(st.reqs) == 1:
        out["kv"] = st.model.kv          # with the pass's own rows behind the prefix
    return out


def work(case):
    s = synth.SHAPES[case["shape"]]
    per_layer = (s.q_dim + 2 * s.kv_dim) * s.d_model + s.d_model * s.q_dim + 3 * s.d_ffn * s.d_model
    kv_row = 2 * s.n_layers * s.kv_dim * 2                       # bytes of one position's K and V
    head = s.vocab * s.d_model
    if case["op"] == "prefill":
        n = case["n"]
        pairs = n * (n + 1) / 2                                  # causal (query, key) pairs
        return {"bytes": 2 * (s.n_layers * per_layer + head) + 2 * n * s.d_model + kv_row * n + 4 * s.vocab,
                "flops": 2 * (n * s.n_layers * per_layer + head) + 4 * s.n_layers * s.q_dim * pairs}
    lens, ks = _requests(case)
    bytes_, flops = 0, 0
    for turn in range(2 if case["commit"] == "device" else 1):
        rows = sum(ks) + len(ks)
        cached = sum(lens) + turn * rows
        pairs = sum((P + turn * (k + 1)) * (k + 1) + (k + 1) * (k + 2) / 2 for P, k in zip(lens, ks))
        q = 4 * sum(ks) * s.vocab if case["mode"] == "stochastic" else 0
        bytes_ += 2 * (s.n_layers * per_layer + head) + 2 * rows * s.d_model + kv_row * (cached + rows) + 4 * rows * s.vocab + q
        flops += 2 * rows * (s.n_layers * per_layer + head) + 4 * s.n_layers * s.q_dim * pairs
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Activations are carried to 2^-17 and sums are fp32, but K and V are stored as bf16: where a value sits at a rounding
    boundary, two correct implementations store neighbours (2^-7 apart at most), and that is what later layers see.  A
    verify pass stores only its own rows that way, a prompt all of them, layer after layer.  Measured between two orders
    of summation (the library's two projection kernels; two chunk sizes of a prefill): logits up to 1.5e-4 and 2.1e-4
    relative, K/V up to 7.4e-4 (a prompt of the 7b shape), single K/V values by one bf16 step (7.8e-3)."""
    return {"rel": 3e-3 if case["op"] == "prefill" else 6e-4, "max": 3.2e-2}
