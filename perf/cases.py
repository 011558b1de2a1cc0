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


# --------------------------------------------------------------------------- inputs, from a generator alone
def _weights(s, gen):
    """Per layer a dict of matrices, the embedding table and the output matrix."""
    def matrix(n, k):
        return torch.empty((n, k), dtype=torch.bfloat16, device="cuda").normal_(0.0, STD, generator=gen)

    sizes = dict(wq=(s.q_dim, s.d_model), wk=(s.kv_dim, s.d_model), wv=(s.kv_dim, s.d_model), wo=(s.d_model, s.q_dim),
                 wg=(s.d_ffn, s.d_model), wu=(s.d_ffn, s.d_model), wd=(s.d_model, s.d_ffn))
    return [{n: matrix(*d) for n, d in sizes.items()} for _ in range(s.n_layers)], matrix(s.vocab, s.d_model), matrix(s.vocab, s.d_model)


def _prefix_block(s, gen, lens):
    """Cached prefixes: random K and V rows (std 0.02 sqrt(d), what a prefill of these weights leaves behind).  One block
    of rows serves all: a request and layer take it from a row of their own, _prefix_row."""
    rows = max(lens) + s.n_layers + 8 * len(lens)
    return torch.empty((2, rows, s.kv_dim), dtype=torch.bfloat16, device="cuda").normal_(0.0, STD * math.sqrt(s.d_model), generator=gen)


def _prefix_row(layer, i):
    return layer + 8 * i


def _round(case, s, ks, gen):
    """Tokens (pending and drafts) and uniforms of all rows; the edge model's distributions, as peaked as the target's,
    and the drafts drawn from them."""
    rows = sum(ks) + len(ks)
    tokens = torch.randint(s.vocab, (rows,), dtype=torch.int32, device="cuda", generator=gen).cpu()
    u = (torch.randint(1 << 24, (rows,), device="cuda", generator=gen).float() * 2.0 ** -24).cpu()
    q = None
    if case["mode"] != "greedy":
        q = torch.empty((sum(ks), s.vocab), device="cuda").normal_(0.0, FINAL_GAIN * STD * math.sqrt(s.d_model), generator=gen)
        q = torch.softmax(q, 1)
        drafts = torch.multinomial(q, 1, generator=gen)[:, 0].to(torch.int32).cpu()
        row = qrow = 0
        for k in ks:
            tokens[row + 1:row + 1 + k] = drafts[qrow:qrow + k]
            row, qrow = row + k + 1, qrow + k
    return tokens, u, q


def _prompt(case, s, gen):
    return torch.randint(s.vocab, (case["n"],), dtype=torch.int32, device="cuda", generator=gen).cpu()


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
        mats, emb, head = _weights(s, gen)
        one, final = (torch.full((s.d_model,), v, device=dev) for v in (1.0, FINAL_GAIN))
        layers = (binding.LayerWeights * s.n_layers)()
        for l, m in zip(layers, mats):
            for name, t in m.items():
                setattr(l, name, t.data_ptr())
            l.attn_norm = l.ffn_norm = one.data_ptr()
        w = binding.Weights(emb.data_ptr(), head.data_ptr(), final.data_ptr(), layers)
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
    block = _prefix_block(shape, gen, lens)
    block = torch.empty(block.shape, dtype=torch.bfloat16, pin_memory=True).copy_(block)
    for i, (req, P) in enumerate(zip(reqs, lens)):
        for layer in range(shape.n_layers):
            at = _prefix_row(layer, i)
            model.check(model.lib.pipesd_debug_write_kv(model.handle, req, layer, 0, P, block[0, at].data_ptr(), block[1, at].data_ptr()))


class Round:
    """The items of one pipesd_verify call and the arrays they point into."""

    def __init__(self, case, shape, reqs, ks, gen):
        greedy, n = case["mode"] == "greedy", len(reqs)
        self.items, self.results = (binding.VerifyItem * n)(), (binding.VerifyResult * n)()
        self.flags = 0
        self.tokens, self.u, self.q = _round(case, shape, ks, gen)
        if not greedy and case["q"] == "host":
            self.flags |= binding.Q_HOST
            self.q = torch.empty(self.q.shape, pin_memory=True).copy_(self.q)
        row = qrow = 0
        for i, (req, k) in enumerate(zip(reqs, ks)):
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
        st.prompt = _prompt(case, shape, gen)
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


class _Plain:
    """The model in 64-bit torch.  K and V are rounded to bf16 where they are cached: that is what the cache holds."""

    def __init__(self, shape, gen):
        self.s = shape
        self.layers, self.emb, self.head = _weights(shape, gen)
        self.cache = []                    # per request, per layer: [K, V], each [positions, kv heads, head_dim]

    def norm(self, x):
        return x * torch.rsqrt((x * x).mean(1, keepdim=True) + self.s.rms_eps)

    def forward(self, chunks):
        """The requests' next tokens (None: none); returns the rows after the last layer, final norm included."""
        s, hd, half, group = self.s, self.s.head_dim, self.s.head_dim // 2, self.s.n_q_heads // self.s.n_kv_heads
        sizes = [len(c) for c in chunks]
        starts = [self.cache[i][0][0].shape[0] for i in range(len(chunks))]
        pos = torch.cat([torch.arange(p, p + n, device="cuda", dtype=torch.float64) for p, n in zip(starts, sizes)])
        angle = pos[:, None, None] * float(s.rope_base) ** (-torch.arange(half, device="cuda", dtype=torch.float64) * 2 / hd)
        c, z = angle.cos(), angle.sin()

        def turn(v):
            a, b = v[..., :half], v[..., half:]
            return torch.cat([a * c - b * z, b * c + a * z], -1)

        x = self.emb[torch.cat(chunks).long().cuda()].double()
        for l, m in enumerate(self.layers):
            h = self.norm(x)
            q, k, v = ((h @ m[n].double().T).view(len(x), -1, hd) for n in ("wq", "wk", "wv"))
            q, k, v = turn(q), turn(k).bfloat16().double(), v.bfloat16().double()
            out, at = [], 0
            for i, (p, n) in enumerate(zip(starts, sizes)):
                kv = self.cache[i][l] = [torch.cat([old, new[at:at + n]]) for old, new in zip(self.cache[i][l], (k, v))]
                kk, vv = (t.repeat_interleave(group, 1).transpose(0, 1) for t in kv)
                score = q[at:at + n].transpose(0, 1) @ kk.transpose(1, 2) / math.sqrt(hd)
                later = torch.arange(p + n, device="cuda")[None, :] > torch.arange(p, p + n, device="cuda")[:, None]
                out.append((score.masked_fill_(later, -math.inf).softmax(2) @ vv).transpose(0, 1).reshape(n, -1))
                del kk, vv, score
                at += n
            x = x + torch.cat(out) @ m["wo"].double().T
            h = self.norm(x)
            x = x + (torch.nn.functional.silu(h @ m["wg"].double().T) * (h @ m["wu"].double().T)) @ m["wd"].double().T
        return self.norm(x) * FINAL_GAIN

    def logits(self, rows):
        return torch.cat([rows @ w.double().T for w in self.head.split(16384)], 1)

    def pool(self, n_pages):
        """The first request's cache as the library lays it out (include/pipesd.h, pages handed out in order)."""
        s, out = self.s, torch.zeros((self.s.n_layers, n_pages, 2, self.s.n_kv_heads, PAGE // 8, self.s.head_dim // 8, 8, 8), dtype=torch.float64)
        for l, kv in enumerate(self.cache[0]):
            for j, t in enumerate(kv):
                t = torch.nn.functional.pad(t, (0, 0, 0, 0, 0, n_pages * PAGE - t.shape[0]))
                out[l, :, j] = t.view(n_pages, PAGE // 8, 8, s.n_kv_heads, s.head_dim // 8, 8).permute(0, 3, 1, 4, 2, 5).cpu()
        return out.view(-1)


def exact(case, seed):
    """`run` in 64 bits: logits, and the cache of a single request.  Decisions (whole numbers) are left out."""
    s = synth.SHAPES[case["shape"]]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    m = _Plain(s, gen)
    empty = torch.zeros((0, s.n_kv_heads, s.head_dim), dtype=torch.float64, device="cuda")
    if case["op"] == "prefill":
        m.cache = [[[empty, empty] for _ in range(s.n_layers)]]
        rows = m.forward([_prompt(case, s, gen)])
        return {"logits": m.logits(rows[-1:])[0].cpu(), "kv": m.pool((case["n"] + PAGE - 1) // PAGE)}
    lens, ks = _requests(case)
    block = _prefix_block(s, gen, lens)
    for i, P in enumerate(lens):
        m.cache.append([[block[j, _prefix_row(l, i):_prefix_row(l, i) + P].double().view(P, s.n_kv_heads, s.head_dim) for j in (0, 1)]
                        for l in range(s.n_layers)])
    turns = 2 if case["commit"] == "device" else 1
    for tokens in [_round(case, s, ks, gen)[0] for _ in range(turns)]:
        rows = m.forward(list(tokens.split([k + 1 for k in ks])))
    out = {"results": [None] * turns, "logits": m.logits(rows).cpu()}
    if len(ks) == 1:
        out["kv"] = m.pool((lens[0] + 2 * (max(ks) + 1)) // PAGE + 1)
    return out


def tolerance(case):
    """Activations are carried to 2^-17 and sums are fp32, but K and V are stored as bf16: where a value sits at a rounding
    boundary, two correct implementations store neighbours (2^-7 apart at most), and that is what later layers see.  A
    verify pass stores only its own rows that way, a prompt all of them, layer after layer.  Measured between two orders
    of summation (the library's two projection kernels; two chunk sizes of a prefill): logits up to 1.5e-4 and 2.1e-4
    relative, K/V up to 7.4e-4 (a prompt of the 7b shape), single K/V values by one bf16 step (7.8e-3)."""
    return {"rel": 3e-3 if case["op"] == "prefill" else 6e-4, "max": 3.2e-2}
