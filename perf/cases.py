"""The work that users of this library have it do, as cases to be timed: decode steps of whole stacks over a latent
cache (every layer's new K/V rows encoded and appended, then attention over the cache through kvcar_step_layer) and
bulk encoding of prompts.  Shapes: the GPT-2-small-shaped stack (12 layers, 12 heads) and the TinyLLaMA-1.1B-shaped
grouped-query stack (22 layers, 32 query / 4 KV heads), the autoencoders halving K and V, a share of the heads reading
the layer below.

A decode case does not advance the sequences, so that it can be run again on the same state: every pass appends at the
same positions.  A prefill case opens its sequences, encodes and closes them again, as a server does with a request.
"""
from __future__ import annotations

import math

import torch

from paper_2512_06727_b200 import binding as B
from paper_2512_06727_b200.session import Session

HEAD_DIM = 64
PAGE = 64
# layers, query heads, KV heads, latent elements per stored head, share of the heads of layers >= 1 that reuse the layer below
SHAPES = {
    "gpt2": (12, 12, 12, 32, 0.25),
    "tinyllama": (22, 32, 4, 32, 0.20),
}


def _decode(name, shape, batch, tokens, **more):
    c = {"name": name, "do": "decode", "shape": shape, "store": "bf16", "batch": batch, "tokens": tokens,
         "ragged": False, "host": False, "layers": SHAPES[shape][0]}
    return {**c, **more}


def _prefill(name, shape, batch, tokens, tensor):
    return {"name": name, "do": "prefill", "shape": shape, "store": "bf16", "batch": batch, "tokens": tokens,
            "tensor": tensor, "layers": SHAPES[shape][0]}


def listed():
    return [
        # one user, a short conversation: the smallest call, all latency and launches
        _decode("gpt2 step b1 t200", "gpt2", 1, 200),
        # a small batch at the full context of the GPT-2 shape
        _decode("gpt2 step b8 t1024", "gpt2", 8, 1024),
        # the same step for a caller whose K, V and q are in host memory and who reads the outputs there
        _decode("gpt2 step b8 t1024 host", "gpt2", 8, 1024, host=True),
        # a serving batch: sequences of every length up to the longest
        _decode("gpt2 step b32 ragged", "gpt2", 32, 4096, ragged=True),
        # the largest batch: throughput
        _decode("gpt2 step b256 t4096", "gpt2", 256, 4096),
        # grouped-query attention, a serving batch
        _decode("tinyllama step b32 t2048", "tinyllama", 32, 2048),
        # grouped-query attention, long documents
        _decode("tinyllama step b4 t32768", "tinyllama", 4, 32768),
        # layers without autoencoders: the uncompressed cache, with head reuse
        _decode("gpt2 raw step b32 t4096", "gpt2", 32, 4096, store="raw"),
        # int8 latent rows: the smallest cache
        _decode("gpt2 int8 step b8 t1024", "gpt2", 8, 1024, store="int8"),
        # fp32 storage: one layer, as a numerics check runs it
        _decode("gpt2 f32 layer b1 t128", "gpt2", 1, 128, store="f32", layers=1),
        # prompts of a batch encoded in one call per layer, fp32 between the encoder's two layers
        _prefill("gpt2 prefill b8 t1024", "gpt2", 8, 1024, False),
        # the same through the bf16 tensor-core encoder, at its usual size
        _prefill("tinyllama prefill tensor b32 t1024", "tinyllama", 32, 1024, True),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gpt2", "gpt2", "gpt2", "tinyllama", "tinyllama", "raw", "int8", "f32", "prefill", "prefill tensor"])
    if kind in ("gpt2", "tinyllama", "raw"):
        shape = "gpt2" if kind == "raw" else kind
        most = {"gpt2": 4096, "tinyllama": 32768, "raw": 4096}[kind]
        tokens = _log(rng, 17, most)
        batch = _log(rng, 1, max(1, min(256 if kind == "gpt2" else 32, (1 << 17) // tokens if kind != "gpt2" else 256)))
        c = _decode("", shape, batch, tokens, ragged=rng.random() < 0.4, store="raw" if kind == "raw" else "bf16",
                    host=kind != "raw" and batch <= 32 and rng.random() < 0.2)
    elif kind == "int8":
        tokens = _log(rng, 17, 2048)
        c = _decode("", "gpt2", _log(rng, 1, max(1, min(16, 8192 // tokens))), tokens, store="int8", ragged=rng.random() < 0.4)
    elif kind == "f32":
        c = _decode("", "gpt2", rng.randint(1, 4), _log(rng, 17, 512), store="f32", layers=rng.randint(1, 2))
    else:
        tokens = _log(rng, 30, 2048)
        c = _prefill("", rng.choice(["gpt2", "tinyllama"]), _log(rng, 1, max(1, min(32, 32768 // tokens))), tokens,
                     kind.endswith("tensor"))
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------------- the stack
def _reuse_map(case):
    """-1 = the head keeps its own rows, else the head of the layer below that it reads; the same spread every time."""
    layers, _, hkv, _, frac = SHAPES[case["shape"]]
    src = [-1] * (case["layers"] * hkv)
    if case["store"] == "f32":
        return src
    cand = [(l, h) for l in range(1, case["layers"]) for h in range(hkv)]
    g = torch.Generator().manual_seed(1)
    order = torch.randperm(len(cand), generator=g).tolist()
    for i in order[:int(frac * len(cand) + 0.5)]:
        l, h = cand[i]
        src[l * hkv + h] = h
    return src


def _autoencoders(case, src, g):
    """Random-init autoencoders over the heads each layer stores: Xavier-uniform weights, BatchNorm statistics of a
    trained layer's order; on the storage grid."""
    _, _, hkv, per_head, _ = SHAPES[case["shape"]]
    out = {}

    def uniform(a, *shape):
        return (torch.rand(*shape, generator=g, device="cuda") * 2 - 1) * a

    def matrix(rows, cols):
        w = uniform(math.sqrt(6.0 / (rows + cols)), rows, cols)
        return w if case["store"] == "f32" else w.bfloat16().float()

    def norm(n):
        u = torch.rand(4, n, generator=g, device="cuda")
        z = torch.randn(4, n, generator=g, device="cuda") * 0.1
        return torch.stack([u[0] + 0.5, z[1], z[2], u[3] + 0.5])

    for l in range(case["layers"]):
        n = sum(1 for h in range(hkv) if src[l * hkv + h] < 0)
        i, d = n * HEAD_DIM, n * per_head
        m = (i + d) // 2
        for which in (B.K, B.V):
            if n == 0:
                continue
            ae = {"enc_w1": matrix(m, i), "enc_b1": uniform(i ** -0.5, m), "enc_bn": norm(m), "enc_w2": matrix(d, m),
                  "enc_b2": uniform(m ** -0.5, d), "dec_w1": matrix(m, d), "dec_b1": uniform(d ** -0.5, m),
                  "dec_bn": norm(m), "dec_w2": matrix(i, m), "dec_b2": uniform(m ** -0.5, i)}
            out[(l, which)] = {**{k: v.cpu().numpy() for k, v in ae.items()}, "in_dim": i, "hidden": m, "latent": d,
                               "leaky_slope": 0.01, "bn_eps": 1e-5}
    return out


def _lengths(case):
    n, top = case["batch"], case["tokens"]
    if not case.get("ragged"):
        return [top] * n
    g = torch.Generator().manual_seed(7)
    return [max(1, int(top * x)) for x in (0.05 + 0.95 * torch.rand(n, generator=g)).tolist()]


_weights = []   # the weights buffers of every context made so far


def _session(case, seqs, pages_per_seq, g):
    _, hq, hkv, _, _ = SHAPES[case["shape"]]
    src = _reuse_map(case)
    aes = {} if case["store"] == "raw" else _autoencoders(case, src, g)
    sess = Session(case["layers"], hq, hkv, HEAD_DIM, PAGE, seqs, seqs * pages_per_seq, pages_per_seq,
                   "f32" if case["store"] == "f32" else "bf16", src, src, aes, latent_quant=case["store"] == "int8")
    # A program makes its context once.  Here many follow one another, and the tensor maps that the kernels read lie in
    # the weights buffer: its memory is not handed out again, so that no map of an earlier context is met there.
    _weights.append(sess.weights)
    return sess


def _rows(sess, g, *shape):
    return torch.randn(*shape, generator=g, device="cuda").to(sess.dtype)


def _pool(sess, rows=slice(None)):
    """The cache rows of every (layer, K/V) that stores any (int8 rows: their scales and zero-points too)."""
    out = []
    for l in range(sess.ctx.cfg.n_layers):
        for which in (B.K, B.V):
            if sess.ctx.pool_layout(l, which)[2] == 0:
                continue
            out.append(sess.pool_rows(l, which)[rows])
            if sess.latent_quant:
                out.append(sess.pool_quant_params(l, which)[rows])
    return out


# ---------------------------------------------------------------------------------------------------- decode steps
def _fill(sess, case, lens, g):
    """The cached tokens, through the library's own encoder; then one page per sequence for the row a step appends.
    The pages being appended to are taken together, last, so that they lie side by side in the pools."""
    ctx = sess.ctx
    width = sess.ctx.cfg.n_kv_heads * HEAD_DIM
    call = ctx.encode_append_tensor if case["store"] == "bf16" else ctx.encode_append
    seqs = list(range(len(lens)))

    def append(which_seqs, n):
        k, v = (_rows(sess, g, len(which_seqs), n, width) for _ in range(2))
        for l in range(case["layers"]):
            # another layer's rows: the same numbers, other places (drawing each layer's own would take most of the time)
            kl, vl = k.roll(l, 1), v.roll(-l, 1)
            call(l, which_seqs, n, kl.data_ptr(), vl.data_ptr(), sess.stream())
        ctx.advance(which_seqs, n, sess.stream())

    whole = [n // PAGE * PAGE for n in lens]
    if len(set(whole)) == 1:
        done, most = 0, max(PAGE, (1 << 15) // len(seqs) // PAGE * PAGE)
        while done < whole[0]:
            n = min(most, whole[0] - done)
            append(seqs, n)
            done += n
    else:
        for s in seqs:
            if whole[s]:
                append([s], whole[s])
    tail = sum(whole) // PAGE
    ctx.reserve(seqs, PAGE)
    if len(set(lens)) == 1:
        if lens[0] > whole[0]:
            append(seqs, lens[0] - whole[0])
    else:
        for s in seqs:
            if lens[s] > whole[s]:
                append([s], lens[s] - whole[s])
    return slice(tail * PAGE, (tail + len(seqs)) * PAGE)


def _prepare_decode(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    _, hq, hkv, _, _ = SHAPES[case["shape"]]
    lens = _lengths(case)
    sess = _session(case, case["batch"], case["tokens"] // PAGE + 1, g)
    for s in range(case["batch"]):
        sess.ctx.seq_open(s)
    tail = _fill(sess, case, lens, g)
    k, v = (_rows(sess, g, case["layers"], case["batch"], hkv * HEAD_DIM) for _ in range(2))
    q = _rows(sess, g, case["layers"], case["batch"], hq, HEAD_DIM)
    if case["host"]:
        k, v, q = (x.cpu().pin_memory() for x in (k, v, q))
    out = torch.empty_like(q, pin_memory=True) if case["host"] else torch.empty_like(q)
    sess.ctx.sync_status(sess.stream())
    at = [(k[l].data_ptr(), v[l].data_ptr(), q[l].data_ptr(), out[l].data_ptr()) for l in range(case["layers"])]
    return {"do": "decode", "host": case["host"], "sess": sess, "seqs": list(range(case["batch"])), "at": at,
            "keep": (k, v, q), "back": {"out": out, "rows": _pool(sess, tail)}}


def _run_decode(state):
    sess, seqs = state["sess"], state["seqs"]
    stream = sess.stream()
    step = sess.ctx.step_layer_host if state["host"] else sess.ctx.step_layer
    for l, (k, v, q, out) in enumerate(state["at"]):
        step(l, seqs, k, v, q, out, B.INCLUDE_CURRENT_EXACT, stream)
    if state["host"]:       # the caller reads the outputs in its own memory
        torch.cuda.current_stream().synchronize()
    return state["back"]


# ---------------------------------------------------------------------------------------------------- prompts
def _prepare_prefill(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    hkv = SHAPES[case["shape"]][2]
    sess = _session(case, case["batch"], (case["tokens"] + PAGE - 1) // PAGE, g)
    k, v = (_rows(sess, g, case["layers"], case["batch"], case["tokens"], hkv * HEAD_DIM) for _ in range(2))
    return {"do": "prefill", "tensor": case["tensor"], "tokens": case["tokens"], "sess": sess,
            "seqs": list(range(case["batch"])), "keep": (k, v),
            "at": [(k[l].data_ptr(), v[l].data_ptr()) for l in range(case["layers"])], "back": _pool(sess)}


def _run_prefill(state):
    ctx, seqs, n = state["sess"].ctx, state["seqs"], state["tokens"]
    stream = state["sess"].stream()
    for s in seqs:
        ctx.seq_open(s)
    encode = ctx.encode_append_tensor if state["tensor"] else ctx.encode_append
    for l, (k, v) in enumerate(state["at"]):
        encode(l, seqs, n, k, v, stream)
    ctx.advance(seqs, n, stream)
    # the request ends: closing in reverse order hands every sequence its own pages again in the next pass
    for s in reversed(seqs):
        ctx.seq_close(s)
    return state["back"]


def prepare(case, seed):
    return _prepare_decode(case, seed) if case["do"] == "decode" else _prepare_prefill(case, seed)


def run(state):
    return _run_decode(state) if state["do"] == "decode" else _run_prefill(state)


# ---------------------------------------------------------------------------------------------------- what it takes
def work(case):
    """Bytes: cache rows of every distinct source layer, each layer's weights, the step's K, V, q and outputs, once
    each.  Operations: the encoder of the new rows; per cached token and source the first decoder layer, and the last
    one (linear) either applied to the restored heads or moved to the query side and the weighted sum, whichever is
    fewer; the attention products."""
    _, hq, hkv, per_head, _ = SHAPES[case["shape"]]
    src, L, elem = _reuse_map(case), case["layers"], 4 if case["store"] == "f32" else 2
    raw, group = case["store"] == "raw", hq // hkv
    stored = [sum(1 for h in range(hkv) if src[l * hkv + h] < 0) for l in range(L)]
    width = [n * HEAD_DIM if raw else n * per_head for n in stored]
    hidden = [(n * HEAD_DIM + n * per_head) // 2 for n in stored]
    enc = [0 if raw else stored[l] * HEAD_DIM * hidden[l] + hidden[l] * width[l] for l in range(L)]   # parameters of one half
    row_elem = 1 if case["store"] == "int8" else elem
    row_more = 8 if case["store"] == "int8" else 0
    by = fl = 0.0
    if case["do"] == "prefill":
        rows = case["batch"] * case["tokens"]
        for l in range(L):
            by += 2 * (rows * (stored[l] * HEAD_DIM * elem + width[l] * row_elem + row_more) + enc[l] * elem)
            fl += 2 * rows * 2 * enc[l]
        return {"bytes": by, "flops": fl}
    tokens, rows = float(sum(_lengths(case))), case["batch"]
    for l in range(L):
        roots = {}
        for h in range(hkv):
            r = l
            while src[r * hkv + h] >= 0:
                r -= 1
            roots[r] = roots.get(r, 0) + 1
        by += rows * elem * HEAD_DIM * 2 * (hkv + hq)
        for r, n in roots.items():
            if raw:
                by += 2 * tokens * n * HEAD_DIM * elem
            else:
                by += 2 * (tokens * (width[r] * row_elem + row_more) + (enc[r] + (enc[l] if r == l else 0)) * elem)
                fl += 2 * tokens * (2 * width[r] * hidden[r] + 2 * hidden[r] * min(n * HEAD_DIM, n * group))
        if raw:
            fl += tokens * 4 * hq * HEAD_DIM
        fl += 2 * rows * 2 * enc[l]
        by += 2 * rows * (width[l] * row_elem + row_more)
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """bf16: outputs lie 1.7e-3 (2-norm) from the fp64 oracle; fp32: a few 1e-6, the order of sums of 64 to 768 terms."""
    if case["store"] == "f32":
        return {"rel": 1e-5, "max": 1e-3}
    if case["store"] == "int8":
        # a code on a rounding boundary may fall on either side
        return {"rel": 8e-3, "max": 0.2, "differ": 2e-3}
    return {"rel": 8e-3, "max": 0.2}
