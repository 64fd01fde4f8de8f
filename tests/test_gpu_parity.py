"""GPU parity: the CUDA library against the CPU oracle, element by element, on
the same seeded inputs, through the C ABI.  Sizes are chosen so that the oracle
finishes in seconds while the kernels still see several tiles, several pages and
ragged tails."""
import numpy as np
import pytest
import torch

import kvcar_synth as synth
from kvcar_harness import Pair, assert_close
from oracle.kvcar_oracle import K, V
from paper_2512_06727_b200 import binding as B

pytestmark = pytest.mark.gpu

KERNELS = [B.KERNEL_GENERIC, B.KERNEL_AUTO]
KNAME = {B.KERNEL_GENERIC: "generic", B.KERNEL_AUTO: "auto"}


def _check_step(res, storage, what):
    worst = 0.0
    for l, (got, ref, rows) in res.items():
        err, rel = assert_close(got[rows], ref, storage, f"{what} layer {l}")
        worst = max(worst, err)
    return worst


def test_config1_fp32_single_layer():
    """Configuration 1 exactly: one GPT-2-small-shaped layer, 768->384, batch 1,
    128 cached tokens, one decode step, fp32, no reuse; max abs error <= 1e-4."""
    w = synth.CONFIGS["c1"]
    p = Pair(w, max_seqs=1, max_pages=4, max_pages_per_seq=4)
    p.open([0])
    p.prefill([0], w.cached_tokens)
    p.check_latents([0])
    res = p.decode_step([0], 0)
    got, ref, rows = res[0]
    err, rel = assert_close(got[rows], ref, "f32", "config 1")
    assert err <= 1e-4
    assert p.s.ctx.cache_bytes_per_token() == (2 * 384 * 4, 2 * 768 * 4)


@pytest.mark.parametrize("kernel", KERNELS, ids=lambda k: KNAME[k])
def test_gpt2_shape_stack_bf16_with_reuse(kernel):
    """Config-2-shaped stack (12 layers x 12 heads, latent 32/head, 25 % reuse),
    reduced batch and ragged lengths, two decode steps with encode-append."""
    w = synth.scaled(synth.CONFIGS["c2"], batch=3, cached_tokens=0, decode_steps=2)
    p = Pair(w, max_seqs=4, max_pages=16, max_pages_per_seq=5, kernel=kernel)
    seqs = [2, 0, 3]
    p.open(seqs)
    p.prefill([2], 200)
    p.prefill([0], 131)
    p.prefill([3], 64)
    p.check_latents(seqs)
    if kernel == B.KERNEL_AUTO:     # the bf16 stack must really run on the tensor-core kernel
        assert all(p.s.ctx.layer_kernel(l) == B.KERNEL_TENSOR for l in range(w.n_layers))
    for step in range(2):
        _check_step(p.decode_step(seqs, step), "bf16", f"step {step}")
    p.check_latents(seqs)
    assert p.s.ctx.cache_bytes_per_token() == p.o.cache_bytes_per_token()


@pytest.mark.parametrize("kernel", KERNELS, ids=lambda k: KNAME[k])
def test_tinyllama_shape_gqa_stack_bf16_with_reuse(kernel):
    """Config-3-shaped GQA stack (22 layers, 32 query / 4 KV heads, latent 32/head,
    20 % reuse), K and V reuse maps different, ragged lengths incl. 1 token."""
    w = synth.scaled(synth.CONFIGS["c3"], batch=4, cached_tokens=0, decode_steps=2)
    src_k = synth.make_reuse_map(w.n_layers, w.n_kv_heads, w.reuse_frac, w.seed)
    src_v = synth.make_reuse_map(w.n_layers, w.n_kv_heads, w.reuse_frac, w.seed + 7)
    p = Pair(w, max_seqs=4, max_pages=20, max_pages_per_seq=6, src_k=src_k, src_v=src_v, kernel=kernel)
    seqs = [0, 1, 2, 3]
    p.open(seqs)
    for s, n in zip(seqs, (300, 257, 128, 1)):
        p.prefill([s], n)
    p.check_latents(seqs)
    if kernel == B.KERNEL_AUTO:
        assert all(p.s.ctx.layer_kernel(l) == B.KERNEL_TENSOR for l in range(w.n_layers))
    for step in range(2):
        _check_step(p.decode_step(seqs, step), "bf16", f"step {step}")


@pytest.mark.parametrize("kernel", KERNELS, ids=lambda k: KNAME[k])
def test_peaked_softmax_and_planted_key(kernel):
    """N(0,1) inputs give near-uniform softmax, under which a token-indexing bug
    hardly moves the output: repeat with queries scaled x8 and with one cached key
    made proportional to the query."""
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=3, batch=2, cached_tokens=0, decode_steps=1, reuse_frac=0.34)
    p = Pair(w, max_seqs=2, max_pages=12, max_pages_per_seq=6, kernel=kernel)
    seqs = [0, 1]
    p.open(seqs)
    p.prefill(seqs, 333)
    res = p.decode_step(seqs, 0, q_scale=8.0)
    _check_step(res, "bf16", "q x8")
    # the softmax really is peaked: the largest probability of some head exceeds 0.5
    out, probs = p.o.decode_attention(2, [0], np.stack([synth.make_q(w, 2, 0, 0, scale=8.0)]),
                                      include_current=False, return_probs=True)
    assert max(float(pr.max()) for pr in probs) > 0.5
    # planted key: make token 77's pre-compression K of every head a multiple of one query head, raw layer 0
    w2 = synth.scaled(w, n_layers=1, reuse_frac=0.0)
    p2 = Pair(w2, max_seqs=1, max_pages=4, max_pages_per_seq=4, compress=False, kernel=kernel)
    p2.open([0])
    q = synth.make_q(w2, 0, 0, 0)
    k = synth.make_kv(w2, 0, K, 0, 0, 150)[None].copy()
    v = synth.make_kv(w2, 0, V, 0, 0, 150)[None].copy()
    for g in range(w2.n_kv_heads):
        k[0, 77, g * 64:(g + 1) * 64] = synth.to_bf16_grid(6.0 * q[g * 8])
    p2.append(0, [0], k, v)
    p2.advance([0], 150)
    got, ref, rows = p2.attention(0, [0], q[None], include_current=False)
    assert_close(got, ref, "bf16", "planted key")
    for g in range(w2.n_kv_heads):   # head g*8 attends almost only to token 77
        assert np.max(np.abs(got[0, g * 8] - v[0, 77, g * 64:(g + 1) * 64])) < 0.05


@pytest.mark.parametrize("kernel", KERNELS, ids=lambda k: KNAME[k])
def test_edge_cases_empty_current_only_and_single_token(kernel):
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, batch=3, reuse_frac=0.5)
    p = Pair(w, max_seqs=3, max_pages=8, max_pages_per_seq=3, kernel=kernel)
    seqs = [0, 1, 2]
    p.open(seqs)
    p.prefill([1], 1)
    p.prefill([2], 65)
    # seq 0 has nothing cached: with the current token the output is that token's exact V
    res = p.decode_step(seqs, 0)
    _check_step(res, "bf16", "current only")
    # nothing cached and no current token: zeros
    p3 = Pair(w, max_seqs=1, max_pages=2, max_pages_per_seq=2, kernel=kernel)
    p3.open([0])
    got, ref, rows = p3.attention(0, [0], synth.make_q(w, 0, 0, 0)[None], include_current=False)
    assert np.all(got == 0) and np.all(ref == 0)
    # cached tokens only (current token attended through its latent after advance)
    got, ref, rows = p.attention(1, seqs, np.stack([synth.make_q(w, 1, s, 9) for s in seqs]), include_current=False)
    assert_close(got, ref, "bf16", "cached only")


@pytest.mark.parametrize("kernel", KERNELS, ids=lambda k: KNAME[k])
def test_uncompressed_twin_and_mixed_stack(kernel):
    """No autoencoders (raw K/V pages, reuse still redirects heads) and a stack
    with autoencoders in some layers only (Table 2's "N layers" rows)."""
    w = synth.scaled(synth.CONFIGS["c2"], n_layers=4, batch=2, reuse_frac=0.3)
    for layers, compress in ((None, False), ([1, 2], True)):
        p = Pair(w, max_seqs=2, max_pages=8, max_pages_per_seq=4, compressed_layers=layers, compress=compress,
                 kernel=kernel)
        p.open([0, 1])
        p.prefill([0], 190)
        p.prefill([1], 70)
        p.check_latents([0, 1])
        _check_step(p.decode_step([0, 1], 0), "bf16", f"layers={layers}")
        assert p.s.ctx.cache_bytes_per_token() == p.o.cache_bytes_per_token()


@pytest.mark.parametrize("heads", [(32, 4), (12, 4), (6, 2)], ids=["group8", "group3", "group3_two_kv_heads"])
def test_uncompressed_twin_with_query_groups(heads):
    """Raw K/V pages with several query heads per KV head: the streaming kernel runs the group's dots on the
    warp-level tensor op (groups of more than two heads).  Ragged tiles: a 32-token step that ends inside a tile,
    a tile of one token, page boundaries inside a step; reuse redirects heads to the lower layer's rows."""
    hq, hkv = heads
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=3, n_q_heads=hq, n_kv_heads=hkv, batch=4, reuse_frac=0.4)
    p = Pair(w, max_seqs=4, max_pages=24, max_pages_per_seq=8, compress=False)
    seqs = [0, 1, 2, 3]
    p.open(seqs)
    for s_, n in zip(seqs, (300, 129, 33, 1)):
        p.prefill([s_], n)
    assert all(p.s.ctx.layer_kernel(l) == B.KERNEL_RAW for l in range(w.n_layers))
    for step in range(2):
        _check_step(p.decode_step(seqs, step), "bf16", f"raw group {hq // hkv} step {step}")


@pytest.mark.parametrize("cfg,slope,int8", [("c2", 0.01, False), ("c2", 1.5, False), ("c2", 1.5, True), ("c3", 1.5, False)])
def test_runs_of_several_tiles(cfg, slope, int8):
    """More tiles than blocks, so that each walks several (the K side one tile ahead) across sequence ends and partial tiles; slopes of
    both sides of 1, of which the upper one is turned round when the weights are laid out.  Three sequences against the oracle."""
    w = synth.scaled(synth.CONFIGS[cfg], n_layers=2, batch=48, reuse_frac=0.3)
    seqs = list(range(48))
    lens = [128 * (5 * s % 8) + (1, 127, 128, 60)[s % 4] for s in seqs]
    assert sum((n + 127) // 128 for n in lens) > 148
    p = Pair(w, max_seqs=48, max_pages=48 * 17, max_pages_per_seq=17, ae_kwargs={"leaky_slope": slope}, latent_quant=int8)
    p.oracle_seqs = {0, 23, 47}
    p.open(seqs)
    for s_, n in zip(seqs, lens):
        p.prefill([s_], n)
    assert all(p.s.ctx.layer_kernel(l) == B.KERNEL_TENSOR for l in range(w.n_layers))
    for step in range(2):
        for l, (got, ref, rows) in p.decode_step(seqs, step, fused=True).items():
            # the bound of slope 0.01 grows with the hidden vector, half of whose features the slope multiplies: rms sqrt((1 + slope^2) / 2)
            grow = max(1.0, (1 + slope * slope) ** 0.5)
            what = f"{cfg} slope {slope} int8 {int8} step {step} layer {l}"
            assert_close(got[rows] / grow, ref / grow, "bf16", what)


@pytest.mark.parametrize("batch", [24, 25])
def test_fp32_merge_on_both_block_sizes(batch):
    """12 heads x 24 sequences merge in blocks of 1024 threads, 12 x 25 (more than two per SM) in blocks of 256."""
    w = synth.scaled(synth.CONFIGS["c2"], n_layers=1, batch=batch, storage="f32", reuse_frac=0.0)
    seqs = list(range(batch))
    p = Pair(w, max_seqs=batch, max_pages=2 * batch, max_pages_per_seq=2)
    p.oracle_seqs = {0, 7, batch - 1}
    p.open(seqs)
    for s_ in seqs:
        p.prefill([s_], (1, 31, 64, 100)[s_ % 4])
    _check_step(p.decode_step(seqs, 0, fused=True), "f32", f"batch {batch}")


@pytest.mark.parametrize("storage,page_tokens,batch", [("bf16", 64, 1), ("bf16", 16, 5), ("bf16", 64, 33), ("f32", 64, 5)])
def test_uncompressed_single_call_steps(storage, page_tokens, batch):
    """Raw layers through the single call, whose tile launch also appends the rows: pages of less than a 32-token step (plain copies)
    and more (tensor loads), fp32 rows, lengths on both sides of a step, a tile and a page."""
    w = synth.scaled(synth.CONFIGS["c2"], n_layers=2, storage=storage, page_tokens=page_tokens, batch=batch, reuse_frac=0.3)
    seqs = list(range(batch))
    lens = [(1, 127, 128, 31, 65)[s % 5] for s in seqs]
    per = (130 + page_tokens) // page_tokens + 1
    p = Pair(w, max_seqs=batch, max_pages=batch * per, max_pages_per_seq=per, compress=False)
    p.open(seqs)
    for s_, n in zip(seqs, lens):
        p.prefill([s_], n)
    for step in range(2):
        _check_step(p.decode_step(seqs, step, fused=True), storage, f"raw {storage} page {page_tokens} batch {batch} step {step}")
    p.check_latents(seqs)


@pytest.mark.parametrize("kernel", KERNELS, ids=lambda k: KNAME[k])
def test_physical_page_permutation_is_bit_invariant(kernel):
    """The same logical cache laid out on different physical pages must give
    bit-identical outputs."""
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, batch=1, reuse_frac=0.25)

    def run(scramble):
        p = Pair(w, max_seqs=3, max_pages=12, max_pages_per_seq=6, kernel=kernel, with_oracle=False)
        if scramble:
            p.open([1, 2])
            p.s.ctx.reserve([1], 130); p.s.ctx.reserve([2], 70)
            p.s.ctx.seq_close(1); p.s.ctx.seq_close(2)
        p.open([0])
        p.prefill([0], 200)
        pages = [p.s.ctx.debug_locate(0, t)[0] for t in range(0, 200, 64)]
        res = p.decode_step([0], 0)
        return pages, {l: r[0] for l, r in res.items()}
    pa, a = run(False)
    pb, b = run(True)
    assert pa != pb
    for l in a:
        assert np.array_equal(a[l], b[l])


def test_large_grid_runs_k_then_v_in_one_cluster():
    """More tile pairs than half of the SM pairs: the tensor-core kernel stops spreading a
    pair over several clusters and each cluster does K, then V (most other tests are
    small enough to take the split paths)."""
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, batch=5, cached_tokens=0, decode_steps=1, reuse_frac=0.25)
    pps = 34
    p = Pair(w, max_seqs=5, max_pages=5 * pps, max_pages_per_seq=pps, kernel=B.KERNEL_TENSOR)
    seqs = [0, 1, 2, 3, 4]
    p.open(seqs)
    for s_, n in zip(seqs, (2100, 2049, 2111, 2050, 2064)):     # 17 tiles each: 85 tiles, 43 pairs
        p.prefill([s_], n)
    _check_step(p.decode_step(seqs, 0), "bf16", "fused clusters")


@pytest.mark.parametrize("shape", ["group2_narrow", "group4_wide", "group3_odd"])
def test_tensor_kernel_variants_walk_several_pairs(shape):
    """The tensor-core kernel is built for 12, 16 or 32 query heads and one to eight blocks of 128 hidden features.  The two paper
    shapes take two of the builds; these shapes take others, with more tiles than CTAs so that each walks several
    (wider shapes: test_runs_of_several_tiles_beyond)."""
    if shape == "group2_narrow":     # 8 query / 4 KV heads, hidden 192: one chunk, two blocks of features
        w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, n_q_heads=8, n_kv_heads=4, latent_full=128, batch=9,
                         cached_tokens=0, decode_steps=1, reuse_frac=0.25)
    elif shape == "group4_wide":     # 32 query / 8 KV heads, hidden 384: two chunks, three blocks
        w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, n_q_heads=32, n_kv_heads=8, latent_full=256, batch=9,
                         cached_tokens=0, decode_steps=1, reuse_frac=0.25)
    else:                            # 6 query / 2 KV heads: a group of three, half of the operand's rows padding
        w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, n_q_heads=6, n_kv_heads=2, latent_full=64, batch=9,
                         cached_tokens=0, decode_steps=1, reuse_frac=0.5)
    pps = 34
    p = Pair(w, max_seqs=9, max_pages=9 * pps, max_pages_per_seq=pps, kernel=B.KERNEL_TENSOR)
    seqs = list(range(9))
    p.open(seqs)
    for s_, n in zip(seqs, (2100, 2049, 2111, 2050, 2064, 2051, 2172, 2090, 2055)):   # 17 tiles each: 77 pairs
        p.prefill([s_], n)
    assert all(p.s.ctx.layer_kernel(l) == B.KERNEL_TENSOR for l in range(w.n_layers))
    _check_step(p.decode_step(seqs, 0), "bf16", shape)


@pytest.mark.parametrize("storage", ["bf16", "f32"])
def test_many_short_sequences_merge_one_warp_per_row(storage):
    """512 (sequence, query head) rows of at most three tiles: the tile partials and the current token are merged
    by the one-warp-per-row kernel (fewer rows or longer sequences take the CTA-per-row kernel of the other tests).
    Lengths include 0 (current token only) and exact tile multiples."""
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, batch=16, cached_tokens=0, decode_steps=1, reuse_frac=0.25,
                     storage=storage)
    p = Pair(w, max_seqs=16, max_pages=16 * 6, max_pages_per_seq=6)
    seqs = list(range(16))
    p.open(seqs)
    for s_, n in zip(seqs, (0, 1, 127, 128, 129, 256, 300, 64, 5, 200, 257, 31, 33, 255, 90, 130)):
        if n:
            p.prefill([s_], n)
    _check_step(p.decode_step(seqs, 0), storage, f"warp merge {storage}")
    _check_step(p.decode_step(seqs, 1, include_current=False), storage, f"warp merge, cached only, {storage}")


@pytest.mark.parametrize("head_dim", [32, 128])
def test_other_head_widths_take_the_generic_kernels(head_dim):
    """Head widths other than 64 run on the generic kernels (fp32 and bf16 storage); 128 exercises the merge
    kernels' upper channel half, 32 their idle lanes.  One sequence is long enough (33 tiles) for the
    CTA-per-row merge, the others take the warp-per-row one."""
    for storage in ("f32", "bf16"):
        w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, n_q_heads=4, n_kv_heads=2, head_dim=head_dim,
                         latent_full=head_dim, batch=2, cached_tokens=0, decode_steps=1, reuse_frac=0.5,
                         storage=storage)
        for lens in ((200, 1), (4200, 130)):
            pps = (max(lens) + 2 + w.page_tokens - 1) // w.page_tokens
            p = Pair(w, max_seqs=2, max_pages=2 * pps, max_pages_per_seq=pps)
            p.open([0, 1])
            for s_, n in zip((0, 1), lens):
                p.prefill([s_], n)
            _check_step(p.decode_step([0, 1], 0), storage, f"head_dim {head_dim} {storage} {lens}")


def test_fp32_stack_with_reuse_generic():
    """fp32 mode on a multi-layer stack with chains of reuse; 1e-4 absolute."""
    w = synth.scaled(synth.CONFIGS["c2"], n_layers=4, batch=2, storage="f32", reuse_frac=0.5)
    p = Pair(w, max_seqs=2, max_pages=8, max_pages_per_seq=4)
    p.open([0, 1])
    p.prefill([0], 150)
    p.prefill([1], 33)
    p.check_latents([0, 1])
    for step in range(2):
        _check_step(p.decode_step([0, 1], step), "f32", f"step {step}")


@pytest.mark.parametrize("cfg", ["c2", "c3"])
def test_single_call_step_matches_oracle_and_the_two_calls(cfg):
    """kvcar_step_layer (tile kernel on the library's side stream beside the encoder) against the oracle, and bit
    for bit against kvcar_encode_append + kvcar_decode_attention on a twin context, over several steps (so that
    later steps read rows appended by earlier ones) and a page boundary."""
    w = synth.scaled(synth.CONFIGS[cfg], n_layers=4, batch=3, cached_tokens=0, decode_steps=3, reuse_frac=0.3)
    seqs = [0, 1, 2]
    pairs = []
    for with_oracle in (True, False):
        p = Pair(w, max_seqs=3, max_pages=24, max_pages_per_seq=8, with_oracle=with_oracle)
        p.open(seqs)
        for s_, n in zip(seqs, (383, 130, 62)):        # the third sequence crosses a page boundary at step 2
            p.prefill([s_], n)
        pairs.append(p)
    fused, split = pairs
    for step in range(3):
        a = fused.decode_step(seqs, step, fused=True)
        b = split.decode_step(seqs, step, fused=False)
        _check_step(a, "bf16", f"single call, step {step}")
        for l in a:
            assert np.array_equal(a[l][0], b[l][0]), (step, l)
    fused.check_latents(seqs)


def test_host_buffer_entry_point_matches_device_entry_points():
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, batch=2, reuse_frac=0.25)
    p = Pair(w, max_seqs=2, max_pages=8, max_pages_per_seq=4)
    seqs = [0, 1]
    p.open(seqs)
    p.prefill(seqs, 100)
    dt = p.s.dtype
    for l in range(w.n_layers):
        k = np.stack([synth.make_kv(w, l, K, s, 100, 1) for s in seqs])
        v = np.stack([synth.make_kv(w, l, V, s, 100, 1) for s in seqs])
        q = np.stack([synth.make_q(w, l, s, 0) for s in seqs])
        hk = torch.from_numpy(k).to(dt).pin_memory(); hv = torch.from_numpy(v).to(dt).pin_memory()
        hq = torch.from_numpy(q).to(dt).pin_memory()
        ho = torch.empty_like(hq).pin_memory()
        p.s.ctx.step_layer_host(l, seqs, hk.data_ptr(), hv.data_ptr(), hq.data_ptr(), ho.data_ptr(),
                                B.INCLUDE_CURRENT_EXACT, p.s.stream())
        p.s.ctx.sync_status(p.s.stream())
        p.o.encode_append(l, seqs, 1, k, v)
        ref = p.o.decode_attention(l, seqs, q)
        assert_close(ho.float().numpy().astype(np.float64), ref, "bf16", f"host entry layer {l}")


@pytest.mark.parametrize("pinned_out", [True, False], ids=["page_locked_out", "pageable_out"])
def test_host_buffer_steps_equal_device_steps(pinned_out):
    """Eleven host-buffer steps of two layers, nothing awaited between them and the inputs overwritten after each call (more calls
    than the library has staging slots), bit for bit against the device entry point on a twin context."""
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, batch=2, reuse_frac=0.25)
    seqs, steps = [0, 1], 11
    host, dev = [Pair(w, max_seqs=2, max_pages=8, max_pages_per_seq=4, with_oracle=False) for _ in range(2)]
    for p in (host, dev):
        p.open(seqs)
        p.prefill(seqs, 50)
    dt = host.s.dtype
    shape = [(2, w.n_kv_heads, w.head_dim)] * 2 + [(2, w.n_q_heads, w.head_dim)]
    buf = [torch.empty(s, dtype=dt).pin_memory() for s in shape]
    out = torch.zeros((steps, 2) + shape[2], dtype=dt)
    out = out.pin_memory() if pinned_out else out
    ref = torch.zeros((steps, 2) + shape[2], dtype=dt, device="cuda")
    gen = torch.Generator().manual_seed(5)
    for step in range(steps):
        for l in range(2):
            x = [torch.randn(s, generator=gen).to(dt) for s in shape]
            for b, t in zip(buf, x):
                b.copy_(t)
            host.s.ctx.step_layer_host(l, seqs, *(b.data_ptr() for b in buf), out[step, l].data_ptr(),
                                       B.INCLUDE_CURRENT_EXACT, host.s.stream())
            for b in buf:
                b.zero_()
            d = [t.cuda() for t in x]
            dev.s.ctx.step_layer(l, seqs, *(t.data_ptr() for t in d), ref[step, l].data_ptr(), B.INCLUDE_CURRENT_EXACT,
                                 dev.s.stream())
        for p in (host, dev):
            p.s.ctx.advance(seqs, 1, p.s.stream())
    host.s.ctx.sync_status(host.s.stream())
    dev.s.ctx.sync_status(dev.s.stream())
    assert torch.equal(out, ref.cpu())


def test_output_buffer_that_is_page_locked_in_part_is_not_written_by_a_kernel():
    """The first page of an output buffer is registered, the rest is not: the output arrives by a copy (or the copy refuses such a
    range), never from a kernel, and the context goes on.  The same buffer registered whole is written in place."""
    import mmap
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=1, batch=2, reuse_frac=0.0)
    seqs = [0, 1]
    p = Pair(w, max_seqs=2, max_pages=4, max_pages_per_seq=2, with_oracle=False)
    p.open(seqs)
    p.prefill(seqs, 50)
    dt, st, page = p.s.dtype, p.s.stream(), mmap.PAGESIZE
    gen = torch.Generator().manual_seed(7)
    ins = [torch.randn(s, generator=gen).to(dt).pin_memory()
           for s in [(2, w.n_kv_heads, w.head_dim)] * 2 + [(2, w.n_q_heads, w.head_dim)]]
    d, ref = [t.cuda() for t in ins], torch.empty_like(ins[2], device="cuda")
    p.s.ctx.step_layer(0, seqs, *(t.data_ptr() for t in d), ref.data_ptr(), B.INCLUDE_CURRENT_EXACT, st)
    mem = mmap.mmap(-1, 4 * page)
    buf = torch.frombuffer(mem, dtype=dt)
    start = (page - 256) // 2                       # 256 bytes of the output lie in the first page
    out = buf[start:start + ins[2].numel()].view(ins[2].shape)
    rt = torch.cuda.cudart()
    for registered in (page, 4 * page):
        assert int(rt.cudaHostRegister(buf.data_ptr(), registered, 0)) == 0
        try:
            p.s.ctx.step_layer_host(0, seqs, *(t.data_ptr() for t in ins), out.data_ptr(), B.INCLUDE_CURRENT_EXACT, st)
            p.s.ctx.sync_status(st)
            assert torch.equal(out, ref.cpu())
        except B.KvcarError as e:
            assert registered == page and e.status == 6
        finally:
            torch.cuda.synchronize()
            rt.cudaHostUnregister(buf.data_ptr())
        buf.zero_()


def test_host_buffer_steps_mix_with_graph_replays():
    """A captured host-buffer step of layer 0, replayed behind queued work, and direct host-buffer steps of layer 1 behind it
    (more than the library has staging slots, whose copies run ahead of the stream): neither reads the other's inputs."""
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, batch=2, reuse_frac=0.0)
    seqs, calls = [0, 1], 9
    p = Pair(w, max_seqs=2, max_pages=8, max_pages_per_seq=4, with_oracle=False)
    p.open(seqs)
    p.prefill(seqs, 50)
    p.decode_step(seqs, 0)
    p.s.ctx.reserve(seqs, 1)
    dt = p.s.dtype
    shape = [(2, w.n_kv_heads, w.head_dim)] * 2 + [(2, w.n_q_heads, w.head_dim)]
    gen = torch.Generator().manual_seed(6)
    sets = [[torch.randn(s, generator=gen).to(dt).pin_memory() for s in shape] for _ in range(1 + calls)]
    outs = [torch.zeros(shape[2], dtype=dt).pin_memory() for _ in sets]

    def call(layer, i):
        p.s.ctx.step_layer_host(layer, seqs, *(t.data_ptr() for t in sets[i]), outs[i].data_ptr(), B.INCLUDE_CURRENT_EXACT, p.s.stream())

    def device(layer, i):
        d, out = [t.cuda() for t in sets[i]], torch.empty(shape[2], dtype=dt, device="cuda")
        p.s.ctx.step_layer(layer, seqs, *(t.data_ptr() for t in d), out.data_ptr(), B.INCLUDE_CURRENT_EXACT, p.s.stream())
        return out.cpu()
    ref = [device(0, 0)] + [device(1, i) for i in range(1, 1 + calls)]
    call(0, 0)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(0, 0)
    x = torch.randn(4096, 4096, device="cuda")
    for _ in range(3):
        for o in outs:
            o.zero_()
        for _ in range(10):
            x = (x @ x).clamp_(-1, 1)
        graph.replay()
        for i in range(1, 1 + calls):
            call(1, i)
        p.s.ctx.sync_status(p.s.stream())
        assert all(torch.equal(a, b) for a, b in zip(outs, ref))


def test_errors_leave_state_untouched():
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=1, batch=1, reuse_frac=0.0)
    p = Pair(w, max_seqs=2, max_pages=2, max_pages_per_seq=2, with_oracle=False)
    p.open([0, 1])
    p.prefill([0], 64)
    big = torch.zeros(1, 100, w.kv_width, dtype=p.s.dtype, device="cuda")
    with pytest.raises(B.KvcarError) as e:      # 100 more tokens need 2 pages, 1 is left
        p.s.ctx.encode_append(0, [0], 100, big.data_ptr(), big.data_ptr(), p.s.stream())
    assert e.value.status == 3
    assert p.s.ctx.seq_len(0) == 64
    p.s.ctx.reserve([1], 64)                    # the last page is still available
    with pytest.raises(B.KvcarError) as e:
        p.s.ctx.decode_attention(0, [5], big.data_ptr(), big.data_ptr(), 0, p.s.stream())
    assert e.value.status == 1


@pytest.mark.parametrize("kernel", KERNELS, ids=lambda k: KNAME[k])
def test_a_list_longer_than_max_seqs_is_refused_before_anything_is_copied(kernel):
    """Staging slots and workspace rows are one per sequence id; a longer list (which names a sequence twice) is an argument error
    of every call that fills them, and the next step of the context is right."""
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=1, batch=1, reuse_frac=0.0)
    p = Pair(w, max_seqs=1, max_pages=2, max_pages_per_seq=2, kernel=kernel)
    p.open([0])
    p.prefill([0], 40)
    n = 9
    host = torch.zeros(n, w.n_q_heads * w.head_dim, dtype=p.s.dtype).pin_memory()
    dev = host.cuda()
    h, d, st, ctx = host.data_ptr(), dev.data_ptr(), p.s.stream(), p.s.ctx
    before = ctx.launch_count()
    for call in (lambda: ctx.step_layer_host(0, [0] * n, h, h, h, h, B.INCLUDE_CURRENT_EXACT, st),
                 lambda: ctx.step_layer(0, [0] * n, d, d, d, d, B.INCLUDE_CURRENT_EXACT, st),
                 lambda: ctx.decode_attention(0, [0] * n, d, d, 0, st),
                 lambda: ctx.encode_append(0, [0] * n, 1, d, d, st)):
        with pytest.raises(B.KvcarError) as e:
            call()
        assert e.value.status == 1
    assert ctx.launch_count() == before
    _check_step(p.decode_step([0], 0, fused=True), "bf16", "after refused calls")


def test_device_side_wait_that_runs_out_is_reported_and_the_context_stays_usable():
    """A bounded device-side wait that nothing completes: the kernel gives up after its limit (1 ms here), records a
    code in the status word and returns; kvcar_sync_status reports KVCAR_ERR_DEVICE_TIMEOUT exactly once, and the
    next decode on the same context is correct.  Nothing traps, faults or waits without a limit."""
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, batch=2, reuse_frac=0.25)
    p = Pair(w, max_seqs=2, max_pages=8, max_pages_per_seq=4)
    p.open([0, 1])
    p.prefill([0], 140)
    p.prefill([1], 65)
    p.s.ctx.debug_expire_wait(1_000_000, p.s.stream())
    with pytest.raises(B.KvcarError) as e:
        p.s.ctx.sync_status(p.s.stream())
    assert e.value.status == 7 and "0x7e57" in str(e.value)
    p.s.ctx.sync_status(p.s.stream())            # the word was cleared: reported once
    _check_step(p.decode_step([0, 1], 0), "bf16", "after a timed-out wait")


@pytest.mark.parametrize("cfg,quant", [("c2", False), ("c3", False), ("c2", True)])
def test_guard_regions_and_device_tables_survive_prefill_and_decode(cfg, quant):
    """Stand-in for a memory checker: 256 guard bytes behind every pool region (K and V pools, int8 row parameters,
    current-token rows) keep their fill through bulk and per-token encoding, decode steps on full and ragged
    pages, and a sequence that fills its last reserved page to the end; the device page table and lengths equal the
    allocator's.  A byte planted by the test just behind layer 0's K pool is then found and located."""
    w = synth.scaled(synth.CONFIGS[cfg], n_layers=3, batch=3, reuse_frac=0.25)
    p = Pair(w, max_seqs=3, max_pages=9, max_pages_per_seq=3, latent_quant=quant)
    p.open([0, 1, 2])
    p.prefill([0], 3 * 64 - 1)          # one step short of the end of its last page
    p.prefill([1], 65)
    p.prefill([2], 1)
    assert p.s.ctx.debug_check(p.s.stream()) == (0, 0, -1)
    p.decode_step([0, 1, 2], 0)         # sequence 0 now ends exactly at the end of the pool rows reserved for it
    assert p.s.ctx.debug_check(p.s.stream()) == (0, 0, -1)
    off, pitch, width = p.s.ctx.pool_layout(0, 0)
    rows = p.s.ctx.cfg.max_pages * p.s.ctx.cfg.page_tokens
    guard = (off + rows * pitch + 255) // 256 * 256
    base = p.s._aligned(p.s.pool) - p.s.pool.data_ptr()
    torch.cuda.synchronize()
    assert int(p.s.pool[base + guard + 7]) == 0xA5
    p.s.pool[base + guard + 7] = 0
    torch.cuda.synchronize()
    st, what, where = p.s.ctx.debug_check(p.s.stream())
    assert (st, what, where) == (8, 1, guard + 7)
    p.s.pool[base + guard + 7] = 0xA5
    torch.cuda.synchronize()
    assert p.s.ctx.debug_check(p.s.stream()) == (0, 0, -1)


@pytest.mark.parametrize("cfg", ["c2", "c3"])
def test_int8_latent_rows_match_the_oracle(cfg):
    """Sec. "Quantization" on top of the autoencoders (Table 5's combination): every cached latent row is stored
    as int8 codes with its own scale and zero-point (Eq. 4) and restored before the decoder.  Cached rows are
    compared as restored values (one code step at most, almost all equal), attention outputs at the bf16
    tolerance, bytes per token exactly."""
    w = synth.scaled(synth.CONFIGS[cfg], batch=3, cached_tokens=0, decode_steps=2)
    p = Pair(w, max_seqs=4, max_pages=16, max_pages_per_seq=6, latent_quant=True)
    seqs = [2, 0, 3]
    p.open(seqs)
    p.prefill([2], 200)
    p.prefill([0], 131)
    p.prefill([3], 1)
    p.check_latents(seqs)
    for step in range(2):
        _check_step(p.decode_step(seqs, step), "bf16", f"int8 step {step}")
    p.check_latents(seqs)
    comp, full = p.s.ctx.cache_bytes_per_token()
    assert (comp, full) == p.o.cache_bytes_per_token()
    plain = Pair(w, max_seqs=1, max_pages=1, max_pages_per_seq=1, with_oracle=False)
    assert comp < 0.55 * plain.s.ctx.cache_bytes_per_token()[0]


@pytest.mark.parametrize("shape", ["gpt2", "group2_narrow", "tinyllama"])
def test_absorbed_last_layer_on_both_sides_matches_the_oracle(shape):
    """KVCAR_ABSORBED | KVCAR_ABSORBED_V: the V side too - a tile hands on sum_t p_t a_t (m values per query head) and
    W4_h is applied once per sequence and head when the tiles are merged; no restored K or V row is ever formed.
    Same tolerance as the plain form; ragged lengths, reuse (several V sources per layer), two steps, and the
    output must also agree with the plain form of the same context."""
    if shape == "gpt2":            # 12 heads, hidden 576: nine slabs, the last feature chunk repeats a slab
        w = synth.scaled(synth.CONFIGS["c2"], n_layers=3, batch=5, cached_tokens=0, decode_steps=2, reuse_frac=0.25)
    elif shape == "tinyllama":     # 32 query / 4 KV heads (two 32-column blocks per chunk), hidden 192
        w = synth.scaled(synth.CONFIGS["c3"], n_layers=3, batch=5, cached_tokens=0, decode_steps=2, reuse_frac=0.25)
    else:                          # 8 query / 4 KV heads, hidden 192: three slabs
        w = synth.scaled(synth.CONFIGS["c3"], n_layers=3, n_q_heads=8, n_kv_heads=4, latent_full=128, batch=5,
                         cached_tokens=0, decode_steps=2, reuse_frac=0.25)
    pps = 34
    p = Pair(w, max_seqs=5, max_pages=5 * pps, max_pages_per_seq=pps, kernel=B.KERNEL_TENSOR)
    seqs = [0, 1, 2, 3, 4]
    p.open(seqs)
    for s_, n in zip(seqs, (2100, 2049, 2111, 2050, 2064)):     # 17 tiles each: 85 tiles, 43 pairs
        p.prefill([s_], n)
    for step in range(2):
        res = p.decode_step(seqs, step, absorbed="kv")
        _check_step(res, "bf16", f"absorbed K and V {shape} step {step}")
    # against the plain form on the same cache (one more layer call each way, no append)
    q = np.stack([synth.make_q(w, 1, s_, 7) for s_ in seqs])
    got_a, _, _ = p.attention(1, seqs, q, absorbed="kv")
    got_p, ref, rows = p.attention(1, seqs, q)
    assert_close(got_a[rows], ref, "bf16", "absorbed K and V, layer 1")
    assert np.max(np.abs(got_a - got_p)) < 2e-2
    assert np.max(np.abs(got_a - got_p)) > 0.0   # the other form did run


@pytest.mark.parametrize("shape", ["gpt2", "tinyllama", "group2_narrow"])
def test_absorbed_last_layer_matches_the_oracle(shape):
    """KVCAR_ABSORBED: a head's scores are taken as a.(W4_h^T q) + q.b4_h from the activated hidden vectors, the
    restored K rows are never formed (the decoder ends in a bare fully connected layer, Sec. "Network Architecture").
    Same result as the plain form up to rounding: compared with the oracle at the usual tolerance, with reuse (several source
    layers per layer).  Every call takes this form; the flag leaves one bf16 term of W4_h^T q instead of two, so it changes some bits
    of the output and no more than that."""
    if shape == "gpt2":            # 12 heads, hidden 576 (three chunks), CUDA-core attention products
        w = synth.scaled(synth.CONFIGS["c2"], n_layers=3, batch=5, cached_tokens=0, decode_steps=2, reuse_frac=0.25)
    elif shape == "tinyllama":     # 32 query / 4 KV heads, hidden 192, tensor-op attention products
        w = synth.scaled(synth.CONFIGS["c3"], n_layers=3, batch=5, cached_tokens=0, decode_steps=2, reuse_frac=0.25)
    else:                          # 8 query / 4 KV heads
        w = synth.scaled(synth.CONFIGS["c3"], n_layers=3, n_q_heads=8, n_kv_heads=4, latent_full=128, batch=5,
                         cached_tokens=0, decode_steps=2, reuse_frac=0.25)
    pps = 34
    p = Pair(w, max_seqs=5, max_pages=5 * pps, max_pages_per_seq=pps, kernel=B.KERNEL_TENSOR)
    seqs = [0, 1, 2, 3, 4]
    p.open(seqs)
    for s_, n in zip(seqs, (2100, 2049, 2111, 2050, 2064)):     # 17 tiles each: 85 tiles, 43 pairs
        p.prefill([s_], n)
    for step in range(2):
        res = p.decode_step(seqs, step, absorbed=True)
        _check_step(res, "bf16", f"absorbed {shape} step {step}")
    q = np.stack([synth.make_q(w, 1, s_, 7) for s_ in seqs])
    one, ref, rows = p.attention(1, seqs, q, absorbed=True)
    two, _, _ = p.attention(1, seqs, q)
    assert 0.0 < np.max(np.abs(one - two)) < 2e-2
    # and on a grid small enough for K and V to be two launches
    w2 = synth.scaled(w, batch=2)
    p2 = Pair(w2, max_seqs=2, max_pages=8, max_pages_per_seq=4, kernel=B.KERNEL_TENSOR)
    p2.open([0, 1])
    p2.prefill([0], 200)
    p2.prefill([1], 130)
    _check_step(p2.decode_step([0, 1], 0, absorbed=True), "bf16", f"absorbed flag on a small grid, {shape}")



@pytest.mark.parametrize("case", ["small_tiles", "large_tiles", "groups", "int8_large_tiles"])
def test_fp32_arithmetic_kernels_at_tile_edges(case):
    """The fp32-FMA attention kernels on fp32 storage: blocks of 32 x 32 with two pieces per partial result, blocks of 64 x 64
    where those fill the machine, and calls of more than 1024 partial results, which are worked through in groups of sequences.
    Lengths around 32, 64 and 128 tokens, one sequence empty; tolerances of the storage type, as everywhere.  (int8_large_tiles is
    the same lengths on the tensor cores; int8 rows on the FMA kernels: the next test.)"""
    lens = {"small_tiles": (31, 32, 33, 0, 63, 64, 65, 129), "large_tiles": (1473, 1, 1472, 0, 1471),
            "int8_large_tiles": (1473, 1, 1472, 0, 1471), "groups": (33000, 65, 0, 32900)}[case]
    if case == "groups":
        w = synth.scaled(synth.CONFIGS["c3"], n_layers=1, n_q_heads=4, n_kv_heads=2, head_dim=32, latent_full=32,
                         batch=len(lens), cached_tokens=0, decode_steps=1, reuse_frac=0.0, storage="f32")
    else:
        quant = case.startswith("int8")
        w = synth.scaled(synth.CONFIGS["c2"], n_layers=2, batch=len(lens), cached_tokens=0, decode_steps=1, reuse_frac=0.25,
                         storage="bf16" if quant else "f32")
    pps = (max(lens) + 2 + w.page_tokens - 1) // w.page_tokens
    p = Pair(w, max_seqs=len(lens), max_pages=len(lens) * pps, max_pages_per_seq=pps, latent_quant=case.startswith("int8"))
    seqs = list(range(len(lens)))
    p.open(seqs)
    for s_, n in zip(seqs, lens):
        if n:
            p.prefill([s_], n)
    _check_step(p.decode_step(seqs, 0), w.storage, case)


@pytest.mark.parametrize("head_dim", [32, 128])
@pytest.mark.parametrize("tiles", ["small", "large"])
def test_int8_rows_on_the_fp32_arithmetic_kernels(head_dim, tiles):
    """int8 rows of other head widths: blocks of 32 x 32 and (from four times the SM count of 64 x 64 blocks on) of 64 x 64.  Four
    launches per attention call show the path (the restoring kernel takes two)."""
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=2, n_q_heads=4, n_kv_heads=2, head_dim=head_dim, latent_full=head_dim, batch=5,
                     cached_tokens=0, decode_steps=1, reuse_frac=0.5)
    lens = (31, 64, 65, 0, 129) if tiles == "small" else (9600, 9537, 1, 9601, 9472)
    blocks = sum((n + 63) // 64 for n in lens) * ((3 * head_dim // 2 + 63) // 64)
    assert (blocks >= 4 * 148) == (tiles == "large")
    pps = (max(lens) + 2 + w.page_tokens - 1) // w.page_tokens
    p = Pair(w, max_seqs=5, max_pages=5 * pps, max_pages_per_seq=pps, latent_quant=True)
    p.oracle_seqs = None if tiles == "small" else {1, 2}
    p.open([0, 1, 2, 3, 4])
    for s_, n in zip(range(5), lens):
        if n:
            p.prefill([s_], n)
    _check_step(p.decode_step([0, 1, 2, 3, 4], 0), "bf16", f"head_dim {head_dim} {tiles}")
    before = p.s.ctx.launch_count()
    p.attention(0, [0, 1, 2, 4], np.stack([synth.make_q(w, 0, s_, 9) for s_ in (0, 1, 2, 4)]))
    assert p.s.ctx.launch_count() - before == 4


@pytest.mark.parametrize("case", ["offset_rows", "groups"])
def test_int8_rows_on_the_tensor_cores_beyond_the_usual(case, monkeypatch):
    """int8 rows are widened to whole numbers that bf16 holds exactly.  offset_rows: K latents far from zero (their zero-points
    do not fit the codes, the rest goes through the weights' row sums); a constant on every K latent adds the same to all
    scores of a head, so the outputs keep their size and the usual tolerance.  groups: more tiles than the widened rows have
    room for at a time (296), worked through in two groups of sequences, an empty sequence among them."""
    if case == "offset_rows":
        real = synth.make_stack_autoencoders

        def shifted(*a, **kw):
            aes = real(*a, **kw)
            for (_, which), ae in aes.items():
                if which == K:
                    ae["enc_b2"] = ae["enc_b2"] + np.float32(6.0)
            return aes
        monkeypatch.setattr(synth, "make_stack_autoencoders", shifted)
        w = synth.scaled(synth.CONFIGS["c2"], n_layers=2, batch=3, cached_tokens=0, decode_steps=1, reuse_frac=0.25)
        lens = (200, 129, 64)
    else:
        w = synth.scaled(synth.CONFIGS["c3"], n_layers=1, batch=4, cached_tokens=0, decode_steps=1, reuse_frac=0.0)
        lens = (13000, 0, 12801, 12929)
    pps = (max(lens) + 2 + w.page_tokens - 1) // w.page_tokens
    p = Pair(w, max_seqs=len(lens), max_pages=len(lens) * pps, max_pages_per_seq=pps, latent_quant=True)
    assert all(p.s.ctx.layer_kernel(l) == B.KERNEL_TENSOR for l in range(w.n_layers))
    seqs = list(range(len(lens)))
    p.open(seqs)
    for s_, n in zip(seqs, lens):
        if n:
            p.prefill([s_], n)
    if case == "offset_rows":
        q = p.s.pool_quant_params(0, 0)[p.o.locate(0, 5)[1]].cpu().numpy()
        assert q[1] < -129      # the zero-point really is out of the codes' reach
    for fused in (False, True):
        _check_step(p.decode_step(seqs, int(fused), fused=fused), "bf16", f"{case} fused={fused}")


@pytest.mark.parametrize("shape", ["gpt2", "tinyllama", "sixteen_heads", "one_slab_tail"])
def test_int8_attention_is_as_precise_as_in_fp32(shape):
    """int8 rows at peaked scores (queries x 8, where what is rounded on the way to a score shows): over the codes that the device
    holds, the tensor-core path (hidden vectors, W4^T q and probabilities as two bf16 terms each) is no further from the fp64 oracle
    than the fp32 kernel, whose whole error is the rounding of the bf16 output (2^-9 relative at most, 1.7e-3 in the norm); one bf16
    term of the hidden vectors alone made it 2.5e-3 to 3.0e-3."""
    kw = {"gpt2": {}, "tinyllama": {}, "sixteen_heads": dict(n_q_heads=16, n_kv_heads=16, latent_full=512),
          "one_slab_tail": dict(n_q_heads=8, n_kv_heads=4, latent_full=128)}[shape]      # hidden 192: a job of one slab at the end
    w = synth.scaled(synth.CONFIGS["c2" if shape in ("gpt2", "sixteen_heads") else "c3"], n_layers=2, batch=4, cached_tokens=0,
                     decode_steps=1, reuse_frac=0.25, **kw)
    seqs, rel = [0, 1, 2, 3], {}
    for kernel in KERNELS:
        p = Pair(w, max_seqs=4, max_pages=64, max_pages_per_seq=16, latent_quant=True, kernel=kernel)
        p.open(seqs)
        for s_, n in zip(seqs, (17, 200, 515, 900)):
            p.prefill([s_], n)
        if kernel == B.KERNEL_AUTO:
            assert all(p.s.ctx.layer_kernel(l) == B.KERNEL_TENSOR for l in range(w.n_layers))
        rows = [p.o.locate(s_, t)[1] for s_ in seqs for t in range(p.o.seq_len[s_])]
        for l in range(w.n_layers):
            for which in (K, V):
                if p.o.stored_width(l, which):
                    codes = p.s.pool_rows(l, which)[torch.tensor(rows, device=p.s.device)].cpu().numpy().astype(np.float64)
                    par = p.s.pool_quant_params(l, which)[torch.tensor(rows, device=p.s.device)].cpu().numpy().astype(np.float64)
                    p.o._pool(l, which)[rows] = (codes - par[:, 1:]) / par[:, :1]
        res = p.decode_step(seqs, 0, q_scale=8.0)
        rel[kernel] = [np.linalg.norm(got[r] - ref) / np.linalg.norm(ref) for got, ref, r in res.values()]
    for auto, fp32 in zip(rel[B.KERNEL_AUTO], rel[B.KERNEL_GENERIC]):
        assert auto <= 1.01 * fp32, (auto, fp32)


# Shapes past what the latent-attention kernels once took, and past what they take: name -> (config, changes, AE hidden width or None)
BEYOND = {
    "latent_576": ("c2", dict(latent_full=576), None),                                   # GPT-2 shape at 25 % compression
    "latent_576_no_reuse": ("c2", dict(latent_full=576, reuse_frac=0.0), None),          # (with reuse a hidden layer is 504 wide)
    "hidden_768": ("c2", {}, 768),                                                       # 12 heads, hidden layer above 640
    "32_heads_of_their_own": ("c3", dict(n_q_heads=32, n_kv_heads=32, latent_full=512), 272),
    "32_heads_in_pairs": ("c3", dict(n_q_heads=32, n_kv_heads=16, latent_full=256), 384),
    "16_heads": ("c2", dict(n_q_heads=16, n_kv_heads=16, latent_full=512), None),
    "32_heads_in_pairs_wide": ("c3", dict(n_q_heads=32, n_kv_heads=16, latent_full=512), None),
    "40_heads": ("c3", dict(n_q_heads=40, n_kv_heads=8, latent_full=256), None),
    "hidden_1040": ("c2", {}, 1040),
    "eight_sources": ("c2", dict(n_layers=8), None),
}


# those of them that the latent-attention kernels take: with jobs of 128 columns (latents above 448), 12 heads padded to 16 (hidden layers
# above 640), probabilities in two operands (32 heads in small groups)
BEYOND_TENSOR = {"latent_576_no_reuse", "hidden_768", "32_heads_in_pairs", "16_heads"}


def _beyond(shape, int8, kernel, monkeypatch):
    cfg, kw, hidden = BEYOND[shape]
    if hidden:
        real = synth.ae_dims
        monkeypatch.setattr(synth, "ae_dims", lambda *a: (real(*a)[0], hidden, real(*a)[2]))
    w = synth.scaled(synth.CONFIGS[cfg], **{**dict(n_layers=2, batch=4, cached_tokens=0, decode_steps=1, reuse_frac=0.25), **kw})
    src = None
    if shape == "eight_sources":       # head h of the top layer reads layer h (heads 7.. the top layer's own)
        src = -np.ones((8, 12), np.int32)
        for h in range(7):
            src[h + 1:, h] = h
        src = src.reshape(-1)
    p = Pair(w, max_seqs=4, max_pages=64, max_pages_per_seq=18, src_k=src, src_v=src, latent_quant=int8, kernel=kernel)
    p.open([0, 1, 2, 3])
    for s_, n in zip(range(4), (1, 127, 0, 1100)):
        if n:
            p.prefill([s_], n)
    return w, p


@pytest.mark.parametrize("shape,kernel", [(s, B.KERNEL_AUTO) for s in sorted(BEYOND)] +
                         [(s, B.KERNEL_TENSOR) for s in ("latent_576_no_reuse", "hidden_768", "32_heads_in_pairs_wide", "40_heads")])
def test_bf16_layers_of_every_shape_have_a_fast_path(shape, kernel, monkeypatch):
    """Wide latents, wide hidden layers, many heads, many source layers: against the oracle, through the two calls and the single one,
    and never on the restoring kernel (which is two launches per call; the others are three or more)."""
    w, p = _beyond(shape, False, kernel, monkeypatch)
    seqs = [0, 1, 2, 3]
    if shape in BEYOND_TENSOR:
        assert all(p.s.ctx.layer_kernel(l) == B.KERNEL_TENSOR for l in range(w.n_layers))
    _check_step(p.decode_step(seqs, 0), "bf16", f"{shape} two calls")
    _check_step(p.decode_step(seqs, 1, fused=True), "bf16", f"{shape} one call")
    q = np.stack([synth.make_q(w, w.n_layers - 1, s_, 9) for s_ in seqs])
    before = p.s.ctx.launch_count()
    got, ref, rows = p.attention(w.n_layers - 1, seqs, q, include_current=False)
    assert p.s.ctx.launch_count() - before >= 3
    assert_close(got[rows], ref, "bf16", f"{shape} cached only")


@pytest.mark.parametrize("shape", sorted(BEYOND))
def test_int8_layers_of_every_shape_have_a_fast_path(shape, monkeypatch):
    """The same with int8 rows."""
    w, p = _beyond(shape, True, B.KERNEL_AUTO, monkeypatch)
    seqs = [0, 1, 2, 3]
    _check_step(p.decode_step(seqs, 0), "bf16", f"int8 {shape} two calls")
    _check_step(p.decode_step(seqs, 1, fused=True), "bf16", f"int8 {shape} one call")
    q = np.stack([synth.make_q(w, w.n_layers - 1, s_, 9) for s_ in seqs])
    before = p.s.ctx.launch_count()
    p.attention(w.n_layers - 1, seqs, q)
    assert p.s.ctx.launch_count() - before >= 3


def test_the_tensor_choice_is_refused_where_it_always_was(monkeypatch):
    """KVCAR_KERNEL_TENSOR: hidden layers above 1024 and more than six source layers stay UNSUPPORTED."""
    with pytest.raises(B.KvcarError) as e:
        _beyond("hidden_1040", False, B.KERNEL_TENSOR, monkeypatch)
    assert e.value.status == 5
    monkeypatch.undo()
    w, p = _beyond("eight_sources", False, B.KERNEL_TENSOR, monkeypatch)
    with pytest.raises(B.KvcarError) as e:
        p.attention(7, [0, 1], np.stack([synth.make_q(w, 7, s_, 9) for s_ in (0, 1)]))
    assert e.value.status == 5


@pytest.mark.parametrize("page_tokens", [16, 48])
def test_bf16_pages_that_are_no_multiple_of_64_tokens(page_tokens):
    """Pages the tensor loads cannot take: the fp32 kernels."""
    w = synth.scaled(synth.CONFIGS["c2"], n_layers=2, batch=3, page_tokens=page_tokens, reuse_frac=0.25)
    per = 320 // page_tokens + 1
    p = Pair(w, max_seqs=3, max_pages=3 * per, max_pages_per_seq=per)
    p.open([0, 1, 2])
    for s_, n in zip(range(3), (300, 49, 1)):
        p.prefill([s_], n)
    before = p.s.ctx.launch_count()
    p.attention(1, [0, 1, 2], np.stack([synth.make_q(w, 1, s_, 9) for s_ in range(3)]))
    assert p.s.ctx.launch_count() - before >= 4
    _check_step(p.decode_step([0, 1, 2], 0, fused=True), "bf16", f"pages of {page_tokens}")


@pytest.mark.parametrize("shape,int8", [("latent_576_no_reuse", False), ("latent_576_no_reuse", True), ("hidden_768", False),
                                        ("32_heads_in_pairs", False), ("16_heads", True)])
def test_runs_of_several_tiles_beyond(shape, int8, monkeypatch):
    """The builds of the wider shapes with more tiles than blocks: each walks several, across sequence ends and partial tiles."""
    cfg, kw, hidden = BEYOND[shape]
    if hidden:
        real = synth.ae_dims
        monkeypatch.setattr(synth, "ae_dims", lambda *a: (real(*a)[0], hidden, real(*a)[2]))
    w = synth.scaled(synth.CONFIGS[cfg], **{**dict(n_layers=1, batch=48, reuse_frac=0.0), **kw, "n_layers": 1})
    seqs = list(range(48))
    lens = [128 * (5 * s % 8) + (1, 127, 128, 60)[s % 4] for s in seqs]
    p = Pair(w, max_seqs=48, max_pages=48 * 17, max_pages_per_seq=17, latent_quant=int8)
    p.oracle_seqs = {0, 23, 47}
    p.open(seqs)
    for s_, n in zip(seqs, lens):
        p.prefill([s_], n)
    assert p.s.ctx.layer_kernel(0) == B.KERNEL_TENSOR
    for step in range(2):
        _check_step(p.decode_step(seqs, step, fused=True), "bf16", f"{shape} int8 {int8} step {step}")


@pytest.mark.parametrize("int8", [False, True], ids=["bf16", "int8"])
@pytest.mark.parametrize("cfg,n", [("c2", 200), ("c2", 2300), ("c3", 200), ("c3", 2300)])
def test_a_stray_value_stays_with_the_heads_that_read_its_source(cfg, n, int8):
    """A NaN in one cached K row of layer 0: in layer 1, the heads that reuse layer 0's K read it, those that read layer 1's own rows
    give the same bits as without it (small grids, where K and V are two launches, and blocks that walk several tiles)."""
    w = synth.scaled(synth.CONFIGS[cfg], n_layers=2, batch=9, cached_tokens=0, decode_steps=1)
    src = -np.ones((2, w.n_kv_heads), np.int32)
    src[1, ::2] = np.arange(w.n_kv_heads)[::2]             # every other KV head of layer 1 reads layer 0's K
    none = -np.ones(2 * w.n_kv_heads, np.int32)
    pps = n // 64 + 2
    p = Pair(w, max_seqs=9, max_pages=9 * pps, max_pages_per_seq=pps, src_k=src.reshape(-1), src_v=none, latent_quant=int8,
             with_oracle=False)
    seqs = list(range(9))
    p.open(seqs)
    p.prefill(seqs, n)
    q = np.stack([synth.make_q(w, 1, s_, 3) for s_ in seqs])
    clean, _, _ = p.attention(1, seqs, q, include_current=False)
    row = p.s.ctx.debug_locate(4, 70)[1]
    if int8:
        p.s.pool_quant_params(0, 0)[row] = float("nan")
    else:
        p.s.pool_rows(0, 0)[row] = float("nan")
    torch.cuda.synchronize()
    got, _, _ = p.attention(1, seqs, q, include_current=False)
    group = w.n_q_heads // w.n_kv_heads
    reads = np.repeat(np.arange(w.n_kv_heads) % 2 == 0, group)
    assert (got[4][reads] != clean[4][reads]).any(axis=-1).all()
    assert np.array_equal(got[4][~reads], clean[4][~reads])
    others = [s_ for s_ in seqs if s_ != 4]
    assert np.array_equal(got[others], clean[others])
