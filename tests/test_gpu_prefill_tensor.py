"""The tensor-core bulk encoder (kvcar_encode_append_tensor) against the CPU oracle: the cache rows it writes,
and decode attention over a cache it filled."""
import numpy as np
import pytest
import torch

import kvcar_synth as synth
from kvcar_harness import Pair, assert_close
from paper_2512_06727_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg", ["c2", "c3"])
def test_tensor_prefill_rows_and_decode_over_them(cfg):
    """A stack with reuse (so encoder widths differ by layer and between K and V), sequences whose rows end
    inside a 128-row tile, a second bulk append on top of the first (rows land behind existing ones, across a page
    boundary), then a decode step through the ordinary path over the cache the tensor-core encoder wrote."""
    w = synth.scaled(synth.CONFIGS[cfg], n_layers=4, batch=3, cached_tokens=0, decode_steps=1, reuse_frac=0.3)
    src_k = synth.make_reuse_map(w.n_layers, w.n_kv_heads, w.reuse_frac, w.seed)
    src_v = synth.make_reuse_map(w.n_layers, w.n_kv_heads, w.reuse_frac, w.seed + 3)
    p = Pair(w, max_seqs=3, max_pages=36, max_pages_per_seq=12, src_k=src_k, src_v=src_v)
    seqs = [0, 1, 2]
    p.open(seqs)
    p.prefill(seqs, 200, tensor=True)              # 600 rows: four full row tiles and one of 88 rows
    p.prefill([1], 77, t0=200, tensor=True)        # behind existing rows, ends inside a page
    p.prefill([0, 2], 1, t0=200, tensor=True)      # a single token per sequence also goes through
    p.check_latents(seqs, bf16_hidden=True)
    res = p.decode_step(seqs, 0)
    for l, (got, ref, rows) in res.items():
        assert_close(got[rows], ref, "bf16", f"{cfg} layer {l} over tensor-prefilled cache")


def test_tensor_prefill_matches_the_fp32_hidden_encoder_closely():
    """The same rows through both encoders: the two caches agree within the bf16-hidden tolerance, row for row."""
    w = synth.scaled(synth.CONFIGS["c2"], n_layers=2, batch=2, cached_tokens=0, decode_steps=1, reuse_frac=0.0)
    caches = []
    for tensor in (False, True):
        p = Pair(w, max_seqs=2, max_pages=8, max_pages_per_seq=4, with_oracle=False)
        p.open([0, 1])
        p.prefill([0, 1], 130, tensor=tensor)
        caches.append([p.s.pool_rows(l, which).float().cpu().numpy() for l in range(w.n_layers) for which in (0, 1)])
    for a, b in zip(*caches):
        used = np.abs(a).sum(axis=-1) > 0            # rows that were written
        assert used.sum() == 260
        scale = np.sqrt(np.mean(np.square(a[used]), axis=-1, keepdims=True))
        assert np.all(np.abs(a[used] - b[used]) <= 2.0 ** -7 * np.abs(a[used]) + 2.0 ** -7 * scale + 1e-6)


def test_tensor_prefill_refuses_what_it_cannot_do():
    w = synth.scaled(synth.CONFIGS["c2"], n_layers=1, batch=1, reuse_frac=0.0)
    p = Pair(w, max_seqs=1, max_pages=4, max_pages_per_seq=4, compress=False, with_oracle=False)   # raw layers
    p.open([0])
    k = torch.zeros(1, 4, w.kv_width, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(B.KvcarError) as e:
        p.s.ctx.encode_append_tensor(0, [0], 4, k.data_ptr(), k.data_ptr(), p.s.stream())
    assert e.value.status == 5          # KVCAR_ERR_UNSUPPORTED
    assert p.s.ctx.seq_len(0) == 0


@pytest.mark.parametrize("batch,tokens", [(1, 2), (1, 127), (1, 129), (3, 86), (2, 5400)])
def test_bulk_append_keeps_the_hidden_activations_in_fp32(batch, tokens):
    """kvcar_encode_append of several tokens (hidden activations as three bf16 terms each on the tensor cores) at the edges
    of a 128-row tile and of a pair of tiles, and past one block of the scratch (10 752 rows): the rows it writes lie within
    one bf16 step of the oracle's, the tolerance of the fp32-hidden encoder, not the wider one of rounded activations."""
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=2 if tokens < 1000 else 1, batch=batch, cached_tokens=0, decode_steps=1,
                     reuse_frac=0.25)
    pps = (tokens + 63) // 64
    p = Pair(w, max_seqs=batch, max_pages=batch * pps, max_pages_per_seq=pps)
    seqs = list(range(batch))
    p.open(seqs)
    p.prefill(seqs, tokens)
    p.check_latents(seqs)


@pytest.mark.parametrize("beta", [3.3e38, float("inf")], ids=["large", "infinite"])
def test_bulk_append_with_hidden_values_at_the_end_of_the_range(beta, monkeypatch):
    """One hidden value of every row is 3.3e38 or infinite.  The rows of the bulk call agree with those of one call per token, whose
    hidden values stay in fp32: within one bf16 step, infinities in the same places."""
    real = synth.make_stack_autoencoders

    def ends(*a, **kw):
        aes = real(*a, **kw)
        for ae in aes.values():
            ae["enc_bn"][1, 7] = beta
            ae["enc_w2"][:, 7] = 2.0 ** -127        # every latent has a share of it, 2 where it is finite
        return aes
    monkeypatch.setattr(synth, "make_stack_autoencoders", ends)
    w = synth.scaled(synth.CONFIGS["c3"], n_layers=1, batch=2, reuse_frac=0.0)
    p = Pair(w, max_seqs=2, max_pages=2, max_pages_per_seq=1, with_oracle=False)
    p.open([0, 1])
    rows = np.stack([synth.make_kv(w, 0, which, 0, 0, 5) for which in (0, 1)])
    p.append(0, [0], rows[0][None], rows[1][None])
    p.advance([0], 5)
    for t in range(5):
        p.append(0, [1], rows[0][None, t:t + 1], rows[1][None, t:t + 1])
        p.advance([1], 1)
    for which in (0, 1):
        c = p.s.pool_rows(0, which).float().cpu().numpy()
        a, b = c[p.s.ctx.debug_locate(0, 0)[1]:][:5], c[p.s.ctx.debug_locate(1, 0)[1]:][:5]
        assert not np.isnan(b).any()
        np.testing.assert_array_equal(np.isinf(a), np.isinf(b))
        assert np.isinf(b).all() == np.isinf(beta)
        if np.isfinite(beta):
            assert np.all(np.abs(a - b) <= 2.0 ** -7 * np.abs(b) + 1e-6)
