"""Decode attention of the shapes the tcgen05 kernels do not take (mma.sync reconstruction, everything after it in fp32).

Operands are bf16 and their products exact; sums of up to 1024 of them in fp32 leave about 2^-24 sqrt(1024) = 2e-6 relative
error in a key, a score error of that size times the score, and as much again in the value sums: 3e-5 of the row rms beside
the rounding of the bf16 output leaves a factor of ten."""
import numpy as np
import pytest

from oracle import lorc_oracle as O
from workloads import synth

import helpers as H

pytestmark = pytest.mark.gpu


def _close(got, want):
    rms = np.sqrt(np.mean(want ** 2, axis=-1, keepdims=True))
    excess = np.abs(got - want) - (0.5 * H.bf16_ulp(want) + 3e-5 * rms)
    assert np.all(excess <= 0.0), float((excess / rms).max())


@pytest.mark.parametrize("D,H_q,H_kv,d_h,r_k,r_v,lens,style,page,n_splits", [
    (256, 4, 2, 64, 32, 32, [129], 0, 0, 0),                  # two shares of whole steps and one of a single token
    (256, 4, 2, 64, 8, 128, [1, 63, 64, 65], 1, 16, 0),       # one block of 32 latent columns, mostly empty
    (256, 2, 2, 64, 40, 24, [128, 300], 2, 48, 3),            # one query head per KV head; a page size no power of two
    (256, 16, 2, 64, 72, 104, [700, 2], 0, 0, 0),             # eight query heads per KV head
    (1024, 16, 16, 64, 1024, 1024, [200], 1, 0, 5),           # 128 column groups: one token group
    (384, 9, 3, 128, 200, 136, [65, 257], 1, 32, 0),          # odd number of KV heads, three query heads each
    (384, 18, 3, 128, 16, 384, [513], 0, 0, 0),
    (256, 2, 2, 128, 256, 8, [31, 192], 0, 0, 200),           # more shares than steps
])
def test_small_decode(D, H_q, H_kv, d_h, r_k, r_v, lens, style, page, n_splits):
    import torch
    prob = H.Problem(D, H_q, H_kv, d_h, r_k, r_v, theta=10000.0, layer=33, style=style)
    b, n_max = len(lens), max(lens) + 3
    sess = H.Session(prob, max_pos=n_max, batch=b)
    L = sess.L
    ck, cv = H.oracle_latents(prob, [synth.hidden_states(n, D, 33, chunk=s).astype(np.float64) for s, n in enumerate(lens)])
    held = H.paged_cache(sess, b, lens, page, 7, ck, cv) if page else H.contiguous_cache(sess, b, n_max, lens, ck, cv)
    for q_scale in (1.0, 8.0, 64.0):
        q = synth.queries(b, H_q, d_h, 33, int(q_scale), q_scale).astype(np.float64)
        want = H.oracle_decode(prob, ck, cv, q)
        for entry in (L.lorc_decode_attn, L.lorc_decode_attn_static):
            out = torch.full((b, H_q, d_h), 3.0, dtype=torch.bfloat16, device="cuda")
            entry(sess.ctx, 0, held[0], H.dev_bf16(q), out, n_splits=n_splits)
            assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
            assert L.lorc_last_path(sess.ctx) == 1
            _close(H.host_f64(out), want)
    sess.close()


@pytest.mark.parametrize("entry,flags,r_v", [("lorc_decode_attn", 0, 1032), ("lorc_decode_attn", 1, 1536), ("lorc_decode_attn_static", 0, 1160)])
def test_value_ranks_above_1024(entry, flags, r_v):
    """Ranks that only the scalar kernel takes: its blocks cover 1024 columns of the latent output each."""
    import torch
    L = H.lib()
    D, H_q, H_kv, d_h, r_k, lens = 64, 32, 32, 64, 16, [70, 33]
    n, b, rng = H_kv * d_h, len(lens), np.random.default_rng(r_v)
    A_k, A_v = (synth.to_bf16_exact(rng.standard_normal((D, r))) for r in (r_k, r_v))
    B_k, B_v = (synth.to_bf16_exact(rng.standard_normal((r, n)) / np.sqrt(n)) for r in (r_k, r_v))
    ctx = L.lorc_create(1, D, H_q, H_kv, d_h, 10000.0, max_pos=72, flags=flags)
    L.lorc_load_factors(ctx, 0, L.LORC_MODE_LATENT, r_k, r_v, *[H.dev_bf16(a) for a in (A_k, B_k, A_v, B_v)])
    ws = torch.full((L.lorc_workspace_bytes(ctx, b, 72),), 255, dtype=torch.uint8, device="cuda")
    L.lorc_set_workspace(ctx, ws)
    ck, cv = ([synth.to_bf16_exact(rng.standard_normal((m, r))) for m in lens] for r in (r_k, r_v))
    kv = [torch.zeros(b, 72, r, dtype=torch.bfloat16, device="cuda") for r in (r_k, r_v)]
    for c, rows in zip(kv, (ck, cv)):
        for s, x in enumerate(rows):
            c[s, :lens[s]] = H.dev_bf16(x)
    sl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    cache = L.make_cache(*kv, sl, b, 72, seq_stride=72)
    q = synth.queries(b, H_q, d_h, 33, 1, 1.0).astype(np.float64)
    for n_splits in (0, 2):
        out = torch.full((b, H_q, d_h), 3.0, dtype=torch.bfloat16, device="cuda")
        getattr(L, entry)(ctx, 0, cache, H.dev_bf16(q), out, n_splits=n_splits)
        assert L.lorc_sync_status(ctx) == 0, L.lorc_last_error(ctx)
        for s in range(b):
            _close(H.host_f64(out[s]), O.decode_attn_latent(ck[s], cv[s], B_k, B_v, q[s], H_kv, 10000.0))
    L.lorc_destroy(ctx)
