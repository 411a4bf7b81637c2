"""Small-shape decode whose context shares merge inside the kernel: both sides of the rule's lines (two heads per KV head, eight
shares, r_v * d_h = 8192, one round of blocks, for 128-wide heads also r_v = 32 and a share per head), shares without tokens, an empty
sequence.  Against the oracle, to the rounding of the output (bound as in test_gpu_small_decode.py); the launches tell which way
a call went."""
import numpy as np
import pytest

from workloads import synth

import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,H_q,H_kv,d_h,r_v,lens,n_splits,launches", [
    (256, 2, 2, 64, 128, [512, 1], 0, 1),           # eight shares; sequences shorter than them
    (256, 6, 2, 64, 120, [513], 0, 2),              # nine shares, three heads
    (256, 4, 2, 64, 120, [513], 0, 2),              # nine shares
    (256, 12, 3, 64, 136, [130], 0, 2),             # four heads, the rank above the line
    (256, 6, 3, 64, 136, [130], 0, 2),              # the rank above the line
    (256, 6, 3, 64, 128, [130], 0, 1),
    (256, 4, 1, 128, 64, [400, 64], 5, 2),          # four heads
    (384, 6, 3, 128, 64, [400, 64], 5, 1),          # shares that do not divide the heads
    (384, 6, 3, 128, 64, [400, 64], 1, 2),          # fewer shares than heads
    (384, 6, 3, 128, 24, [400, 64], 5, 2),          # a rank below the line
    (384, 24, 3, 128, 56, [70, 300], 3, 2),         # eight heads
    (384, 24, 3, 128, 72, [70, 300], 3, 2),
    (256, 4, 2, 64, 8, [17], 1, 1),                 # one share: no cluster; two heads in series
    (256, 16, 2, 64, 32, [40], 0, 2),               # eight heads, one share
    (256, 4, 2, 64, 8, [70] * 98, 2, 2),             # 396 blocks, of 394 that merge
    (256, 4, 2, 64, 8, [70] * 97, 2, 1),            # 392
    (256, 2, 2, 64, 8, [400] * 12, 6, 2),           # 156 blocks in clusters of six, of 148 that merge
    (256, 2, 2, 64, 8, [400] * 11, 6, 1),
])
def test_merge_inside(D, H_q, H_kv, d_h, r_v, lens, n_splits, launches):
    import torch
    prob = H.Problem(D, H_q, H_kv, d_h, 40, r_v, theta=10000.0, layer=34)
    b, n_max = len(lens), max(lens)
    sess = H.Session(prob, max_pos=n_max, batch=b + 1)
    L = sess.L
    ck, cv = H.oracle_latents(prob, [synth.hidden_states(n, D, 34, chunk=s).astype(np.float64) for s, n in enumerate(lens)])
    q = synth.queries(b + 1, H_q, d_h, 34, 1, 8.0).astype(np.float64)
    want = H.oracle_decode(prob, ck, cv, q[:b])
    none = [np.zeros((0, c[0].shape[1])) for c in (ck, cv)]
    held = H.contiguous_cache(sess, b + 1, n_max, lens + [0], ck + [none[0]], cv + [none[1]])
    for entry in (L.lorc_decode_attn, L.lorc_decode_attn_static):
        out = torch.full((b + 1, H_q, d_h), 3.0, dtype=torch.bfloat16, device="cuda")
        before = L.lorc_launch_count(sess.ctx)
        entry(sess.ctx, 0, held[0], H.dev_bf16(q), out, n_splits=n_splits)
        if entry is L.lorc_decode_attn and torch.cuda.get_device_properties(0).multi_processor_count == 148:
            assert L.lorc_launch_count(sess.ctx) - before == launches
        assert L.lorc_sync_status(sess.ctx) == L.LORC_ERR_EMPTY and L.lorc_last_path(sess.ctx) == 1
        got, rms = H.host_f64(out), np.sqrt(np.mean(want ** 2, axis=-1, keepdims=True))
        assert np.all(np.abs(got[:b] - want) <= 0.5 * H.bf16_ulp(want) + 3e-5 * rms)
        assert np.all(got[b] == 0.0)
    sess.close()
