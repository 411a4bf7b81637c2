"""Prompt kernels whose units shrink for short launches: reconstruction by single heads (up to four pairs of 128-token tiles with eight
KV heads, nine with four) against units of two heads; rank tails, odd tile counts, pages.  Bound as in the other prompt tests."""
import numpy as np
import pytest

from oracle import lorc_oracle as O
from workloads import synth

import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H_q,H_kv,r_k,r_v,lens,T,page", [
    (32, 8, 200, 72, [450, 130], 60, 16),         # four pairs of tiles: single heads; rank tails below a slice
    (64, 8, 72, 200, [385], 385, 0),              # eight heads per KV head
    (32, 8, 72, 200, [300, 200, 129], 40, 128),   # six pairs: two heads per unit
    (64, 8, 72, 72, [257], 257, 0),               # single heads, an odd number of tiles: the pair's second tile lies past the end
    (32, 8, 136, 64, [384, 129], 50, 64),
    (32, 8, 64, 72, [1100], 33, 0),               # five pairs, nine tiles: two heads per unit
    (32, 4, 72, 64, [130] * 9, 20, 0),            # nine pairs with four KV heads: single heads, 72 units for 74 pairs of SMs
    (32, 4, 72, 64, [130] * 10, 20, 32),          # ten: two heads
])
def test_reconstruction_units(H_q, H_kv, r_k, r_v, lens, T, page):
    import torch
    prob = H.Problem(1024, H_q, H_kv, 128, r_k, r_v, theta=500000.0, layer=24)
    b, n_max = len(lens), max(lens)
    sess = H.Session(prob, max_pos=n_max, batch=b)
    ck, cv = H.oracle_latents(prob, [synth.hidden_states(n, prob.D, 24, chunk=s).astype(np.float64) for s, n in enumerate(lens)])
    held = H.paged_cache(sess, b, lens, page, 5, ck, cv) if page else H.contiguous_cache(sess, b, n_max, lens, ck, cv)
    q = synth.to_bf16_exact(8.0 * synth.gaussian((b, T, H_q, 128), 24, 78)).astype(np.float64)
    ws = torch.zeros(sess.L.lorc_prefill_workspace_bytes(sess.ctx, b, n_max, T), dtype=torch.uint8, device="cuda")
    sess.L.lorc_set_workspace(sess.ctx, ws)
    out = torch.zeros(b, T, H_q, 128, dtype=torch.bfloat16, device="cuda")
    sess.L.lorc_prefill_attn(sess.ctx, 0, held[0], H.dev_bf16(q), out, T)
    assert sess.L.lorc_sync_status(sess.ctx) == 0 and sess.L.lorc_last_path(sess.ctx) == 2
    want = np.stack([O.prefill_attn_latent(ck[s], cv[s], prob.B_k, prob.B_v, q[s], prob.H_kv, prob.theta) for s in range(b)])
    H.assert_rows_close(H.host_f64(out), want, 1e-2)
    sess.close()
