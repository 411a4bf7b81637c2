"""Prompt kernels whose units shrink for short launches: reconstruction by single heads (up to four pairs of 128-token tiles with eight
KV heads) against units of two heads; rank tails, odd tile counts, pages.  Bound as in the other prompt tests."""
import numpy as np
import pytest

from oracle import lorc_oracle as O
from workloads import synth

import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H_q,r_k,r_v,lens,T,page", [
    (32, 200, 72, [450, 130], 60, 16),         # four pairs of tiles: single heads; rank tails below a slice
    (64, 72, 200, [385], 385, 0),              # odd number of tiles; eight heads per KV head
    (32, 72, 200, [300, 200, 129], 40, 128),   # six pairs: two heads per unit
])
def test_reconstruction_units(H_q, r_k, r_v, lens, T, page):
    import torch
    prob = H.Problem(1024, H_q, 8, 128, r_k, r_v, theta=500000.0, layer=24)
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
