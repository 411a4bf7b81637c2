"""Context shares of the P.C_V kernel as clusters: the largest cluster, share counts above it, counts that divide neither the
tiles nor the groups of columns that a share adds up."""
import numpy as np
import pytest

from workloads import synth

import helpers as H

pytestmark = pytest.mark.gpu

TOL = 1e-2      # three bf16 roundings of about 2e-3 each (numerators, latent output, output), as in the other decode tests


@pytest.mark.parametrize("H_q,r_v,lens", [
    (32, 264, [2600, 33, 1]),      # 21 tiles, three column blocks, the last of 8 columns; shares without tiles
    (64, 128, [2200]),
])
def test_share_counts_around_the_largest_cluster(H_q, r_v, lens):
    import torch
    prob = H.Problem(1024, H_q, 8, 128, 64, r_v, theta=500000.0, layer=23)
    b, rng = len(lens), np.random.default_rng(r_v)
    ck, cv = ([synth.to_bf16_exact(rng.standard_normal((n, r)) * np.arange(1, r + 1) ** -0.8) for n in lens] for r in (64, r_v))
    q = synth.queries(b, H_q, 128, 23, 1, 8.0).astype(np.float64)
    sess = H.Session(prob, max_pos=max(lens), batch=b)
    held = H.contiguous_cache(sess, b, max(lens), lens, ck, cv)
    want = H.oracle_decode(prob, ck, cv, q)
    outs = {}
    for S in (2, 5, 7, 9, 15, 16, 17, 64):
        out = torch.zeros(b, H_q, 128, dtype=torch.bfloat16, device="cuda")
        sess.L.lorc_decode_attn(sess.ctx, 0, held[0], H.dev_bf16(q), out, n_splits=S)
        assert sess.L.lorc_sync_status(sess.ctx) == 0, S
        H.assert_rows_close(H.host_f64(out), want, TOL, S)
        outs[S] = out
    assert torch.equal(outs[16], outs[17]) and torch.equal(outs[16], outs[64])      # no more shares than the largest cluster
    sess.close()
