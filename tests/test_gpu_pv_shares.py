"""Context shares of the P.C_V kernel: one cluster, several clusters, counts that divide neither the tiles nor the groups of columns
that a share adds up; the number of shares that the library takes by itself for long contexts."""
import numpy as np
import pytest

from workloads import synth

import helpers as H

pytestmark = pytest.mark.gpu

TOL = 1e-2      # three bf16 roundings of about 2e-3 each (numerators, latent output, output), as in the other decode tests


def _case(H_q, r_v, lens, style):
    prob = H.Problem(1024, H_q, 8, 128, 64, r_v, theta=500000.0, layer=23, style=style)
    rng = np.random.default_rng(r_v)
    ck, cv = ([synth.to_bf16_exact(rng.standard_normal((n, r)) * np.arange(1, r + 1) ** -0.8) for n in lens] for r in (64, r_v))
    q = synth.queries(len(lens), H_q, 128, 23, 1, 8.0).astype(np.float64)
    sess = H.Session(prob, max_pos=max(lens), batch=len(lens))
    return sess, H.contiguous_cache(sess, len(lens), max(lens), lens, ck, cv), q, ck, cv


def _run(sess, held, q, lens, S):
    """The result, and the denominators [b, H_q] that the call gives as the only shard of the context, with the same result.
    (Sums in fp32 over the shares: with interleaved pairs, whose numerators have 16 bits, they show the number of shares to the
    bit; sums of a few thousand 8-bit numerators are mostly exact.)"""
    import torch
    L, b = sess.L, len(lens)
    outs = [torch.full(q.shape, 3.0, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    pos = torch.tensor([[0] * b, [n - 1 for n in lens]], dtype=torch.int32, device="cuda")
    ml = torch.zeros(*q.shape[:2], 2, dtype=torch.float32, device="cuda")
    L.lorc_decode_attn(sess.ctx, 0, held[0], H.dev_bf16(q), outs[0], n_splits=S)
    L.lorc_decode_attn_shard(sess.ctx, 0, held[0], H.dev_bf16(q), pos[0], pos[1], outs[1], ml, n_splits=S)
    assert L.lorc_sync_status(sess.ctx) == 0, (S, L.lorc_last_error(sess.ctx))
    assert L.lorc_last_path(sess.ctx) == 2 and torch.equal(*outs)
    return outs[0], ml[..., 1]


def _same(a, b):
    import torch
    return torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("H_q,r_v,lens,style", [
    (32, 264, [4096, 33, 1], 0),      # 32 tiles, three column blocks, the last of 8 columns; shares without tiles
    (64, 128, [4090], 0),
    (32, 136, [4096, 700], 1),        # numerators in two parts
    (64, 72, [4050], 1),
])
def test_share_counts(H_q, r_v, lens, style):
    import torch
    sess, held, q, ck, cv = _case(H_q, r_v, lens, style)
    b, L = len(lens), sess.L
    want = H.oracle_decode(sess.prob, ck, cv, q)
    # room for 32 shares of every block, and nothing finite in it to begin with
    blocks = b * ((r_v + 127) // 128)
    room = torch.full((sess.ws.numel() + blocks * 32 * H_q * 129 * 4,), 255, dtype=torch.uint8, device="cuda")
    L.lorc_set_workspace(sess.ctx, room)
    outs = {}
    for S in (2, 5, 7, 8, 9, 15, 16, 17, 31, 32, 64, 17, 32):
        got = _run(sess, held, q, lens, S)
        H.assert_rows_close(H.host_f64(got[0]), want, TOL, S)
        assert S not in outs or _same(outs[S], got), S        # what counts the clusters is left at zero
        outs[S] = got
    # 16 shares (all with two tiles) in one cluster where the GPU takes it, 17 (the last without tiles) in several: the same sums
    assert _same(outs[16], outs[17])
    assert _same(outs[32], outs[64])                          # never more shares than tiles
    for a, c in ((8, 16), (16, 32)) if style else ():
        assert not _same(outs[a], outs[c]), (a, c)
    # the least workspace (tile images, latent output) takes the shares that run at once as one cluster (interleaved: up to four
    # blocks, whose clusters of 16 do; otherwise fewer shares); below that the call is refused
    img = b * 32 * (2 * H_q * (1 + style) * 128 + 8 * H_q * 4)
    least = -(-img // 256) * 256 + b * H_q * (1 + style) * 1024 * 2
    L.lorc_set_workspace(sess.ctx, room[:least])
    for S in (16, 32):
        got = _run(sess, held, q, lens, S)
        assert _same(got, outs[16]) if style else True
        H.assert_rows_close(H.host_f64(got[0]), want, TOL, S)
    if not style:
        L.lorc_set_workspace(sess.ctx, room[:least - 256])
        with pytest.raises(L.LorcError) as e:
            _run(sess, held, q, lens, 1)
        assert e.value.code == L.LORC_ERR_WORKSPACE
    sess.close()


@pytest.mark.parametrize("H_q,r_v,lens,shares,fewer", [
    (32, 128, [32777], 20, 16),                    # more shares than the largest cluster has blocks
    (64, 264, [8201, 90, 1, 4000, 17, 300, 64, 2000], 6, 5),      # as many blocks as there are SMs, nearly
])
def test_share_count_does_not_depend_on_the_clusters(H_q, r_v, lens, shares, fewer):
    """Without a share count the plan follows from the sizes and the number of SMs: to the bit what that number of shares gives."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the expected counts are those of 148 SMs")
    sess, held, q, ck, cv = _case(H_q, r_v, lens, 1)
    outs = [_run(sess, held, q, lens, S) for S in (0, shares, fewer)]
    H.assert_rows_close(H.host_f64(outs[0][0]), H.oracle_decode(sess.prob, ck, cv, q), TOL)
    assert _same(outs[0], outs[1]) and not _same(outs[0], outs[2])
    sess.close()


def test_share_counts_first_seen_under_stream_capture():
    """A plan may ask for cluster sizes that no call before has asked for while the stream is being captured."""
    import torch
    sess, held, q, ck, cv = _case(32, 136, [4096], 1)
    L, qd, stream = sess.L, H.dev_bf16(q), torch.cuda.Stream()
    _run(sess, held, q, [4096], 1)                       # sets the context's tables up
    outs = {S: torch.zeros(q.shape, dtype=torch.bfloat16, device="cuda") for S in (7, 17)}
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for S, out in outs.items():
            L.lorc_decode_attn(sess.ctx, 0, held[0], qd, out, n_splits=S)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
    for S, out in outs.items():
        assert torch.equal(out, _run(sess, held, q, [4096], S)[0]), S
    del graph
    sess.close()
