"""Interleaved rotary pairs on the tensor-core decode path: numerators and latent outputs in two bf16 parts.

The path took over from the plain fp32 kernels, so its results carry no more error than theirs: the rounding of the bf16
output, and beside it 2e-4 of the row rms.  (Two bf16 parts hold 16 significant bits: 2^-17 = 8e-6 relative per numerator
and per latent output; fp32 sums of up to 1024 products add about 2^-24 sqrt(1024) = 2e-6 per score unit.  An element is a
sum of many such terms of random sign, the row rms their common scale; 2e-4 leaves a factor of ten.)"""
import numpy as np
import pytest

from oracle import lorc_oracle as O
from workloads import synth

import helpers as H

pytestmark = pytest.mark.gpu

INTERLEAVED = 1
G8B = dict(D=1024, H_q=32, H_kv=8, d_h=128)
G70B = dict(D=1024, H_q=64, H_kv=8, d_h=128)
G_N512 = dict(D=512, H_q=32, H_kv=4, d_h=128)      # eight query heads per KV head on 32 heads


def _problem(geom, r_k, r_v, lens, flags=0):
    prob = H.Problem(r_k=r_k, r_v=r_v, theta=500000.0, layer=31, style=INTERLEAVED, **geom)
    sess = H.Session(prob, max_pos=max(lens) + 3, batch=len(lens), flags=flags)
    xs = [synth.hidden_states(n, prob.D, 31, chunk=s).astype(np.float64) for s, n in enumerate(lens)]
    return prob, sess, *H.oracle_latents(prob, xs)


def _close(got, want):
    rms = np.sqrt(np.mean(want ** 2, axis=-1, keepdims=True))
    excess = np.abs(got - want) - (0.5 * H.bf16_ulp(want) + 2e-4 * rms)
    assert np.all(excess <= 0.0), float((excess / rms).max())


@pytest.mark.parametrize("geom,r_k,r_v,lens,page,n_splits", [
    (G8B, 72, 136, [1, 37, 128, 129], 0, 0),        # rank tails, a sequence that ends a tile, one that starts the next
    (G8B, 512, 512, [700, 2], 0, 1),                # one share per column block
    (G8B, 264, 64, [513, 300, 5], 16, 0),
    (G70B, 136, 248, [257, 640], 64, 0),            # 64 heads: 128 rows of numerators, three stages
    (G70B, 64, 128, [385, 1], 0, 2),
    (G_N512, 192, 96, [200, 511], 128, 0),
])
def test_interleaved_decode(geom, r_k, r_v, lens, page, n_splits):
    import torch
    prob, sess, ck, cv = _problem(geom, r_k, r_v, lens)
    L, b = sess.L, len(lens)
    if page:
        held = H.paged_cache(sess, b, lens, page, order_seed=5, k_rows=ck, v_rows=cv)
    else:
        held = H.contiguous_cache(sess, b, max(lens) + 3, lens, ck, cv)
    for q_scale in (1.0, 8.0, 64.0):
        q = synth.queries(b, prob.H_q, 128, 31, int(q_scale), q_scale).astype(np.float64)
        out = torch.zeros(b, prob.H_q, 128, dtype=torch.bfloat16, device="cuda")
        L.lorc_decode_attn(sess.ctx, 0, held[0], H.dev_bf16(q), out, n_splits=n_splits)
        assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
        assert L.lorc_last_path(sess.ctx) == 2, "the tensor-core path was not taken"
        _close(H.host_f64(out), H.oracle_decode(prob, ck, cv, q))
    lat = torch.zeros(b, prob.H_q, r_v, dtype=torch.bfloat16, device="cuda")
    L.lorc_decode_attn_latent_out(sess.ctx, 0, held[0], H.dev_bf16(q), lat, n_splits=n_splits)
    assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
    for s in range(b):
        _close(H.host_f64(lat[s]), O.decode_attn_latent_out(ck[s], cv[s], prob.B_k, q[s], prob.H_kv, prob.theta, INTERLEAVED))
    sess.close()


def test_interleaved_falls_back_to_plain_kernels():
    """A workspace that only holds the plain kernels' partial results, and a first call under stream capture (no table may
    be allocated then), run the plain kernels; the call after it may take the tensor-core path."""
    import torch
    lens = [300, 40]
    prob, sess, ck, cv = _problem(G8B, 96, 96, lens)
    L, b = sess.L, len(lens)
    held = H.contiguous_cache(sess, b, max(lens) + 3, lens, ck, cv)
    q = synth.queries(b, prob.H_q, 128, 31, 1, 8.0).astype(np.float64)
    qd, want = H.dev_bf16(q), H.oracle_decode(prob, ck, cv, q)
    out = torch.zeros(b, prob.H_q, 128, dtype=torch.bfloat16, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        L.lorc_decode_attn(sess.ctx, 0, held[0], qd, out)
        assert L.lorc_last_path(sess.ctx) == 1
    graph.replay()
    assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
    _close(H.host_f64(out), want)
    for nbytes, path in ((b * prob.H_q * (96 + 2) * 4 + 512, 1), (None, 2)):
        L.lorc_set_workspace(sess.ctx, sess.ws, nbytes)
        out.zero_()
        L.lorc_decode_attn(sess.ctx, 0, held[0], qd, out)
        assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
        assert L.lorc_last_path(sess.ctx) == path
        _close(H.host_f64(out), want)
    with torch.cuda.graph(graph2 := torch.cuda.CUDAGraph()):
        L.lorc_decode_attn(sess.ctx, 0, held[0], qd, out)
        assert L.lorc_last_path(sess.ctx) == 2
    for _ in range(2):
        out.zero_()
        graph2.replay()
        assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
        _close(H.host_f64(out), want)
    del graph, graph2
    sess.close()


def test_interleaved_context_shards():
    import torch
    from paper_2410_03111_b200 import sharded
    lens, world = [700, 130, 17], 2
    prob, sess, ck, cv = _problem(G8B, 160, 96, lens)
    L, b = sess.L, len(lens)
    q = synth.queries(b, prob.H_q, 128, 31, 2, 8.0).astype(np.float64)
    qd = H.dev_bf16(q)
    pos0, cnt = sharded.shard_bounds(lens, world)
    q_pos = torch.tensor([n - 1 for n in lens], dtype=torch.int32, device="cuda")
    outs = torch.zeros(world, b, prob.H_q, 128, dtype=torch.bfloat16, device="cuda")
    mls = torch.zeros(world, b, prob.H_q, 2, dtype=torch.float32, device="cuda")
    for r in range(world):
        rows = [[c[s][pos0[r][s]:pos0[r][s] + cnt[r][s]] for s in range(b)] for c in (ck, cv)]
        held = H.contiguous_cache(sess, b, max(lens) + 3, cnt[r], *rows)
        p0 = torch.tensor(pos0[r], dtype=torch.int32, device="cuda")
        L.lorc_decode_attn_shard(sess.ctx, 0, held[0], qd, p0, q_pos, outs[r], mls[r])
        assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
        assert L.lorc_last_path(sess.ctx) == 2
        for s in range(b):
            a, n = pos0[r][s], cnt[r][s]
            if n:
                pos = np.arange(a, a + n)
                _close(H.host_f64(outs[r, s]), O.decode_attn_latent(ck[s][a:a + n], cv[s][a:a + n], prob.B_k, prob.B_v, q[s],
                                                                    prob.H_kv, prob.theta, INTERLEAVED, pos, lens[s] - 1))
                lse = O.shard_log2_sum_exp(ck[s][a:a + n], prob.B_k, q[s], prob.H_kv, prob.theta, pos, lens[s] - 1, INTERLEAVED)
                ml = H.host_f64(mls[r, s])
                assert np.max(np.abs(ml[:, 0] + np.log2(ml[:, 1]) - lse)) <= 2e-4
    merged = torch.zeros(b, prob.H_q, 128, dtype=torch.bfloat16, device="cuda")
    L.lorc_merge_shards(sess.ctx, world, outs, mls, merged, b)
    assert L.lorc_sync_status(sess.ctx) == 0
    H.assert_rows_close(H.host_f64(merged), H.oracle_decode(prob, ck, cv, q), 1e-2)
    sess.close()


@pytest.mark.parametrize("geom,page,n_splits", [(G8B, 0, 1), (G8B, 16, 2), (G70B, 64, 0), (G70B, 0, 3)])
def test_interleaved_rows_past_the_end_may_hold_anything(geom, page, n_splits):
    """Cache rows past a sequence's end, and pages that no sequence uses (the pool's first among them), hold NaN."""
    import torch
    lens = [385, 128, 17, 250]
    prob, sess, ck, cv = _problem(geom, 72, 200, lens)
    L, b = sess.L, len(lens)
    n_max, nan = max(lens) + 3, float("nan")
    q = synth.queries(b, prob.H_q, 128, 31, 5, 8.0).astype(np.float64)
    sl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    kv = []
    if page:
        per = (n_max + page - 1) // page
        table = 1 + np.random.default_rng(3).permutation(b * per).reshape(b, per).astype(np.int32)
        for rows, r in ((ck, 72), (cv, 200)):
            c = torch.full((b * per + 1, page, r), nan, dtype=torch.bfloat16, device="cuda")
            for s in range(b):
                for i in range(0, lens[s], page):
                    part = H.dev_bf16(rows[s][i:i + page])
                    c[int(table[s, i // page]), :part.shape[0]] = part
            kv.append(c)
        tab = torch.from_numpy(table).cuda()
        cache = L.make_cache(*kv, sl, b, max(lens), page_table=tab, page_size=page, max_pages_per_seq=per, n_pages=b * per + 1)
    else:
        for rows, r in ((ck, 72), (cv, 200)):
            c = torch.full((b, n_max, r), nan, dtype=torch.bfloat16, device="cuda")
            for s in range(b):
                c[s, :lens[s]] = H.dev_bf16(rows[s])
            kv.append(c)
        cache = L.make_cache(*kv, sl, b, max(lens), seq_stride=n_max)
    out = torch.zeros(b, prob.H_q, 128, dtype=torch.bfloat16, device="cuda")
    L.lorc_decode_attn(sess.ctx, 0, cache, H.dev_bf16(q), out, n_splits=n_splits)
    assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
    assert L.lorc_last_path(sess.ctx) == 2
    _close(H.host_f64(out), H.oracle_decode(prob, ck, cv, q))
    sess.close()


@pytest.mark.parametrize("geom,page,n_splits", [(G8B, 16, 1), (G8B, 64, 0), (G70B, 32, 2), (G_N512, 128, 0)])
def test_interleaved_pages_outside_the_pool_are_left_out(geom, page, n_splits):
    import torch
    lens = [500, 300, 20]
    prob, sess, ck, cv = _problem(geom, 96, 136, lens)
    L, b = sess.L, len(lens)
    held = H.paged_cache(sess, b, lens, page, order_seed=6, k_rows=ck, v_rows=cv)
    cache, k, v, sl, ptd, pt = held
    live = [np.ones(n, dtype=bool) for n in lens]
    for s, i, entry in ((0, 0, -1), (0, (lens[0] - 1) // page, 10 ** 6), (1, 1, cache.n_pages)):
        ptd[s, i] = entry
        live[s][i * page:(i + 1) * page] = False
    q = synth.queries(b, prob.H_q, 128, 31, 6, 8.0).astype(np.float64)
    out = torch.zeros(b, prob.H_q, 128, dtype=torch.bfloat16, device="cuda")
    L.lorc_decode_attn(sess.ctx, 0, cache, H.dev_bf16(q), out, n_splits=n_splits)
    assert L.lorc_sync_status(sess.ctx) == L.LORC_ERR_CAPACITY
    assert L.lorc_last_path(sess.ctx) == 2
    for s in range(b):
        pos = np.flatnonzero(live[s])
        _close(H.host_f64(out[s]), O.decode_attn_latent(ck[s][pos], cv[s][pos], prob.B_k, prob.B_v, q[s], prob.H_kv, prob.theta,
                                                        INTERLEAVED, pos, lens[s] - 1))
    sess.close()


@pytest.mark.parametrize("page", [0, 16])
def test_interleaved_length_beyond_the_capacity(page):
    """The rows that exist are attended, by a query at the end of the length given; the status word reports it."""
    import torch
    rows = 208 if page else 203
    prob, sess, ck, cv = _problem(G8B, 96, 64, [rows, rows])
    L, lens = sess.L, [rows + 2, 90]
    if page:
        held = H.paged_cache(sess, 2, [rows, rows], page, order_seed=6, k_rows=ck, v_rows=cv)
    else:
        held = H.contiguous_cache(sess, 2, rows, [rows, rows], ck, cv)
    held[3][:] = torch.tensor(lens, dtype=torch.int32)
    q = synth.queries(2, prob.H_q, 128, 31, 7, 8.0).astype(np.float64)
    out = torch.zeros(2, prob.H_q, 128, dtype=torch.bfloat16, device="cuda")
    L.lorc_decode_attn(sess.ctx, 0, held[0], H.dev_bf16(q), out)
    assert L.lorc_sync_status(sess.ctx) == L.LORC_ERR_CAPACITY
    assert L.lorc_last_path(sess.ctx) == 2
    for s, n in enumerate((rows, 90)):
        _close(H.host_f64(out[s]), O.decode_attn_latent(ck[s][:n], cv[s][:n], prob.B_k, prob.B_v, q[s], prob.H_kv, prob.theta,
                                                        INTERLEAVED, np.arange(n), lens[s] - 1))
    sess.close()


@pytest.mark.parametrize("style", [0, INTERLEAVED])
def test_nan_in_a_cached_row_is_an_argument_error_for_both_pairings(style):
    import torch
    prob = H.Problem(r_k=64, r_v=64, theta=500000.0, layer=31, style=style, **G8B)
    sess = H.Session(prob, max_pos=300, batch=2)
    L, lens = sess.L, [290, 40]
    rng = np.random.default_rng(1)
    rows = [[synth.to_bf16_exact(rng.standard_normal((n, 64))) for n in lens] for _ in "kv"]
    cache, k, v, sl = H.contiguous_cache(sess, 2, 300, lens, *rows)
    q = H.dev_bf16(synth.queries(2, prob.H_q, 128, 31, 8, 8.0))
    out = torch.zeros(2, prob.H_q, 128, dtype=torch.bfloat16, device="cuda")
    L.lorc_decode_attn(sess.ctx, 0, cache, q, out)
    assert L.lorc_sync_status(sess.ctx) == 0
    k[0, 133, 5] = float("nan")
    L.lorc_decode_attn(sess.ctx, 0, cache, q, out)
    assert L.lorc_sync_status(sess.ctx) == L.LORC_ERR_ARG
    assert L.lorc_last_path(sess.ctx) == 2
    sess.close()


@pytest.mark.parametrize("style", [0, INTERLEAVED])
def test_shards_that_are_empty_or_end_behind_the_query(style):
    """An empty shard is no error wherever it starts; a shard whose last token lies behind the query is treated as empty and
    reported, whatever the workspace holds."""
    import torch
    prob = H.Problem(r_k=64, r_v=64, theta=500000.0, layer=31, style=style, **G8B)
    sess = H.Session(prob, max_pos=400, batch=2)
    L = sess.L
    rng = np.random.default_rng(1)
    rows = [[synth.to_bf16_exact(rng.standard_normal((200, 64))) for _ in range(2)] for _ in "kv"]
    cache, k, v, sl = H.contiguous_cache(sess, 2, 200, [200, 200], *rows)
    q = H.dev_bf16(synth.queries(2, prob.H_q, 128, 31, 9, 8.0))

    def shard(lens, pos0, q_pos):
        sl[:] = torch.tensor(lens, dtype=torch.int32)
        out = torch.full((2, prob.H_q, 128), 3.0, dtype=torch.bfloat16, device="cuda")
        ml = torch.full((2, prob.H_q, 2), 3.0, dtype=torch.float32, device="cuda")
        at = [torch.tensor(p, dtype=torch.int32, device="cuda") for p in (pos0, q_pos)]
        sess.ws.fill_(255)                                       # NaN in every stale tile image
        L.lorc_decode_attn_shard(sess.ctx, 0, cache, q, *at, out, ml)
        status = L.lorc_sync_status(sess.ctx)
        assert L.lorc_last_path(sess.ctx) == 2
        return status, H.host_f64(out), H.host_f64(ml)

    status, ref, _ = shard([0, 150], [0, 100], [99, 260])
    assert status == 0 and np.all(ref[0] == 0.0)
    status, out, ml = shard([0, 150], [256, 100], [99, 260])     # the empty shard starts behind the query
    assert status == 0, L.lorc_last_error(sess.ctx)
    assert np.all(out[0] == 0.0) and np.all(ml[0, :, 1] == 0.0) and np.array_equal(out[1], ref[1])
    status, out, ml = shard([200, 150], [100, 100], [298, 260])  # the first shard's last token sits at 299
    assert status == L.LORC_ERR_CAPACITY
    assert np.all(out[0] == 0.0) and np.all(ml[0, :, 1] == 0.0) and np.array_equal(out[1], ref[1])
    sess.close()


@pytest.mark.parametrize("geom,lens,page,n_splits", [
    (G8B, [2049, 1990, 17, 128], 0, 0),             # the default plan: six shares at 17 tiles
    (G8B, [2100, 600], 64, 2),
    (G8B, [2049, 40], 0, 7),                        
    (G8B, [2049, 1500], 16, 8),                     
    (G_N512, [1700, 900, 1], 0, 12),
    (G70B, [1300, 130], 0, 3),                      # two parts of 64 heads
    (G70B, [1100, 700], 128, 5),
])
def test_interleaved_several_context_shares(geom, lens, page, n_splits):
    """Each share leaves the sum of both parts behind the memory that the parts' exchange used, and adds up its columns of all."""
    import torch
    prob = H.Problem(r_k=64, r_v=136, theta=500000.0, layer=31, style=INTERLEAVED, **geom)
    L, b = H.lib(), len(lens)
    sess = H.Session(prob, max_pos=max(lens) + 3, batch=b)
    rng = np.random.default_rng(n_splits)
    ck, cv = ([synth.to_bf16_exact(rng.standard_normal((n, r)) * np.arange(1, r + 1) ** -0.8) for n in lens] for r in (64, 136))
    if page:
        held = H.paged_cache(sess, b, lens, page, order_seed=8, k_rows=ck, v_rows=cv)
    else:
        held = H.contiguous_cache(sess, b, max(lens) + 3, lens, ck, cv)
    q = synth.queries(b, prob.H_q, 128, 31, 10, 8.0).astype(np.float64)
    out = torch.zeros(b, prob.H_q, 128, dtype=torch.bfloat16, device="cuda")
    lat = torch.zeros(b, prob.H_q, 136, dtype=torch.bfloat16, device="cuda")
    for _ in range(2):                               # (the row maxima are left empty)
        out.fill_(3.0)
        L.lorc_decode_attn(sess.ctx, 0, held[0], H.dev_bf16(q), out, n_splits=n_splits)
        L.lorc_decode_attn_latent_out(sess.ctx, 0, held[0], H.dev_bf16(q), lat, n_splits=n_splits)
        assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
        assert L.lorc_last_path(sess.ctx) == 2
        _close(H.host_f64(out), H.oracle_decode(prob, ck, cv, q))
        for s in range(b):
            _close(H.host_f64(lat[s]), O.decode_attn_latent_out(ck[s], cv[s], prob.B_k, q[s], prob.H_kv, prob.theta, INTERLEAVED))
    sess.close()
