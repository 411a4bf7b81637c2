"""Streaming decode kernel of uncompressed layers: edges of steps and shares, page sizes that cut a step into boxes, head
counts, and cache rows past the sequence that hold NaN.

Probabilities are carried in two bf16 parts and the output is rounded to bf16: the observed row error is 1.7e-3, the bound the
repository's bf16 tolerance of 1e-2; test_error_beside_the_output_rounding holds what lies beside the rounding closer."""
import numpy as np
import pytest

from oracle import lorc_oracle as O
from workloads import synth

import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H_q,H_kv,lens,style,page,n_splits", [
    (8, 1, [1, 15, 16, 17, 63, 64, 65], 0, 0, 0),
    (8, 8, [129, 700], 1, 48, 3),                  # one head per KV head; four boxes of 16 rows, pages no power of two
    (12, 4, [200, 64], 0, 32, 0),                  # three heads per KV head, boxes of 32
    (32, 8, [1000, 1], 1, 64, 1),                  # one share: every stage is reused
    (64, 8, [333, 448], 2, 128, 40),               # eight heads per KV head, more shares than steps
    (6, 3, [97], 0, 16, 2),
])
def test_full_decode(H_q, H_kv, lens, style, page, n_splits):
    import torch
    L = H.lib()
    rng = np.random.default_rng(H_q + len(lens))
    n, b, n_max = H_kv * 128, len(lens), max(lens) + 70
    ctx = L.lorc_create(1, 256, H_q, H_kv, 128, 10000.0, rope_style=style, max_pos=n_max)
    w = torch.zeros(256, n, dtype=torch.bfloat16, device="cuda")
    L.lorc_load_factors(ctx, 0, L.LORC_MODE_FULL, 0, 0, w, None, w, None)
    ws = torch.zeros(L.lorc_workspace_bytes(ctx, b, n_max), dtype=torch.uint8, device="cuda")
    L.lorc_set_workspace(ctx, ws)
    rows = [[synth.to_bf16_exact(rng.standard_normal((m, n))) for m in lens] for _ in "kv"]
    sl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    if page:
        per = (n_max + page - 1) // page
        table = rng.permutation(b * per + 1)[:b * per].reshape(b, per).astype(np.int32)
        kv = []
        for which in rows:
            c = torch.full((b * per + 1, page, n), float("nan"), dtype=torch.bfloat16, device="cuda")
            for s, r in enumerate(which):
                for i in range(0, lens[s], page):
                    part = H.dev_bf16(r[i:i + page])
                    c[int(table[s, i // page]), :part.shape[0]] = part
            kv.append(c)
        tab = torch.from_numpy(table).cuda()
        cache = L.make_cache(*kv, sl, b, max(lens), page_table=tab, page_size=page, max_pages_per_seq=per, n_pages=b * per + 1)
    else:
        kv = []
        for which in rows:
            c = torch.full((b, n_max, n), float("nan"), dtype=torch.bfloat16, device="cuda")
            for s, r in enumerate(which):
                c[s, :lens[s]] = H.dev_bf16(r)
            kv.append(c)
        cache = L.make_cache(*kv, sl, b, max(lens), seq_stride=n_max)
    for q_scale in (1.0, 8.0):
        q = synth.queries(b, H_q, 128, 35, int(q_scale), q_scale).astype(np.float64)
        for entry in (L.lorc_decode_attn, L.lorc_decode_attn_static):
            out = torch.full((b, H_q, 128), 3.0, dtype=torch.bfloat16, device="cuda")
            entry(ctx, 0, cache, H.dev_bf16(q), out, n_splits=n_splits)
            assert L.lorc_sync_status(ctx) == 0, L.lorc_last_error(ctx)
            assert L.lorc_last_path(ctx) == 3
            for s, m in enumerate(lens):
                k, v = (which[s].astype(np.float64).reshape(m, H_kv, 128) for which in rows)
                qs = q[s]
                if style == H.ROPE_NONE:
                    want = O.attention_one_query(qs, k, v)
                else:
                    want = O.decode_attn_cached_kv(k, v, qs, 10000.0, style)
                H.assert_rows_close(H.host_f64(out[s]), want, 1e-2, (lens, s))
    L.lorc_destroy(ctx)


@pytest.mark.parametrize("page,n_splits", [(16, 1), (32, 0), (64, 3), (96, 1)])
def test_pages_outside_the_pool_are_left_out(page, n_splits):
    """Tokens whose page-table entry lies outside the pool take no part, whatever the pool's first page holds; the status word
    reports them."""
    import torch
    L = H.lib()
    rng = np.random.default_rng(page)
    H_q, H_kv, lens = 8, 2, [400, 70]
    n, b, per = H_kv * 128, len(lens), (max(lens) + page - 1) // page
    ctx = L.lorc_create(1, 256, H_q, H_kv, 128, 10000.0, max_pos=512)
    w = torch.zeros(256, n, dtype=torch.bfloat16, device="cuda")
    L.lorc_load_factors(ctx, 0, L.LORC_MODE_FULL, 0, 0, w, None, w, None)
    ws = torch.zeros(L.lorc_workspace_bytes(ctx, b, 512), dtype=torch.uint8, device="cuda")
    L.lorc_set_workspace(ctx, ws)
    rows = [[synth.to_bf16_exact(rng.standard_normal((m, n))) for m in lens] for _ in "kv"]
    kv = [torch.full((b * per + 1, page, n), 50.0, dtype=torch.bfloat16, device="cuda") for _ in "kv"]     # page 0 is not in use
    table = np.arange(1, b * per + 1, dtype=np.int32).reshape(b, per)
    for c, which in zip(kv, rows):
        for s, r in enumerate(which):
            for i in range(0, lens[s], page):
                part = H.dev_bf16(r[i:i + page])
                c[int(table[s, i // page]), :part.shape[0]] = part
    live = [np.ones(m, dtype=bool) for m in lens]
    for s, i, entry in ((0, 0, -1), (0, 2, b * per + 1), (0, (lens[0] - 1) // page, 10 ** 6)):
        table[s, i] = entry
        live[s][i * page:(i + 1) * page] = False
    sl, tab = torch.tensor(lens, dtype=torch.int32, device="cuda"), torch.from_numpy(table).cuda()
    cache = L.make_cache(*kv, sl, b, max(lens), page_table=tab, page_size=page, max_pages_per_seq=per, n_pages=b * per + 1)
    q = synth.queries(b, H_q, 128, 36, 1, 8.0).astype(np.float64)
    out = torch.full((b, H_q, 128), 3.0, dtype=torch.bfloat16, device="cuda")
    L.lorc_decode_attn(ctx, 0, cache, H.dev_bf16(q), out, n_splits=n_splits)
    assert L.lorc_sync_status(ctx) == L.LORC_ERR_CAPACITY
    assert L.lorc_last_path(ctx) == 3
    for s, m in enumerate(lens):
        k, v = (which[s].astype(np.float64).reshape(m, H_kv, 128)[live[s]] for which in rows)
        want = O.decode_attn_cached_kv(k, v, q[s], 10000.0, q_position=m - 1)
        H.assert_rows_close(H.host_f64(out[s]), want, 1e-2, (page, s))
    L.lorc_destroy(ctx)


@pytest.mark.parametrize("page", [0, 16, 48])
def test_length_beyond_the_capacity(page):
    """A length beyond the rows that exist: the query sits at the end of that length, the rows that exist are attended, and
    the status word reports it."""
    import torch
    L = H.lib()
    rng = np.random.default_rng(7)
    H_q, H_kv, rows_max = 4, 1, 96 if page else 101
    n, lens = H_kv * 128, [rows_max + 9, 50]
    ctx = L.lorc_create(1, 256, H_q, H_kv, 128, 10000.0, max_pos=128)
    w = torch.zeros(256, n, dtype=torch.bfloat16, device="cuda")
    L.lorc_load_factors(ctx, 0, L.LORC_MODE_FULL, 0, 0, w, None, w, None)
    ws = torch.zeros(L.lorc_workspace_bytes(ctx, 2, 128), dtype=torch.uint8, device="cuda")
    L.lorc_set_workspace(ctx, ws)
    rows = [[synth.to_bf16_exact(rng.standard_normal((rows_max, n))) for _ in lens] for _ in "kv"]
    sl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    kv = [torch.stack([H.dev_bf16(r) for r in which]) for which in rows]
    if page:
        per = rows_max // page
        tab = torch.arange(2 * per, dtype=torch.int32, device="cuda").view(2, per)
        cache = L.make_cache(*[c.view(2 * per, page, n) for c in kv], sl, 2, rows_max, page_table=tab, page_size=page,
                             max_pages_per_seq=per, n_pages=2 * per)
    else:
        cache = L.make_cache(*kv, sl, 2, rows_max, seq_stride=rows_max)
    q = synth.queries(2, H_q, 128, 36, 2, 8.0).astype(np.float64)
    out = torch.full((2, H_q, 128), 3.0, dtype=torch.bfloat16, device="cuda")
    L.lorc_decode_attn(ctx, 0, cache, H.dev_bf16(q), out)
    assert L.lorc_sync_status(ctx) == L.LORC_ERR_CAPACITY
    for s, m in enumerate(lens):
        k, v = (which[s].astype(np.float64).reshape(-1, H_kv, 128)[:m] for which in rows)
        want = O.decode_attn_cached_kv(k, v, q[s], 10000.0, q_position=m - 1)
        H.assert_rows_close(H.host_f64(out[s]), want, 1e-2, (page, s))
    L.lorc_destroy(ctx)


@pytest.mark.parametrize("n_splits", [0, 1, 9])
@pytest.mark.parametrize("q_scale", [1.0, 8.0])
def test_error_beside_the_output_rounding(q_scale, n_splits):
    """Half an ulp of the bf16 output, and beside it 2e-4 of the row rms: two bf16 parts leave 2^-17 = 8e-6 in a probability
    and 2^-18 in a query element (about 8 * 2^-18 = 3e-5 in a score of standard deviation 8), random in sign over the
    tokens.  (One bf16 part leaves 2e-3.)"""
    import torch
    L = H.lib()
    rng = np.random.default_rng(11)
    H_q, H_kv, lens = 32, 8, [2100, 600]
    n, b = H_kv * 128, len(lens)
    ctx = L.lorc_create(1, 256, H_q, H_kv, 128, 10000.0, max_pos=2112)
    w = torch.zeros(256, n, dtype=torch.bfloat16, device="cuda")
    L.lorc_load_factors(ctx, 0, L.LORC_MODE_FULL, 0, 0, w, None, w, None)
    ws = torch.zeros(L.lorc_workspace_bytes(ctx, b, 2112), dtype=torch.uint8, device="cuda")
    L.lorc_set_workspace(ctx, ws)
    rows = [[synth.to_bf16_exact(rng.standard_normal((2112, n))) for _ in lens] for _ in "kv"]
    kv = [torch.stack([H.dev_bf16(r) for r in which]) for which in rows]
    sl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    cache = L.make_cache(*kv, sl, b, max(lens), seq_stride=2112)
    q = synth.queries(b, H_q, 128, 36, 3, q_scale).astype(np.float64)
    out = torch.zeros(b, H_q, 128, dtype=torch.bfloat16, device="cuda")
    L.lorc_decode_attn(ctx, 0, cache, H.dev_bf16(q), out, n_splits=n_splits)
    assert L.lorc_sync_status(ctx) == 0, L.lorc_last_error(ctx)
    for s, m in enumerate(lens):
        k, v = (which[s].astype(np.float64).reshape(-1, H_kv, 128)[:m] for which in rows)
        want = O.decode_attn_cached_kv(k, v, q[s], 10000.0)
        rms = np.sqrt(np.mean(want ** 2, axis=-1, keepdims=True))
        excess = np.abs(H.host_f64(out[s]) - want) - (0.5 * H.bf16_ulp(want) + 2e-4 * rms)
        assert np.all(excess <= 0.0), float((excess / rms).max())
    L.lorc_destroy(ctx)


@pytest.mark.parametrize("lens,H_q,H_kv", [
    ([3000] + [64, 0, 1, 65] * 8, 16, 8),            # 33 sequences: the second group of 32 is searched too
    ([130, 9000] * 20, 8, 1),                        # more resident blocks than sequences
    ([130, 2000] * 35, 8, 1),                        # equal parts of them are short enough
    ([100] * 40 + [2500], 64, 8),                    # fewer; the long one comes last
    ([64], 4, 4),
])
def test_shares_by_length(lens, H_q, H_kv):
    """Sequences of very unequal length in one call: the blocks that are resident at once are dealt out by length."""
    import torch
    L = H.lib()
    n, b, n_max = H_kv * 128, len(lens), max(lens)
    ctx = L.lorc_create(1, 256, H_q, H_kv, 128, 10000.0, max_pos=n_max)
    w = torch.zeros(256, n, dtype=torch.bfloat16, device="cuda")
    L.lorc_load_factors(ctx, 0, L.LORC_MODE_FULL, 0, 0, w, None, w, None)
    ws = torch.full((L.lorc_workspace_bytes(ctx, b, n_max),), 255, dtype=torch.uint8, device="cuda")     # NaN everywhere
    L.lorc_set_workspace(ctx, ws)
    g = torch.Generator(device="cuda").manual_seed(5)
    kv = [torch.randn(b, n_max, n, generator=g, device="cuda", dtype=torch.bfloat16) for _ in "kv"]
    sl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    cache = L.make_cache(*kv, sl, b, n_max, seq_stride=n_max)
    q = synth.queries(b, H_q, 128, 36, 4, 8.0).astype(np.float64)
    out = torch.full((b, H_q, 128), 3.0, dtype=torch.bfloat16, device="cuda")
    L.lorc_decode_attn(ctx, 0, cache, H.dev_bf16(q), out)
    assert L.lorc_sync_status(ctx) == (L.LORC_ERR_EMPTY if 0 in lens else 0)
    # share results sit at the front of the workspace: [sequence][head][room for shares] of (reference, denominator)
    slots = 2 * torch.cuda.get_device_properties(0).multi_processor_count // H_kv
    equal = max(1, slots // b)
    room = min((n_max + 63) // 64, max(equal, min((n_max + 511) // 512, slots)) if n_max > 1024 * equal else equal)
    ml = ws[:b * H_q * room * 8].view(torch.float32).view(b, H_q, room, 2).cpu().numpy()
    steps = np.array([(m + 63) // 64 for m in lens])
    if room > equal:
        up, total = max(slots - b + 1, 0), steps.sum()
        want_shares = np.clip(np.maximum(steps * slots // total, -(-steps * up // total)), 1, room)
    else:
        want_shares = np.full(b, room)                   # equal parts
    for s, m in enumerate(lens):
        per = -(-steps[s] // want_shares[s])
        assert np.all((ml[s, :, :, 1] > 0).sum(axis=1) == (-(-steps[s] // per) if m else 0)), s
        if m == 0:
            assert float(out[s].abs().max()) == 0.0
            continue
        k, v = (c[s, :m].double().cpu().numpy().reshape(m, H_kv, 128) for c in kv)
        H.assert_rows_close(H.host_f64(out[s]), O.decode_attn_cached_kv(k, v, q[s], 10000.0), 1e-2, s)
    again = torch.zeros_like(out)
    L.lorc_decode_attn(ctx, 0, cache, H.dev_bf16(q), again)
    L.lorc_sync_status(ctx)
    assert torch.equal(out, again)
    L.lorc_destroy(ctx)
