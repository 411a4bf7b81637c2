"""Prompt-sized cache writes: unit widths, narrow last column blocks, token remainders, paged and contiguous rows.

A stored element is the fp32 sum of D exact products, rounded once: half a bf16 ulp, and 2^-20 of the sum of magnitudes for
the order of the fp32 additions (D = 256 terms: 2^-24 sqrt(256) is the expected size)."""
import numpy as np
import pytest

import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r_k,r_v,b,T,page", [
    (8, 8, 16, 447, 0),           # 16 columns: units of 32, half a block per CTA
    (96, 72, 2, 357, 16),         # 168 columns: a last block of 40, rounded up to 64; tokens of two sequences in a tile
    (264, 256, 1, 257, 0),        # a third token block of one row
    (512, 512, 5, 333, 64),       # full-width units
    (928, 416, 1, 129, 128),
    (928, 928, 1, 49, 0),         # fewer tokens than a CTA's half of a unit
    (160, 128, 1, 200, 0),        # the warp-level kernel: fewer than three rounds of its blocks
    (1024, 1000, 16, 520, 0),     # more units than pairs: several rounds, both accumulators
])
def test_prompt_sized_append(r_k, r_v, b, T, page):
    import torch
    D, H_q, H_kv = 256, 32, 8
    rng = np.random.default_rng(r_k + T)
    dev = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).to(torch.bfloat16).cuda()
    L = H.lib()
    lens = [T + int(x) for x in rng.integers(0, 40, size=b)]
    n_max = max(lens) + 5
    ctx = L.lorc_create(1, D, H_q, H_kv, 128, 500000.0, max_pos=n_max)
    A_k, A_v, x = dev(D, r_k), dev(D, r_v), dev(b, T, D)
    L.lorc_load_factors(ctx, 0, L.LORC_MODE_LATENT, r_k, r_v, A_k, dev(r_k, 1024), A_v, dev(r_v, 1024))
    sl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    if page:
        per = (n_max + page - 1) // page
        table = torch.from_numpy(rng.permutation(b * per + 2)[:b * per].astype(np.int32)).view(b, per).cuda()
        shape = (b * per + 2, page)
        k, v = (torch.full((*shape, r), 3.0, dtype=torch.bfloat16, device="cuda") for r in (r_k, r_v))
        cache = L.make_cache(k, v, sl, b, n_max, page_table=table, page_size=page, max_pages_per_seq=per, n_pages=shape[0])
    else:
        k, v = (torch.full((b, n_max, r), 3.0, dtype=torch.bfloat16, device="cuda") for r in (r_k, r_v))
        cache = L.make_cache(k, v, sl, b, n_max, seq_stride=n_max)
    L.lorc_append(ctx, 0, cache, x, T)
    assert L.lorc_sync_status(ctx) == 0, L.lorc_last_error(ctx)
    assert L.lorc_last_path(ctx) == 2
    for c, A in ((k, A_k), (v, A_v)):
        rows = c.view(-1, c.shape[-1]).clone()
        for s in range(b):
            pos = torch.arange(lens[s] - T, lens[s], device="cuda")
            at = (table[s, pos // page].long() * page + pos % page) if page else s * n_max + pos
            got, want = rows[at].double(), x[s].double() @ A.double()
            ulp = torch.from_numpy(H.bf16_ulp(want.cpu().numpy())).cuda()
            assert torch.all((got - want).abs() <= 0.5 * ulp + 2.0 ** -20 * (x[s].double().abs() @ A.double().abs()))
            rows[at] = 3.0
        assert torch.all(rows == 3.0)              # nothing else was written
    L.lorc_destroy(ctx)
