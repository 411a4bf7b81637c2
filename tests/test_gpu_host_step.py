"""lorc_decode_step_host on every kind of host buffer gives what the device calls give, bit for bit: pinned buffers are read
and written by kernels, others go through copies."""
import numpy as np
import pytest

from workloads import synth

import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom", [dict(D=1024, H_q=32, H_kv=8, d_h=128, r_k=160, r_v=96), dict(D=264, H_q=4, H_kv=2, d_h=64, r_k=32, r_v=24)])
@pytest.mark.parametrize("kind", ["pinned", "pinned_misaligned", "pageable", "mixed", "result_over_queries"])
def test_step_from_host_buffers(geom, kind):
    import torch
    lens = [130, 17, 64]
    prob = H.Problem(geom["D"], geom["H_q"], geom["H_kv"], geom["d_h"], geom["r_k"], geom["r_v"], layer=34)
    b, n_max = len(lens), 140
    sess = H.Session(prob, max_pos=n_max, batch=b)
    L = sess.L
    ck, cv = H.oracle_latents(prob, [synth.hidden_states(n, prob.D, 34, chunk=s).astype(np.float64) for s, n in enumerate(lens)])
    x, q = H.dev_bf16(synth.hidden_states(b, prob.D, 34, chunk=9)), H.dev_bf16(synth.queries(b, prob.H_q, prob.d_h, 34, 1, 8.0))

    def host(t, i):
        pin = kind != "pageable" and not (kind == "mixed" and i == 1)
        skip = 2 if kind == "pinned_misaligned" else 0
        buf = torch.empty(t.numel() + skip, dtype=t.dtype)
        buf = buf.pin_memory() if pin else buf
        out = buf[skip:].view(t.shape)
        out.copy_(t.cpu())
        return out

    results = []
    for step in range(2):
        held = H.contiguous_cache(sess, b, n_max, lens, ck, cv)
        out = torch.full_like(q, 3.0)
        if step == 0:
            L.lorc_append(sess.ctx, 0, held[0], x)
            L.lorc_decode_attn(sess.ctx, 0, held[0], q, out)
        else:
            xh, qh = host(x, 0), host(q, 1)
            oh = qh if kind == "result_over_queries" else host(out, 2)
            for _ in range(2):
                if kind == "result_over_queries":
                    torch.cuda.synchronize()
                    qh.copy_(q.cpu())
                L.lorc_decode_step_host(sess.ctx, 0, held[0], xh, qh, oh)
            torch.cuda.current_stream().synchronize()
            out = oh
        assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
        results.append((out.cpu(), held[1].cpu(), held[2].cpu()))
    for a, c in zip(*results):
        assert torch.equal(a, c)
    sess.close()


def test_pinned_buffers_need_one_staging_launch():
    """A slice of a pinned allocation is staged by a kernel (one launch more than the copies need), a pageable buffer is not."""
    import torch
    prob = H.Problem(264, 4, 2, 64, 32, 24, layer=34)
    sess = H.Session(prob, max_pos=64, batch=2)
    L = sess.L
    held = H.contiguous_cache(sess, 2, 64, [9, 40])
    launches = []
    for pinned in (True, False):
        buf = torch.zeros(4096, dtype=torch.bfloat16)
        buf = buf.pin_memory() if pinned else buf
        x, q, out = buf[8:8 + 528].view(2, 264), buf[1024:1536].view(2, 4, 64), buf[2048:2560].view(2, 4, 64)
        before = L.lorc_launch_count(sess.ctx)
        L.lorc_decode_step_host(sess.ctx, 0, held[0], x, q, out)
        assert L.lorc_sync_status(sess.ctx) == 0, L.lorc_last_error(sess.ctx)
        launches.append(L.lorc_launch_count(sess.ctx) - before)
    assert launches[0] == launches[1] + 1
    sess.close()
