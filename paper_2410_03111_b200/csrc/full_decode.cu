// Decode attention of the uncompressed reference mode (ordinary KV cache: keys stored rotated, values as they are)
// on the warp-level tensor cores.  The work is one pass over 2 n bf16 numbers per token and is bound by HBM, so the
// kernel is shaped for streaming: a CTA owns one (sequence, KV head, context share), see lorc_full_decode_splits; a producer
// warp keeps three 64-token stages of keys and values in flight by TMA; each of four consumer warps owns 16 of a stage's tokens
// with its own running softmax (no block-wide synchronisation inside the loop).  The tokens (scores) and the dimensions (output)
// are the M side of the m16n8k16 tiles, the G <= 8 query heads the N side, so no row of a tile is padding:
//
//   S^T[16 tok x 8]   = K[16 tok x 128] . Q^^T            q^ = RoPE(q, N-1)/sqrt(d_h) split into bf16 hi + lo parts,
//                                                          so the scores keep fp32-level accuracy
//   p = exp(S - m) as two bf16 parts, rounded value and rounded remainder (16 significant bits)
//   O^T[128 x 8]     += V^T[128 x 16 tok] . P^T[16 tok x 8]
//
// What is left of the error against fp64 is the rounding of the bf16 output, 1.7e-3.  With one part it was 2.3e-3, and grew
// with the length of a share, because a higher reference moves p to other places between powers of two.  The second part
// costs 0.5 % where HBM sets the pace and 3 to 4 % where a single block's stream does.
//
// b 16, 8 KV heads of 128, 4129 tokens (271 MB): 45 us, 6.0 TB/s, 0.93 of the measured copy rate.  (With per-lane
// asynchronous copies and the heads on the M side, half of them padding, a warp issued seven times the instructions per tile
// and the issue slots, not HBM, set the pace: 55 us.)
// Each CTA leaves (m, l, un-normalised O) per query head for the merge kernel of the plain family.
#include <math.h>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "tc_kernels.cuh"

using namespace sm100;

namespace {

constexpr int FD_DH = 128;
constexpr int FD_TILE = 64;          // tokens per stage (16 per consumer warp)
constexpr int FD_STAGES = 3;
constexpr int FD_THREADS = 160;      // warps 0..3 consumers, warp 4 TMA
constexpr int FD_BLOCKS_PER_SM = 2;

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

// transpose of an 8 x 8 matrix of 16-bit elements spread over the warp (row lane / 4, columns 2 (lane % 4), + 1)
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// e^x for x <= 0 (relative error 2^-22 + 2^-24 |x|; 16 bits of the result are kept)
__device__ __forceinline__ float exp_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x * 1.4426950408889634f));
    return y;
}

struct FdSmem {
    // a stage: keys, then values, each in two 64-column halves [64 tokens][128 bytes], 128-byte swizzle
    union {
        bf16 kv[FD_STAGES][2][2][FD_TILE * 64];
        float o[4][8][FD_DH + 4];                    // after the loop: every warp's un-normalised output
    } u;
    float qs[8][FD_DH];                              // rotated, scaled queries of the G heads (rows G..7 zero)
    float m[4][8], l[4][8];
    uint64_t full[FD_STAGES], empty[FD_STAGES];
    uint32_t dead[FD_STAGES];                        // boxes of the stage whose page lies outside the pool, one bit each
};

struct FdParams {
    const bf16* q;
    CacheView cv;
    const float2* rope_table;
    float* part_ml;
    float* part_o;
    int* status;
    int G, n_kv, n_splits, rope_style, max_pos, box_rows;
    int slots;                     // 0: every sequence has n_splits shares; else at most as many, and `slots` together
};

// Shares of a sequence of `weight` steps when all of them have `total` (with `slots`): in proportion to its length, so that the
// blocks of a launch are resident at once and about equally long whatever the lengths are.  Its part of `slots`, rounded down,
// or its part of slots - batch + 1, rounded up (which adds up to at most `slots` too), whichever is more; for equal lengths
// both are slots / batch.  In all at most slots + batch.  (Steps are counted up to 2^15 a sequence, which keeps the sums of any
// batch in 32 bits.)
__device__ __forceinline__ int fd_weight(const FdParams& p, int len) {
    return len <= 0 || len > p.max_pos ? 0 : min((len - 1) / FD_TILE + 1, 1 << 15);
}
__device__ __forceinline__ int fd_shares(const FdParams& p, int weight, int total) {
    const int d = max(total, 1), up = max(p.slots - p.cv.batch + 1, 0);
    return max(1, min(p.n_splits, max(weight * p.slots / d, (weight * up + d - 1) / d)));
}

// Block `f` of a KV head -> sequence (-1: none), its length, share, number of shares; executed by whole warps.  (The result
// comes from warp reductions: those leave it in uniform registers, where loop bounds and TMA coordinates want it.)
__device__ __forceinline__ int4 fd_locate(const FdParams& p, int f, int lane) {
    const CacheView& cv = p.cv;
    if (p.slots == 0) return make_int4(f / p.n_splits, cv.seq_lens[f / p.n_splits], f % p.n_splits, p.n_splits);
    const int len0 = lane < cv.batch ? cv.seq_lens[lane] : 0;
    int sum = fd_weight(p, len0);
    for (int i = lane + 32; i < cv.batch; i += 32) sum += fd_weight(p, cv.seq_lens[i]);
    const int total = __reduce_add_sync(0xffffffffu, sum);
    int first = 0;
    for (int i0 = 0; i0 < cv.batch; i0 += 32) {
        const int i = i0 + lane, len = i0 == 0 ? len0 : i < cv.batch ? cv.seq_lens[i] : 0;
        const int n = i < cv.batch ? fd_shares(p, fd_weight(p, len), total) : 0;
        int end = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += x;
        }
        const unsigned hit = __ballot_sync(0xffffffffu, f < first + end);
        if (hit) {
            const bool mine = lane == __ffs(hit) - 1;
            return make_int4(i0 + __ffs(hit) - 1, __reduce_add_sync(0xffffffffu, mine ? len : 0),
                             __reduce_add_sync(0xffffffffu, mine ? f - first - (end - n) : 0),
                             __reduce_add_sync(0xffffffffu, mine ? n : 0));
        }
        first += __shfl_sync(0xffffffffu, end, 31);
    }
    return make_int4(-1, 0, 0, 1);
}

__global__ void __launch_bounds__(FD_THREADS, FD_BLOCKS_PER_SM)
full_decode_mma_kernel(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV, const FdParams p) {
    extern __shared__ uint8_t fd_raw[];
    FdSmem& sm = *reinterpret_cast<FdSmem*>((reinterpret_cast<uintptr_t>(fd_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3;            // fragment row / column group of this lane
    const int kvh = (int)blockIdx.x % p.n_kv;
    const CacheView& cv = p.cv;
    const int G = p.G, H_q = G * p.n_kv;
    if (tid == 0) {
        for (int i = 0; i < FD_STAGES; ++i) {
            mbar_init(&sm.full[i], 1);
            mbar_init(&sm.empty[i], 4);
        }
        fence_barrier_init();
        prefetch_tensormap(&mapK);
        prefetch_tensormap(&mapV);
    }
    grid_dep_wait();
    grid_dep_launch();
    const int4 share = fd_locate(p, (int)blockIdx.x / p.n_kv, lane);
    const int s = share.x, split = share.z, n_shares = share.w;
    int len = share.y;
    if (s < 0) return;
    // the slots of the shares that this sequence does not have
    if (split == 0)
        for (int i = tid; i < G * (p.n_splits - n_shares); i += FD_THREADS) {
            const int h = i / (p.n_splits - n_shares), c = n_shares + i % (p.n_splits - n_shares);
            *reinterpret_cast<float2*>(p.part_ml + (((long long)s * H_q + kvh * G + h) * p.n_splits + c) * 2) =
                make_float2(-INFINITY, 0.f);
        }
    if ((len > p.max_pos || len > cv.capacity) && tid == 0) lorc_set_status(p.status, LORC_ERR_CAPACITY);
    if (len < 0 || len > p.max_pos) len = 0;
    const int q_pos = len - 1;
    // tokens past the capacity, and those whose page lies outside the pool, are left out of the attention
    if (len > cv.capacity) len = (int)cv.capacity;
    // this CTA's share of the context, in whole 64-token tiles
    const int tiles = (len + FD_TILE - 1) / FD_TILE;
    const int tps = (tiles + n_shares - 1) / n_shares;
    const int t_begin = min(len, split * tps * FD_TILE), t_end = min(len, (split + 1) * tps * FD_TILE);
    const int n_steps = (t_end - t_begin + FD_TILE - 1) / FD_TILE;
    const int col0 = kvh * FD_DH;
    __syncthreads();                                  // the barriers are initialised
    bool ok = true;

    if (warp == 4) {
        // ------------------------------------------------------------------ producer (one elected lane issues)
        const int nbox = FD_TILE / p.box_rows;        // boxes per tile and half: 1, or up to 4 on small pages
        // lane i < nbox: the page of the tile's i-th box, -1 for a table entry outside the pool (reported).  Such a box, and one
        // past the end of the sequence, is fetched from behind the pool, where it reads as zero.
        auto lookup = [&](int t0) {
            int page = cv.page_table ? cv.n_pages : 0;
            if (cv.page_table != nullptr && lane < nbox && t0 + lane * p.box_rows < len) {
                page = cv.page_table[(long long)s * cv.max_pages_per_seq + (t0 + lane * p.box_rows) / cv.page_size];
                if (page < 0 || page >= cv.n_pages) {
                    lorc_set_status(p.status, LORC_ERR_CAPACITY);
                    page = -1;
                }
            }
            return page;
        };
        int mine = n_steps > 0 ? lookup(t_begin) : 0;
        int i = 0;
        for (; i < n_steps; ++i) {
            const int st = i % FD_STAGES, t0 = t_begin + i * FD_TILE;
            int pages[4];
            const uint32_t dead = __ballot_sync(0xffffffffu, mine < 0);
            if (mine < 0) mine = cv.n_pages;
#pragma unroll
            for (int j = 0; j < 4; ++j) pages[j] = __shfl_sync(0xffffffffu, mine, j);
            if (i + 1 < n_steps) mine = lookup(t0 + FD_TILE);
            if (!mbar_wait(&sm.empty[st], ((i / FD_STAGES) & 1) ^ 1)) { ok = false; break; }
            if (elect_one()) {
                sm.dead[st] = dead;
                mbar_arrive_expect_tx(&sm.full[st], 2 * 2 * FD_TILE * 64 * 2);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (j >= nbox) break;
                    const int tok = t0 + j * p.box_rows;
                    const int y = cv.page_table ? tok % cv.page_size : tok, z = cv.page_table ? pages[j] : s;
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        tma_load_3d(sm.u.kv[st][0][half] + j * p.box_rows * 64, &mapK, &sm.full[st], col0 + half * 64, y, z);
                        tma_load_3d(sm.u.kv[st][1][half] + j * p.box_rows * 64, &mapV, &sm.full[st], col0 + half * 64, y, z);
                    }
                }
            }
            __syncwarp();
        }
        // The block stays until the copies into its shared memory have landed (or the limit has passed once more), also when a
        // wait has run out.  Otherwise the consumers wait for all of them anyhow.
        for (int j = max(i - FD_STAGES, 0); j < i; ++j)
            if (!mbar_wait(&sm.full[j % FD_STAGES], (j / FD_STAGES) & 1)) ok = false;
        if (!ok && lane == 0) lorc_set_status(p.status, LORC_ERR_TIMEOUT);
    } else {
        // ------------------------------------------------------------------ consumers
        // q^ = RoPE(q, N - 1) / sqrt(d_h) for the G heads of this KV head
        for (int i = tid; i < 8 * (FD_DH / 2); i += 128) {
            const int h = i / (FD_DH / 2), jj = i - h * (FD_DH / 2);
            const int ia = (p.rope_style == LORC_ROPE_HALF_SPLIT) ? jj : 2 * jj;
            const int ib = (p.rope_style == LORC_ROPE_HALF_SPLIT) ? jj + FD_DH / 2 : 2 * jj + 1;
            float ra = 0.f, rb = 0.f;
            if (h < G && len > 0) {
                const bf16* qp = p.q + ((long long)s * H_q + kvh * G + h) * FD_DH;
                const float a = __bfloat162float(qp[ia]), b = __bfloat162float(qp[ib]);
                const float2 cs = p.rope_table[(long long)q_pos * (FD_DH / 2) + jj];
                const float scale = rsqrtf((float)FD_DH);
                ra = (a * cs.x - b * cs.y) * scale;
                rb = (a * cs.y + b * cs.x) * scale;
            }
            sm.qs[h][ia] = ra;
            sm.qs[h][ib] = rb;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        // Query fragments of head g: k-step ks covers the dimensions 16 ks .. + 15, split into bf16 hi + lo parts.
        uint32_t qhi[8][2], qlo[8][2];
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int d0 = 16 * ks + 8 * half + 2 * t;
                const float v0 = sm.qs[g][d0], v1 = sm.qs[g][d0 + 1];
                const float h0 = __bfloat162float(__float2bfloat16_rn(v0)), h1 = __bfloat162float(__float2bfloat16_rn(v1));
                qhi[ks][half] = pack_bf16(h0, h1);
                qlo[ks][half] = pack_bf16(v0 - h0, v1 - h1);
            }
        }
        float o[8][4];                                // dimensions 16 db + g (+ 8: [2], [3]), heads 2 t, 2 t + 1
#pragma unroll
        for (int db = 0; db < 8; ++db) o[db][0] = o[db][1] = o[db][2] = o[db][3] = 0.f;
        float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};   // heads 2 t, 2 t + 1 (l: this lane's tokens)

        // byte offset of this lane's row in a half stage, and the row's swizzle; ldmatrix.x4 takes four 8 x 8 matrices, lane
        // mi = lane / 8 addresses a row of matrix mi: keys (tokens 0..7 | 8..15) x (dims 0..7), then (dims 8..15); values
        // (dims 0..7 | 8..15) x (tokens 0..7), then (tokens 8..15)
        const int mi = lane >> 3, lr = lane & 7;
        const int box = warp * 16 / p.box_rows;          // the box of a stage that holds this warp's tokens
        const uint32_t k_row = (uint32_t)(warp * 16 + (mi & 1) * 8 + lr) * 128, v_row = (uint32_t)(warp * 16 + (mi >> 1) * 8 + lr) * 128;
        for (int i = 0; i < n_steps; ++i) {
            const int st = i % FD_STAGES, tw = t_begin + i * FD_TILE + warp * 16;     // first token of this warp
            if (!mbar_wait(&sm.full[st], (i / FD_STAGES) & 1)) { ok = false; break; }
            const int t_live = (sm.dead[st] >> box) & 1 ? 0 : t_end;
            const uint32_t k0 = smem_u32(sm.u.kv[st][0][0]), v0 = smem_u32(sm.u.kv[st][1][0]);
            // scores of tokens g, g + 8 against heads 2 t, 2 t + 1; four short chains
            float sc[4][4];
#pragma unroll
            for (int j = 0; j < 4; ++j) sc[j][0] = sc[j][1] = sc[j][2] = sc[j][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                uint32_t a[4];
                const int piece = 2 * (ks & 3) + (mi >> 1);
                ldmatrix_x4(a, k0 + (ks >> 2) * (FD_TILE * 128) + k_row + ((piece ^ lr) << 4));
                mma_bf16_16816(sc[ks & 1], a[0], a[1], a[2], a[3], qhi[ks][0], qhi[ks][1]);
                mma_bf16_16816(sc[2 + (ks & 1)], a[0], a[1], a[2], a[3], qlo[ks][0], qlo[ks][1]);
            }
            float x[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                x[j] = (sc[0][j] + sc[1][j]) + (sc[2][j] + sc[3][j]);
                if (tw + g + (j >> 1) * 8 >= t_live) x[j] = -INFINITY;
            }
            // running softmax over this warp's tokens
            float m_new[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float mx = fmaxf(x[e], x[2 + e]);
#pragma unroll
                for (int w = 4; w < 32; w <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
                m_new[e] = fmaxf(m_run[e], mx);
            }
            if (__any_sync(0xffffffffu, m_new[0] > m_run[0] || m_new[1] > m_run[1])) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float alpha = m_run[e] == -INFINITY ? 0.f : expf(m_run[e] - m_new[e]);
                    l_run[e] *= alpha;
#pragma unroll
                    for (int db = 0; db < 8; ++db) {
                        o[db][e] *= alpha;
                        o[db][2 + e] *= alpha;
                    }
                    m_run[e] = m_new[e];
                }
            }
            // p = e^(x - m) in two bf16 parts, pairs of heads: the rounded value and the rounded remainder
            uint32_t ph[2], pl[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float e[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float m = m_run[i] == -INFINITY ? 0.f : m_run[i];          // nothing seen yet: e^(-inf) = 0
                    e[i] = exp_approx(x[2 * j + i] - m);
                    l_run[i] += e[i];
                }
                ph[j] = pack_bf16(e[0], e[1]);
                pl[j] = pack_bf16(e[0] - __uint_as_float(ph[j] << 16), e[1] - __uint_as_float(ph[j] & 0xffff0000u));
            }
            const uint32_t b0 = movmatrix_trans(ph[0]), b1 = movmatrix_trans(ph[1]);
            const uint32_t c0 = movmatrix_trans(pl[0]), c1 = movmatrix_trans(pl[1]);
            if (tw + 16 > t_end) {
                // rows past the share's end: their probabilities are zero, and zero their values (they may hold anything)
                for (int r = max(t_end - tw, 0); r < 16; ++r)
                    *reinterpret_cast<uint2*>(reinterpret_cast<uint8_t*>(sm.u.kv[st][1][lane >> 4]) + (warp * 16 + r) * 128 +
                                              (lane & 15) * 8) = make_uint2(0u, 0u);
                fence_proxy_async_smem();              // before the stage's next copy
                __syncwarp();
            }
            // O^T += V^T P^T
#pragma unroll
            for (int db = 0; db < 8; ++db) {
                uint32_t a[4];
                const int piece = 2 * (db & 3) + (mi & 1);
                ldmatrix_x4_trans(a, v0 + (db >> 2) * (FD_TILE * 128) + v_row + ((piece ^ lr) << 4));
                mma_bf16_16816(o[db], a[0], a[1], a[2], a[3], b0, b1);
                mma_bf16_16816(o[db], a[0], a[1], a[2], a[3], c0, c1);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.empty[st]);
        }
        if (!ok && lane == 0) lorc_set_status(p.status, LORC_ERR_TIMEOUT);
        __syncwarp();
        asm volatile("bar.sync 1, 128;" ::: "memory");   // every warp is done with the stages (the union is reused)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
#pragma unroll
            for (int w = 4; w < 32; w <<= 1) l_run[e] += __shfl_xor_sync(0xffffffffu, l_run[e], w);
            if (g == 0) {
                sm.m[warp][2 * t + e] = m_run[e];
                sm.l[warp][2 * t + e] = l_run[e];
            }
#pragma unroll
            for (int db = 0; db < 8; ++db) {
                sm.u.o[warp][2 * t + e][16 * db + g] = o[db][e];
                sm.u.o[warp][2 * t + e][16 * db + 8 + g] = o[db][2 + e];
            }
        }
        __syncwarp();
        asm volatile("bar.sync 1, 128;" ::: "memory");
        // merge the four warps of the CTA (thread = dimension)
        for (int h = 0; h < G; ++h) {
            float M = -INFINITY;
#pragma unroll
            for (int w = 0; w < 4; ++w)
                if (sm.l[w][h] > 0.f) M = fmaxf(M, sm.m[w][h]);
            float L = 0.f, acc = 0.f;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const float wgt = (sm.l[w][h] > 0.f) ? expf(sm.m[w][h] - M) : 0.f;
                L += wgt * sm.l[w][h];
                acc += wgt * sm.u.o[w][h][tid];
            }
            const long long unit = ((long long)s * H_q + kvh * G + h) * p.n_splits + split;
            if (tid == 0) {
                p.part_ml[unit * 2 + 0] = M;
                p.part_ml[unit * 2 + 1] = L;
            }
            p.part_o[unit * FD_DH + tid] = acc;
        }
    }
}

}  // namespace

bool lorc_full_decode_supported(const lorc_ctx* ctx, const LorcLayer& L) {
    return L.mode == LORC_MODE_FULL && ctx->desc.d_head == FD_DH && ctx->group >= 1 && ctx->group <= 8 &&
           !(ctx->desc.flags & LORC_FLAG_DEBUG_FP32);
}

// Blocks of a KV head that are resident at once.
static int fd_slots(const lorc_ctx* ctx) { return FD_BLOCKS_PER_SM * ctx->sm_count / ctx->desc.n_kv_heads; }

// Most context shares of a sequence: an equal part of the resident blocks, so that every block streams from the start to the
// end of the launch (down to one 64-token step each).  Where that makes shares of more than 1024 tokens, which take a block
// longer than 17 us, there is room for shares of 512 tokens and the kernel deals the resident blocks out by length.  (With
// equal parts alone one sequence of 8200 tokens among 23 of 256, 8 KV heads, is streamed by 8 blocks: 74 us, dealt out 19.
// Shares of 512 tokens for all make 1152 blocks in 3.9 rounds at b 16, 8 KV heads, 4129 tokens: 56 us against 49.  Dealing
// costs 0.5 to 1 us where all lengths are equal.)
int lorc_full_decode_splits(const lorc_ctx* ctx, int batch, int max_seq_len) {
    const int slots = fd_slots(ctx), steps = (max_seq_len - 1) / FD_TILE + 1, room = (max_seq_len - 1) / 512 + 1;
    int n = slots / batch > 1 ? slots / batch : 1;
    if (max_seq_len > 1024ll * n && n < room) n = room < slots ? room : slots;
    return n < 1 ? 1 : n < steps ? n : steps;
}

cudaError_t lorc_full_decode(lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, const bf16* q, int n_splits, bool by_length,
                             float* part_ml, float* part_o, cudaStream_t st, int* launches) {
    const lorc_model_desc& d = ctx->desc;
    const size_t smem = sizeof(FdSmem) + 1024;
    // the attribute belongs to a device's copy of the kernel: one flag per device (devices beyond the table set it
    // on every call, which is only slower)
    static bool attr[64] = {false};
    const bool known = ctx->device >= 0 && ctx->device < 64;
    if (!known || !attr[ctx->device]) {
        cudaError_t e = cudaFuncSetAttribute(full_decode_mma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (known) attr[ctx->device] = true;
    }
    // nothing to deal where an equal part of the resident blocks is as many shares as a sequence has room for
    const int slots = by_length && n_splits > fd_slots(ctx) / cv.batch && n_splits > 1 ? fd_slots(ctx) : 0;
    // a box never leaves its page: page sizes are multiples of 16
    FdParams p;
    p.box_rows = !cv.page_table || cv.page_size % 64 == 0 ? 64 : cv.page_size % 32 == 0 ? 32 : 16;
    CUtensorMap *mapK, *mapV;
    if (!lorc_tc_full_maps(ctx, L, cv, p.box_rows, &mapK, &mapV)) return cudaErrorInvalidValue;
    p.q = q; p.cv = cv; p.rope_table = ctx->rope_table; p.part_ml = part_ml; p.part_o = part_o; p.status = ctx->status_dev;
    p.G = ctx->group; p.n_kv = d.n_kv_heads; p.n_splits = n_splits; p.slots = slots; p.rope_style = ctx->pair_style; p.max_pos = d.max_pos;
    const long long even = (long long)cv.batch * n_splits, most = (long long)slots + cv.batch;
    const dim3 grid((unsigned)(d.n_kv_heads * (slots > 0 && most < even ? most : even)));
    *launches += 1;
    return lorc_launch_dependent(full_decode_mma_kernel, grid, dim3(FD_THREADS), smem, st, *mapK, *mapV, p);
}
