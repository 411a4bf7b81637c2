// Decode attention over the latent cache for the shapes the tcgen05 kernels do not take (64-wide heads, other head counts),
// with the arithmetic of the plain kernels: products of bf16 operands summed in fp32, fp32 rotation, scores, softmax and
// probabilities.
//
// A CTA owns one (sequence, KV head, context share) and walks it 64 tokens at a time; a warp owns 16 of them.
//   K[16 tokens, d_h] = C_K . B_K[:, g]   on mma.sync m16n8k16 (bf16 operands as they are stored, fp32 sums), operands
//                                         straight from global memory: a lane's 16 bytes are 8 consecutive latent columns
//                                         of a token (A) or of a feature of B_K^T (B), the same slot order on both sides
//   rotation and q.k in registers (the accumulator columns of a rotary pair belong to one thread), softmax over the 64
//   tokens, then O_lat += P . C_V with fp32 FMAs, thread = (8 latent columns, group of tokens).
// Such calls are small: the kernel is bound by its chain of dependent loads, so shares are short (64 tokens when that
// fills the chip).  Where a call is small in every way (see SD_MERGE_SHARES) its shares form a cluster that merges them through
// distributed shared memory and up-projects the result: one launch less.  At 129 tokens, rank 32, 4 heads of 64 the kernel takes
// 11 us where the scalar kernel took 99 us; the step with cache write and merge took 72 us with that one, then 19; one step among
// many, launched from Python: 11.8 us with the merge kernel, 9.5 with the merge inside.
#include <math.h>

#include "common.cuh"
#include "sm100_pair.cuh"
#include "sm100_ptx.cuh"
#include "tc_kernels.cuh"

using namespace sm100;

namespace {

constexpr int SD_THREADS = 128;
constexpr int SD_TILE = LORC_SMALL_TILE;             // tokens per step: 16 per warp
// Merge inside: as many shares as every GPU takes in a cluster, and r_v * d_h at most this, so that a thread holds its 64 or
// fewer elements of B_V in registers before the shares meet.  Its blocks hold more registers and shared memory, and one of them
// takes the heads of a KV head in series, so the line lies where this was faster than the merge kernel throughout a sweep of
// heads, ranks, lengths and batches (one call among many, graph replay, merge kernel -> inside; where the rule keeps that kernel
// the second figure is what merging inside took):
//   up to two query heads per KV head: d_h 64, r 32, 129 tokens 9.2 -> 7.1 us; r 128, 500 tokens 17.0 -> 11.1.
//   more: d_h 64, r 32, 40 tokens, four heads 7.9 -> 10.8, eight 9.8 -> 16.1; with as many shares as heads 0.93 to 1.06.
//   blocks that all run at once (8 / 3 per SM): 320 blocks 18.1 -> 14.8, 384 13.1 -> 11.3, 432 17.5 -> 22.9, 512 14.8 -> 22.5;
//   clusters of more than five do not pack as well: 256 blocks 10.8 -> 11.3.
//   d_h 128, where a thread holds a pair's whole row: r 64, 129 tokens 11.0 -> 9.4, r 16 7.8 -> 8.1; one share of two heads
//   10.0 -> 10.1; 240 blocks 12.7 -> 13.4.
constexpr int SD_MERGE_SHARES = 8, SD_MERGE_WORK = 64 * SD_THREADS, SD_MERGE_HEADS = 2;

struct SdParams {
    const bf16* q;
    CacheView cv;
    const bf16* B_kT;              // [n, r_k], every head in half-split order (see LorcLayer)
    const float2* rope_table;
    const int32_t* pos0;
    const int32_t* q_pos;
    float* part_ml;
    float* part_o;
    bf16* out;                     // MERGE: [b, H_q, DH]
    const bf16* B_v;               // MERGE: [r_v, n]
    int* status;
    int r_k, r_v, G, n_splits, rope_style, max_pos, n;
};

// GM: query heads per KV head rounded up to 2, 4 or 8 (rows past p.G hold zero queries and are not written)
// MERGE: the shares of a (sequence, KV head) form a cluster
template <int DH, int GM, bool MERGE>
__global__ void __launch_bounds__(SD_THREADS)
small_decode_kernel(const SdParams p) {
    constexpr int HALF = DH / 2, NT = DH / 8;
    __shared__ __align__(16) float qs[GM][DH];        // rotated, scaled queries, half-split order
    __shared__ float P[GM][SD_TILE];
    __shared__ float wmax[4][GM], m_s[2][GM], l_s[GM];
    __shared__ long long row_s[SD_TILE];
    __shared__ float red[SD_THREADS * GM * 8];        // token groups' partial outputs
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g8 = lane >> 2, t = lane & 3;
    const int split = blockIdx.x, g = blockIdx.y, s = blockIdx.z;
    const int H_q = p.G * (int)gridDim.y;
    const CacheView& cv = p.cv;

    grid_dep_wait();
    grid_dep_launch();
    int len = cv.seq_lens[s];
    // context shards: the cached rows sit at positions p0 .. p0 + len - 1, the query at qpos (not before the last row)
    const int p0 = p.pos0 ? p.pos0[s] : 0;
    const int qpos = p.q_pos ? p.q_pos[s] : p0 + len - 1;
    if (len > 0 && (len > p.max_pos || p0 < 0 || qpos < p0 + len - 1 || qpos >= p.max_pos)) {
        if (tid == 0) lorc_set_status(p.status, LORC_ERR_CAPACITY);
        len = 0;
    }
    if (len < 0) len = 0;
    const int tiles = (len + SD_TILE - 1) / SD_TILE, tps = (tiles + p.n_splits - 1) / p.n_splits;
    const int t_begin = min(len, split * tps * SD_TILE), t_end = min(len, (split + 1) * tps * SD_TILE);

    if (len > 0) {
        const float scale = rsqrtf((float)DH);
        for (int i = tid; i < GM * HALF; i += SD_THREADS) {
            const int h = i / HALF, j = i - h * HALF;
            float a = 0.f, b = 0.f;
            if (h < p.G) {
                const bf16* qp = p.q + ((long long)s * H_q + g * p.G + h) * DH;
                const bool hs = p.rope_style == LORC_ROPE_HALF_SPLIT;
                a = __bfloat162float(qp[hs ? j : 2 * j]);
                b = __bfloat162float(qp[hs ? j + HALF : 2 * j + 1]);
            }
            const float2 cs = p.rope_table[(long long)qpos * HALF + j];
            qs[h][j] = (a * cs.x - b * cs.y) * scale;
            qs[h][j + HALF] = (a * cs.y + b * cs.x) * scale;
        }
    }
    if (tid < GM) {
        m_s[0][tid] = -INFINITY;
        l_s[tid] = 0.f;
    }

    // P . C_V: column group (8 latent columns) and token group of this thread
    const int ncg = p.r_v / 8, ntg = SD_THREADS / ncg;
    const int cg = tid % ncg, tg = tid / ncg;
    float acc[GM][8];
#pragma unroll
    for (int h = 0; h < GM; ++h)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[h][e] = 0.f;

    int it = 0;
    for (int t0 = t_begin; t0 < t_end; t0 += SD_TILE, ++it) {
        if (tid < SD_TILE) {
            long long row = -1;
            if (t0 + tid < t_end) {
                row = lorc_row_index(cv, s, t0 + tid);
                if (row < 0) lorc_set_status(p.status, LORC_ERR_CAPACITY);
            }
            row_s[tid] = row;
        }
        __syncthreads();
        // ---- keys of this warp's 16 tokens
        const long long ra = row_s[warp * 16 + g8], rb = row_s[warp * 16 + 8 + g8];
        float k[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) k[nt][e] = 0.f;
        {
            const uint4 zero = make_uint4(0, 0, 0, 0);
            const bf16* bp = p.B_kT + (long long)(g * DH + g8) * p.r_k + 8 * t;
#pragma unroll 1
            for (int k0 = 0; k0 < p.r_k; k0 += 32) {
                const bool in = k0 + 8 * t < p.r_k;       // ranks are multiples of 8
                const uint4 x = in && ra >= 0 ? *reinterpret_cast<const uint4*>(cv.k + ra * cv.w_k + k0 + 8 * t) : zero;
                const uint4 y = in && rb >= 0 ? *reinterpret_cast<const uint4*>(cv.k + rb * cv.w_k + k0 + 8 * t) : zero;
#pragma unroll
                for (int n0 = 0; n0 < NT; n0 += 8) {
                    uint4 w[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        w[i] = in ? __ldg(reinterpret_cast<const uint4*>(bp + (long long)(n0 + i) * 8 * p.r_k + k0)) : zero;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        mma_bf16_16816(k[n0 + i], x.x, y.x, x.y, y.y, w[i].x, w[i].y);
                        mma_bf16_16816(k[n0 + i], x.z, y.z, x.w, y.w, w[i].z, w[i].w);
                    }
                }
            }
        }
        // ---- rotation and dots: this thread holds features 8 nt + 2 t, + 1 of tokens g8 (k[..][0, 1]) and g8 + 8 (k[..][2, 3])
        float sc[2][GM];
#pragma unroll
        for (int h = 0; h < GM; ++h) sc[0][h] = sc[1][h] = 0.f;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
            const int tok = warp * 16 + hf * 8 + g8;
            const float2* cs = p.rope_table + (long long)min(p0 + t0 + tok, p.max_pos - 1) * HALF;
#pragma unroll
            for (int nt = 0; nt < NT / 2; ++nt) {
                const int j = 8 * nt + 2 * t;
                const float4 c = __ldg(reinterpret_cast<const float4*>(cs + j));       // (cos, sin) of pairs j, j + 1
                const float a0 = k[nt][2 * hf], a1 = k[nt][2 * hf + 1];
                const float b0 = k[nt + NT / 2][2 * hf], b1 = k[nt + NT / 2][2 * hf + 1];
                const float x0 = a0 * c.x - b0 * c.y, y0 = a0 * c.y + b0 * c.x;
                const float x1 = a1 * c.z - b1 * c.w, y1 = a1 * c.w + b1 * c.z;
#pragma unroll
                for (int h = 0; h < GM; ++h) {
                    const float2 qa = *reinterpret_cast<const float2*>(&qs[h][j]);
                    const float2 qb = *reinterpret_cast<const float2*>(&qs[h][j + HALF]);
                    sc[hf][h] = fmaf(qa.x, x0, fmaf(qa.y, x1, fmaf(qb.x, y0, fmaf(qb.y, y1, sc[hf][h]))));
                }
            }
        }
#pragma unroll
        for (int h = 0; h < GM; ++h) {
            float mx = -INFINITY;
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                float v = sc[hf][h];
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                if ((hf ? rb : ra) < 0) v = -INFINITY;
                if (t == 0) P[h][warp * 16 + hf * 8 + g8] = v;
                mx = fmaxf(mx, v);
            }
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (lane == 0) wmax[warp][h] = mx;
        }
        __syncthreads();
        // ---- running softmax: a warp takes a head
        float alpha[GM];
#pragma unroll
        for (int h = 0; h < GM; ++h) {
            const float m_old = m_s[it & 1][h];
            const float m_new = fmaxf(fmaxf(fmaxf(wmax[0][h], wmax[1][h]), fmaxf(wmax[2][h], wmax[3][h])), m_old);
            alpha[h] = m_old == -INFINITY ? 0.f : expf(m_old - m_new);
            if ((h & 3) == warp) {
                const float m_use = m_new == -INFINITY ? 0.f : m_new;
                const float e0 = expf(P[h][lane] - m_use), e1 = expf(P[h][lane + 32] - m_use);
                P[h][lane] = e0;
                P[h][lane + 32] = e1;
                float sum = e0 + e1;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (lane == 0) {
                    l_s[h] = l_s[h] * alpha[h] + sum;
                    m_s[(it + 1) & 1][h] = m_new;
                }
            }
        }
        __syncthreads();
        // ---- O_lat = alpha O_lat + P . C_V
        if (tg < ntg) {
#pragma unroll
            for (int h = 0; h < GM; ++h)
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[h][e] *= alpha[h];
            const int n_tok = min(SD_TILE, t_end - t0);
#pragma unroll 4
            for (int tok = tg; tok < n_tok; tok += ntg) {
                const long long row = row_s[tok];
                if (row < 0) continue;
                const uint4 v = *reinterpret_cast<const uint4*>(cv.v + row * cv.w_v + cg * 8);
                const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int h = 0; h < GM; ++h) {
                    const float pr = P[h][tok];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        acc[h][2 * e] = fmaf(pr, __uint_as_float(w[e] << 16), acc[h][2 * e]);
                        acc[h][2 * e + 1] = fmaf(pr, __uint_as_float(w[e] & 0xffff0000u), acc[h][2 * e + 1]);
                    }
                }
            }
        }
        __syncthreads();
    }

    // ---- add the token groups' parts, write this share's partial result
    if (tg < ntg) {
#pragma unroll
        for (int h = 0; h < GM; ++h)
#pragma unroll
            for (int e = 0; e < 8; ++e) red[(h * ntg + tg) * p.r_v + cg * 8 + e] = acc[h][e];
    }
    __syncthreads();
    __shared__ float part[MERGE ? GM * (SD_MERGE_WORK / DH) : 1];        // MERGE: [G][r_v]
    for (int i = tid; i < p.G * p.r_v; i += SD_THREADS) {
        const int h = i / p.r_v, col = i - h * p.r_v;
        float a = 0.f;
        for (int x = 0; x < ntg; ++x) a += red[(h * ntg + x) * p.r_v + col];
        if (MERGE)
            part[i] = a;
        else
            p.part_o[(((long long)s * H_q + g * p.G + h) * p.n_splits + split) * p.r_v + col] = a;
    }
    if constexpr (!MERGE) {
        if (tid < p.G) {
            const long long unit = ((long long)s * H_q + g * p.G + tid) * p.n_splits + split;
            p.part_ml[unit * 2] = m_s[it & 1][tid];
            p.part_ml[unit * 2 + 1] = l_s[tid];
        }
    } else {
        // The arithmetic is that of the merge kernel, and so is the order of the sums, but for the denominator's (in double).  A share's CTA takes every n_splits-th head;
        // thread = (output column j, slices sl and sl + SL of the rank), its elements of B_V on their way while the shares meet.
        constexpr int SL = SD_THREADS / DH, SLICES = 256 / DH, NW = 64 / 2;
        __shared__ float ml[GM][2];
        __shared__ float o_lat[SD_MERGE_WORK / DH], sums[SLICES][DH];
        if (tid < GM) {
            ml[tid][0] = m_s[it & 1][tid];
            ml[tid][1] = l_s[tid];
        }
        const int j = tid % DH, sl = tid / DH;
        bf16 w[2][NW];
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                const int k = i * SLICES + sl + x * SL;
                w[x][i] = k < p.r_v ? p.B_v[(long long)k * p.n + g * DH + j] : __float2bfloat16_rn(0.f);
            }
        __syncwarp();
        cluster_arrive_release();
        cluster_wait_acquire();
        const uint32_t part0 = smem_u32(part), ml0 = smem_u32(&ml[0][0]);
        for (int h = split; h < p.G; h += p.n_splits) {
            float m[SD_MERGE_SHARES], l[SD_MERGE_SHARES], M = -INFINITY;
#pragma unroll
            for (int c = 0; c < SD_MERGE_SHARES; ++c) {
                m[c] = -INFINITY;
                l[c] = 0.f;
                if (c < p.n_splits) {
                    m[c] = ld_cluster_f1(mapa_shared(ml0 + h * 8, c));
                    l[c] = ld_cluster_f1(mapa_shared(ml0 + h * 8 + 4, c));
                }
                if (l[c] > 0.f) M = fmaxf(M, m[c]);
            }
            double L = 0.0;
#pragma unroll
            for (int c = 0; c < SD_MERGE_SHARES; ++c) {
                m[c] = l[c] > 0.f ? expf(m[c] - M) : 0.f;                // the share's weight
                L += (double)m[c] * (double)l[c];
            }
            const float Lf = (float)L, inv = Lf > 0.f ? 1.f / Lf : 0.f;
            if (tid == 0 && !(L > 0.0)) lorc_set_status(p.status, LORC_ERR_EMPTY);
            for (int col = tid; col < p.r_v; col += SD_THREADS) {
                float x[SD_MERGE_SHARES], a = 0.f;
#pragma unroll
                for (int c = 0; c < SD_MERGE_SHARES; ++c)
                    x[c] = c < p.n_splits ? ld_cluster_f1(mapa_shared(part0 + (h * p.r_v + col) * 4, c)) : 0.f;
#pragma unroll
                for (int c = 0; c < SD_MERGE_SHARES; ++c)
                    if (m[c] != 0.f) a = fmaf(m[c], x[c], a);
                o_lat[col] = a * inv;
            }
            __syncthreads();
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                float a = 0.f;
#pragma unroll
                for (int i = 0; i < NW; ++i) {
                    const int k = i * SLICES + sl + x * SL;
                    if (k < p.r_v) a = fmaf(o_lat[k], __bfloat162float(w[x][i]), a);
                }
                sums[sl + x * SL][j] = a;
            }
            __syncthreads();
            if (tid < DH) {
                float a = sums[0][tid];
#pragma unroll
                for (int x = 1; x < SLICES; ++x) a += sums[x][tid];
                p.out[((long long)s * H_q + g * p.G + h) * DH + tid] = __float2bfloat16_rn(a);
            }
        }
        __syncwarp();
        cluster_arrive_release();                        // no CTA leaves while another may still read its part
        cluster_wait_acquire();
    }
}

}  // namespace

bool lorc_small_decode_supported(const lorc_ctx* ctx, const LorcLayer& L) {
    // (a thread of the kernel holds 8 latent columns of every head: 128 threads cover 1024)
    return L.mode == LORC_MODE_LATENT && L.r_v <= 8 * SD_THREADS && !(ctx->desc.flags & LORC_FLAG_DEBUG_FP32);
}

cudaError_t lorc_small_decode(const lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, const bf16* q, int n_splits,
                              float* part_ml, float* part_o, bf16* out, bool may_merge, bool* merged, cudaStream_t st,
                              int* launches, const int32_t* pos0, const int32_t* q_pos) {
    const lorc_model_desc& d = ctx->desc;
    SdParams p;
    p.q = q; p.cv = cv; p.B_kT = L.B_kT; p.rope_table = ctx->rope_table; p.pos0 = pos0; p.q_pos = q_pos;
    p.part_ml = part_ml; p.part_o = part_o; p.status = ctx->status_dev;
    p.r_k = L.r_k; p.r_v = L.r_v; p.G = ctx->group; p.n_splits = n_splits; p.rope_style = ctx->pair_style;
    p.max_pos = d.max_pos; p.out = out; p.B_v = L.B_v; p.n = ctx->n;
    const bool wide = d.d_head == 128;
    const long long blocks = (long long)n_splits * d.n_kv_heads * cv.batch;
    const bool one_round = wide || n_splits > 5 ? blocks <= ctx->sm_count : 3 * blocks <= 8ll * ctx->sm_count;
    *merged = may_merge && ctx->group <= SD_MERGE_HEADS && n_splits <= SD_MERGE_SHARES && L.r_v * d.d_head <= SD_MERGE_WORK &&
              one_round && (!wide || (L.r_v >= 32 && n_splits >= ctx->group));
    auto kernel = ctx->group <= 2 ? (*merged ? (wide ? small_decode_kernel<128, 2, true> : small_decode_kernel<64, 2, true>)
                                             : (wide ? small_decode_kernel<128, 2, false> : small_decode_kernel<64, 2, false>))
                  : ctx->group <= 4 ? (wide ? small_decode_kernel<128, 4, false> : small_decode_kernel<64, 4, false>)
                                    : (wide ? small_decode_kernel<128, 8, false> : small_decode_kernel<64, 8, false>);
    *launches += 1;
    const dim3 grid(n_splits, d.n_kv_heads, cv.batch), block(SD_THREADS);
    return lorc_launch_dependent_cluster(kernel, grid, block, 0, dim3(*merged ? n_splits : 1), st, p);
}
