// Cache write for prompt-sized token counts on the tensor cores (sm_100a: TMA + tcgen05 + TMEM).
//
// C_K, C_V[new tokens] = bf16(x . [A_K | A_V])  (Sec. 3.1: the cache keeps X times the Sigma-carrying factor), one GEMM
// with M = tokens, N = r_k + r_v, K = D.  At decode (a token per sequence) the call is bound by the factor stream and
// runs on the warp-level kernel; with more tokens it is a dense contraction and runs here.
//
// Persistent CTA pairs (clusters of two, cta_group::2 MMAs) walk units of 256 tokens x up to NB columns of [A_K | A_V].
// K = D in 64-wide TMA stages; x rows are the K-major A operand (128 tokens per CTA), the factor rows (D index) with their
// contiguous columns are the MN-major B operand (each CTA stages half of the unit's columns), so the factor needs no
// transposed copy.  fp32 accumulation in TMEM, two buffers: the epilogue of one unit (one rounding to bf16, transposed
// through shared memory so that a token's columns leave in 128-byte runs to its row of the contiguous or paged cache) runs
// under the MMAs of the next.  The last column block of the matrix is as narrow as what is left (a multiple of 32).
// 16384 tokens x 1344 columns, D 4096: 142 us (one CTA per 128 x 256 block, row-wise stores: 163); 777 tokens x 1856
// columns: 20 us (27).
#include <math.h>

#include "sm100_pair.cuh"
#include "sm100_ptx.cuh"
#include "tc_kernels.cuh"

using namespace sm100;

namespace {

constexpr int TILE = 128;            // tokens per CTA
constexpr int KC = 64;               // D elements per stage
constexpr int NB_MAX = 256;          // columns of [A_K | A_V] per unit
constexpr int W_STAGES = 5;
constexpr int W_THREADS = 384;       // warp 0 TMA, warp 1 MMA (leader CTA issues), warps 4..11 epilogue
constexpr int T_LD = 144;            // bytes per token of a warp's transposition buffer (64 columns and padding)

struct AppSmem {
    bf16 X[W_STAGES][TILE * KC];          // [128 tokens][64]                                               16 KiB
    bf16 A[W_STAGES][2][KC * KC];         // this CTA's half of the columns: two blocks of [64 D rows][64]  16 KiB
    uint8_t T[8][32 * T_LD];              // per epilogue warp: 32 tokens x 64 columns
    uint64_t full[W_STAGES], empty[W_STAGES], acc_full[2], acc_empty[2];
    uint32_t tmem_base;
};

struct AppParams {
    CacheView cv;
    int D, r_k, r_v, T, n_tok, max_pos, nb, m_units, n_units;
    int* status;
};

// Unit u -> token block, first column and number of columns (a multiple of 32).  First the blocks of full width, column
// blocks fastest (the pairs that work at the same time share the x rows in L2: with the token blocks fastest x came from
// HBM once per column block, 242 instead of 142 us at 16384 tokens x 1344 columns), then the narrow ones, which even out
// the last round.
__device__ __forceinline__ void app_unit(const AppParams& p, int u, int& mt, int& col0, int& cols) {
    const int R = p.r_k + p.r_v, nf = R / p.nb;
    if (u < p.m_units * nf) {
        mt = u / nf;
        col0 = (u - mt * nf) * p.nb;
        cols = p.nb;
    } else {
        mt = u - p.m_units * nf;
        col0 = nf * p.nb;
        cols = (R - col0 + 31) & ~31;
    }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(W_THREADS, 1)
lorc_append_tc_kernel(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapA, const AppParams p) {
    extern __shared__ uint8_t raw[];
    AppSmem& sm = *reinterpret_cast<AppSmem*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int rank = (int)cluster_ctarank();           // 0 = leader (issues the MMAs, owns the full / acc_empty barriers)
    const int pair_id = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const int R = p.r_k + p.r_v, nkc = p.D / KC, total = p.m_units * p.n_units;

    if (tid == 0) {
        for (int i = 0; i < W_STAGES; ++i) {
            mbar_init(&sm.full[i], 1);
            mbar_init(&sm.empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sm.acc_full[i], 1);
            mbar_init(&sm.acc_empty[i], 2 * 8);             // one arrival per epilogue warp, both CTAs
        }
        fence_barrier_init();
        prefetch_tensormap(&mapX);
        prefetch_tensormap(&mapA);
    }
    grid_dep_wait();
    if (warp == 1) {
        tmem_alloc_pair(&sm.tmem_base, 512);
        tmem_relinquish_pair();
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_arrive_release();                            // the peer's barriers are initialised before anyone signals them
    cluster_wait_acquire();
    tc_fence_after_sync();
    grid_dep_launch();
    const uint32_t tmem = sm.tmem_base;
    bool ok = true;

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer (both CTAs)
        const uint32_t x_base = smem_u32(sm.X[0]), a_base = smem_u32(sm.A[0][0]);
        const uint32_t empty0 = smem_u32(&sm.empty[0]), full0 = smem_u32(&sm.full[0]);
        const uint32_t lead_full0 = mapa_shared(full0, 0);   // all bytes of a stage are counted on the leader's barrier
        uint32_t st = 0, par = 1;
        for (int u = pair_id; u < total && ok; u += n_pairs) {
            int mt, col0, cols;
            app_unit(p, u, mt, col0, cols);
            const int tok0 = mt * 2 * TILE + rank * TILE, half = cols / 2, acol = col0 + rank * half;
            const int blocks = (half + KC - 1) / KC;
            const uint32_t bytes = 2 * (TILE + blocks * KC) * KC * 2;
            for (int kc = 0; kc < nkc; ++kc) {
                if (!mbar_wait_addr(empty0 + st * 8, par)) { ok = false; break; }
                const uint32_t lead_bar = lead_full0 + st * 8, a_dst = a_base + st * (2 * KC * KC * 2);
                if (elect_one()) {
                    // columns past r_k + r_v and token rows past the launch read as zero, but still deliver their bytes
                    if (rank == 0) mbar_arrive_expect_tx_addr(full0 + st * 8, bytes);
                    tma_load_2d_pair_addr(x_base + st * (TILE * KC * 2), &mapX, lead_bar, kc * KC, tok0);
                    tma_load_2d_pair_addr(a_dst, &mapA, lead_bar, acol, kc * KC);
                    if (blocks > 1) tma_load_2d_pair_addr(a_dst + KC * KC * 2, &mapA, lead_bar, acol + KC, kc * KC);
                }
                __syncwarp();
                if (++st == W_STAGES) { st = 0; par ^= 1; }
            }
        }
        if (!ok && lane == 0) lorc_set_status(p.status, LORC_ERR_TIMEOUT);
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (leader CTA only)
        // A: x rows (K-major), a k-step is 32 bytes.  B: factor blocks (MN-major: a D row's 64 columns are contiguous),
        // 64-column blocks 8 KiB apart, 16 D rows (one k-step) 2 KiB apart.
        if (rank == 0) {
            const uint64_t da0 = make_smem_desc_sw128(smem_u32(sm.X[0]), 0, 1024);
            const uint64_t db0 = make_smem_desc_sw128(smem_u32(sm.A[0][0]), KC * KC * 2, 1024);
            const uint32_t a_lo0 = (uint32_t)da0, a_hi = (uint32_t)(da0 >> 32);
            const uint32_t b_lo0 = (uint32_t)db0, b_hi = (uint32_t)(db0 >> 32);
            const uint32_t full0 = smem_u32(&sm.full[0]), empty0 = smem_u32(&sm.empty[0]);
            uint32_t st = 0, par = 0, uc = 0;
            for (int u = pair_id; u < total && ok; u += n_pairs, ++uc) {
                int mt, col0, cols;
                app_unit(p, u, mt, col0, cols);
                const uint32_t idesc = make_idesc_bf16(256, cols, 0, 1);
                const int buf = uc & 1;
                if (!mbar_wait(&sm.acc_empty[buf], ((uc >> 1) & 1) ^ 1)) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t d = tmem + buf * NB_MAX;
                for (int kc = 0; kc < nkc; ++kc) {
                    if (!mbar_wait_addr(full0 + st * 8, par)) { ok = false; break; }
                    tc_fence_after_sync();
                    const uint32_t a_lo = a_lo0 + st * (TILE * KC * 2 / 16), b_lo = b_lo0 + st * (2 * KC * KC * 2 / 16);
                    if (elect_one()) {
                        if (kc == 0)
                            tc_mma_bf16_pair_set(d, a_lo, a_hi, b_lo, b_hi, idesc);
                        else
                            tc_mma_bf16_pair_acc(d, a_lo, a_hi, b_lo, b_hi, idesc);
#pragma unroll
                        for (int k = 1; k < 4; ++k)
                            tc_mma_bf16_pair_acc(d, a_lo + 2 * k, a_hi, b_lo + 128 * k, b_hi, idesc);
                        tc_commit_pair_addr(empty0 + st * 8);        // frees the stage in both CTAs
                    }
                    __syncwarp();
                    if (++st == W_STAGES) { st = 0; par ^= 1; }
                }
                if (!ok) break;
                if (elect_one()) tc_commit_pair(&sm.acc_full[buf]);
                __syncwarp();
            }
            if (!ok && lane == 0) lorc_set_status(p.status, LORC_ERR_TIMEOUT);
        }
    } else if (warp >= 4) {
        // ------------------------------------------------------------------ epilogue (both CTAs): this CTA's 128 tokens
        // Warps 4..7 take the even 64-column chunks of the unit, warps 8..11 the odd ones; a warp's 32 tokens are its
        // tensor-memory lanes.  A chunk goes through the warp's own buffer: written with thread = token, read back with
        // eight lanes per token.
        const int quarter = warp % 4, part = (warp - 4) >> 2;
        uint8_t* buf_t = sm.T[warp - 4];
        const uint32_t lead_acc_empty[2] = {mapa_shared(smem_u32(&sm.acc_empty[0]), 0),
                                            mapa_shared(smem_u32(&sm.acc_empty[1]), 0)};
        uint32_t uc = 0;
        for (int u = pair_id; u < total && ok; u += n_pairs, ++uc) {
            int mt, col0, cols;
            app_unit(p, u, mt, col0, cols);
            const int buf = uc & 1;
            // where this lane's token lives: token i of sequence s goes to position seq_lens[s] - T + i
            const int tok = mt * 2 * TILE + rank * TILE + quarter * 32 + lane;
            long long row = -1;
            if (tok < p.n_tok) {
                const int s = tok / p.T, i = tok - s * p.T;
                const int pos = p.cv.seq_lens[s] - p.T + i;
                if (pos >= 0 && pos < p.max_pos) row = lorc_row_index(p.cv, s, pos);
                if (row < 0) lorc_set_status(p.status, LORC_ERR_CAPACITY);
            }
            if (!mbar_wait(&sm.acc_full[buf], (uc >> 1) & 1)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + buf * NB_MAX;
            const int n64 = (cols + KC - 1) / KC;
#pragma unroll 1
            for (int b = part; b < n64; b += 2) {
#pragma unroll
                for (int c0 = 0; c0 < KC; c0 += 32) {
                    uint32_t r[32];
                    tmem_ld32(tbase + b * KC + c0, r);       // (columns past the unit's hold stale numbers, not stored below)
                    tmem_wait_ld();
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        uint32_t w[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(r[v * 8 + 2 * e]),
                                                                            __uint_as_float(r[v * 8 + 2 * e + 1]));
                            w[e] = *reinterpret_cast<const uint32_t*>(&b2);
                        }
                        *reinterpret_cast<uint4*>(buf_t + lane * T_LD + c0 * 2 + v * 16) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
                __syncwarp();
                // eight columns per lane: ranks are multiples of eight, so a piece lies wholly in C_K or wholly in C_V
                const int pc = lane & 7, in_unit = b * KC + pc * 8, col = col0 + in_unit;
                const bool live = in_unit < cols && col < R;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int t = 4 * i + (lane >> 3);
                    const long long trow = __shfl_sync(0xffffffffu, row, t);
                    const uint4 w = *reinterpret_cast<const uint4*>(buf_t + t * T_LD + pc * 16);
                    if (live && trow >= 0) {
                        bf16* dst = col < p.r_k ? p.cv.k + trow * p.cv.w_k + col : p.cv.v + trow * p.cv.w_v + (col - p.r_k);
                        *reinterpret_cast<uint4*>(dst) = w;
                    }
                }
                __syncwarp();
            }
            // this warp has read its part of the accumulator
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(lead_acc_empty[buf]);
        }
        if (!ok && lane == 0) lorc_set_status(p.status, LORC_ERR_TIMEOUT);
    }
    // both CTAs are done with tensor memory and with each other's barriers before either lets go
    tc_fence_before_sync();
    __syncthreads();
    cluster_arrive_release();
    cluster_wait_acquire();
    if (warp == 1) tmem_dealloc_pair(tmem, 512);
}

}  // namespace

// Whether a launch runs here.  The warp-level kernel takes one block per 8 columns and 16 tokens, two at a time on an SM, and its
// time goes with the rounds of them; this one takes a time of its own up to 256 tokens (about 18 us at D 4096).  They cross at
// three rounds, whatever the rank and D.  Cache write and attention of one prompt, warp-level against here: 8B shape, r 928,
// 48 tokens 34.1 / 34.9 us, 64 tokens 38.9 / 35.9, 127 tokens 51.6 / 36.1; r 416, 127 tokens 33.2 / 33.4; r 128, 127 tokens
// 22.8 / 31.7; D 8192, r 928, 64 tokens 50.8 / 46.3.  Where the warp-level kernel does not run (D not a multiple of 256), from
// 128 tokens on.
bool lorc_tc_append_gemm_supported(const lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, int T) {
    if (L.mode != LORC_MODE_LATENT || ctx->desc.d_model % KC || L.r_k % 8 || L.r_v % 8 || !lorc_get_tmap_encode()) return false;
    const long long n_tok = (long long)cv.batch * T;
    if (!lorc_tc_append_supported(ctx, L, cv, T)) return n_tok >= TILE;
    return (L.r_k + L.r_v) / 8 * ((n_tok + 15) / 16) > 6ll * ctx->sm_count;
}

cudaError_t lorc_tc_append_gemm(lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, const bf16* x, int T,
                                cudaStream_t st, int* launches) {
    static bool attr[64] = {false};
    const bool known = ctx->device >= 0 && ctx->device < 64;
    if (!known || !attr[ctx->device]) {
        cudaError_t e = cudaFuncSetAttribute(lorc_append_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(AppSmem) + 1024);
        if (e != cudaSuccess) return e;
        if (known) attr[ctx->device] = true;
    }
    const int D = ctx->desc.d_model, R = L.r_k + L.r_v;
    const long long n_tok = (long long)cv.batch * T;
    CUtensorMap mapX, mapA;
    {
        uint64_t xd[2] = {(uint64_t)D, (uint64_t)n_tok}, xs[1] = {(uint64_t)D * 2};
        uint32_t xb[2] = {KC, TILE};
        if (!lorc_make_tmap_bf16(&mapX, x, 2, xd, xs, xb)) return cudaErrorInvalidValue;
        uint64_t ad[2] = {(uint64_t)R, (uint64_t)D}, as[1] = {(uint64_t)R * 2};
        uint32_t ab[2] = {KC, KC};
        if (!lorc_make_tmap_bf16(&mapA, L.A_cat, 2, ad, as, ab)) return cudaErrorInvalidValue;
    }
    AppParams p;
    p.cv = cv; p.D = D; p.r_k = L.r_k; p.r_v = L.r_v; p.T = T; p.n_tok = (int)n_tok; p.max_pos = ctx->desc.max_pos;
    p.status = ctx->status_dev;
    // Width of a unit: the widest (fewest operand bytes per product), unless narrower ones finish the rounds of the
    // persistent pairs in less time: a unit's time goes with its width, and below about 64 columns with the x rows.
    const int slots = ctx->sm_count / 2;
    p.m_units = (int)((n_tok + 2 * TILE - 1) / (2 * TILE));
    long long best = 0;
    for (int nb = NB_MAX; nb >= 64; nb /= 2) {
        const int nf = R / nb;
        const long long full = (long long)p.m_units * nf, rest = R > nf * nb ? p.m_units : 0;
        // rounds of full units; what is narrow fills the last round's idle pairs, or takes a round of its own
        const long long rounds = (full + slots - 1) / slots, idle = rounds * slots - full;
        const long long cost = rounds * (nb + 32) + (rest > idle ? R - nf * nb + 32 : 0);
        if (nb == NB_MAX || cost < best) {
            best = cost;
            p.nb = nb;
        }
    }
    p.n_units = (R + p.nb - 1) / p.nb;
    const long long total = (long long)p.m_units * p.n_units;
    const int pairs = total < slots ? (int)total : slots;
    *launches += 1;
    return lorc_launch_dependent(lorc_append_tc_kernel, dim3(2 * pairs), dim3(W_THREADS), sizeof(AppSmem) + 1024, st, mapX, mapA, p);
}
