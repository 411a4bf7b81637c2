// P.C_V split by LATENT COLUMNS, and the value up-projection; both contractions run on the tensor cores.
//
// PV kernel.  A CTA owns one 128-column block of C_V (rho in [128 blk, 128 blk + 128)) of one sequence and one share
// of its context.  A block of latent columns is disjoint from every other block, so the CTA's accumulator
// O_lat^T[128 rho, H_q] (fp32 in TMEM) needs no merge with other column blocks.  The score kernel left, per tile of
// 128 tokens, the softmax numerators p = bf16(2^(s - m)) against an integer reference m per 32-token quarter and head
// (as the swizzled K-major image the MMA reads), m itself and the sums of p.  While the tile sits in shared memory the
// epilogue warps multiply it by 2^(m - M), M the reference of the whole sequence (exact: only the exponent changes),
// and add up the denominator; then
//       O_lat^T += C_V[tile, block]^T . P^T                    tcgen05, MN-major A
// and at the end the CTA writes its 128 x H_q piece of the latent output, normalised, as bf16.  Several context shares of a
// block form one cluster or several: each leaves its piece in shared memory (several: in memory), and each adds up and writes its
// part of the heads and columns.  The pieces are always added in the order of the shares, so the result depends on their number,
// which follows from the sizes and the number of SMs, and not on the clusters, which follow from how a GPU's SMs are grouped.
//
// Up-projection.  One CTA per (KV head g, 64 output rows = 64 / G sequences, quarter of the head's columns)
// multiplies those rows by B_V[:, g] (TMA-staged from a transposed copy): out = o . B_V[:, g] in TMEM, then bf16.
#include <math.h>

#include "sm100_pair.cuh"
#include "sm100_ptx.cuh"
#include "tc_kernels.cuh"

using namespace sm100;

namespace {

constexpr int TILE = 128;
constexpr int KC = 64;
// one CTA per SM; 5 stages x 40 KiB with 32 query heads (200 KiB in flight), 4 x 48 KiB with 64
// (NR rows of numerators per tile: the heads, or twice as many where they are carried in two parts)
template <int NR>
struct PvStages { static constexpr int value = NR <= 32 ? 5 : NR <= 64 ? 4 : 3; };
constexpr int P_THREADS = 192;       // warp 0 TMA, warp 1 MMA, warps 2..5 epilogue
constexpr int PV_MAX_CLUSTER = LORC_PV_MAX_CLUSTER, PV_MAX_SHARES = 64;

// ------------------------------------------------------------------------------------------------
// PV kernel
// ------------------------------------------------------------------------------------------------
// Tile image written by the score kernel, fetched with one bulk copy per tile:
//   [2 chunks of 64 tokens][NR rows of 128 bytes]   p = bf16(2^(s - m)), 128-byte swizzle (the MMA's A operand); SPLIT:
//                                                   rows HQ .. 2 HQ - 1 hold the remainders bf16(2^(s - m) - p)
//   float m[4][HQ]   integer reference of every 32-token quarter and head (log2 units; -inf: no token)
//   float l[4][HQ]   sum of the quarter's rounded p
template <int HQ, bool SPLIT>
struct Pv2Smem {
    static constexpr int NR = SPLIT ? 2 * HQ : HQ;
    static constexpr int P_STAGES = PvStages<NR>::value;
    static constexpr int IMG = 2 * NR * KC * 2 + 8 * HQ * 4;
    // tile images (IMG is a multiple of 1 KiB).  They come first: with 32 rows the MMA's 64-row A operand runs
    // 4 KiB past a chunk of the image, into the next image or into V, never past the allocation
    uint8_t P[P_STAGES][IMG];
    bf16 V[P_STAGES][2][TILE * KC];       // C_V block: two 64-column halves of [128 tokens][64]; 32 KiB / stage
    float red[128 / HQ][HQ];
    float m_row[HQ];                      // row maximum over the whole sequence
    float l_inv[HQ];
    uint64_t vfull[P_STAGES], pfull[P_STAGES], fixed[P_STAGES], empty[P_STAGES], o_full;
    uint32_t tmem_base;
    int last;
};

struct Pv2Params {
    const uint8_t* pimg;           // [b, tiles, image]
    unsigned* rowmax;              // [b, H_q]   row maxima of the softmax (order-preserving keys of integers)
    bf16* o_norm;                  // [b, H_q, r_pad]      normalised latent output; SPLIT: [b, H_q, 2, r_pad], remainders second
    float* ml_out;                 // NULL, or [b, H_q, 2]: reference M (log2 units) and denominator sum_n 2^(s_n - M)
    float* o_part;                 // several clusters: [b, n_blk, n_csplit, H_q * 128 + H_q]   every share's piece and denominators
    unsigned* arrived;             // several clusters: [b * n_blk, PV_MAX_CLUSTER]   clusters whose pieces are there; zero between calls
    const int32_t* seq_lens;
    const int32_t* page_table;
    int* status;
    int batch, H_q, n_kv, r_v, tiles, n_blk, n_csplit, max_pos;
    int cluster, n_clusters;       // shares per cluster, clusters per column block: at least n_csplit together
    int max_rows;                  // SPLIT: rows of a sequence that exist
    const int32_t* pos0;           // as in the score kernel
    const int32_t* q_pos;
    int page_size, max_pages_per_seq, n_pages;
};

// A share's piece in memory: [H_q][128] outputs, then [H_q] denominators.
__host__ __device__ constexpr int share_floats(int n_q_heads) { return n_q_heads * 128 + n_q_heads; }

// Biased exponent of 2^d for an integer-valued d <= 0 (0, i.e. the number zero, below 2^-126 and for d = -inf).
__device__ __forceinline__ uint32_t pow2_exponent(float d) { return d >= -126.f ? (uint32_t)(127 + (int)d) : 0u; }

// MANY: the shares of a column block in several clusters
template <int HQ, bool SPLIT, bool MANY>
__global__ void __launch_bounds__(P_THREADS, 1)
lorc_pv2_kernel(const __grid_constant__ CUtensorMap mapCV, const Pv2Params p) {
    extern __shared__ uint8_t raw[];
    typedef Pv2Smem<HQ, SPLIT> S;
    constexpr int P_STAGES = S::P_STAGES, NR = S::NR;
    S& sm = *reinterpret_cast<S*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    constexpr uint32_t TM_COLS = 128;
    constexpr uint32_t P_BYTES = S::IMG;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int blk = blockIdx.x, cs = blockIdx.y, s = blockIdx.z;

    int len = p.seq_lens[s];
    if (len > p.max_pos) len = 0;                             // the score kernel reports the capacity errors
    if (SPLIT) len = min(len, p.max_rows);
    if (len > p.tiles * TILE || (len > 0 && !lorc_query_ok(p.pos0, p.q_pos, s, p.seq_lens[s], p.max_pos))) len = 0;
    if (len < 0) len = 0;
    // this CTA's share of the context: whole 128-token tiles, dealt evenly over the context shares (a CTA past them: none)
    const int tiles_s = (len + TILE - 1) / TILE;
    const int per = (tiles_s + p.n_csplit - 1) / p.n_csplit;
    const int tile_lo = min(tiles_s, cs * per), tile_hi = min(tiles_s, tile_lo + per);
    const int ntiles = tile_hi - tile_lo;
    const int rho0 = blk * 128;

    if (tid == 0) {
        for (int i = 0; i < P_STAGES; ++i) {
            mbar_init(&sm.vfull[i], 1);
            mbar_init(&sm.pfull[i], 1);
            mbar_init(&sm.fixed[i], 4);
            mbar_init(&sm.empty[i], 1);
        }
        mbar_init(&sm.o_full, 1);
        fence_barrier_init();
        prefetch_tensormap(&mapCV);
    }
    if (warp == 1) {
        tmem_alloc(&sm.tmem_base, TM_COLS);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = sm.tmem_base;
    bool ok = true;
    constexpr int XLD = 132;                              // floats per row of the exchanges (16-byte rows, spread over the banks)
    constexpr int SHARE_FLOATS = share_floats(HQ);
    const int r_pad = p.n_blk * 128;
    const int r_ld = SPLIT ? 2 * r_pad : r_pad;           // row of o_norm

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        // The whole warp walks the loop and one elected lane issues: the asynchronous instructions take their
        // operands from uniform registers, which the compiler only uses in warp-uniform code.
        // The kernel before this one only writes the tile images; the latent values were complete before IT could
        // start.  So the first stages' C_V boxes are requested right away, and only the images wait for that kernel
        // to finish.
        {
            const bool paged = p.page_table != nullptr;
            const int ppt = paged ? TILE / p.page_size : 0;
            auto tile_page = [&](int tile) {
                return lorc_tile_page(p.page_table, s, tile, lane, len, p.page_size, p.max_pages_per_seq, p.n_pages, p.status,
                                      SPLIT ? p.n_pages : 0);
            };
            int mine = paged && ntiles > 0 ? tile_page(tile_lo) : 0;
            for (int i = 0; i < ntiles && ok; ++i) {
                const int tile = tile_lo + i;
                const int n0 = tile * TILE;
                const int st = i % P_STAGES;
                int pages[8];
                if (paged) {
#pragma unroll
                    for (int pg = 0; pg < 8; ++pg) pages[pg] = __shfl_sync(0xffffffffu, mine, pg);
                    if (i + 1 < ntiles) mine = tile_page(tile + 1);      // on its way while this tile's boxes go out
                }
                if (i == P_STAGES) {
                    // images of the stages whose C_V boxes went out before the wait
                    grid_dep_wait();
                    if (elect_one()) {
                        for (int j = 0; j < P_STAGES; ++j) {
                            mbar_arrive_expect_tx(&sm.pfull[j], P_BYTES);
                            bulk_load(sm.P[j], p.pimg + ((long long)s * p.tiles + tile_lo + j) * P_BYTES, P_BYTES, &sm.pfull[j]);
                        }
                    }
                    __syncwarp();
                }
                if (!mbar_wait(&sm.empty[st], ((i / P_STAGES) & 1) ^ 1)) { ok = false; break; }
                if (elect_one()) {
                // the image (from L2, where the score kernel just left it) and the C_V block (from HBM) are counted on
                // barriers of their own: the exponent shift of the image runs while the block is still in flight
                if (i >= P_STAGES) {
                    mbar_arrive_expect_tx(&sm.pfull[st], P_BYTES);
                    bulk_load(sm.P[st], p.pimg + ((long long)s * p.tiles + tile) * P_BYTES, P_BYTES, &sm.pfull[st]);
                }
                mbar_arrive_expect_tx(&sm.vfull[st], 2 * TILE * KC * 2);
                if (p.page_table == nullptr) {
                    tma_load_3d(sm.V[st][0], &mapCV, &sm.vfull[st], rho0, n0, s);
                    tma_load_3d(sm.V[st][1], &mapCV, &sm.vfull[st], rho0 + 64, n0, s);
                } else {
                    // One box per page.  (Pages past the end of the sequence come from page 0, SPLIT: from behind the pool: their
                    // probabilities are zero, but the rows must hold finite numbers, which stale shared memory would not
                    // guarantee.)
#pragma unroll
                    for (int pg = 0; pg < 8; ++pg) {
                        if (pg >= ppt) break;
                        tma_load_3d(sm.V[st][0] + pg * p.page_size * KC, &mapCV, &sm.vfull[st], rho0, 0, pages[pg]);
                        tma_load_3d(sm.V[st][1] + pg * p.page_size * KC, &mapCV, &sm.vfull[st], rho0 + 64, 0, pages[pg]);
                    }
                }
                }
                __syncwarp();
            }
            if (ntiles <= P_STAGES) {
                grid_dep_wait();
                if (elect_one()) {
                    for (int j = 0; j < ntiles; ++j) {
                        mbar_arrive_expect_tx(&sm.pfull[j], P_BYTES);
                        bulk_load(sm.P[j], p.pimg + ((long long)s * p.tiles + tile_lo + j) * P_BYTES, P_BYTES, &sm.pfull[j]);
                    }
                }
                __syncwarp();
            }
            if (!ok && lane == 0) lorc_set_status(p.status, LORC_ERR_TIMEOUT);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (warp-uniform, elected lane)
        if (ntiles > 0) {
            // O_lat[64 rows (heads; 32 of them unused with 32 heads), 128 rho] += P[heads, 16 tokens] . C_V[16 tokens, 128 rho]:
            // the heads are the M side (a small M costs few cycles per MMA), the latent columns the N side
            const uint32_t idesc = make_idesc_bf16(NR <= 64 ? 64 : 128, 128, 0, 1);
            for (int i = 0; i < ntiles && ok; ++i) {
                const int st = i % P_STAGES;
                if (!mbar_wait(&sm.fixed[st], (i / P_STAGES) & 1)) { ok = false; break; }
                if (!mbar_wait(&sm.vfull[st], (i / P_STAGES) & 1)) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t p0 = smem_u32(sm.P[st]), v0 = smem_u32(sm.V[st][0]);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        // A: P [rows][128 tokens] (K-major), 64-token chunks of NR*128 bytes
                        const uint64_t ad = make_smem_desc_sw128(p0 + (k >> 2) * (NR * KC * 2) + (k & 3) * 32, 0, 1024);
                        // B: C_V block (MN-major: a token's 64 latent columns are contiguous): 16 token rows per step,
                        // the two 64-column halves 16 KiB apart
                        const uint64_t bd = make_smem_desc_sw128(v0 + k * 2048, TILE * KC * 2, 1024);
                        tc_mma_bf16(tmem, ad, bd, idesc, (i | k) != 0);
                    }
                    tc_commit(&sm.empty[st]);
                }
                __syncwarp();
            }
            if (elect_one()) tc_commit(&sm.o_full);
            __syncwarp();
            if (!ok && lane == 0) lorc_set_status(p.status, LORC_ERR_TIMEOUT);
        }
    } else {
        // ------------------------------------------------------------------ exponent shift, then epilogue
        const int t = tid - 64;
        const int quarter = warp % 4;
        constexpr int PARTS = 128 / HQ;                   // threads per head in the denominator sums
        grid_dep_wait();                                  // images and row maxima come from the kernel before this one
        grid_dep_launch();
        if (t < HQ) {
            const unsigned key = p.rowmax[(long long)s * p.H_q + t];
            sm.m_row[t] = key ? lorc_key_float(key) : 0.f;
        }
        __syncwarp();   // a named barrier counts a warp once only if the warp arrives converged
        asm volatile("bar.sync 2, 128;" ::: "memory");
        // While the tiles stream: every tile image holds p against the integer reference m of its own 32-token
        // quarter; multiplying by 2^(m - M), M the reference of the whole sequence, is exact in bf16 (a change of the
        // exponent) unless the product is too small to matter.  Thread t owns 2 NR bytes of the image: with 32 rows per
        // chunk half a row (one head, one quarter), with 64 a whole row (one head, both quarters of a chunk), with 128
        // the same row of both chunks.
        constexpr int RPT = NR == 128 ? 2 : 1;            // rows per thread
        constexpr int NP = (NR == 32 ? 64 : 128) / 16;    // 16-byte pieces of a row per thread
        const int frow0 = NR == 128 ? t : (t * 2 * NR) >> 7;   // (first) row of the image: chunk * NR + row in chunk
        const int fh = (frow0 % NR) % HQ;
        const int fpiece0 = NR == 32 ? ((t * 64) & 127) >> 4 : 0;   // first 16-byte piece (physical) of this thread
        const int frot = NR == 32 ? (t >> 1) & 3 : t & 7;  // rotation of the order in which it takes its pieces
        const float m_mine = sm.m_row[fh];
        const int lh = t % HQ, lpart = t / HQ;            // denominator: head, and which quarters of a tile
        const float m_l = sm.m_row[lh];
        float lacc = 0.f;
        for (int i = 0; i < ntiles && ok; ++i) {
            const int st = i % P_STAGES;
            if (!mbar_wait(&sm.pfull[st], (i / P_STAGES) & 1)) { ok = false; break; }
            const float* mt = reinterpret_cast<const float*>(sm.P[st] + 2 * NR * KC * 2);
            const float* lt = mt + 4 * HQ;
#pragma unroll
            for (int qq = 0; qq < 4 / PARTS; ++qq) {
                const int qrt = lpart * (4 / PARTS) + qq;
                lacc += lt[qrt * HQ + lh] * __uint_as_float(pow2_exponent(mt[qrt * HQ + lh] - m_l) << 23);
            }
#pragma unroll
            for (int rr = 0; rr < RPT; ++rr) {
                const int frow = frow0 + rr * 128, fchunk = frow / NR;
                // 2^(m - M) of the quarter(s) this thread's pieces belong to, as a bf16 pair (built from the exponent: m and M
                // are integers).  A piece's quarter is bit 2 of its logical index, physical index xor (row & 7).
                uint32_t scb[2];
#pragma unroll
                for (int hq = 0; hq < 2; ++hq) {
                    const uint32_t e = pow2_exponent(mt[(fchunk * 2 + hq) * HQ + fh] - m_mine) << 7;
                    scb[hq] = e | (e << 16);
                }
                uint4* prow = reinterpret_cast<uint4*>(sm.P[st] + frow * 128);
                uint4 v[NP];
                // (the pieces are taken in an order rotated by the thread index: the threads of a quarter warp, whose
                // pieces lie 64 or 128 bytes apart, then touch different banks)
#pragma unroll
                for (int j = 0; j < NP; ++j) v[j] = prow[fpiece0 + ((j + frot) & (NP - 1))];
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const int pp = fpiece0 + ((j + frot) & (NP - 1));
                    const uint32_t sb = scb[((pp ^ (fh & 7)) >> 2) & 1];
                    const __nv_bfloat162 sc = *reinterpret_cast<const __nv_bfloat162*>(&sb);
                    __nv_bfloat162* e = reinterpret_cast<__nv_bfloat162*>(&v[j]);
#pragma unroll
                    for (int k = 0; k < 4; ++k) e[k] = __hmul2(e[k], sc);
                    prow[pp] = v[j];
                }
            }
            if (SPLIT && (tile_lo + i + 1) * TILE > len) {
                // The rows of C_V past the end of the sequence may hold anything, as for the plain kernels, whose place this
                // path takes: their probabilities are zero, and zero the rows.  (Thread = row; the last tile of a sequence only.)
                if (!mbar_wait(&sm.vfull[st], (i / P_STAGES) & 1)) { ok = false; break; }
                if ((tile_lo + i) * TILE + t >= len) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        *reinterpret_cast<uint4*>(&sm.V[st][j >> 3][t * KC + (j & 7) * 8]) = make_uint4(0u, 0u, 0u, 0u);
                }
            }
            fence_proxy_async_smem();      // the MMA reads the image through the asynchronous proxy
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.fixed[st]);
        }
        // this share's part of the softmax denominator
        sm.red[lpart][lh] = lacc;
        __syncwarp();
        asm volatile("bar.sync 2, 128;" ::: "memory");
        float l_share = 0.f;
        if (t < HQ) {
#pragma unroll
            for (int i = 0; i < PARTS; ++i) l_share += sm.red[i][t];
        }
        if (ntiles > 0 && ok) {
            if (!mbar_wait(&sm.o_full, 0)) ok = false;
        }
        // A 64-row accumulator holds row 16 q + i (i < 16) in lane i of lane quarter q, a 128-row one row 32 q + i; it is
        // 128 latent columns wide.  The rows are the heads; SPLIT: quarters 2 and 3 hold the heads' remainders.
        constexpr int QROWS = NR <= 64 ? 16 : 32;
        const int hrow = (SPLIT ? quarter & 1 : quarter) * QROWS + lane;     // the head this thread reads
        const bool has_row = lane < QROWS && hrow < HQ && (!SPLIT || quarter < 2);
        float* xch = reinterpret_cast<float*>(&sm.V[0][0][0]);
        if (SPLIT) {
            // the products of the remainders go to the threads that hold the heads' other part (the C_V stages are free:
            // every MMA that reads them has completed)
            if (quarter >= 2) {
#pragma unroll
                for (int c0 = 0; c0 < 128; c0 += 32) {
                    uint32_t r[32];
                    if (ntiles > 0 && ok) {
                        tmem_ld32(tmem + ((uint32_t)(quarter * 32) << 16) + c0, r);
                        tmem_wait_ld();
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i) r[i] = 0u;
                    }
                    if (lane < QROWS) {
#pragma unroll
                        for (int q4 = 0; q4 < 8; ++q4)
                            *reinterpret_cast<uint4*>(xch + hrow * XLD + c0 + q4 * 4) =
                                make_uint4(r[q4 * 4], r[q4 * 4 + 1], r[q4 * 4 + 2], r[q4 * 4 + 3]);
                    }
                }
            }
            __syncwarp();
            asm volatile("bar.sync 2, 128;" ::: "memory");
        }
        // this thread's 32 columns from c0: the accumulator, with the remainders' part added
        auto take = [&](int c0, uint32_t (&r)[32]) {
            if (ntiles > 0 && ok) {
                tmem_ld32(tmem + ((uint32_t)(quarter * 32) << 16) + c0, r);
                tmem_wait_ld();
            } else {
#pragma unroll
                for (int i = 0; i < 32; ++i) r[i] = 0u;
            }
            if (SPLIT && has_row) {
#pragma unroll
                for (int i4 = 0; i4 < 8; ++i4) {
                    const float4 x = *reinterpret_cast<const float4*>(xch + hrow * XLD + c0 + i4 * 4);
                    r[i4 * 4] = __float_as_uint(__uint_as_float(r[i4 * 4]) + x.x);
                    r[i4 * 4 + 1] = __float_as_uint(__uint_as_float(r[i4 * 4 + 1]) + x.y);
                    r[i4 * 4 + 2] = __float_as_uint(__uint_as_float(r[i4 * 4 + 2]) + x.z);
                    r[i4 * 4 + 3] = __float_as_uint(__uint_as_float(r[i4 * 4 + 3]) + x.w);
                }
            }
        };
        if (!MANY && p.n_csplit == 1) {
            if (t < HQ) {
                sm.l_inv[t] = l_share > 0.f ? 1.f / l_share : 0.f;
                if (!(l_share > 0.f) && blk == 0 && !p.ml_out) lorc_set_status(p.status, LORC_ERR_EMPTY);
                if (p.ml_out && blk == 0) {
                    p.ml_out[((long long)s * p.H_q + t) * 2] = sm.m_row[t];
                    p.ml_out[((long long)s * p.H_q + t) * 2 + 1] = l_share;
                }
            }
            __syncwarp();
            asm volatile("bar.sync 2, 128;" ::: "memory");
            const float li = has_row ? sm.l_inv[hrow] : 0.f;
            bf16* on = p.o_norm + ((long long)s * p.H_q + (has_row ? hrow : 0)) * r_ld + rho0;
#pragma unroll
            for (int c0 = 0; c0 < 128; c0 += 32) {
                uint32_t r[32];
                take(c0, r);
                if (has_row) {
#pragma unroll
                    for (int q4 = 0; q4 < 4; ++q4) {
                        uint32_t w[4], wl[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float x0 = __uint_as_float(r[q4 * 8 + 2 * e]) * li, x1 = __uint_as_float(r[q4 * 8 + 2 * e + 1]) * li;
                            const __nv_bfloat162 b2 = __floats2bfloat162_rn(x0, x1);
                            w[e] = *reinterpret_cast<const uint32_t*>(&b2);
                            if (SPLIT) {
                                const float2 h2 = __bfloat1622float2(b2);
                                const __nv_bfloat162 l2 = __floats2bfloat162_rn(x0 - h2.x, x1 - h2.y);
                                wl[e] = *reinterpret_cast<const uint32_t*>(&l2);
                            }
                        }
                        *reinterpret_cast<uint4*>(on + c0 + q4 * 8) = make_uint4(w[0], w[1], w[2], w[3]);
                        if (SPLIT) *reinterpret_cast<uint4*>(on + r_pad + c0 + q4 * 8) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
                    }
                }
            }
        } else {
            // this share's piece, for the CTAs of the cluster, or in memory for those of all clusters
            float* share = MANY ? p.o_part + (((long long)s * p.n_blk + blk) * p.n_csplit + cs) * SHARE_FLOATS
                                     : xch + (SPLIT ? HQ * XLD : 0);
            constexpr int ld = MANY ? 128 : XLD;
#pragma unroll
            for (int c0 = 0; c0 < 128; c0 += 32) {
                uint32_t r[32];
                take(c0, r);
                if (has_row && (!MANY || cs < p.n_csplit)) {
#pragma unroll
                    for (int q4 = 0; q4 < 8; ++q4)
                        *reinterpret_cast<uint4*>(share + hrow * ld + c0 + q4 * 4) =
                            make_uint4(r[q4 * 4], r[q4 * 4 + 1], r[q4 * 4 + 2], r[q4 * 4 + 3]);
                }
            }
            if (t < HQ && (!MANY || cs < p.n_csplit)) (MANY ? share + HQ * 128 : sm.l_inv)[t] = l_share;
        }
        if (!ok && lane == 0) lorc_set_status(p.status, LORC_ERR_TIMEOUT);
    }
    if (MANY || p.n_csplit > 1) {
        // One cluster: behind its barrier the pieces of all shares are there.  Several: those of this cluster are, and of the CTAs
        // of one rank the last to arrive goes on, when those of the others are there too.  Each rank takes every cluster-th group of
        // 128 x four columns and adds the shares up in their order.  (Through memory, with the last share to arrive adding all of
        // them, this took 5 us for two shares and 9 for eighteen.  Interleaved pairs, b 4, 2049 tokens, six shares: step 33.6 ->
        // 31.1 us.)
        __syncwarp();
        cluster_arrive_release();
        cluster_wait_acquire();
        const int rank = MANY ? cs % p.cluster : cs;
        bool mine = warp >= 2;
        if (MANY && mine) {
            if (tid == 64) {
                __threadfence();
                // (counts up to the number of clusters and wraps, so the word is zero again for the next call)
                const unsigned before = atomicInc(p.arrived + ((long long)s * p.n_blk + blk) * PV_MAX_CLUSTER + rank, p.n_clusters - 1);
                sm.last = before == (unsigned)p.n_clusters - 1;
                __threadfence();
            }
            __syncwarp();   // a named barrier counts a warp once only if the warp arrives converged
            asm volatile("bar.sync 2, 128;" ::: "memory");
            mine = sm.last != 0;
        }
        if (mine) {
            const uint32_t share0 = smem_u32(&sm.V[0][0][0]) + (SPLIT ? HQ * XLD * 4 : 0), l0 = smem_u32(sm.l_inv);
            auto finish = [&](int i, float4 x, float l) {         // element group i: head i / 32, columns 4 (i % 32) ..
                const int h = i >> 5, c = (i & 31) * 4;
                if (blk == 0 && c == 0) {
                    if (p.ml_out) {
                        p.ml_out[((long long)s * p.H_q + h) * 2] = sm.m_row[h];
                        p.ml_out[((long long)s * p.H_q + h) * 2 + 1] = l;
                    } else if (!(l > 0.f)) {
                        lorc_set_status(p.status, LORC_ERR_EMPTY);
                    }
                }
                const float li = l > 0.f ? 1.f / l : 0.f;
                const float y[4] = {x.x * li, x.y * li, x.z * li, x.w * li};
                bf16* on = p.o_norm + ((long long)s * p.H_q + h) * r_ld + rho0 + c;
                uint32_t w[2], wl[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const __nv_bfloat162 b2 = __floats2bfloat162_rn(y[2 * e], y[2 * e + 1]);
                    w[e] = *reinterpret_cast<const uint32_t*>(&b2);
                    const float2 h2 = __bfloat1622float2(b2);
                    const __nv_bfloat162 l2 = __floats2bfloat162_rn(y[2 * e] - h2.x, y[2 * e + 1] - h2.y);
                    wl[e] = *reinterpret_cast<const uint32_t*>(&l2);
                }
                *reinterpret_cast<uint2*>(on) = make_uint2(w[0], w[1]);
                if (SPLIT) *reinterpret_cast<uint2*>(on + r_pad) = make_uint2(wl[0], wl[1]);
            };
            const int t = tid - 64;
            if (!MANY) {
                for (int i = rank * 128 + t; i < HQ * 32; i += p.n_csplit * 128) {
                    const int h = i >> 5, c = (i & 31) * 4;
                    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                    float l = 0.f;
#pragma unroll 4
                    for (int j = 0; j < p.n_csplit; ++j) {
                        const float4 v = ld_cluster_f4(mapa_shared(share0 + (h * XLD + c) * 4, j));
                        l += ld_cluster_f1(mapa_shared(l0 + h * 4, j));
                        x.x += v.x; x.y += v.y; x.z += v.z; x.w += v.w;
                    }
                    finish(i, x, l);
                }
            } else {
                // (up to E x U loads of a thread are in flight at once; with bulk copies into the C_V stages instead a call took
                // 2 us more)
                constexpr int E = 4, U = 8;
                const int step = p.cluster * 128;
                const float* part = p.o_part + ((long long)s * p.n_blk + blk) * p.n_csplit * SHARE_FLOATS;
                for (int i0 = rank * 128 + t; i0 < HQ * 32; i0 += E * step) {
                    float4 x[E];
                    float l[E];
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        x[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                        l[e] = 0.f;
                    }
                    for (int j0 = 0; j0 < p.n_csplit; j0 += U) {
                        float4 v[U][E];
                        float lv[U][E];
#pragma unroll
                        for (int u = 0; u < U; ++u)
#pragma unroll
                            for (int e = 0; e < E; ++e) {
                                const int i = i0 + e * step;
                                v[u][e] = make_float4(0.f, 0.f, 0.f, 0.f);
                                lv[u][e] = 0.f;
                                if (j0 + u < p.n_csplit && i < HQ * 32) {
                                    const float* piece = part + (long long)(j0 + u) * SHARE_FLOATS;
                                    v[u][e] = __ldcg(reinterpret_cast<const float4*>(piece) + i);
                                    lv[u][e] = __ldcg(piece + HQ * 128 + (i >> 5));
                                }
                            }
#pragma unroll
                        for (int u = 0; u < U; ++u)
#pragma unroll
                            for (int e = 0; e < E; ++e) {
                                x[e].x += v[u][e].x; x[e].y += v[u][e].y; x[e].z += v[u][e].z; x[e].w += v[u][e].w;
                                l[e] += lv[u][e];
                            }
                    }
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (i0 + e * step < HQ * 32) finish(i0 + e * step, x[e], l[e]);
                }
            }
        }
        __syncwarp();
        cluster_arrive_release();                        // no CTA leaves while another may still read its piece
        cluster_wait_acquire();
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, TM_COLS);
}

}  // namespace

namespace {

// ------------------------------------------------------------------------------------------------
// value up-projection: out[(s, h), :] = o_norm[s, h, :] . B_V[:, g(h)], a plain TMA-fed tcgen05 GEMM.
// grid (n_kv_heads, ceil(batch * G / 64), 4): 64 output rows (s, i) x 32 of the head's 128 columns, K = r_v in
// slices of 64.  (Splitting the columns gives four times the CTAs and small stages, so a whole rank is in flight.)
// ------------------------------------------------------------------------------------------------
constexpr int U_STAGES = 16;         // 16 x 12 KiB: every rank up to 1024 fits in one round of loads
constexpr int U_THREADS = 192;
constexpr int U_NCOL = 32;           // output columns per CTA (a quarter of a head)
constexpr int U_ROWS = 64;           // output rows (sequence, head of the KV head) per CTA: the M of the MMA

constexpr int U_LD = 80;             // bytes per row of the transposition buffer (64 and padding)

template <bool HOST>
struct UpSmem {
    bf16 A[U_STAGES][U_ROWS * KC];        // o_norm rows [64 rows (s, i)][64 rho]
    bf16 B[U_STAGES][U_NCOL * KC];        // B_V^T slice [32 columns j][64 rho]
    uint8_t O[HOST ? 4 : 0][16 * U_LD];   // HOST: per epilogue warp: 16 finished rows of 64 bytes
    uint64_t full[U_STAGES], empty[U_STAGES], d_full;
    uint32_t tmem_base;
};

struct UpParams {
    bf16* out;                     // [b, H_q, 128]
    unsigned* rowmax;              // [b, H_q]   left empty for the next call's score kernel
    int* status;
    int batch, H_q, G, r_v;
    int parts, r_pad;              // bf16 parts of the latent rows (the second one r_pad columns after the first)
};

// HOST: `out` is mapped host memory
template <bool HOST>
__global__ void __launch_bounds__(U_THREADS, 1)
lorc_upproj_kernel(const __grid_constant__ CUtensorMap mapON, const __grid_constant__ CUtensorMap mapBVT,
                   const UpParams p) {
    extern __shared__ uint8_t raw[];
    typedef UpSmem<HOST> S;
    S& sm = *reinterpret_cast<S*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int g = blockIdx.x, chunk = blockIdx.y, cq = blockIdx.z;     // KV head, block of 64 rows, column quarter
    const int nslice = (p.r_v + KC - 1) / KC, nkc = nslice * p.parts;    // slices of the rank, of the contraction
    const int seqs_per_cta = U_ROWS / p.G;
    constexpr uint32_t STAGE_BYTES = (U_ROWS + U_NCOL) * KC * 2;
    if (tid == 0) {
        for (int i = 0; i < U_STAGES; ++i) {
            mbar_init(&sm.full[i], 1);
            mbar_init(&sm.empty[i], 1);
        }
        mbar_init(&sm.d_full, 1);
        fence_barrier_init();
        prefetch_tensormap(&mapON);
        prefetch_tensormap(&mapBVT);
    }
    if (warp == 1) {
        tmem_alloc(&sm.tmem_base, 32);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = sm.tmem_base;
    bool ok = true;

    if (warp == 0) {
        // (warp-uniform loops, one elected lane issues)
        // The factor slices of the first stages do not depend on the kernel before this one: they are requested
        // before the wait, the latent rows after it.
        const int npre = nkc < U_STAGES ? nkc : U_STAGES;
        if (elect_one()) {
            for (int kc = 0; kc < npre; ++kc) {
                mbar_arrive_expect_tx(&sm.full[kc], STAGE_BYTES);
                tma_load_2d(sm.B[kc], &mapBVT, &sm.full[kc], (kc % nslice) * KC, g * 128 + cq * U_NCOL);
            }
        }
        __syncwarp();
        grid_dep_wait();                             // the normalised latent rows come from the kernel before
        grid_dep_launch();
        for (int kc = 0; kc < nkc; ++kc) {
            const int st = kc % U_STAGES;
            if (kc >= npre && !mbar_wait(&sm.empty[st], ((kc / U_STAGES) & 1) ^ 1)) { ok = false; break; }
            if (elect_one()) {
                if (kc >= npre) {
                    mbar_arrive_expect_tx(&sm.full[st], STAGE_BYTES);
                    tma_load_2d(sm.B[st], &mapBVT, &sm.full[st], (kc % nslice) * KC, g * 128 + cq * U_NCOL);
                }
                // rows (s, i): box of G heads x 128/G sequences (sequences past the batch read as zero)
                tma_load_3d(sm.A[st], &mapON, &sm.full[st], (kc / nslice) * p.r_pad + (kc % nslice) * KC, g * p.G,
                            chunk * seqs_per_cta);
            }
            __syncwarp();
        }
        if (!ok && lane == 0) lorc_set_status(p.status, LORC_ERR_TIMEOUT);
    } else if (warp == 1) {
        const uint32_t idesc = make_idesc_bf16(U_ROWS, U_NCOL, 0, 0);    // 64 rows: half the cycles of a 128-row MMA
        for (int kc = 0; kc < nkc; ++kc) {
            const int st = kc % U_STAGES;
            if (!mbar_wait(&sm.full[st], (kc / U_STAGES) & 1)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t a0 = smem_u32(sm.A[st]), b0 = smem_u32(sm.B[st]);
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    tc_mma_bf16(tmem, make_smem_desc_sw128(a0 + k * 32, 0, 1024), make_smem_desc_sw128(b0 + k * 32, 0, 1024),
                                idesc, (kc | k) != 0);
                tc_commit(&sm.empty[st]);
            }
            __syncwarp();
        }
        if (elect_one()) tc_commit(&sm.d_full);
        __syncwarp();
        if (!ok && lane == 0) lorc_set_status(p.status, LORC_ERR_TIMEOUT);
    } else {
        grid_dep_wait();
        // every reader of the row maxima (the kernel before this one) has completed
        if (g == 0 && chunk == 0 && cq == 0)
            for (int i = tid - 64; i < p.batch * p.H_q; i += 128) p.rowmax[i] = 0u;
        if (!mbar_wait(&sm.d_full, 0)) ok = false;
        if (ok) {
            tc_fence_after_sync();
            // A 64-row accumulator keeps row 16 q + i (i < 16) in lane i of lane quarter q; row = s_local * G + i.  A lane stores
            // its row's 64 bytes, unless `out` lies in host memory, where a store of 16 bytes is a bus transaction of
            // its own (20 us for 131 KB): there the rows go through shared memory and leave with four lanes per row (12 us).
            const int quarter = warp % 4;
            uint32_t r[32];
            tmem_ld32(tmem + ((uint32_t)(quarter * 32) << 16), r);
            tmem_wait_ld();
            auto row_of = [&](int row) -> uint4* {
                const int s = chunk * seqs_per_cta + row / p.G, h = g * p.G + row % p.G;
                return s < p.batch ? reinterpret_cast<uint4*>(p.out + ((long long)s * p.H_q + h) * 128 + cq * U_NCOL) : nullptr;
            };
            uint4* dst = row_of(quarter * 16 + (lane & 15));
            if constexpr (HOST) dst = reinterpret_cast<uint4*>(sm.O[warp - 2] + lane * U_LD);
            if (lane < 16 && dst) {
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) {
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        __nv_bfloat162 b = __floats2bfloat162_rn(__uint_as_float(r[q4 * 8 + 2 * e]),
                                                                 __uint_as_float(r[q4 * 8 + 2 * e + 1]));
                        w[e] = *reinterpret_cast<uint32_t*>(&b);
                    }
                    dst[q4] = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            if constexpr (HOST) {
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int lr = i * 8 + (lane >> 2);
                    uint4* to = row_of(quarter * 16 + lr);
                    if (to) to[lane & 3] = *reinterpret_cast<const uint4*>(sm.O[warp - 2] + lr * U_LD + (lane & 3) * 16);
                }
            }
        }
        if (!ok && lane == 0) lorc_set_status(p.status, LORC_ERR_TIMEOUT);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, 32);
}

// Result of lorc_decode_attn_latent_out: the normalised latent output without the padding columns, and the row maxima
// left empty for the next call (what the up-projection kernel does otherwise).
__global__ void latent_out_kernel(const bf16* __restrict__ o_norm, bf16* __restrict__ o_lat, unsigned* rowmax, int rows,
                                  int r_v, int r_ld) {
    grid_dep_wait();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < rows) rowmax[i] = 0u;
    const int vec = r_v / 8;                              // r_v is a multiple of 8: 16-byte pieces
    if (i < (long long)rows * vec) {
        const long long row = i / vec, c = i % vec;
        reinterpret_cast<uint4*>(o_lat + row * r_v)[c] = reinterpret_cast<const uint4*>(o_norm + row * r_ld)[c];
    }
}

// Scratch: the normalised latent output [b][H_q][parts][r_pad] of a layer with n_blk column blocks.
size_t on_bytes(const lorc_ctx* ctx, int batch, int n_blk) {
    return lorc_align_up((size_t)batch * ctx->desc.n_q_heads * (lorc_tc_split(ctx) ? 2 : 1) * n_blk * 128 * sizeof(bf16), 256);
}

template <bool MANY, class Fn>
cudaError_t with_pv_kernel(const lorc_ctx* ctx, Fn fn) {
    const bool split = lorc_tc_split(ctx);
    if (ctx->desc.n_q_heads == 32)
        return split ? fn(lorc_pv2_kernel<32, true, MANY>, sizeof(Pv2Smem<32, true>) + 1024)
                     : fn(lorc_pv2_kernel<32, false, MANY>, sizeof(Pv2Smem<32, false>) + 1024);
    return split ? fn(lorc_pv2_kernel<64, true, MANY>, sizeof(Pv2Smem<64, true>) + 1024)
                 : fn(lorc_pv2_kernel<64, false, MANY>, sizeof(Pv2Smem<64, false>) + 1024);
}

// Scratch of `shares` shares whose pieces go through memory.
size_t part_bytes(const lorc_ctx* ctx, long long blocks, int shares) {
    return (size_t)blocks * shares * share_floats(ctx->desc.n_q_heads) * sizeof(float);
}

// Clusters of `blocks` blocks that are resident at once (0: no such launch).  Asked for once per context, when a plan first wants
// to know: the fifteen sizes together take as long as a small layer.
int pv_clusters(lorc_ctx* ctx, int blocks) {
    if (blocks == 1) return ctx->sm_count;
    int& known = ctx->pv_clusters[blocks];
    if (known == 0) {
        int n = 0;
        const cudaError_t e = with_pv_kernel<false>(ctx, [&](auto kernel, size_t smem) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(1, blocks, 1);
            cfg.blockDim = dim3(P_THREADS);
            cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 1;
            attr[0].val.clusterDim.y = (unsigned)blocks;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            return cudaOccupancyMaxActiveClusters(&n, kernel, &cfg);
        });
        if (e != cudaSuccess) {
            cudaGetLastError();      // (a size that the GPU does not take)
            n = 0;
        }
        known = n > 0 ? n : -1;
    }
    return known > 0 ? known : 0;
}

}  // namespace

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
size_t lorc_tc_pv_scratch_least(const lorc_ctx* ctx, int batch) { return on_bytes(ctx, batch, (ctx->n + 127) / 128); }

// The pieces of as many shares as the plan takes by itself, for any rank.
size_t lorc_tc_pv_scratch_bytes(const lorc_ctx* ctx, int batch, int max_seq_len) {
    const int tiles = (max_seq_len + TILE - 1) / TILE;
    size_t most = 0;
    for (int n_blk = 1; n_blk <= (ctx->n + 127) / 128; ++n_blk) {
        const long long blocks = (long long)batch * n_blk;
        int shares = (int)(ctx->sm_count / blocks);
        if (shares > tiles) shares = tiles;
        if (shares > PV_MAX_SHARES) shares = PV_MAX_SHARES;
        if (shares > 1 && part_bytes(ctx, blocks, shares) > most) most = part_bytes(ctx, blocks, shares);
    }
    return lorc_tc_pv_scratch_least(ctx, batch) + most;
}

cudaError_t lorc_tc_pv_set_attrs(const lorc_ctx* ctx) {
    // (one context's kernels; the attributes are the device's, and another context sets those of its own)
    auto attr = [](auto kernel, size_t bytes) {
        return cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    auto pv_attr = [&](auto kernel, size_t bytes) {
        const cudaError_t e = cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        return e == cudaSuccess ? attr(kernel, bytes) : e;
    };
    cudaError_t e = with_pv_kernel<false>(ctx, pv_attr);
    if (e == cudaSuccess) e = with_pv_kernel<true>(ctx, pv_attr);
    if (e == cudaSuccess) e = attr(lorc_upproj_kernel<false>, sizeof(UpSmem<false>) + 1024);
    if (e == cudaSuccess) e = attr(lorc_upproj_kernel<true>, sizeof(UpSmem<true>) + 1024);
    return e;
}

// One CTA per SM at most, and the number of shares whose chain is shortest.  In units of one tile (about 0.45 us of a CTA's
// stream): the tiles of a share, and with more than one share 8 and 0.8 per share.  So up to 15 tiles one CTA takes a block.
// (The constants were measured with shares that met in memory, where the last to arrive added all of them; inside one cluster the
// exchange takes about 2 us less.)  The shares of a block are dealt to as few clusters of equal size as are resident at once.
void lorc_tc_pv_plan(lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, int n_splits_hint, size_t scratch_bytes,
                     LorcPvPlan* plan) {
    const int tiles = (cv.max_seq_len + TILE - 1) / TILE;
    plan->n_blk = (L.r_v + 127) / 128;
    plan->off_part = on_bytes(ctx, cv.batch, plan->n_blk);
    plan->fits = plan->off_part <= scratch_bytes;
    const long long blocks = (long long)cv.batch * plan->n_blk;
    long long most = n_splits_hint > 0 ? n_splits_hint : ctx->sm_count / blocks;
    if (most > tiles) most = tiles;
    if (most > PV_MAX_SHARES) most = PV_MAX_SHARES;
    int shares = n_splits_hint > 0 ? (int)most : 1;
    if (n_splits_hint <= 0) {
        int best = 5 * tiles;                                 // five times the cost, in tiles
        for (int cs = 2; cs <= most; ++cs) {
            const int cost = 5 * ((tiles + cs - 1) / cs + 8) + 4 * cs;
            if (cost < best) {
                best = cost;
                shares = cs;
            }
        }
    }
    for (; shares > 1; --shares) {
        int clusters = (shares + PV_MAX_CLUSTER - 1) / PV_MAX_CLUSTER;
        while (clusters <= shares && pv_clusters(ctx, (shares + clusters - 1) / clusters) < blocks * clusters) ++clusters;
        // (a count that was asked for, of more blocks than run at once: pairs, which leave no SM idle.  b 4, r 256, 32777 tokens, 24
        // and 64 shares: 94 and 113 us before clusters, 103 and 123 in clusters of 12 and 16, 95 and 109 in pairs; b 16, r 512, 4129
        // tokens, as many as the workspace holds: 83, 114 and 90)
        if (clusters > shares) clusters = pv_clusters(ctx, 2) > 0 ? (shares + 1) / 2 : shares;
        if (clusters > 1 && plan->off_part + part_bytes(ctx, blocks, shares) > scratch_bytes) continue;
        plan->n_csplit = shares;
        plan->n_clusters = clusters;
        plan->cluster = (shares + clusters - 1) / clusters;
        return;
    }
    plan->n_csplit = plan->cluster = plan->n_clusters = 1;
}

// scratch: the normalised latent output, then the pieces of shares in several clusters
cudaError_t lorc_tc_pv_launch(lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, const CUtensorMap& mapCV,
                              const CUtensorMap& mapBVT, const uint8_t* pimg, unsigned* rowmax, unsigned* arrived, int tiles,
                              const LorcPvPlan& plan, void* scratch, bf16* out, bool latent_out, const int32_t* pos0,
                              const int32_t* q_pos, float* ml_out, cudaStream_t st, int* launches) {
    const lorc_model_desc& d = ctx->desc;
    const int n_blk = plan.n_blk;
    const int r_pad = n_blk * 128;
    const bool split = lorc_tc_split(ctx);
    const int r_ld = split ? 2 * r_pad : r_pad;        // row of o_norm
    bf16* o_norm = (bf16*)scratch;
    cudaError_t e;
    {
        LorcStageTimer timer(ctx, LORC_STAGE_PV, st);
        Pv2Params p;
        p.pimg = pimg; p.rowmax = rowmax; p.o_norm = o_norm; p.ml_out = ml_out;
        p.seq_lens = cv.seq_lens; p.page_table = cv.page_table; p.status = ctx->status_dev;
        p.batch = cv.batch; p.H_q = d.n_q_heads; p.n_kv = d.n_kv_heads; p.r_v = L.r_v; p.tiles = tiles;
        p.o_part = (float*)((char*)scratch + plan.off_part); p.arrived = arrived;
        p.n_blk = n_blk; p.n_csplit = plan.n_csplit; p.cluster = plan.cluster; p.n_clusters = plan.n_clusters; p.max_pos = d.max_pos; p.max_rows = lorc_tc_max_rows(cv);
        p.pos0 = pos0; p.q_pos = q_pos;
        p.page_size = cv.page_size; p.max_pages_per_seq = cv.max_pages_per_seq; p.n_pages = cv.n_pages;
        dim3 grid(n_blk, plan.cluster * plan.n_clusters, cv.batch);
        auto launch = [&](auto kernel, size_t smem) {
            return lorc_launch_dependent_cluster(kernel, grid, dim3(P_THREADS), smem, dim3(1, plan.cluster, 1), st, mapCV, p);
        };
        e = plan.n_clusters > 1 ? with_pv_kernel<true>(ctx, launch) : with_pv_kernel<false>(ctx, launch);
        *launches += 1;
        if (e != cudaSuccess) return e;
    }
    LorcStageTimer timer(ctx, LORC_STAGE_COMBINE, st);
    if (latent_out) {
        const int rows = cv.batch * d.n_q_heads;
        const long long work = (long long)rows * (L.r_v / 8);
        e = lorc_launch_dependent(latent_out_kernel, dim3((unsigned)((work + 255) / 256)), dim3(256), 0, st,
                                  (const bf16*)o_norm, out, rowmax, rows, L.r_v, r_ld);
        *launches += 1;
        return e;
    }
    // o_norm [b, H_q, r_ld] as (rho, head, sequence) with boxes of 64 rho x G heads x 64/G sequences
    CUtensorMap mapON;
    {
        uint64_t dims[3] = {(uint64_t)r_ld, (uint64_t)d.n_q_heads, (uint64_t)cv.batch};
        uint64_t str[2] = {(uint64_t)r_ld * 2, (uint64_t)d.n_q_heads * r_ld * 2};
        uint32_t box[3] = {KC, (uint32_t)ctx->group, (uint32_t)(U_ROWS / ctx->group)};
        if (!lorc_make_tmap_bf16(&mapON, o_norm, 3, dims, str, box)) return cudaErrorInvalidValue;
    }
    UpParams u;
    u.out = out; u.rowmax = rowmax; u.status = ctx->status_dev;
    u.batch = cv.batch; u.H_q = d.n_q_heads; u.G = ctx->group; u.r_v = L.r_v;
    u.parts = split ? 2 : 1; u.r_pad = r_pad;
    dim3 ugrid(d.n_kv_heads, (cv.batch * ctx->group + U_ROWS - 1) / U_ROWS, 128 / U_NCOL);
    e = ctx->host_out ? lorc_launch_dependent(lorc_upproj_kernel<true>, ugrid, dim3(U_THREADS), sizeof(UpSmem<true>) + 1024, st, mapON, mapBVT, u)
                      : lorc_launch_dependent(lorc_upproj_kernel<false>, ugrid, dim3(U_THREADS), sizeof(UpSmem<false>) + 1024, st, mapON, mapBVT, u);
    *launches += 1;
    return e;
}
