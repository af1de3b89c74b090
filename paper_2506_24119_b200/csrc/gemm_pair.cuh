// Dense GEMM of the context append on pairs of SMs (tcgen05 cta_group::2, sm_100a):
//     Y[t][r] = sum_k X[t][k] * W[r][k]     X fp16 [T][K], W fp16 (the k-block-major copy of gemm_tc.cuh), fp32 sums
//
// A cluster of two CTAs works on one output tile of 256 weight rows x N token rows (N <= 256, a multiple of 32): CTA r
// of the pair holds weight rows 128 r .. + 127 and token rows (N / 2) r .. of the tile in its shared memory, one
// tcgen05.mma (M = 256) of the leader CTA reads both halves of both, and each CTA's tensor memory receives its 128
// weight rows x N token columns.  What bounds a dense contraction here is shared memory: with a tile of 128 x 256 per
// CTA every k step of 16 fills and reads 12 KB in the 128 cycles its MMA takes; with the token rows halved between the
// CTAs of a pair 8 KB.  One CTA, six warps:
//   warp 0      TMA producer of its CTA's half; both CTAs' copies are counted on the leader's "stage full" barriers
//   warp 1      MMA issuer (leader CTA): four MMAs per k block; completion frees the stage in both CTAs (commit with
//               multicast) and, at a tile's last block, releases the accumulator to both epilogues
//   warps 2..5  epilogue under the next tile's main loop (two accumulators of N columns): 32 token rows at a time
//               through a staging buffer and out by TMA: plain store, reduction into the residual stream (every
//               element receives exactly one addition per launch, so the result does not depend on any order), or
//               SwiGLU gating to fp16
// Work is dealt to the pairs in one of two forms:
//   whole tiles, round-robin, when they fill the pairs evenly: the epilogue sees complete sums;
//   stream-K when they do not (few token rows: 331 rows give the 2560-row matrices 20 tiles for 74 pairs): the
//   flattened (tile, k block) space in equal contiguous ranges, each touched tile leaving one "piece" per range, summed
//   in k order by the kernel that reads it (Pieces of kernels_small.cuh).
#pragma once
#include "gemm_tc.cuh"

namespace spiral {

constexpr int PG_BM = 2 * TC_BM;                     // weight rows per pair tile
constexpr int PG_MAX_N = 256;                        // token rows per pair tile
constexpr int PG_THREADS = 192;
constexpr int PG_MAX_STAGES = 8;
constexpr int PG_BPS = 2;                            // k blocks per stage = per TMA box
constexpr size_t PG_SMEM_BUDGET = 227 * 1024 - 1024;           // less the static part (barriers)
enum { PG_STORE = 0, PG_ADD = 1, PG_SILU = 2 };

struct PgParams {
    int row_tiles, tok_tiles, KB;   // 256-row tiles of W, N-row tiles of X, 64-wide k blocks
    int T, N;                       // token rows; token rows per tile
    int whole, row_fastest;         // whole tiles or stream-K; order of whole tiles (see pg_tile_of)
    int stages;                     // ring depth
    int w_once;                     // 1: weight tiles are read by few token tiles and leave L2 first
    float unscale;                  // what the sums are multiplied with (TcWeight::unscale)
    int* status;
};

// consecutive tiles share a weight tile (token tile fastest: each weight tile comes from HBM once and is shared through
// L2) or an activation tile (row tile fastest: where the activations are the larger operand)
__device__ __forceinline__ void pg_tile_of(int L, const PgParams& p, int& rt, int& tt) {
    if (p.row_fastest) { tt = L / p.row_tiles; rt = L - tt * p.row_tiles; }
    else { rt = L / p.tok_tiles; tt = L - rt * p.tok_tiles; }
}

// one part of a tile: k blocks [kb0, kb1)
struct PgSeg { int tile, kb0, kb1, piece; };
// the work of pair c of G
struct PgSchedule {
    long long u, u1, U;
    int tiles, KB, c, G, whole, L;
    __host__ __device__ PgSchedule(int tiles_, int KB_, int whole_, int c_, int G_) {
        tiles = tiles_; KB = KB_; whole = whole_; c = c_; G = G_; L = c_;
        U = (long long)tiles * KB;
        u = U * c / G;
        u1 = U * (c + 1) / G;
    }
    __host__ __device__ bool next(PgSeg& sg) {
        if (whole) {
            if (L >= tiles) return false;
            sg.tile = L; sg.kb0 = 0; sg.kb1 = KB; sg.piece = 0;
            L += G;
            return true;
        }
        if (u >= u1) return false;
        const int tile = (int)(u / KB), off = (int)(u - (long long)tile * KB);
        const long long left = u1 - u;
        const int len = (int)(left < KB - off ? left : KB - off);
        sg.tile = tile; sg.kb0 = off; sg.kb1 = off + len;
        sg.piece = c - streamk_cta_of((long long)tile * KB, G, U);
        u += len;
        return true;
    }
};

// ---- cta_group::2 forms --------------------------------------------------------------------------
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst_smem, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_mma_f16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// one arrival on the barrier at this address in both CTAs once every MMA issued so far by this thread has completed
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
    const uint16_t both = 3;
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"(both) : "memory");
}
// tiled load into this CTA's shared memory whose bytes are counted on a barrier of the leader CTA
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t leader_bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3, %4}], [%5], %6;"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(leader_bar), "l"(policy) : "memory");
}
// element-wise addition of a dense fp32 box in shared memory to global memory (same rules as tma_store_3d)
__device__ __forceinline__ void tma_reduce_add_3d(const CUtensorMap* map, uint32_t src, int x, int y, int z) {
    asm volatile("cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3, %4}], [%1];"
                 ::"l"(map), "r"(src), "r"(x), "r"(y), "r"(z) : "memory");
}

// tmOut: STORE: [piece][T][rows] floats; ADD: [1][T][rows] floats; box 1 x 32 x 32.  SILU: [1][T][rows / 2] fp16, box 1 x 32 x 16.
template <int EPI, bool SCALED>           // SCALED: p.unscale != 1
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PG_THREADS, 1)
    pg_gemm_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                   const __grid_constant__ CUtensorMap tmOut, PgParams p) {
    extern __shared__ uint8_t pg_smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[PG_MAX_STAGES], empty_bar[PG_MAX_STAGES], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base_sm;
    __shared__ int abort_sm;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int pair = (int)(blockIdx.x >> 1), G = (int)(gridDim.x >> 1);
    grid_launch_dependents();
    constexpr int BPS = PG_BPS;
    const int S = p.stages, N = p.N;
    // a stage: the W halves of PG_BPS k blocks, then their X halves, each group one TMA box
    const uint32_t x_bytes = (uint32_t)(N / 2) * 128u, stage_bytes = PG_BPS * (TC_W_BYTES + x_bytes);
    const uint32_t ring = (smem_u32(pg_smem_raw) + 1023u) & ~1023u;
    const uint32_t out_stage = ring + (uint32_t)S * stage_bytes;
    uint32_t tmem_cols = 32;
    while (tmem_cols < 2u * (uint32_t)N) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(smem_u32(&acc_full[a]), 1); mbar_init(smem_u32(&acc_empty[a]), 8); }
        abort_sm = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tmap_prefetch(&tmW);
        tmap_prefetch(&tmX);
        tmap_prefetch(&tmOut);
    }
    if (warp == 1) tmem_alloc_pair(smem_u32(&tmem_base_sm), tmem_cols);
    tc_fence_before();
    __syncthreads();
    cluster_sync();                     // both CTAs' barriers exist before either's copies or commits reach them
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_sm;
    volatile int* abort_flag = &abort_sm;

    if (warp == 0) {
        // ---------------- TMA producer (the whole warp walks the loop, one elected lane issues) ----------------
        const uint64_t pol_w = p.w_once ? l2_policy_evict_first() : l2_policy_evict_last(), pol_x = l2_policy_evict_last();
        const uint32_t full_leader = map_to_rank(smem_u32(&full_bar[0]), 0), full_own = smem_u32(&full_bar[0]);
        const uint32_t empty_own = smem_u32(&empty_bar[0]);
        const int n_tiles = p.row_tiles * p.tok_tiles;
        // weights are written by nobody: the W halves of the first ring-full go out before the dependency wait
        int pre = 0;
        {
            PgSchedule sched(n_tiles, p.KB, p.whole, pair, G);
            PgSeg sg;
            bool more = sched.next(sg);
            int kb = more ? sg.kb0 : 0;
            while (more && pre < S) {
                int rt, tt;
                pg_tile_of(sg.tile, p, rt, tt);
                // (a stage never crosses a segment: where one has an odd number of blocks, its last stage fetches a block
                // that is not used)
                const int y_w = (2 * rt + (int)rank) * TC_BM;
                const uint32_t dst = ring + (uint32_t)pre * stage_bytes;
                if (elect_one()) {
                    if (rank == 0) mbar_expect_tx(full_own + 8u * (uint32_t)pre, 2u * stage_bytes);
                    tma_load_3d_pair(dst, &tmW, 0, y_w, kb, full_leader + 8u * (uint32_t)pre, pol_w);
                }
                __syncwarp();
                ++pre;
                kb += BPS;
                if (kb >= sg.kb1) { more = sched.next(sg); kb = more ? sg.kb0 : 0; }
            }
        }
        grid_dependency_wait();                                  // X is written by the preceding kernel
        PgSchedule sched(n_tiles, p.KB, p.whole, pair, G);
        PgSeg sg;
        bool ok = true;
        int st = 0;
        uint32_t s = 0, ph = 0;
        while (ok && sched.next(sg)) {
            int rt, tt;
            pg_tile_of(sg.tile, p, rt, tt);
            const int y_x = tt * N + (int)rank * (N / 2), y_w = (2 * rt + (int)rank) * TC_BM;
            for (int kb = sg.kb0; kb < sg.kb1; kb += BPS, ++st) {
                const uint32_t dst = ring + s * stage_bytes, fb = full_leader + 8u * s;
                const bool with_w = st >= pre;
                if (with_w && !mbar_wait_warp(empty_own + 8u * s, ph ^ 1u, abort_flag, p.status, STATUS_TIMEOUT_MMA)) { ok = false; break; }
                if (elect_one()) {
                    if (with_w) {
                        if (rank == 0) mbar_expect_tx(full_own + 8u * s, 2u * stage_bytes);
                        tma_load_3d_pair(dst, &tmW, 0, y_w, kb, fb, pol_w);
                    }
                    tma_load_3d_pair(dst + PG_BPS * TC_W_BYTES, &tmX, 0, y_x, kb, fb, pol_x);
                }
                __syncwarp();
                if (++s == (uint32_t)S) { s = 0; ph ^= 1u; }
            }
        }
        if (!ok && rank == 0 && lane == 0) {
            // copies already issued still land in the pair's shared memory: bounded wait for them
            for (int back = 1; back <= S && back <= st; ++back) {
                const int j = st - back;
                const uint32_t sj = (uint32_t)(j % S), pj = (uint32_t)(j / S) & 1u;
                unsigned long long t1 = global_ns();
                while (!mbar_try(full_own + 8u * sj, pj) && global_ns() - t1 < g_wait_limit_ns) {}
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (leader CTA) ----------------
        if (rank == 0) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(PG_BM >> 4) << 24);
            const uint64_t desc0 = smem_desc_sw128(ring);
            const uint64_t d_x0 = (uint64_t)((PG_BPS * TC_W_BYTES) >> 4), d_x = (uint64_t)(x_bytes >> 4), d_stage = (uint64_t)(stage_bytes >> 4);
            PgSchedule sched(p.row_tiles * p.tok_tiles, p.KB, p.whole, pair, G);
            PgSeg sg;
            uint32_t s = 0, ph = 0, a = 0, aph = 0;
            bool ok = true;
            while (ok && sched.next(sg)) {
                if (!mbar_wait_warp(smem_u32(&acc_empty[a]), aph ^ 1u, abort_flag, p.status, STATUS_TIMEOUT_EPI)) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + a * (uint32_t)N;
                uint32_t acc = 0u;
                for (int kb = sg.kb0; kb < sg.kb1; kb += BPS) {
                    const int nb = min(BPS, sg.kb1 - kb);
                    if (!mbar_wait_warp(smem_u32(&full_bar[s]), ph, abort_flag, p.status, STATUS_TIMEOUT_TMA)) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t da = desc0 + d_stage * s;
                    if (elect_one()) {
                        for (int b = 0; b < nb; ++b) {
                            const uint64_t dab = da + (uint64_t)(b * (TC_W_BYTES >> 4)), db = da + d_x0 + d_x * (uint64_t)b;
#pragma unroll
                            for (int k = 0; k < TC_BK / 16; ++k)
                                tc_mma_f16_pair(d_tmem, dab + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc,
                                                (acc | (uint32_t)b | (uint32_t)k) ? 1u : 0u);
                        }
                        tc_commit_pair(smem_u32(&empty_bar[s]));
                    }
                    __syncwarp();
                    acc = 1u;
                    if (++s == (uint32_t)S) { s = 0; ph ^= 1u; }
                }
                if (ok && elect_one()) tc_commit_pair(smem_u32(&acc_full[a]));
                __syncwarp();
                if ((a ^= 1u) == 0u) aph ^= 1u;
            }
        }
    } else {
        // ---------------- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 = weight rows of this CTA's half ----------------
        const int q = warp & 3;
        grid_dependency_wait();              // the output may still be read (or, ADD, written) by earlier kernels
        const uint32_t release0 = map_to_rank(smem_u32(&acc_empty[0]), 0);
        PgSchedule sched(p.row_tiles * p.tok_tiles, p.KB, p.whole, pair, G);
        PgSeg sg;
        uint32_t a = 0, aph = 0, out_it = 0;
        while (sched.next(sg)) {
            int rt, tt;
            pg_tile_of(sg.tile, p, rt, tt);
            if (!mbar_wait(smem_u32(&acc_full[a]), aph, abort_flag, p.status, STATUS_TIMEOUT_MMA)) break;
            tc_fence_after();
            const int row0 = rt * PG_BM + (int)rank * TC_BM;
            const uint32_t t_addr = tmem_base + ((uint32_t)(q * 32) << 16) + a * (uint32_t)N;
            for (int c0 = 0; c0 < N && tt * N + c0 < p.T; c0 += TC_OUT_ROWS, ++out_it) {
                uint32_t v[2][16];
                tmem_ld16_async(t_addr + (uint32_t)c0, v[0]);
                tmem_ld16_async(t_addr + (uint32_t)(c0 + 16), v[1]);
                const uint32_t buf = out_stage + (uint32_t)(2 * q + (int)(out_it & 1u)) * TC_OUT_BYTES;
                if (out_it >= 2) {
                    if (lane == 0) tma_store_wait_read<1>();
                    __syncwarp();
                }
                tmem_ld_wait();
                if (SCALED) tc_unscale(v, p.unscale);
                if (EPI == PG_SILU) {
                    // even lanes hold gate features, odd lanes the matching up features: per pair of token columns the
                    // even lane finishes the first and the odd lane the second
                    const bool odd = lane & 1;
                    const uint32_t base = buf + (uint32_t)(lane >> 1) * 2u + (odd ? 32u : 0u);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int j = 0; j < 16; j += 2) {
                            const float m0 = __uint_as_float(v[h][j]), m1 = __uint_as_float(v[h][j + 1]);
                            const float got = __shfl_xor_sync(0xffffffffu, odd ? m0 : m1, 1);
                            const float gate = odd ? got : m0, up = odd ? m1 : got;
                            const unsigned short r = (unsigned short)float_to_f16_bits(__fdividef(gate, 1.f + __expf(-gate)) * up);
                            asm volatile("st.shared.b16 [%0], %1;" ::"r"(base + (uint32_t)(16 * h + j) * 32u), "h"(r) : "memory");
                        }
                } else {
                    const uint32_t base = buf + (uint32_t)lane * 4u;
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            asm volatile("st.shared.b32 [%0], %1;" ::"r"(base + (uint32_t)(16 * h + j) * 128u), "r"(v[h][j]) : "memory");
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    const int y = tt * N + c0, x = row0 + q * 32;
                    if (EPI == PG_ADD) tma_reduce_add_3d(&tmOut, buf, x, y, 0);
                    else if (EPI == PG_SILU) tma_store_3d(&tmOut, buf, x >> 1, y, 0);
                    else tma_store_3d(&tmOut, buf, x, y, sg.piece);
                    tma_store_commit();
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(release0 + 8u * a);
            if ((a ^= 1u) == 0u) aph ^= 1u;
        }
        if (lane == 0) tma_store_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();                     // the peer's shared and tensor memory is in use until the leader's last MMA is done
    if (warp == 1) tmem_dealloc_pair(tmem_base, tmem_cols);
}

// ---- host side -----------------------------------------------------------------------------------
struct PgPlan {
    int N = 0, tok_tiles = 0, row_tiles = 0, KB = 0, G = 0, whole = 1, max_pieces = 1, stages = 0;
    size_t smem = 0;
};

// Time of one 64-wide k block of a pair tile of N token rows, us: measured on a pair working alone (the 9728-wide down
// projection, T = N).  Up to N = 128 the weight half of the tile sets it (an SM takes at most 67 bytes per clock from L2).
inline double pg_block_us(int N) {
    static const double at[][2] = {{32, 0.195}, {64, 0.20}, {128, 0.208}, {160, 0.27}, {192, 0.295}, {224, 0.31}, {256, 0.325}};
    for (int i = 1; i < 7; ++i)
        if (N <= at[i][0]) return at[i - 1][1] + (at[i][1] - at[i - 1][1]) * (N - at[i - 1][0]) / (at[i][0] - at[i - 1][0]);
    return at[6][1];
}

// How a [rows][K] matrix meets T token rows: the token tile N and whole tiles or stream-K, whichever the estimate below
// makes shorter.  Whole tiles cost their waves over the pairs; stream-K fills every pair but writes each piece and has it
// read again (both at about 3 TB/s, from L2), and where the epilogue would have gated (`gated`) the gating becomes a
// kernel of its own.  E.g. 331 rows of the Qwen3-4B matrices, all with N = 128 (estimates, us, whole against stream-K):
// gate/up whole (4 waves of 76 x 3 tiles; 33 against 51 with the gating kernel that stream-K needs), QKV whole (72 tiles; 8
// against 12), output and down projection stream-K (10 and 18 against 13 and 32).
constexpr int PG_SPLIT_MAX_T = 1024;                 // bounds the pieces buffer
constexpr int PG_SEARCH_MAX_T = 2048;                // beyond: many waves, and the widest tile moves the fewest bytes per flop
enum { PG_OUT_PIECES = 0, PG_OUT_ADD = 1, PG_OUT_GATED = 2 };      // what a whole tile's epilogue writes
// Stream-K over `tiles` tiles: pairs that take part, and its estimated time (fixed + per_row x token rows, us)
struct PgSplit { int G; double fixed, per_row; };
inline PgSplit pg_split(int pairs, int tiles, int KB, int N, int rows, int out) {
    const long long U = (long long)tiles * KB;
    int G = (int)std::min<long long>(pairs, std::max<long long>(1, U / 4));       // no ranges under four k blocks
    // Whole numbers of equal k ranges per tile where they use nearly all pairs (10 tiles x 7, 24 x 3 of 74): one segment
    // and one epilogue per pair, as in tc_get_plan.  Qwen3-4B shape, us per call: 100 tokens 3519 -> 3347, 2 x 25
    // 3348 -> 3239; Llama-3.1-8B shape 2 x 60 4272 -> 4183, Qwen2.5-7B shape 3871 -> 3730.
    const int aligned = tiles <= G ? tiles * (G / tiles) : 0;
    if (aligned * 100 >= G * 94) G = aligned;
    const double pieces = 1.0 + (double)G / tiles, one = (double)rows * 4 / 3e6;
    return PgSplit{G, (double)U / G * pg_block_us(N) + (out == PG_OUT_GATED ? 5.0 : 1.0),
                   one * (out == PG_OUT_PIECES ? pieces - 1.0 : out == PG_OUT_GATED ? pieces + 1.0 : pieces)};
}
inline int pg_max_pieces(int tiles, int KB, int G) {
    const long long U = (long long)tiles * KB;
    int most = 0;
    for (int t = 0; t < tiles; ++t) {
        const long long first = (long long)t * KB;
        most = std::max(most, streamk_cta_of(first + KB - 1, G, U) - streamk_cta_of(first, G, U) + 1);
    }
    return most;
}
inline PgPlan pg_plan(int n_sm, int rows, int K, int T, int out) {
    PgPlan pl;
    pl.row_tiles = (rows + PG_BM - 1) / PG_BM;
    pl.KB = (K + TC_BK - 1) / TC_BK;
    const int pairs = std::max(1, n_sm / 2), fewest = (T + PG_MAX_N - 1) / PG_MAX_N;
    double best = -1;
    const int most = T <= PG_SEARCH_MAX_T ? fewest + 3 : fewest;
    for (int tt = fewest; tt <= most; ++tt) {
        const int N = ((T + tt - 1) / tt + 31) & ~31, tok_tiles = (T + N - 1) / N;
        if (tok_tiles != tt) continue;
        const int tiles = pl.row_tiles * tok_tiles, waves = (tiles + pairs - 1) / pairs;
        const double whole = (double)waves * pl.KB * pg_block_us(N);
        if (best < 0 || whole < best) { best = whole; pl.N = N; pl.tok_tiles = tok_tiles; pl.whole = 1; }
        const PgSplit sp = pg_split(pairs, tiles, pl.KB, N, rows, out);
        const double split = sp.fixed + sp.per_row * T;
        if (T <= PG_SPLIT_MAX_T && split < best) { best = split; pl.N = N; pl.tok_tiles = tok_tiles; pl.whole = 0; pl.G = sp.G; }
    }
    const int tiles = pl.row_tiles * pl.tok_tiles;
    if (pl.whole) {
        pl.G = std::min(pairs, tiles);
    } else {
        pl.max_pieces = pg_max_pieces(tiles, pl.KB, pl.G);
    }
    const size_t blk = TC_W_BYTES + (size_t)(pl.N / 2) * 128, budget = PG_SMEM_BUDGET - 1024 - TC_OUT_BUFS * TC_OUT_BYTES;
    pl.stages = (int)std::min<size_t>(PG_MAX_STAGES, budget / (PG_BPS * blk));
    pl.smem = (size_t)pl.stages * PG_BPS * blk + TC_OUT_BUFS * TC_OUT_BYTES + 1024;
    return pl;
}

// The most floats a plan for up to `cap` token rows leaves in pieces: what the buffer has to hold for every call that the
// rest of a workspace of `cap` rows holds.  For each token tile: the largest T at which stream-K is still estimated shorter
// than whole tiles (pg_plan takes it for no other), times its pieces.
inline size_t pg_piece_elems(int n_sm, int rows, int K, int cap, int out) {
    const int row_tiles = (rows + PG_BM - 1) / PG_BM, KB = (K + TC_BK - 1) / TC_BK, pairs = std::max(1, n_sm / 2);
    size_t most = out == PG_OUT_PIECES ? (size_t)cap * rows : 0;
    for (int tt = 1; tt <= PG_SPLIT_MAX_T / PG_MAX_N + 3; ++tt)
        for (int N = 32; N <= PG_MAX_N; N += 32) {
            const int tiles = row_tiles * tt, waves = (tiles + pairs - 1) / pairs;
            const PgSplit sp = pg_split(pairs, tiles, KB, N, rows, out);
            const double slack = (double)waves * KB * pg_block_us(N) - sp.fixed;
            int T = std::min(std::min(N * tt, cap), PG_SPLIT_MAX_T);
            if (slack <= 0) continue;
            if (sp.per_row * T > slack) T = (int)(slack / sp.per_row) + 1;
            if (T > (N - 32) * tt && tt <= (T + PG_MAX_N - 1) / PG_MAX_N + 3)
                most = std::max(most, (size_t)pg_max_pieces(tiles, KB, sp.G) * T * rows);
        }
    return most;
}

// a tensor of fp16 values as [outer][mid][64] with a box of box_outer x box_mid x 64, 128-byte swizzle (none for the weight
// copies, which are stored swizzled)
inline int pg_encode(TcState& tc, CUtensorMap* m, const void* base, uint64_t mid, uint64_t mid_bytes, uint64_t outer, uint64_t outer_bytes,
                     uint32_t box_mid, uint32_t box_outer, bool swizzle = true) {
    cuuint64_t dims[3] = {(cuuint64_t)TC_BK, (cuuint64_t)mid, (cuuint64_t)outer};
    cuuint64_t strides[2] = {(cuuint64_t)mid_bytes, (cuuint64_t)outer_bytes};
    cuuint32_t box[3] = {(cuuint32_t)TC_BK, box_mid, box_outer};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = tc.encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        g_tc_error = "cuTensorMapEncodeTiled (pair operand) failed (" + std::to_string((int)r) + ")";
        return SPIRAL_ERR_CUDA;
    }
    return SPIRAL_OK;
}
// X [T][K] as [k block][T][64]: one box is PG_BPS k blocks of box_rows rows.  Where K is no multiple of 64 the last block of
// a row runs into the next row (the buffer is that much longer and zeroed once): finite values that meet the zeros of the
// weight copy.
inline int pg_get_xmap(TcState& tc, const __half* X, int K, int T, int box_rows, const CUtensorMap** out) {
    auto key = std::make_tuple((const void*)X, K, T, -box_rows);
    auto it = tc.xmaps.find(key);
    if (it == tc.xmaps.end()) {
        if (tc.xmaps.size() > 4096) tc.xmaps.clear();
        CUtensorMap m;
        int rc = pg_encode(tc, &m, X, (uint64_t)T, (uint64_t)K * 2, (uint64_t)((K + TC_BK - 1) / TC_BK), 128, (uint32_t)box_rows, PG_BPS);
        if (rc) return rc;
        it = tc.xmaps.emplace(key, m).first;
    }
    *out = &it->second;
    return SPIRAL_OK;
}
// the weight copy as [k block][row][64], a box of PG_BPS k blocks of a 128-row tile (beyond the last row or block: zeros)
inline int tc_weight_map(TcState& tc, const TcWeight& w, CUtensorMap* map, int box_rows, int box_kb) {
    const uint64_t slab = (uint64_t)((w.rows + TC_BM - 1) / TC_BM) * TC_BM;
    return pg_encode(tc, map, w.w16, slab, 128, (uint64_t)((w.K + TC_BK - 1) / TC_BK), slab * 128, (uint32_t)box_rows, (uint32_t)box_kb, false);
}
inline int pg_get_wmap(TcState& tc, TcWeight& w, const CUtensorMap** out) {
    if (!w.has_map2) {
        int rc = tc_weight_map(tc, w, &w.map2, TC_BM, PG_BPS);
        if (rc) return rc;
        w.has_map2 = true;
    }
    *out = &w.map2;
    return SPIRAL_OK;
}

// fp16 output [T][cols] with a 1 x 32 x 16 box (SILU epilogue)
inline int pg_get_actmap(TcState& tc, const __half* base, int cols, int T, const CUtensorMap** out) {
    auto key = std::make_tuple((const void*)base, cols, T, -1);
    auto it = tc.omaps.find(key);
    if (it == tc.omaps.end()) {
        if (tc.omaps.size() > 4096) tc.omaps.clear();
        CUtensorMap m;
        cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)T, 1};
        cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)T * cols * 2};
        cuuint32_t box[3] = {16, (cuuint32_t)TC_OUT_ROWS, 1};
        cuuint32_t estr[3] = {1, 1, 1};
        CUresult r = tc.encode(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half*>(base), dims, strides, box, estr,
                               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) {
            g_tc_error = "cuTensorMapEncodeTiled (activations) failed (" + std::to_string((int)r) + ")";
            return SPIRAL_ERR_CUDA;
        }
        it = tc.omaps.emplace(key, m).first;
    }
    *out = &it->second;
    return SPIRAL_OK;
}

// EPI over T token rows.  W: the caller's bf16 matrix, registered (its fp16 copy is read).  out: STORE: fp32
// [max_pieces][T][rows]; ADD: fp32 [T][rows], added to; SILU: fp16 [T][rows / 2].  pieces (STORE): what a consumer needs.
template <int EPI>
inline int pg_gemm(TcState& tc, const PgPlan& pl, const __nv_bfloat16* W, int rows, int K, const __half* X, int T, void* out,
                   Pieces* pieces, int* status, cudaStream_t st, int64_t* launches) {
    if (!tc_resident(tc, W, rows, K)) return SPIRAL_ERR_UNSUPPORTED;
    auto it = tc.weights.find(W);
    const CUtensorMap *xm = nullptr, *om = nullptr;
    int rc = pg_get_xmap(tc, X, K, T, pl.N / 2, &xm);
    if (rc) return rc;
    const CUtensorMap* wm = nullptr;
    rc = pg_get_wmap(tc, it->second, &wm);
    if (rc) return rc;
    if (EPI == PG_SILU) rc = pg_get_actmap(tc, (const __half*)out, rows / 2, T, &om);
    else rc = tc_get_omap(tc, (const float*)out, rows, T, EPI == PG_STORE ? pl.max_pieces : 1, &om);
    if (rc) return rc;
    PgParams p{};
    p.row_tiles = pl.row_tiles; p.tok_tiles = pl.tok_tiles; p.KB = pl.KB; p.T = T; p.N = pl.N; p.whole = pl.whole;
    p.row_fastest = (pl.whole && T > rows) ? 1 : 0;              // re-read the smaller operand: weights rows x K, activations T x K
    p.stages = pl.stages; p.w_once = pl.tok_tiles <= 2; p.status = status; p.unscale = it->second.unscale;
    TC_TRY(launch_kernel(true, it->second.unscale != 1.f ? pg_gemm_kernel<EPI, true> : pg_gemm_kernel<EPI, false>, dim3(2 * pl.G), dim3(PG_THREADS), pl.smem, st, *wm, *xm, *om, p));
    if (launches) ++*launches;
    if (pieces) {
        pieces->base = (const float*)out; pieces->stride = (size_t)T * rows; pieces->ld = rows; pieces->n_pieces = pl.max_pieces;
        pieces->sk_KB = pl.KB; pieces->sk_G = pl.whole ? 0 : pl.G;
        pieces->sk_shift = 8; pieces->sk_tt = pl.tok_tiles; pieces->sk_BN = pl.N;
    }
    return SPIRAL_OK;
}

inline int pg_gemm_setup() {
    for (auto kern : {pg_gemm_kernel<PG_STORE, false>, pg_gemm_kernel<PG_STORE, true>, pg_gemm_kernel<PG_ADD, false>,
                      pg_gemm_kernel<PG_ADD, true>, pg_gemm_kernel<PG_SILU, false>, pg_gemm_kernel<PG_SILU, true>})
        TC_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PG_SMEM_BUDGET));
    return SPIRAL_OK;
}

}  // namespace spiral
