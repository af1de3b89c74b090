// All layers of a decode step for few games in one persistent kernel.
//
// With few games a step reads the weights once and little else; the per-layer kernels then spend more time at their
// boundaries (release of the dependency, first tile, epilogue, partial sums through L2) than streaming: 62 us per layer of
// the Qwen3-4B shape with one game, of which 28 are the weights.  Here one CTA per SM stays for the whole step:
//
//   warps 8, 9  producers.  Every byte that a layer reads from memory in bulk -- the four weight matrices, the cached keys
//               and values -- is known before the step starts, so it is asked for in the order of use, through a ring of
//               shared memory that knows no layer or phase boundary: while the CTAs wait for each other, the weights of the
//               phases behind are on their way (about 150 KB per SM, three microseconds of memory).
//   warp 10     norms.
//   warps 0..7  consumers: products, attention, element-wise work.
//
// us per step, kernel per operation -> this kernel (contexts of 200 to 1000 tokens): Qwen3-4B shape, 1 game 2297 -> 1940, 2
// games 2331 -> 2009, 4 games 2398 -> 2189, 8 games 2471 -> 2342 (contexts to 5000: 2970 -> 2851); Llama-3.1-8B shape 3177 ->
// 2862, 3205 -> 2894, 3261 -> 3119, 3349 -> 3213 (3781 -> 3725); two layers of 256 columns, 4 games 74 -> 56.  Of a layer's 52 us
// with one game the memory is idle for about a fifth: the attention's chain (queries from L2, first page, partial results of
// several CTAs) is longer than what the ring holds.  Nine and more games, as two tiles of the products, were slower here than
// as kernels (11 games 3757 against 2254): every CTA reads all activations of a phase, and a stage of the attention costs the
// same however many there are.
//
// A CTA owns whole rows of every matrix (rows c R / G .. (c + 1) R / G), so no partial sum leaves it: the eight warps
// split the k blocks (and, where a CTA has more than 80 rows, the rows), and add up in shared memory.  What a phase passes
// to the next is a vector per game through global memory and one barrier of all CTAs; five per layer:
//
//   QKV       x stored by the owners as fp16 (x gain 2^e), see below                   -> raw q, k, v in fp32
//   attention q/k-norm, rotation, the append of the new key and value, paged attention -> heads in fp16
//   output    residual += ..., kept by the owner in shared memory for the whole step   -> x in fp16
//   gate/up   SiLU(gate) up                                                            -> fp16
//   down      residual += ...                                                          -> x in fp16
//
// RMSNorm needs the sum of squares of a whole row, which no CTA has when it stores its columns.  They are stored as
// fp16(x gain 2^e) with 2^e about 1/256 of the reciprocal norm of the row's previous state, beside the CTA's part of the
// sum of squares; whoever reads them adds the parts up (in CTA order, so everybody gets the same) and multiplies the sums
// by norm / 2^e.  The rounding is that of fp16(x norm gain), since powers of two are exact.  Should a row have grown more than
// 256-fold or shrunk more than fourfold in between, fp16 might no longer hold it like the normalised value: then the owners
// store their columns again (every CTA sees the same sums and comes to the same conclusion).
//
// The products use mma.sync.m16n8k16 (weight rows are the M side, games the N side): 18 to 132 rows per CTA do not fill a
// tcgen05 tile, whose activations would have to pass through shared memory as well, and at eight games the legacy pipe needs a
// fraction of the time the weights need to arrive.  Activations go from L2 straight into registers, three 64-wide k blocks
// ahead of their use (us per step, Qwen3-4B shape with 1 and 4 games, Llama-3.1-8B shape with 2: two blocks 2035, 2202, 2937;
// three 1981, 2187, 2923; four 1966, 2222, 3000; eight 8 % more than four: moves cost more than latency); they are stored in an order (fs_perm) in
// which one 16-byte load is two B fragments.
//
// CTAs wait for one another, so the launch is cooperative.  Every wait is bounded: after a timeout the CTA records a status
// and walks through the rest of the step without waiting (its results are garbage and the status says so), arriving at
// every barrier, so that nobody is left behind.
#pragma once
#include <cuda.h>

#include "attn_decode.cuh"
#include "common.cuh"
#include "gemm_pair.cuh"
#include "gemm_tc.cuh"
#include "kernels_small.cuh"
#include "tma.cuh"

namespace spiral {

constexpr int FS_WARPS = 8;                        // consumer warps
// A third warpgroup carries the producer and the norms: with nine warps a thread could have 168 registers (three warps on one
// of the four schedulers), with twelve the two consumer warpgroups take over what the third does not need: 256 x 224 +
// 128 x 56 registers are the 384 x 168 of the launch.
constexpr int FS_THREADS = 32 * (FS_WARPS + 4);
constexpr int FS_REG_CONSUMER = 224, FS_REG_PRODUCER = 56;
constexpr int FS_MAX_GAMES = 8;                    // one 8-column tile of the products (figures above)
// Slots of the ring, two per consumer warp: stage q of the step lies in slot q % 16 and is taken by warp q % 8, always.  (A
// warp may wait for a parity of a barrier only if it has seen every earlier phase of it complete.)
constexpr int FS_SLOTS = 2 * FS_WARPS;
constexpr int FS_PRODUCERS = 2;                    // warps that ask for the stages, in turn: about 0.3 us each (with one: 1 game
                                                   // of the Qwen3-4B shape 2460 us per step instead of 2226)
// Items of at most this many pages are not shared by CTAs: two pages per warp cost less than adding up partial results
// through the L2 (5 us).
constexpr int FS_WHOLE = 16;
constexpr int FS_MT = 5;                           // 16-row tiles of a warp: row groups of up to 80 weight rows
constexpr int FS_COLS = 64;                        // residual columns a CTA can own
constexpr int FS_EXP_BIAS = 8;                     // activations are stored 2^-8 below their normalised size

// how one of a layer's matrices is dealt: CTA c of G owns the row units [U c / G, U (c + 1) / G), U = rows / unit, cut into
// `groups` groups; warp w works on group w % groups and every (8 / groups)-th stage of it
struct FsMat {
    int rows, K, KB;
    int unit;               // rows that stay together (gate and up rows are interleaved: 2)
    int groups;             // 1, 2 or 4
    int h;                  // rows of a group: the most any CTA has, and what a stage holds of every k block
    int m, stages;          // k blocks per stage, stages per group
    int pitch;              // row stride (floats) of a warp's sums in shared memory
    int ldx;                // row stride of the activations: whole stages, zeros behind the last k
};
enum { FS_QKV = 0, FS_O = 1, FS_GU = 2, FS_DOWN = 3, FS_ATT = 4 };

struct FsVectors {
    const __nv_bfloat16* vec[4];    // per phase: bias of the QKV rows, gain of the norm behind the residual (or none)
    const __nv_bfloat16* qk_norm[2];
    const __half* w[2];             // the copies of the two matrices behind a norm (QKV, gate/up), see FsGemm::again
    float unscale[4];
};
struct FsLayer {
    CUtensorMap w[4];       // the fp16 copies as [k block][row][64], a box of FsMat::m k blocks of FsMat::h rows
    FsVectors v;
};

struct FsParams {
    const FsLayer* layers;
    int n_layers, n;
    FsMat mat[4];
    int d_model, d_ff, vocab;
    float eps, inv_d;       // inv_d: 1 / d_model
    const __nv_bfloat16 *embed, *first_norm;
    int qk_norm;
    const StepArgs* args;
    StepMeta meta;
    int32_t* block_table;
    const float *cos_tab, *sin_tab;
    uint16_t* pool;
    AttnParams at{};        // schedule, scratch and status of the attention (q, layer and len_add unused)
    float* qkv;             // [n][qkv rows]
    __half *xn, *heads, *act;       // activations [n][ldx], in the order of fs_perm
    __half* h;              // [n][d_model] after the final norm, in plain order
    float* ss_part;         // [grid][FS_MAX_GAMES]
    unsigned int* bar;      // arrivals, CTAs that have left; both zero between launches
    int slot_bytes, red_bytes;
};

__device__ __forceinline__ void fs_bar_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
// the norms of a phase: given by the norm warp, taken by the consumers (both wait: after an abort neither may run ahead)
__device__ __forceinline__ void fs_norms_sync() { asm volatile("bar.sync 2, 288;" ::: "memory"); }
// A value the compiler cannot reason about: keeps it from making a copy of a loop for every case of a condition that does not
// change in it (code that is run once per phase and layer comes from the L2 every time: about 300 cycles per 128 bytes).
__device__ __forceinline__ int fs_opaque(int v) {
    asm volatile("" : "+r"(v));
    return v;
}

// Where element k of an activation row is stored: inside 32 elements the pairs (2 c, 2 c + 1) of the four 8-element chunks
// lie together, which is what lane c of a quad needs for two k steps of 16.
__host__ __device__ inline int fs_perm(int k) { return (k & ~30) | ((k & 6) << 2) | ((k & 24) >> 2); }

// rows of group j of CTA c
__host__ __device__ inline void fs_rows(const FsMat& M, int c, int G, int j, int& a, int& h) {
    const long long U = M.rows / M.unit;
    const int u0 = (int)(U * c / G), un = (int)(U * (c + 1) / G) - u0;
    const int g0 = un * j / M.groups, g1 = un * (j + 1) / M.groups;
    a = (u0 + g0) * M.unit;
    h = (g1 - g0) * M.unit;
}

// How a matrix is dealt.  False where the matrix does not fit this kernel.
inline bool fs_plan(FsMat& M, int rows, int K, int unit, int G, int slot_bytes) {
    M.rows = rows; M.K = K; M.unit = unit; M.KB = (K + TC_BK - 1) / TC_BK;
    if (rows % unit || K % 8) return false;
    const int units = (rows / unit + G - 1) / G;
    for (M.groups = 1; M.groups <= 4; M.groups *= 2)
        if ((units + M.groups - 1) / M.groups * unit <= 16 * FS_MT) break;
    if (M.groups > 4) return false;
    M.h = (units + M.groups - 1) / M.groups * unit;
    const int kparts = FS_WARPS / M.groups;
    // A stage costs its producer and its consumer a barrier round trip each: as many k blocks as a slot holds and as leave
    // the warp with the longest share little more than the others.
    if (M.h * 128 > slot_bytes) return false;
    int best = 1 << 30;
    for (int m = 1; m <= 32 && m * M.h * 128 <= slot_bytes; ++m) {
        const int rounds = (M.KB + kparts * m - 1) / (kparts * m), cost = rounds * (2 * m + 1);
        if (cost <= best) { best = cost; M.m = m; }
    }
    M.stages = (M.KB + M.m - 1) / M.m;
    M.pitch = ((M.h + 15) & ~15) + 4;
    return true;
}

struct FsShared {
    FsMat mat[4];
    uint64_t full[FS_SLOTS], empty[FS_SLOTS];
    int row[FS_SLOTS];                             // attention stages: first pool row of the unit, or -1
    int cum[FS_MAX_GAMES + 2], len[FS_MAX_GAMES], game[FS_MAX_GAMES], newp[FS_MAX_GAMES];
    float mult[FS_MAX_GAMES];                      // norm / 2^e of each game's stored activations
    float scale[FS_MAX_GAMES];                     // 2^e of the activations stored next
    float inv[FS_MAX_GAMES];                       // reciprocal norm of each game's row
    int misfit;                                    // a row has left the window in which fp16 holds it like the normalised one
    float vec[16 * FS_MT * 4];                     // bias of the CTA's rows, gains of its columns
    alignas(16) float qk_gain[2][128];
    FsVectors lay[2];                              // this layer's and the next one's
    int2 rows[4][4];                               // first row and number of rows of each matrix and row group
    // Partial results that the warps leave for each other: [0] of an item that began before the warp's units, [1] of one that
    // begins in them.
    struct Part {
        int item;                                  // slot * n_kv_heads + kv head, or -1
        int side;                                  // 0: began before this CTA's units, 1: goes on after them, 2: neither
        int first_cta, n_cta;                      // CTAs that share it
        float m[8], l[8];
        const float* o;                            // [group][head_dim] in shared memory
    } part[FS_WARPS][2];
    int last[2], open_item[2], open_first[2], open_n[2];   // items shared with earlier / later CTAs: the item or -1, its CTAs
    int abort;
};

// The slow half of a wait for an mbarrier phase: false when the time limit ran out or the CTA has given up.
__device__ __forceinline__ bool fs_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status, int code) {
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
#pragma unroll 1
    for (uint32_t spin = 1; !mbar_try(bar, parity); ++spin) {
        if (*abort_flag) return false;
        if ((spin & 63u) == 0 && global_ns() - t0 > g_wait_limit_ns) {
            record_status(status, code);
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}

// The producers: everything the layers read in bulk, in the order of use, through the ring's slots.  Warp `which` of them
// asks for every FS_PRODUCERS-th stage.
template <int HD>
__device__ __forceinline__ void fs_produce(const FsParams& p, const CUtensorMap* tmKV, FsShared* sh, uint32_t ring, int c0, int c1, int which) {
    constexpr int HALVES = HD / 64;
    constexpr uint32_t UNIT = HD * 64;             // 16 keys and 16 values of one head
    const int lane = threadIdx.x & 31;
    const uint64_t pol_w = l2_policy_evict_first();
    // attention: warp w (counted from the one that takes the phase's first stage) has u_base contiguous units, one more if
    // w < u_rem; a stage is a unit
    const int cnt = c1 - c0, u_base = cnt / FS_WARPS, u_rem = cnt % FS_WARPS;
    int pool_row = -1;                             // first pool row of the unit of stage `lane` of the window, or -1
    int q = 0;
    bool ok = true;
#pragma unroll 1
    for (int l = 0; l < p.n_layers && ok; ++l)
#pragma unroll 1
        for (int k = 0; k < 5 && ok; ++k) {
            const int phase = k == 0 ? FS_QKV : k == 1 ? FS_ATT : k - 1;
            const FsMat& M = sh->mat[phase & 3];
            const CUtensorMap* map = &p.layers[l].w[phase & 3];
            // (descriptors come from memory: the next phase's is on its way while this one's are in use)
            if (lane == 0 && phase < 4 && (phase < 3 || l + 1 < p.n_layers)) tmap_prefetch(phase < 3 ? map + 1 : &p.layers[l + 1].w[0]);
            const uint32_t w_bytes = (uint32_t)(M.h * M.m) * 128u;
            const int count = phase == FS_ATT ? cnt : M.stages * M.groups;
            const int step = M.m, groups = M.groups;
            int kb = 0, j = 0;
#pragma unroll 1
            for (int i = 0; i < count; ++i) {
                const bool att = fs_opaque(phase) == FS_ATT;
                if (att && (i & 31) == 0) {
                    const int w = lane & (FS_WARPS - 1), u = c0 + u_base * w + min(w, u_rem) + (i + lane) / FS_WARPS;
                    pool_row = -1;
                    if (i + lane < count) {
                        int slot = 0;
#pragma unroll 1
                        while (slot + 1 < p.n && sh->cum[slot + 1] <= u) ++slot;
                        const int pages = (sh->len[slot] + ATTN_PAGE - 1) / ATTN_PAGE, off = u - sh->cum[slot];
                        const int kvh = off / pages, pg = off - kvh * pages;
                        // a page that begins with this step's token is not in the table yet
                        const int page = (pg + 1 == pages && sh->newp[slot] >= 0) ? sh->newp[slot] : __ldcg(p.block_table + (size_t)sh->game[slot] * p.at.max_pages + pg);
                        if (page < 0 || page >= p.at.n_pages) record_status(p.at.status, STATUS_BAD_PAGE);
                        else pool_row = ((l * p.at.n_pages + page) * p.at.n_kv_heads + kvh) * 32;
                    }
                }
                const int at_j = j, at_kb = kb;
                if (!att && ++j == groups) { j = 0; kb += step; }
                if ((q & (FS_PRODUCERS - 1)) != which) { ++q; continue; }
                const int s = q & (FS_SLOTS - 1);
                const uint32_t dst = ring + (uint32_t)(s * p.slot_bytes);
                const uint32_t fb = smem_u32(&sh->full[s]);
                if (!__all_sync(0xffffffffu, fs_wait(smem_u32(&sh->empty[s]), ((uint32_t)(q / FS_SLOTS) & 1u) ^ 1u, &sh->abort, p.at.status, STATUS_TIMEOUT_EPI))) { ok = false; break; }
                if (att) {
                    const int y = __shfl_sync(0xffffffffu, pool_row, i & 31);
                    if (elect_one()) {
                        sh->row[s] = y;
                        mbar_expect_tx(fb, UNIT);
#pragma unroll
                        for (int hf = 0; hf < HALVES; ++hf) tma_load_2d_nohint(dst + hf * 4096, tmKV, 64 * hf, max(y, 0), fb);
                    }
                } else if (elect_one()) {
                    mbar_expect_tx(fb, w_bytes);
                    tma_load_3d(dst, map, 0, sh->rows[phase][at_j].x, at_kb, fb, pol_w);
                }
                __syncwarp();
                ++q;
            }
        }
    if (!ok) {
        // copies in flight still land in this CTA's shared memory: bounded time to complete before it may exit
#pragma unroll 1
        for (int t = max(0, q - FS_SLOTS); t < q; ++t) {
            if ((t & (FS_PRODUCERS - 1)) != which) continue;
            const unsigned long long t0 = global_ns();
            while (!mbar_try(smem_u32(&sh->full[t & (FS_SLOTS - 1)]), (uint32_t)(t / FS_SLOTS) & 1u) && global_ns() - t0 < g_wait_limit_ns) {}
        }
    }
}

// ---- consumers ---------------------------------------------------------------------------------------------------
// waits for stage q (one of this warp's)
__device__ __forceinline__ void fs_take(const FsParams& p, FsShared* sh, int q) {
    fs_wait(smem_u32(&sh->full[q & (FS_SLOTS - 1)]), (uint32_t)(q / FS_SLOTS) & 1u, &sh->abort, p.at.status, STATUS_TIMEOUT_TMA);
    __syncwarp();
}
__device__ __forceinline__ void fs_release(FsShared* sh, int q) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(smem_u32(&sh->empty[q & (FS_SLOTS - 1)]));
}

// barrier of all CTAs, in two halves; every consumer thread calls both
__device__ __forceinline__ void fs_grid_poll(const unsigned int* bar, unsigned int target, volatile int* abort_flag, int* status) {
    unsigned long long t0 = 0;
#pragma unroll 1
    for (uint32_t spin = 1;; ++spin) {
        unsigned int v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        if (v >= target || *abort_flag) return;
        if ((spin & 63u) == 0) {
            const unsigned long long t = global_ns();
            if (t0 == 0) t0 = t;
            if (t - t0 > g_wait_limit_ns) {
                record_status(status, STATUS_TIMEOUT_EPI);
                *abort_flag = 1;
                return;
            }
        }
    }
}
struct FsGrid {
    unsigned int* bar;
    volatile int* abort_flag;
    int* status;
    unsigned int target = 0;
    __device__ __forceinline__ void arrive() {
        fs_bar_sync();
        target += gridDim.x;
        if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    }
    __device__ __forceinline__ void wait() {
        if (threadIdx.x == 0) fs_grid_poll(bar, target, abort_flag, status);
        fs_bar_sync();
    }
};

// The products of one matrix.  prefetch() asks for the first activations, run() multiplies.  Games beyond the last are read
// as the last one; their sums are not used.
struct FsGemm {
    static constexpr int P = 3;                    // k blocks of activations in flight
    const FsMat& M;
    const int2* rows;                              // [groups]
    int vw, q;                                     // this warp counted from the one with the phase's first stage; its first stage
    int a, kp, kparts, j, m;
    int total;                                     // k blocks of this warp (a multiple of m)
    const uint4* x_at;                             // next block's activations of game g
    int ask_left, x_jump;                          // blocks left in the stage that is asked for; from its end to the next one's start
    uint4 x[P][2];                                 // [..][first / second half of the 64 k]

    __device__ __forceinline__ FsGemm(const FsMat& M_, const int2* rows_, const __half* X, int n, int q0) : M(M_), rows(rows_) {
        const int sh = M.groups >> 1, lane = threadIdx.x & 31;        // (1, 2, 4: shifts 0, 1, 2)
        vw = ((threadIdx.x >> 5) - q0) & (FS_WARPS - 1); q = q0 + vw;
        j = vw & (M.groups - 1); kp = vw >> sh; kparts = FS_WARPS >> sh;
        a = rows[j].x;
        m = M.m;
        total = ((M.stages - kp + kparts - 1) >> (3 - sh)) * m;
        x_at = reinterpret_cast<const uint4*>(X + (size_t)min(lane >> 2, n - 1) * M.ldx + kp * m * TC_BK + 8 * (lane & 3));
        x_jump = (kparts - 1) * m * (TC_BK / 8);
        ask_left = m;
    }
    __device__ __forceinline__ void ask(int u) {
        x[u][0] = __ldcg(x_at);
        x[u][1] = __ldcg(x_at + 4);
        x_at += TC_BK / 8;
        if (--ask_left == 0) { x_at += x_jump; ask_left = m; }
    }
    __device__ __forceinline__ void prefetch() {
#pragma unroll
        for (int u = 0; u < P; ++u)
            if (u < total) ask(u);
    }
    // MT: 16-row tiles that a group has at most
    template <int MT>
    __device__ __forceinline__ void run_tiles(const FsParams& p, FsShared* sh, uint32_t ring, float (&acc)[FS_MT][4]) {
        constexpr int H = MT <= 3 ? 4 : 2;         // k steps whose weights are loaded ahead of their products (the warp issues in
                                                   // order: a product right behind its load would wait for it)
        const int lane = threadIdx.x & 31;
        // this lane's row and 16-byte chunk of the ldmatrix (chunk ch of row r sits at ch ^ (r & 7)); a k step further on:
        // chunk + 2, the same row
        const int r = lane & 15;
        const uint32_t o0 = ring + (uint32_t)(r * 128 + (((lane >> 4) ^ ((a + r) & 7)) << 4));
        const uint32_t per = (uint32_t)M.h * 128u;
        int left = 0;
        uint32_t at = 0;
        float odd[MT][4];                          // sums of the odd k steps: half as long a chain of dependent products
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) { odd[mt][0] = 0.f; odd[mt][1] = 0.f; odd[mt][2] = 0.f; odd[mt][3] = 0.f; }
#pragma unroll 1
        for (int done = 0; done < total; ++done) {
            if (left == 0) {
                fs_take(p, sh, q);
                at = o0 + (uint32_t)((q & (FS_SLOTS - 1)) * p.slot_bytes);
                left = m;
            }
#pragma unroll
            for (int k0 = 0; k0 < 4; k0 += H) {
                uint32_t w[H][MT][4];
#pragma unroll
                for (int ks = 0; ks < H; ++ks)
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)          // (the k step's bits are the chunk's bits of `at`)
                        ldmatrix_x4((at ^ (uint32_t)((k0 + ks) << 5)) + mt * 2048, w[ks][mt][0], w[ks][mt][1], w[ks][mt][2], w[ks][mt][3]);
#pragma unroll
                for (int ks = 0; ks < H; ks += 2) {
                    const uint4 v = x[0][(k0 + ks) >> 1];
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        mma_16816<true>(acc[mt], w[ks][mt][0], w[ks][mt][1], w[ks][mt][2], w[ks][mt][3], v.x, v.y);
                        mma_16816<true>(odd[mt], w[ks + 1][mt][0], w[ks + 1][mt][1], w[ks + 1][mt][2], w[ks + 1][mt][3], v.z, v.w);
                    }
                }
            }
            at += per;
            if (--left == 0) { fs_release(sh, q); q += FS_WARPS; }
            // (one copy of the block's code, activations moved down a register set per block)
#pragma unroll
            for (int u = 0; u + 1 < P; ++u) { x[u][0] = x[u + 1][0]; x[u][1] = x[u + 1][1]; }
            if (done + P < total) ask(P - 1);
        }
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[mt][e] += odd[mt][e];
    }
    __device__ __forceinline__ void run(const FsParams& p, FsShared* sh, uint32_t ring, float (&acc)[FS_MT][4]) {
#pragma unroll
        for (int mt = 0; mt < FS_MT; ++mt) { acc[mt][0] = 0.f; acc[mt][1] = 0.f; acc[mt][2] = 0.f; acc[mt][3] = 0.f; }
        if (M.h <= 32) run_tiles<2>(p, sh, ring, acc);
        else if (M.h <= 48) run_tiles<3>(p, sh, ring, acc);
        else if (M.h <= 64) run_tiles<4>(p, sh, ring, acc);
        else run_tiles<5>(p, sh, ring, acc);
    }
    // Leaves the warps' sums in `red` (row pitch 4 modulo 16: the 32 lanes hit 32 banks).
    __device__ __forceinline__ void publish(float* red, const float (&acc)[FS_MT][4]) const {
        const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
        const int hp = M.pitch, tiles = (M.h + 15) >> 4;
        float* dst = red + vw * (8 * hp) + 2 * c * hp + g;
#pragma unroll
        for (int mt = 0; mt < FS_MT; ++mt)
            if (mt < tiles) {
#pragma unroll
                for (int e = 0; e < 4; ++e) dst[(e & 1) * hp + 16 * mt + 8 * (e >> 1)] = acc[mt][e];
            }
    }
    // row lr of group jj for game b, summed over the warps
    __device__ __forceinline__ float sum(const float* red, int b, int jj, int lr) const {
        const int hp = M.pitch, step = M.groups * 8 * hp;
        const float* src = red + (jj * 8 + b) * hp + lr;
        float v[FS_WARPS], s = 0.f;
#pragma unroll
        for (int k = 0; k < FS_WARPS; ++k) v[k] = k < kparts ? src[k * step] : 0.f;
#pragma unroll
        for (int k = 0; k < FS_WARPS; ++k) s += v[k];
        return s;
    }
    // The sums once more, from the activations as they are stored now and weights from memory: into part 0, the other
    // parts zero.  For the rare phase whose activations had to be stored again after their weights had been used up.
    __device__ __noinline__ static void again(const FsMat& M, const int2* rows, const __half* W, const __half* X, int n, float* red) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, hp = M.pitch;
        const size_t slab = (size_t)((M.rows + TC_BM - 1) / TC_BM) * TC_BM;
#pragma unroll 1
        for (int jj = 0; jj < M.groups; ++jj)
#pragma unroll 1
            for (int e = warp; e < n * rows[jj].y; e += FS_WARPS) {
                const int lr = e / n, b = e - lr * n, row = rows[jj].x + lr;
                float s = 0.f;
#pragma unroll 1
                for (int k = lane; k < M.K; k += 32) {
                    const int ch = ((k >> 3) & 7) ^ (row & 7);
                    const float w = __half2float(W[((size_t)(k >> 6) * slab + row) * TC_BK + 8 * ch + (k & 7)]);
                    s += w * __half2float(__ushort_as_half(__ldcg(reinterpret_cast<const unsigned short*>(X) + (size_t)b * M.ldx + fs_perm(k))));
                }
                s = warp_sum(s);
                if (lane < FS_WARPS / M.groups) red[(lane * M.groups + jj) * 8 * hp + b * hp + lr] = lane == 0 ? s : 0.f;
            }
    }
};

// reciprocal root mean square of a row
__device__ __forceinline__ float fs_size(float ms) { return rsqrtf(fmaxf(ms, 1e-36f)); }
// 2^-8 times the power of two below v
__device__ __forceinline__ float fs_pow2(float v) {
    const int e = max(-100, min(100, (int)((__float_as_uint(v) >> 23) & 255u) - 127));
    return __uint_as_float((uint32_t)(e - FS_EXP_BIAS + 127) << 23);
}
// 1 / v of a power of two
__device__ __forceinline__ float fs_recip_pow2(float v) { return __uint_as_float((254u << 23) - __float_as_uint(v)); }

// Reciprocal norms from the CTAs' sums of squares (every CTA adds them up in the same order), the factor that belongs to the
// activations as they are stored, the power of two for the ones stored next, and whether a row has left the window in which
// fp16 holds the stored values like the normalised ones.  One warp; the games' sums are in flight together.
__device__ __forceinline__ void fs_norms(const FsParams& p, FsShared* sh) {
    const int lane = threadIdx.x & 31, G = gridDim.x;
    float v[FS_MAX_GAMES];
#pragma unroll
    for (int e = 0; e < FS_MAX_GAMES; ++e) v[e] = 0.f;
    const float4* src = reinterpret_cast<const float4*>(p.ss_part);
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int i0 = lane; i0 - lane < G; i0 += 5 * 32) {     // (five CTAs' sums per lane in flight; games beyond the last: zeros)
        float4 a[5], b[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const int i = i0 + 32 * k;
            a[k] = i < G ? __ldcg(src + 2 * i) : none;
            b[k] = i < G && p.n > 4 ? __ldcg(src + 2 * i + 1) : none;
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            v[0] += a[k].x; v[1] += a[k].y; v[2] += a[k].z; v[3] += a[k].w;
            v[4] += b[k].x; v[5] += b[k].y; v[6] += b[k].z; v[7] += b[k].w;
        }
    }
    // eight sums over 32 lanes: halves are exchanged, lane l ends up with game l & 7
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int e = 0; e < o; ++e) {
            const float got = __shfl_xor_sync(0xffffffffu, up ? v[e] : v[e + o], o);
            v[e] = (up ? v[e + o] : v[e]) + got;
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 8);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 16);
    int misfit = 0;
    if (lane < p.n) {
        // (the power of two follows the row's size itself, the norm has eps in it)
        const float ms = v[0] * p.inv_d, inv = rsqrtf(ms + p.eps), size = fs_size(ms), sc = sh->scale[lane];
        misfit = sc > size || sc < size * 9.765625e-4f;
        sh->inv[lane] = inv;
        sh->mult[lane] = inv * fs_recip_pow2(sc);
        sh->scale[lane] = fs_pow2(size);
    }
    misfit = __any_sync(0xffffffffu, misfit);
    if (lane == 0) sh->misfit = misfit;
    __syncwarp();
}

// A residual value as the next product reads it.
__device__ __forceinline__ void fs_put_x(const FsParams& p, const FsShared* sh, int b, int a, int col, float x) {
    p.xn[(size_t)b * sh->mat[FS_QKV].ldx + fs_perm(a + col)] = __ushort_as_half((unsigned short)float_to_f16_bits(x * sh->vec[col] * sh->scale[b]));
}

// two values as packed high and low parts of the 2-byte type (see split2)
template <bool F16>
__device__ __forceinline__ void fs_split_pair(float a, float b, uint32_t& hi, uint32_t& lo) {
    if (F16) {
        const __half2 h = __floats2half2_rn(a, b);
        const float2 f = __half22float2(h);
        const __half2 r = __floats2half2_rn(a - f.x, b - f.y);
        hi = *reinterpret_cast<const uint32_t*>(&h);
        lo = *reinterpret_cast<const uint32_t*>(&r);
    } else {
        const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        hi = *reinterpret_cast<const uint32_t*>(&h);
        const __nv_bfloat162 r = __floats2bfloat162_rn(a - bf16_lo(hi), b - bf16_hi(hi));
        lo = *reinterpret_cast<const uint32_t*>(&r);
    }
}

// The attention of one layer: units [c0, c1) of the step's (game, KV head, page) list are this CTA's.  See attn_decode.cuh
// for the arithmetic; what differs: the pages come from the producer's ring; queries are normalised and rotated here; the new token's key and value, which the last page of a game
// does not hold yet, are computed by the warp that has this page, put into the page's copy in shared memory and appended to
// the cache.
template <int HD, bool F16>
__device__ __forceinline__ void fs_attend(const FsParams& p, FsShared* sh, uint32_t ring, float* red, int q0,
                                          int c0, int c1, int Rc) {
    constexpr int HALVES = HD / 64, KSTEPS = HD / 16, NT = HD / 8, HALF = HD / 2, EL = HD / 64;
    const AttnParams& A = p.at;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
    const int vw = (warp - q0) & (FS_WARPS - 1);           // the order of the warps' units
    const int G = A.group, Hkv = A.n_kv_heads, Hq = A.n_q_heads, QR = p.mat[FS_QKV].rows;
    const int n_units = c1 - c0, u_base = n_units / FS_WARPS, u_rem = n_units % FS_WARPS;
    const int cnt = u_base + (vw < u_rem ? 1 : 0), u0 = c0 + u_base * vw + min(vw, u_rem), u1 = u0 + cnt;
    if (lane < 2) {
        sh->part[vw][lane].item = -1;
        if (warp == 0) sh->open_item[lane] = -1;
    }
    if (n_units <= 0) return;
    __syncwarp();
    float* const part0 = red + 2 * warp * G * HD;          // (and the [1] partial behind it)
    // rows of the output in the order of fs_perm: element 2 c + 8 t of a head sits at 32 (t / 4) + 8 c + 2 (t % 4)
    const int ldx = sh->mat[FS_O].ldx;
    int slot = 0, T = 0, pages = 1, kvh = 0, pg = 0;
    if (cnt > 0) {
        while (slot + 1 < p.n && sh->cum[slot + 1] <= u0) ++slot;
        T = sh->len[slot];
        pages = (T + ATTN_PAGE - 1) / ATTN_PAGE;
        kvh = (u0 - sh->cum[slot]) / pages;
        pg = (u0 - sh->cum[slot]) - kvh * pages;
    }
    int q = q0 + vw;
    uint32_t qa[KSTEPS][4];
    float m = -INFINITY, l = 0.f;
    float o[NT][4];
    int fresh = 1;
    const int lr = lane & 7, lm = lane >> 3;
    const int k_tok = lr + 8 * (lm >> 1), k_chk = lm & 1;
    const int v_tok = lr + 8 * (lm & 1), v_chk = lm >> 1;
    const uint32_t k_row_off = (uint32_t)(k_tok * 128), v_row_off = (uint32_t)((16 + v_tok) * 128);
#pragma unroll 1
    for (int i = 0; i < cnt; ++i) {
        const int last_page = fs_opaque(pg + 1 == pages);
        const float* raw = p.qkv + (size_t)slot * QR;
        // the new token's key and value, elements EL lane .. of either half of the head
        float nk[2][EL], nv[2][EL], ncs[EL], nsn[EL];
        if (fs_opaque(last_page)) {
#pragma unroll
            for (int e = 0; e < EL; ++e) {
                const int x = EL * lane + e;
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    nk[hf][e] = __ldcg(raw + (Hq + kvh) * HD + x + hf * HALF);
                    nv[hf][e] = __ldcg(raw + (Hq + Hkv + kvh) * HD + x + hf * HALF);
                }
                ncs[e] = __ldg(p.cos_tab + (size_t)(T - 1) * HALF + x);
                nsn[e] = __ldg(p.sin_tab + (size_t)(T - 1) * HALF + x);
            }
        }
        if (fs_opaque(fresh)) {
            // query head g of the group: elements 16 ks + 2 c + {0, 1, 8, 9}; rotation partners sit KSTEPS / 2 further on
            float qv[KSTEPS][4];
            const float* qp = raw + (size_t)(kvh * G + g) * HD + 2 * c;
#pragma unroll
            for (int ks = 0; ks < KSTEPS; ++ks) {
                float2 a = make_float2(0.f, 0.f), b = make_float2(0.f, 0.f);
                if (g < G) {
                    a = __ldcg(reinterpret_cast<const float2*>(qp + 16 * ks));
                    b = __ldcg(reinterpret_cast<const float2*>(qp + 16 * ks + 8));
                }
                qv[ks][0] = a.x; qv[ks][1] = a.y; qv[ks][2] = b.x; qv[ks][3] = b.y;
            }
            if (fs_opaque(p.qk_norm)) {
                float ss = 0.f;
#pragma unroll
                for (int ks = 0; ks < KSTEPS; ++ks)
#pragma unroll
                    for (int e = 0; e < 4; ++e) ss += qv[ks][e] * qv[ks][e];
                ss += __shfl_xor_sync(0xffffffffu, ss, 1);
                ss += __shfl_xor_sync(0xffffffffu, ss, 2);
                const float inv = rsqrtf(ss / (float)HD + p.eps);
#pragma unroll
                for (int ks = 0; ks < KSTEPS; ++ks) {
                    const float2 ga = *reinterpret_cast<const float2*>(&sh->qk_gain[0][16 * ks + 2 * c]), gb = *reinterpret_cast<const float2*>(&sh->qk_gain[0][16 * ks + 2 * c + 8]);
                    qv[ks][0] = qv[ks][0] * inv * ga.x; qv[ks][1] = qv[ks][1] * inv * ga.y;
                    qv[ks][2] = qv[ks][2] * inv * gb.x; qv[ks][3] = qv[ks][3] * inv * gb.y;
                }
            }
#pragma unroll
            for (int ks = 0; ks < KSTEPS / 2; ++ks) {
                const size_t at = (size_t)(T - 1) * HALF + 16 * ks + 2 * c;
                const float2 ca = __ldg(reinterpret_cast<const float2*>(p.cos_tab + at)), cb = __ldg(reinterpret_cast<const float2*>(p.cos_tab + at + 8));
                const float2 sa = __ldg(reinterpret_cast<const float2*>(p.sin_tab + at)), sb = __ldg(reinterpret_cast<const float2*>(p.sin_tab + at + 8));
                const float cs[4] = {ca.x, ca.y, cb.x, cb.y}, sn[4] = {sa.x, sa.y, sb.x, sb.y};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float a = qv[ks][e], b = qv[ks + KSTEPS / 2][e];
                    qv[ks][e] = a * cs[e] - b * sn[e];
                    qv[ks + KSTEPS / 2][e] = b * cs[e] + a * sn[e];
                }
            }
#pragma unroll
            for (int ks = 0; ks < KSTEPS; ++ks) {
                fs_split_pair<F16>(qv[ks][0] * A.scale_log2, qv[ks][1] * A.scale_log2, qa[ks][0], qa[ks][1]);
                fs_split_pair<F16>(qv[ks][2] * A.scale_log2, qv[ks][3] * A.scale_log2, qa[ks][2], qa[ks][3]);
            }
            m = -INFINITY; l = 0.f;
#pragma unroll
            for (int t = 0; t < NT; ++t) { o[t][0] = 0.f; o[t][1] = 0.f; o[t][2] = 0.f; o[t][3] = 0.f; }
            fresh = 0;
        }
        fs_take(p, sh, q);
        const uint32_t base = ring + (uint32_t)((q & (FS_SLOTS - 1)) * p.slot_bytes);
        const int valid = T - pg * ATTN_PAGE;              // tokens of this page that exist, the new one included (>= 1)
        if (fs_opaque(last_page)) {
            if (fs_opaque(p.qk_norm)) {
                float ss = 0.f;
#pragma unroll
                for (int e = 0; e < EL; ++e) ss += nk[0][e] * nk[0][e] + nk[1][e] * nk[1][e];
                const float inv = rsqrtf(warp_sum(ss) / (float)HD + p.eps);
#pragma unroll
                for (int e = 0; e < EL; ++e) {
                    nk[0][e] = nk[0][e] * inv * sh->qk_gain[1][EL * lane + e];
                    nk[1][e] = nk[1][e] * inv * sh->qk_gain[1][EL * lane + e + HALF];
                }
            }
            const int y = *(volatile int*)&sh->row[q & (FS_SLOTS - 1)], r = valid - 1;
            uint16_t* dst = p.pool + ((size_t)max(y, 0) + r) * HD;
#pragma unroll
            for (int e = 0; e < EL; ++e) {
                const float lo = nk[0][e] * ncs[e] - nk[1][e] * nsn[e], hi = nk[1][e] * ncs[e] + nk[0][e] * nsn[e];
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int x = EL * lane + e + hf * HALF;
                    const float kf = hf ? hi : lo;
                    const uint32_t kk = F16 ? float_to_f16_bits(kf) : float_to_bf16_bits(kf), vv = F16 ? float_to_f16_bits(nv[hf][e]) : float_to_bf16_bits(nv[hf][e]);
                    const uint32_t at = base + (uint32_t)((x >> 6) * 4096 + r * 128 + ((((x & 63) >> 3) ^ (r & 7)) << 4) + (x & 7) * 2);
                    asm volatile("st.shared.u16 [%0], %1;" ::"r"(at), "h"((unsigned short)kk) : "memory");
                    asm volatile("st.shared.u16 [%0], %1;" ::"r"(at + 2048u), "h"((unsigned short)vv) : "memory");
                    if (y >= 0) { dst[x] = (uint16_t)kk; dst[16 * HD + x] = (uint16_t)vv; }
                }
            }
            // value rows of positions that do not exist yet hold stale pool bytes: zero them so that weight 0 times
            // garbage cannot produce NaN
            for (int idx = lane; idx < (ATTN_PAGE - valid) * 8 * HALVES; idx += 32) {
                const int rw = valid + idx / (8 * HALVES), rem = idx % (8 * HALVES);
                asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(base + (rem >> 3) * 4096 + (16 + rw) * 128 + (rem & 7) * 16), "r"(0u) : "memory");
            }
            __syncwarp();
        }
        // ---- scores: S[16 x 16 tokens] = Q[16 x HD] K^T ----
        float s[2][4];
#pragma unroll
        for (int t = 0; t < 2; ++t) { s[t][0] = 0.f; s[t][1] = 0.f; s[t][2] = 0.f; s[t][3] = 0.f; }
        // (four loads, then the products of the four: the warp issues in order, a product right behind its load would wait)
#pragma unroll
        for (int k4 = 0; k4 < KSTEPS; k4 += 4) {
            uint32_t b[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                ldmatrix_x4(base + (k4 >> 2) * 4096 + k_row_off + (uint32_t)((((2 * u + k_chk) ^ (k_tok & 7)) << 4)), b[u][0], b[u][1], b[u][2], b[u][3]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                mma_16816<F16>(s[0], qa[k4 + u][0], qa[k4 + u][1], qa[k4 + u][2], qa[k4 + u][3], b[u][0], b[u][1]);
                mma_16816<F16>(s[1], qa[k4 + u][0], qa[k4 + u][1], qa[k4 + u][2], qa[k4 + u][3], b[u][2], b[u][3]);
            }
        }
        float sc[4];
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float v = s[t][e] + s[t][2 + e];
                sc[2 * t + e] = (8 * t + 2 * c + e) < valid ? v : -INFINITY;
            }
        float mx = fmaxf(fmaxf(sc[0], sc[1]), fmaxf(sc[2], sc[3]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m, mx);
        float pr[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) pr[k] = fast_exp2(sc[k] - m_new);
        const float alpha = fast_exp2(m - m_new);
        l = l * alpha + (pr[0] + pr[1]) + (pr[2] + pr[3]);
        if (__any_sync(0xffffffffu, m_new > m)) {
#pragma unroll
            for (int t = 0; t < NT; ++t) { o[t][0] *= alpha; o[t][1] *= alpha; o[t][2] *= alpha; o[t][3] *= alpha; }
        }
        m = m_new;
        uint32_t a0, a1, a2, a3;
        fs_split_pair<F16>(pr[0], pr[1], a0, a1);
        fs_split_pair<F16>(pr[2], pr[3], a2, a3);
        // ---- O[16 x HD] += P[16 x 16 tokens] V ----
#pragma unroll
        for (int n4 = 0; n4 < NT / 2; n4 += 4) {
            uint32_t b[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                ldmatrix_x4_trans(base + (n4 >> 2) * 4096 + v_row_off + (uint32_t)((((2 * u + v_chk) ^ (v_tok & 7)) << 4)), b[u][0], b[u][1], b[u][2], b[u][3]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                mma_16816<F16>(o[2 * (n4 + u)], a0, a1, a2, a3, b[u][0], b[u][1]);
                mma_16816<F16>(o[2 * (n4 + u) + 1], a0, a1, a2, a3, b[u][2], b[u][3]);
            }
        }
        if (fs_opaque(last_page)) fence_proxy_async_smem();           // (written above; the ring's next copy is the asynchronous proxy's)
        fs_release(sh, q);
        q += FS_WARPS;
        ++pg;
        const int item_end = fs_opaque(pg == pages);
        if (fs_opaque(item_end | (i + 1 == cnt))) {
            l += __shfl_xor_sync(0xffffffffu, l, 1);
            l += __shfl_xor_sync(0xffffffffu, l, 2);
            const int ua = sh->cum[slot] + kvh * pages;
            if (ua >= u0 && ua + pages <= u1) {
                if (g < G) {
                    const float inv = 1.f / l;
                    uint32_t* dst = reinterpret_cast<uint32_t*>(p.heads + (size_t)slot * ldx + (kvh * G + g) * HD + 8 * c);
#pragma unroll
                    for (int t = 0; t < NT; ++t) dst[16 * (t >> 2) + (t & 3)] = pack_f16((o[t][0] + o[t][2]) * inv, (o[t][1] + o[t][3]) * inv);
                }
            } else {
                const int sd = ua >= u0 ? 1 : 0;
                FsShared::Part& P = sh->part[vw][sd];
                float* op = part0 + sd * G * HD;
                if (lane == 0) {
                    const int first = ua / Rc;
                    P.item = slot * Hkv + kvh;
                    P.side = ua < c0 ? 0 : ua + pages > c1 ? 1 : 2;
                    P.first_cta = first; P.n_cta = (ua + pages - 1) / Rc - first + 1;
                    P.o = op;
                }
                if (g < G) {
                    op += g * HD + 2 * c;
#pragma unroll
                    for (int t = 0; t < NT; ++t)
                        *reinterpret_cast<float2*>(op + 8 * t) = make_float2(o[t][0] + o[t][2], o[t][1] + o[t][3]);
                    if (c == 0) { P.m[g] = m; P.l[g] = l; }
                }
            }
            fresh = 1;
        }
        if (fs_opaque(item_end)) {
            pg = 0;
            if (++kvh == Hkv) {
                kvh = 0;
                ++slot;
                if (slot < p.n) { T = sh->len[slot]; pages = (T + ATTN_PAGE - 1) / ATTN_PAGE; }
            }
        }
    }
    // Items shared by warps are added up, a query head per warp at a time: in the first pass the warps' partials of this
    // CTA, which are an item's result or, where other CTAs have a part in it, this CTA's partial in global memory; in the
    // second pass, by the CTA that was the last to publish, the CTAs' partials in CTA order.
    fs_bar_sync();
    // groups of the first pass: bit 0, the item that began before the CTA's units; bit 1 + w, the one that begins in warp w's
    const unsigned groups0 = __ballot_sync(0xffffffffu, lane <= FS_WARPS && sh->part[max(lane - 1, 0)][lane > 0 ? 1 : 0].item >= 0);
#pragma unroll 1
    for (int pass_ = 0; pass_ < 2; ++pass_) {
        const int pass = fs_opaque(pass_);
        unsigned groups = pass ? (sh->last[0] ? 1u : 0u) | (sh->last[1] ? 2u : 0u) : groups0;
#pragma unroll 1
        for (int gi = 0; groups; ++gi, groups &= groups - 1) {
            const int grp = __ffs(groups) - 1;
#pragma unroll 1
            for (int gq = (warp - gi * G) & (FS_WARPS - 1); gq < G; gq += FS_WARPS) {
            int item, first, cnt_p, side = 2;      // pass 0: partials in [first][fs], then [first + 1 ..][0]; pass 1: CTAs first ..
            const int fs = pass == 0 && grp > 0 ? 1 : 0;
            if (pass == 0) {
                first = max(grp - 1, 0);
                const FsShared::Part& P = sh->part[first][fs];
                item = P.item; side = P.side;
                cnt_p = 1;
#pragma unroll 1
                while (first + cnt_p < FS_WARPS && sh->part[first + cnt_p][0].item == item) ++cnt_p;
            } else {
                item = sh->open_item[grp]; first = sh->open_first[grp]; cnt_p = sh->open_n[grp];
            }
            constexpr int E4 = HD / 32;            // elements E4 lane .. of the head
            float M = -INFINITY, ls = 0.f, acc[E4];
#pragma unroll
            for (int e = 0; e < E4; ++e) acc[e] = 0.f;
#pragma unroll 1
            for (int i0 = 0; i0 < cnt_p; i0 += 8) {
                // eight partials at a time, all their loads in flight together (from global memory each is a trip to the L2):
                // lane i looks at the maximum, the sum and the place of partial i0 + i
                const int k = i0 + lane;
                float mi = -INFINITY, li = 0.f;
                const float* oi = nullptr;
                if (lane < 8 && k < cnt_p) {
                    if (pass == 0) {
                        const FsShared::Part& P = sh->part[first + k][k ? 0 : fs];
                        mi = P.m[gq]; li = P.l[gq]; oi = P.o + gq * HD;
                    } else {
                        const size_t at = (size_t)(2 * (first + k) + (k ? 0 : 1)) * G + gq;       // (the first CTA keeps it as "goes on")
                        oi = A.o_part + at * HD;
                        mi = __ldcg(A.m_part + at); li = __ldcg(A.l_part + at);
                    }
                }
                float v[8][E4];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float* src = reinterpret_cast<const float*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(oi), u)) + E4 * lane;
#pragma unroll
                    for (int e = 0; e < E4; e += 2) {
                        v[u][e] = 0.f; v[u][e + 1] = 0.f;              // (shared memory or, written by other SMs, global memory)
                        if (i0 + u < cnt_p) asm volatile("ld.volatile.v2.f32 {%0,%1}, [%2];" : "=f"(v[u][e]), "=f"(v[u][e + 1]) : "l"(src + e) : "memory");
                    }
                }
                const float Mn = fmaxf(warp_max(mi), M), al = fast_exp2(M - Mn), w = fast_exp2(mi - Mn);
                ls = ls * al + warp_sum(w * li);
                M = Mn;
#pragma unroll
                for (int e = 0; e < E4; ++e) acc[e] *= al;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float wq = __shfl_sync(0xffffffffu, w, u);
#pragma unroll
                    for (int e = 0; e < E4; ++e) acc[e] += wq * v[u][e];
                }
            }
            if (side == 2) {
                const float inv = 1.f / ls;
                const int sl = item / Hkv, el = ((item - sl * Hkv) * G + gq) * HD + E4 * lane;
#pragma unroll
                for (int e = 0; e < E4; e += 2)
                    *reinterpret_cast<uint32_t*>(p.heads + (size_t)sl * ldx + fs_perm(el + e)) = pack_f16(acc[e] * inv, acc[e + 1] * inv);
            } else {
                const size_t at = (size_t)(2 * blockIdx.x + side) * G + gq;
#pragma unroll
                for (int e = 0; e < E4; ++e) A.o_part[at * HD + E4 * lane + e] = acc[e];
                if (lane == 0) {
                    const FsShared::Part& P = sh->part[first][fs];
                    A.m_part[at] = M; A.l_part[at] = ls;
                    sh->open_item[side] = item; sh->open_first[side] = P.first_cta; sh->open_n[side] = P.n_cta;     // (every head the same)
                }
            }
            }
        }
        if (pass == 1) break;
        fs_bar_sync();
        if (warp == 0) {
            int last = 0;
            const int item = lane < 2 ? sh->open_item[lane] : -1;
            if (item >= 0) {
                __threadfence();
                last = atomicAdd(A.item_cnt + item, 1) == sh->open_n[lane] - 1;
                if (last) A.item_cnt[item] = 0;
                __threadfence();
            }
            if (lane < 2) sh->last[lane] = last;
        }
        fs_bar_sync();
        if (!sh->last[0] && !sh->last[1]) break;
    }
}

template <int HD, bool F16>
__global__ void __launch_bounds__(FS_THREADS, 1) few_step_kernel(const __grid_constant__ CUtensorMap tmKV, const __grid_constant__ FsParams p) {
    extern __shared__ uint8_t fs_smem_raw[];
    __shared__ FsShared sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n = p.n, G = gridDim.x, cta = blockIdx.x;
    uint8_t* const ring_p = fs_smem_raw + ((1024u - (smem_u32(fs_smem_raw) & 1023u)) & 1023u);
    const uint32_t ring = smem_u32(ring_p);
    float* const red = reinterpret_cast<float*>(ring_p + FS_SLOTS * p.slot_bytes);  // (row tiles read past a stage's end, at most into here)
    float* const xs = red + p.red_bytes / 4;               // [n][cols] residual stream of this CTA's columns
    if (tid == 0) {
        for (int s = 0; s < FS_SLOTS; ++s) { mbar_init(smem_u32(&sh.full[s]), 1); mbar_init(smem_u32(&sh.empty[s]), 1); }
        sh.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 4 * (int)(sizeof(FsMat) / 4)) reinterpret_cast<int*>(sh.mat)[tid] = reinterpret_cast<const int*>(p.mat)[tid];
    if (tid < (int)(sizeof(FsVectors) / 8)) reinterpret_cast<unsigned long long*>(&sh.lay[0])[tid] = reinterpret_cast<const unsigned long long*>(&p.layers[0].v)[tid];
    if (tid < 16 && (tid & 3) < p.mat[tid >> 2].groups) fs_rows(p.mat[tid >> 2], cta, G, tid & 3, sh.rows[tid >> 2][tid & 3].x, sh.rows[tid >> 2][tid & 3].y);
    if (tid <= n) {
        sh.cum[tid] = p.at.cum[tid];
        if (tid < n) { sh.len[tid] = p.meta.pos[tid] + 1; sh.game[tid] = p.meta.game[tid]; sh.newp[tid] = p.meta.new_page[tid]; }
    }
    __syncthreads();
    // The attention's units of this CTA: whole (game, KV head) items where they are short (FS_WHOLE), else equal shares of all
    // units.  (One game at 900 tokens, 57 pages: whole items 2206 us per step, equal shares of eight pages 2088.)
    const int U = sh.cum[n], Hkv = p.at.n_kv_heads, items = n * Hkv, per_cta = (items + G - 1) / G;
    int longest = 0, c0, c1, Rc = max(ATTN_CTA_MIN, (U + G - 1) / G);
    for (int b = 0; b < n; ++b) longest = max(longest, (sh.len[b] + ATTN_PAGE - 1) / ATTN_PAGE);
    if (per_cta * longest <= FS_WHOLE) {
        auto begin = [&](int item) {
            const int b = min(item / Hkv, n);
            return b == n ? U : sh.cum[b] + (item - b * Hkv) * ((sh.len[b] + ATTN_PAGE - 1) / ATTN_PAGE);
        };
        c0 = begin(min(items, cta * per_cta));
        c1 = begin(min(items, (cta + 1) * per_cta));
    } else {
        c0 = min(U, cta * Rc);
        c1 = min(U, c0 + Rc);
    }
    if (warp >= FS_WARPS) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(FS_REG_PRODUCER));
        if (warp < FS_WARPS + FS_PRODUCERS) {
            if (lane == 0) tmap_prefetch(&tmKV);
            fs_produce<HD>(p, &tmKV, &sh, ring, c0, c1, warp - FS_WARPS);
        } else if (warp == FS_WARPS + FS_PRODUCERS) {
            // the norms of the phases that need them, while the consumers multiply
            unsigned int target = (unsigned)G;             // the barrier behind the embedding rows
#pragma unroll 1
            for (int l = 0; l < p.n_layers; ++l)
#pragma unroll 1
                for (int k = 0; k < 2; ++k) {              // in front of QKV, in front of gate/up
                    if (l > 0 || k > 0) {
                        target += (unsigned)G * (k ? 3u : 2u);
                        fs_grid_poll(p.bar, target, &sh.abort, p.at.status);
                        __syncwarp();
                        fs_norms(p, &sh);
                        // (a misfit takes the CTAs through one more barrier)
                        if (sh.misfit) target += (unsigned)G;
                    }
                    fs_norms_sync();
                }
            target += 2u * (unsigned)G;
            fs_grid_poll(p.bar, target, &sh.abort, p.at.status);
            __syncwarp();
            fs_norms(p, &sh);
            fs_norms_sync();
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(FS_REG_CONSUMER));
        FsGrid grid{p.bar, &sh.abort, p.at.status};
        const int a_d = sh.rows[FS_O][0].x, cols = sh.rows[FS_O][0].y;
        // embedding rows: this CTA's columns, the sum of squares of the whole row
        if (tid < cols) sh.vec[tid] = __bfloat162float(p.first_norm[a_d + tid]);
        if (tid == 0) sh.misfit = 0;
        fs_bar_sync();
        const int32_t* tokens = p.args->tokens;
        if (warp < n) {
            const int b = warp, ti = p.meta.tok_index[b];
            int tok = tokens[ti >= 0 ? ti : b];
            if (tok < 0 || tok >= p.vocab) {
                if (cta == 0 && lane == 0) record_status(p.at.status, STATUS_BAD_TOKEN);
                tok = 0;
            }
            const __nv_bfloat16* row = p.embed + (size_t)tok * p.d_model;
            float ss = 0.f;
            for (int i = lane; i < p.d_model / 8; i += 32) {
                const uint4 v = ldg_v4(row + 8 * i);
                const uint32_t in[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) ss += bf16_lo(in[e]) * bf16_lo(in[e]) + bf16_hi(in[e]) * bf16_hi(in[e]);
            }
            const float ms = warp_sum(ss) * p.inv_d, inv = rsqrtf(ms + p.eps), sc = fs_pow2(fs_size(ms));
            if (lane == 0) { sh.scale[b] = sc; sh.mult[b] = inv * fs_recip_pow2(sc); }
            __syncwarp();
            for (int col = lane; col < cols; col += 32) {
                const float x = __bfloat162float(row[a_d + col]);
                xs[b * cols + col] = x;
                fs_put_x(p, &sh, b, a_d, col, x);
            }
        }
        if (cta == 0 && tid < n && sh.newp[tid] >= 0)
            p.block_table[(size_t)sh.game[tid] * p.at.max_pages + (sh.len[tid] - 1) / ATTN_PAGE] = sh.newp[tid];
        grid.arrive();

        int q = 0;                                         // first stage of the phase
#pragma unroll 1
        for (int l = 0; l < p.n_layers; ++l) {
            const FsVectors& W = sh.lay[l & 1];
#pragma unroll 1
            for (int phase = 0; phase < 4; ++phase) {
                const int ph = fs_opaque(phase);
                if (ph == FS_O) {
                    grid.wait();
                    fs_attend<HD, F16>(p, &sh, ring, red, q, c0, c1, Rc);
                    q += c1 - c0;
                    grid.arrive();
                }
                float acc[FS_MT][4];
                FsGemm gm(sh.mat[ph], sh.rows[ph], ph == FS_O ? p.heads : ph == FS_DOWN ? p.act : p.xn, n, q);
                const int groups = gm.M.groups, a0 = gm.rows[0].x, rows = gm.rows[groups - 1].x + gm.rows[groups - 1].y - a0;
                // bias of the rows, or gains of the norm behind the residual columns, gains of the query and key norms, the
                // next layer's pointers: on their way while the CTAs meet
                const bool last = l + 1 == p.n_layers, normed = ph == FS_QKV || ph == FS_GU;
                const __nv_bfloat16* vec = W.vec[ph];
                float qkg = 0.f;
                if (ph == FS_QKV && p.qk_norm && tid < 2 * HD) qkg = __bfloat162float(W.qk_norm[tid / HD][tid & (HD - 1)]);
                unsigned long long ahead = 0;
                if (ph == FS_QKV && !last && tid < (int)(sizeof(FsVectors) / 8)) ahead = __ldg(reinterpret_cast<const unsigned long long*>(&p.layers[l + 1].v) + tid);
                const float v0 = vec && tid < rows ? __bfloat162float(vec[a0 + tid]) : 0.f;
                const float v1 = vec && tid + 256 < rows ? __bfloat162float(vec[a0 + tid + 256]) : 0.f;
                const float unscale = W.unscale[ph];
                grid.wait();
                gm.prefetch();
                gm.run(p, &sh, ring, acc);
                q += gm.M.stages * groups;
                gm.publish(red, acc);
                if (normed) {
                    fs_norms_sync();
                    if (sh.misfit) {
                        // the rows just multiplied are stored again with a power of two that fits them, and multiplied again
                        // (rare: a row has changed its size 256-fold, or shrunk fourfold, in one half of a layer)
                        if (warp < n) {
                            if (lane == 0) sh.mult[warp] = sh.inv[warp] * fs_recip_pow2(sh.scale[warp]);
#pragma unroll 1
                            for (int col = lane; col < cols; col += 32) fs_put_x(p, &sh, warp, a_d, col, xs[warp * cols + col]);
                        }
                        grid.arrive();
                        grid.wait();
                        FsGemm::again(gm.M, gm.rows, W.w[ph >> 1], p.xn, n, red);
                        if (tid == 0) sh.misfit = 0;
                        fs_bar_sync();
                    }
                }
                if (vec || ph == FS_QKV) {
                    if (tid < rows) sh.vec[tid] = v0;
                    if (tid + 256 < rows) sh.vec[tid + 256] = v1;
                }
                if (ph == FS_QKV) {
                    if (tid < 2 * HD) sh.qk_gain[tid / HD][tid & (HD - 1)] = qkg;
                    if (tid < (int)(sizeof(FsVectors) / 8)) reinterpret_cast<unsigned long long*>(&sh.lay[(l + 1) & 1])[tid] = ahead;
                }
                fs_bar_sync();
                if (ph == FS_QKV) {
                    // a thread per (game, row), groups one after the other
#pragma unroll 1
                    for (int jj = 0; jj < groups; ++jj) {
                        const int a = gm.rows[jj].x, h = gm.rows[jj].y;
#pragma unroll 1
                        for (int e = tid; e < n * h; e += 32 * FS_WARPS) {
                            const int b = e / h, lr = e - b * h;
                            p.qkv[(size_t)b * gm.M.rows + a + lr] = gm.sum(red, b, jj, lr) * (unscale * sh.mult[b]) + sh.vec[a - a0 + lr];
                        }
                    }
                } else if (ph == FS_GU) {
                    // a thread per (game, pair of a gate and an up row); the groups hold equally many up to one pair
                    const int half = gm.M.h >> 1, all = n * groups * half;
#pragma unroll 1
                    for (int e = tid; e < all; e += 32 * FS_WARPS) {
                        const int bj = e / half, pr = e - bj * half, jj = bj & (groups - 1), b = bj >> (groups >> 1);
                        const int a = gm.rows[jj].x;
                        if (2 * pr < gm.rows[jj].y) {
                            const float f = unscale * sh.mult[b];
                            const float gate = gm.sum(red, b, jj, 2 * pr) * f, up = gm.sum(red, b, jj, 2 * pr + 1) * f;
                            p.act[(size_t)b * sh.mat[FS_DOWN].ldx + fs_perm((a >> 1) + pr)] = __ushort_as_half((unsigned short)float_to_f16_bits(gate / (1.f + expf(-gate)) * up));
                        }
                    }
                } else if (warp < n) {
                    const int b = warp;
                    float ss = 0.f;
#pragma unroll 1
                    for (int col = lane; col < cols; col += 32) {
                        const float v = xs[b * cols + col] + gm.sum(red, b, 0, col) * unscale;
                        xs[b * cols + col] = v;
                        ss += v * v;
                        if (ph == FS_O || !last) fs_put_x(p, &sh, b, a_d, col, v);
                    }
                    ss = warp_sum(ss);
                    if (lane == 0) p.ss_part[(size_t)cta * FS_MAX_GAMES + b] = ss;
                }
                grid.arrive();
            }
        }
        // final norm
        fs_norms_sync();
        if (warp < n)
            for (int col = lane; col < cols; col += 32)
                p.h[(size_t)warp * p.d_model + a_d + col] = __ushort_as_half((unsigned short)float_to_f16_bits(xs[warp * cols + col] * sh.inv[warp] * sh.vec[col]));
    }
    __syncthreads();
    grid_launch_dependents();
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(p.bar + 1, 1u) == (unsigned)G - 1u) { p.bar[0] = 0u; p.bar[1] = 0u; }
    }
}

}  // namespace spiral
