// Context append ("prefill"): the tokens an environment adds to a game's context between two turns
// of Algorithm 1 enter the model many at a time.  With hundreds to thousands of token rows per
// weight matrix the linear layers are dense contractions -- compute-bound on the tensor cores, not
// weight-streaming like the decode step -- and attention reads each cached key once per block of
// queries instead of once per query.  Kernels:
//
//   pg_gemm_kernel<EPI>   (gemm_pair.cuh) the linear layers on pairs of SMs, with the residual addition or the SwiGLU
//                         gating in the epilogue; partial sums where few token rows make stream-K the better split.
//   attn_append_tc_kernel causal grouped-query attention of a block of new positions of one game against
//                         everything cached for it (earlier turns and the new tokens up to each query's own
//                         position) on tcgen05: scores and the output accumulator in tensor memory, one
//                         softmax thread per query row, keys/values streamed page by page by TMA.
//   attn_append_kernel    the same attention on mma.sync.m16n8k16, flash-style with the fp32 online softmax in
//                         registers: bf16 pages (queries and weights in two bf16 parts), and an option for fp16 pages.
//   pf_rmsnorm_kernel, pf_qkv_post_kernel   the element-wise steps for thousands of token rows.
//
// Every wait is bounded as in the decode kernels.
#pragma once
#include "attn_decode.cuh"
#include "gemm_pair.cuh"
#include "gemm_tc.cuh"

namespace spiral {

// ------------------------------------------------------------------------------------------------
// element-wise kernels over thousands of token rows (the decode step's versions are built for a
// few hundred rows at most: one CTA per row, half a warp per head)
// ------------------------------------------------------------------------------------------------

// h[t][:] = x[t][:] * rsqrt(mean(x[t]^2) + eps) * gain as fp16, one CTA of four warps per token row: the row stays in
// registers between the reduction and the scaling, and a row's loads are spread thin enough (NV4 float4 per thread)
// for ten CTAs per SM.  Bound by memory: 6 bytes read and written per element.  (With a warp per row, 20 float4 per
// lane at d_model 2560 left room for 16 warps per SM, which went through their rows in lockstep: 54 us for 9984 rows.)
// PIECES: the row is x + the pieces a projection has left (written back to x), added piece by piece over the whole row.
constexpr int PF_RMS_THREADS = 128;
template <int NV4, bool PIECES>         // float4 per thread
__global__ void __launch_bounds__(PF_RMS_THREADS) pf_rmsnorm_kernel(float* __restrict__ x, Pieces pieces,
                                                                    const __nv_bfloat16* __restrict__ gain, float eps,
                                                                    int d_model, __half* __restrict__ h) {
    grid_launch_dependents();
    __shared__ float red[PF_RMS_THREADS / 32];
    __shared__ unsigned char cnt_tab[PIECES ? PIECE_TABLE : 1];
    const int nc = d_model >> 2;
    uint2 g[NV4];                       // (weights: nobody writes them)
#pragma unroll
    for (int k = 0; k < NV4; ++k) {
        const int c = threadIdx.x + PF_RMS_THREADS * k;
        g[k] = c < nc ? __ldg(reinterpret_cast<const uint2*>(gain) + c) : make_uint2(0u, 0u);
    }
    PieceCounts pcnt{cnt_tab};
    if (PIECES) pcnt = piece_counts_init(pieces, cnt_tab);             // (parameters only: before the wait)
    grid_dependency_wait();
    const size_t t = blockIdx.x;
    float4* xr = reinterpret_cast<float4*>(x + t * d_model);
    float4 v[NV4];
#pragma unroll
    for (int k = 0; k < NV4; ++k) {
        const int c = threadIdx.x + PF_RMS_THREADS * k;
        v[k] = c < nc ? __ldcs(xr + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (PIECES) {
        int most = 0, cnt[NV4];
#pragma unroll
        for (int k = 0; k < NV4; ++k) {
            const int c = threadIdx.x + PF_RMS_THREADS * k;
            cnt[k] = c < nc ? pcnt.of(pieces, (int)t, 4 * c) : 0;
            most = max(most, cnt[k]);
        }
        for (int i = 0; i < most; ++i) {
            const float* pr = pieces.base + (size_t)i * pieces.stride + t * pieces.ld;
            float4 w[NV4];
#pragma unroll
            for (int k = 0; k < NV4; ++k)
                w[k] = i < cnt[k] ? __ldcg(reinterpret_cast<const float4*>(pr) + threadIdx.x + PF_RMS_THREADS * k) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < NV4; ++k) { v[k].x += w[k].x; v[k].y += w[k].y; v[k].z += w[k].z; v[k].w += w[k].w; }
        }
#pragma unroll
        for (int k = 0; k < NV4; ++k) {
            const int c = threadIdx.x + PF_RMS_THREADS * k;
            if (c < nc) xr[c] = v[k];
        }
    }
    float ss = 0.f;
#pragma unroll
    for (int k = 0; k < NV4; ++k) ss += v[k].x * v[k].x + v[k].y * v[k].y + v[k].z * v[k].z + v[k].w * v[k].w;
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    const float inv = rsqrtf((red[0] + red[1] + red[2] + red[3]) / (float)d_model + eps);
    uint2* hr = reinterpret_cast<uint2*>(h + t * d_model);
#pragma unroll
    for (int k = 0; k < NV4; ++k) {
        const int c = threadIdx.x + PF_RMS_THREADS * k;
        if (c < nc) {
            uint2 o;
            o.x = pack_f16(v[k].x * inv * bf16_lo(g[k].x), v[k].y * inv * bf16_hi(g[k].x));
            o.y = pack_f16(v[k].z * inv * bf16_lo(g[k].y), v[k].w * inv * bf16_hi(g[k].y));
            hr[c] = o;
        }
    }
}

// The QKV projection [T][(Hq + 2 Hkv) * HD] (pieces, summed here): bias, per-head RMSNorm of q and k, rotate-half RoPE at
// the token's position; then q -> fp16 [T][Hq][HD] already multiplied by log2(e) / sqrt(HD) (the attention kernel works in
// the exp2 domain), k and v -> the token's slot in its page, rounded once to fp16.  One warp per token row and PF_QKV_HEADS
// heads of one kind (q, k or v): the loads of all its heads, the rotation and the page look-up are in flight together.
// Lane l holds elements {E l .. E l + E - 1} and their rotation partners HD/2 further on (E = HD / 64).  Bound by memory
// (4 bytes read, 2 written per element); with a warp per single head the chain position -> page -> store of every head
// was what took the time (208 us for 9984 rows of 48 heads).
// bf16 pages (F16 = false): q leaves as a high and a low bf16 part (q_out, q_lo), k and v are rounded once to bf16.
// fp16 pages: q leaves as a high and a low fp16 part where q_lo is given (see attn_append_tc_kernel's TWO), else as one.
constexpr int PF_QKV_THREADS = 256;
constexpr int PF_QKV_HEADS = 4;
inline int pf_qkv_groups(int n_q_heads, int n_kv_heads) {        // tasks per token row
    return (n_q_heads + PF_QKV_HEADS - 1) / PF_QKV_HEADS + 2 * ((n_kv_heads + PF_QKV_HEADS - 1) / PF_QKV_HEADS);
}
template <int HD, bool F16>
__global__ void __launch_bounds__(PF_QKV_THREADS) pf_qkv_post_kernel(
    Pieces pieces, const __nv_bfloat16* __restrict__ bias, const __nv_bfloat16* __restrict__ q_gain,
    const __nv_bfloat16* __restrict__ k_gain, float eps, const float* __restrict__ cos_tab,
    const float* __restrict__ sin_tab, const int32_t* __restrict__ game, const int32_t* __restrict__ pos_of,
    const int32_t* __restrict__ block_table, int max_pages, int n_pages, int layer, int T, int n_q_heads,
    int n_kv_heads, float q_scale, __half* __restrict__ q_out, __half* __restrict__ q_lo, uint16_t* __restrict__ pool,
    int* status) {
    constexpr int E = HD / 64, HALF = HD / 2, NH = PF_QKV_HEADS;
    grid_launch_dependents();
    __shared__ unsigned char cnt_tab[PIECE_TABLE];
    const PieceCounts pcnt = piece_counts_init(pieces, cnt_tab);       // (parameters only: before the wait)
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    const int gq = (n_q_heads + NH - 1) / NH, gk = (n_kv_heads + NH - 1) / NH, groups = gq + 2 * gk;
    const int total = T * groups;
    const int task0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    // position, page, rotation and gains of a task: uploaded before the pass or never written, so the first task's are
    // fetched while the projection still runs
    int pos = 0, page = 0;
    float cs[E], sn[E], gl[E], gh[E];
    auto fetch_ahead = [&](int task) {
        const int t = task / groups, grp = task - t * groups;
        const bool is_q = grp < gq, is_k = !is_q && grp < gq + gk;
        pos = __ldg(pos_of + t);
        page = 0;
        if (!is_q) page = __ldg(block_table + (size_t)__ldg(game + t) * max_pages + pos / ATTN_PAGE);
        const __nv_bfloat16* gain = is_q ? q_gain : is_k ? k_gain : nullptr;
        if (is_q || is_k) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                cs[e] = __ldg(cos_tab + (size_t)pos * HALF + E * lane + e);
                sn[e] = __ldg(sin_tab + (size_t)pos * HALF + E * lane + e);
                gl[e] = gain ? __bfloat162float(gain[E * lane + e]) : 1.f;
                gh[e] = gain ? __bfloat162float(gain[E * lane + e + HALF]) : 1.f;
            }
        }
    };
    if (task0 < total) fetch_ahead(task0);
    grid_dependency_wait();
    for (int task = task0; task < total; task += warps) {
        if (task != task0) fetch_ahead(task);
        const int t = task / groups, grp = task - t * groups;
        const bool is_q = grp < gq, is_k = !is_q && grp < gq + gk;
        const int first = is_q ? grp * NH : (is_k ? grp - gq : grp - gq - gk) * NH;             // head within its kind
        const int nh = min(NH, (is_q ? n_q_heads : n_kv_heads) - first);
        const int head0 = first + (is_q ? 0 : is_k ? n_q_heads : n_q_heads + n_kv_heads);       // row of the projection
        const float* yr = pieces.base + (size_t)t * pieces.ld + head0 * HD + E * lane;
        float lo[NH][E], hi[NH][E];
        auto fetch = [&](const float* yh, float (&l)[E], float (&h)[E]) {
            if (E == 2) {
                const float2 a = __ldcs(reinterpret_cast<const float2*>(yh)), b = __ldcs(reinterpret_cast<const float2*>(yh + HALF));
                l[0] = a.x; l[E - 1] = a.y; h[0] = b.x; h[E - 1] = b.y;
            } else {
                l[0] = __ldcs(yh); h[0] = __ldcs(yh + HALF);
            }
        };
        // the first piece of every head, then (stream-K) the second of every head, ...: no head's sum is waited for before
        // the next head's loads are out
        int most = 0;
#pragma unroll
        for (int u = 0; u < NH; ++u)
            if (u < nh) {
                fetch(yr + u * HD, lo[u], hi[u]);
                most = max(most, pcnt.of(pieces, t, (head0 + u) * HD));
            }
        for (int i = 1; i < most; ++i) {
            float l2[NH][E], h2[NH][E];
#pragma unroll
            for (int u = 0; u < NH; ++u) {
                const bool in = u < nh && i < pcnt.of(pieces, t, (head0 + u) * HD);
#pragma unroll
                for (int e = 0; e < E; ++e) { l2[u][e] = 0.f; h2[u][e] = 0.f; }
                if (in) fetch(yr + u * HD + (size_t)i * pieces.stride, l2[u], h2[u]);
            }
#pragma unroll
            for (int u = 0; u < NH; ++u)
#pragma unroll
                for (int e = 0; e < E; ++e) { lo[u][e] += l2[u][e]; hi[u][e] += h2[u][e]; }
        }
        const __nv_bfloat16* gain = is_q ? q_gain : is_k ? k_gain : nullptr;
#pragma unroll
        for (int u = 0; u < NH; ++u) {
            if (u >= nh) break;
            if (bias) {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    lo[u][e] += __bfloat162float(bias[(head0 + u) * HD + E * lane + e]);
                    hi[u][e] += __bfloat162float(bias[(head0 + u) * HD + E * lane + e + HALF]);
                }
            }
            if (is_q || is_k) {
                if (gain) {
                    float ss = 0.f;
#pragma unroll
                    for (int e = 0; e < E; ++e) ss += lo[u][e] * lo[u][e] + hi[u][e] * hi[u][e];
                    ss = warp_sum(ss);
                    const float inv = rsqrtf(ss / (float)HD + eps);
#pragma unroll
                    for (int e = 0; e < E; ++e) { lo[u][e] = lo[u][e] * inv * gl[e]; hi[u][e] = hi[u][e] * inv * gh[e]; }
                }
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const float a = lo[u][e], b = hi[u][e];
                    lo[u][e] = a * cs[e] - b * sn[e];
                    hi[u][e] = b * cs[e] + a * sn[e];
                }
            }
        }
        if (!is_q && (page < 0 || page >= n_pages)) {
            if (lane == 0) record_status(status, STATUS_BAD_PAGE);
            continue;
        }
#pragma unroll
        for (int u = 0; u < NH; ++u) {
            if (u >= nh) break;
            const float sc = is_q ? q_scale : 1.f;
            uint16_t* dst = is_q ? reinterpret_cast<uint16_t*>(q_out) + ((size_t)t * n_q_heads + first + u) * HD + E * lane
                                 : pool + kv_block_offset(layer, page, first + u, n_pages, n_kv_heads, ATTN_PAGE, HD) +
                                       (is_k ? 0 : (size_t)ATTN_PAGE * HD) + (size_t)(pos % ATTN_PAGE) * HD + E * lane;
            if (!F16) {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    uint32_t h0, l0, h1, l1;
                    split2<false>(lo[u][e] * sc, h0, l0);
                    split2<false>(hi[u][e] * sc, h1, l1);
                    dst[e] = (uint16_t)h0;
                    dst[e + HALF] = (uint16_t)h1;
                    if (is_q) {
                        uint16_t* dl = reinterpret_cast<uint16_t*>(q_lo) + ((size_t)t * n_q_heads + first + u) * HD + E * lane;
                        dl[e] = (uint16_t)l0;
                        dl[e + HALF] = (uint16_t)l1;
                    }
                }
            } else {
                auto put = [&](uint16_t* at, const float (&l)[E], const float (&h)[E]) {
                    if (E == 2) {
                        *reinterpret_cast<uint32_t*>(at) = pack_f16(l[0], l[E - 1]);
                        *reinterpret_cast<uint32_t*>(at + HALF) = pack_f16(h[0], h[E - 1]);
                    } else {
                        at[0] = (uint16_t)float_to_f16_bits(l[0]);
                        at[HALF] = (uint16_t)float_to_f16_bits(h[0]);
                    }
                };
                float l[E], h[E];
#pragma unroll
                for (int e = 0; e < E; ++e) { l[e] = lo[u][e] * sc; h[e] = hi[u][e] * sc; }
                put(dst, l, h);
                if (is_q && q_lo) {             // what the rounding left, rounded again
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        l[e] -= unpack_f16(float_to_f16_bits(l[e])).x;
                        h[e] -= unpack_f16(float_to_f16_bits(h[e])).x;
                    }
                    put(reinterpret_cast<uint16_t*>(q_lo) + (dst - reinterpret_cast<uint16_t*>(q_out)), l, h);
                }
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------
// causal append attention
// ------------------------------------------------------------------------------------------------
constexpr int APP_ROWS = 176;              // query rows (position x head of the KV group) per CTA: 11 consumer warps +
                                           // the producer warp = three warps per scheduler, the register file's limit at
                                           // the ~168 registers the consumers need
constexpr int APP_CWARPS = APP_ROWS / 16;  // consumer warps; one more warp issues the TMA loads
// bf16 pages: a warp's 16 MMA rows are eight query rows, high parts in rows 0..7 and low parts in rows 8..15 (products
// with a query and a softmax weight of twice bf16's mantissa, as in the decode kernel)
constexpr int app_rows(bool f16) { return f16 ? APP_ROWS : APP_ROWS / 2; }
constexpr int APP_THREADS = (APP_CWARPS + 1) * 32;
constexpr int APP_BLK_PAGES = 4;           // pages (16 keys each) per ring stage
constexpr int APP_STAGES = 4;

// One block of consecutive new positions of one game: queries at positions pos0 .. pos0 + n_pos - 1
// (rows row0 .. of the chunk's q / output buffers); kv_len = positions of the game whose keys and
// values have been written (everything beyond is stale pool memory).
// tcgen05 kernel: the CTA takes the key blocks blk0 .. blk1 - 1 of the item; slot >= 0: they are a part of it, whose result
// goes to that partial slot for attn_append_merge_kernel.
struct AppendItem { int game, pos0, n_pos, row0, kv_len, blk0, blk1, slot; };
// a split item: its partials are slots slot .. slot + parts - 1
struct AppendMerge { int n_pos, row0, slot, parts; };

struct AppendParams {
    const __half* q;                // [T][n_q_heads][head_dim] fp16: normalised, rotated, times log2(e)/sqrt(head_dim)
    const __half* q_lo;             // bf16 pages: q and q_lo are the high and low bf16 parts of the same; fp16 pages in two
                                    // parts: the high and low fp16 parts
    const AppendItem* items;
    const int32_t* block_table;     // [max_games][max_pages]
    int max_pages, n_pages, layer, n_q_heads, n_kv_heads, group;
    __half* out;                    // [T][n_q_heads * head_dim]
    float* o_part;                  // [slot][kv head][256 rows][head_dim] partial outputs of split items, not normalised
    float2* ml_part;                // [slot][kv head][256 rows] their (maximum, sum)
    int* status;
};

inline int app_positions_per_item(int group, bool f16) { return app_rows(f16) / group; }
__device__ __forceinline__ uint32_t pack_unit_f16(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}
inline size_t app_smem_bytes(int head_dim) {
    return (size_t)APP_STAGES * APP_BLK_PAGES * (head_dim / 64) * 4096 + 1024;
}

template <int HD, bool F16>
__global__ void __launch_bounds__(APP_THREADS, 1) attn_append_kernel(const __grid_constant__ CUtensorMap tmKV,
                                                                     AppendParams p) {
    constexpr int HALVES = HD / 64;
    constexpr int PAGE_BYTES = HALVES * 4096;          // 16 K rows + 16 V rows of one (page, head), 128-byte rows
    constexpr int STAGE_BYTES = APP_BLK_PAGES * PAGE_BYTES;
    constexpr int KSTEPS = HD / 16;
    constexpr int NT = HD / 8;
    extern __shared__ uint8_t app_smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[APP_STAGES], empty_bar[APP_STAGES];
    __shared__ int abort_sm;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    grid_launch_dependents();
    if (threadIdx.x == 0) {
        for (int s = 0; s < APP_STAGES; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), APP_CWARPS); }
        abort_sm = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tmap_prefetch(&tmKV);
    }
    __syncthreads();
    volatile int* abort_flag = &abort_sm;
    grid_dependency_wait();            // items, queries and the new keys/values come from earlier kernels / copies

    const AppendItem item = p.items[blockIdx.y];          // (all heads of the longest items come first)
    const int kvh = blockIdx.x;
    const int G = p.group;
    const int last_pos = item.pos0 + item.n_pos - 1;
    const int n_pg = last_pos / ATTN_PAGE + 1;                         // pages holding keys 0 .. last_pos
    const int n_blk = (n_pg + APP_BLK_PAGES - 1) / APP_BLK_PAGES;
    const uint32_t ring = (smem_u32(app_smem_raw) + 1023u) & ~1023u;

    if (warp == APP_CWARPS) {
        // ---------------- TMA producer (one warp: lanes look page ids up, lane 0 issues) ----------------
        int my_page = 0;
        for (int j = 0; j < n_blk; ++j) {
            if ((j & 7) == 0) {          // page ids of the next eight blocks, one per lane
                const int pg = APP_BLK_PAGES * j + lane;
                my_page = 0;
                if (pg < n_pg) {
                    my_page = __ldcg(p.block_table + (size_t)item.game * p.max_pages + pg);
                    if (my_page < 0 || my_page >= p.n_pages) {
                        record_status(p.status, STATUS_BAD_PAGE);
                        my_page = 0;
                    }
                }
            }
            const int s = j % APP_STAGES;
            bool ok = true;
            if (j >= APP_STAGES && lane == 0)
                ok = mbar_wait(smem_u32(&empty_bar[s]), (uint32_t)((j / APP_STAGES) - 1) & 1u, abort_flag, p.status,
                               STATUS_TIMEOUT_MMA);
            if (!__shfl_sync(0xffffffffu, ok ? 1 : 0, 0)) break;
            const int npg = min(APP_BLK_PAGES, n_pg - APP_BLK_PAGES * j);
            if (lane == 0) mbar_expect_tx(smem_u32(&full_bar[s]), (uint32_t)(npg * PAGE_BYTES));
#pragma unroll
            for (int k = 0; k < APP_BLK_PAGES; ++k) {
                const int page = __shfl_sync(0xffffffffu, my_page, (j & 7) * APP_BLK_PAGES + k);
                if (lane == 0 && k < npg) {
                    const int y = (((p.layer * p.n_pages + page) * p.n_kv_heads) + kvh) * 32;
#pragma unroll
                    for (int h = 0; h < HALVES; ++h)
                        tma_load_2d_nohint(ring + (uint32_t)(s * STAGE_BYTES + k * PAGE_BYTES + h * 4096), &tmKV, 64 * h, y,
                                           smem_u32(&full_bar[s]));
                }
            }
        }
        // every load issued is waited for by the consumers unless they gave up: then give the copies a bounded time
        if (*abort_flag && lane == 0) {
            for (int s = 0; s < APP_STAGES; ++s) {
                unsigned long long t0 = global_ns();
                while (!mbar_try(smem_u32(&full_bar[s]), 0) && !mbar_try(smem_u32(&full_bar[s]), 1) &&
                       global_ns() - t0 < TMA_WAIT_NS) {}
            }
        }
        return;
    }

    // ---------------- consumers: warp w owns query rows 16 w .. 16 w + 15 (bf16 pages: 8 w .. 8 w + 7) ----------------
    const int g = lane >> 2, c = lane & 3;
    const int r0 = (F16 ? 16 : 8) * warp + g, r1 = F16 ? r0 + 8 : r0;   // this thread's two rows (bf16: one, in two parts)
    const int po0 = r0 / G, hh0 = r0 - po0 * G;                  // position offset and head within the group
    const int po1 = r1 / G, hh1 = r1 - po1 * G;
    const bool ok0 = po0 < item.n_pos, ok1 = po1 < item.n_pos;
    const int pos_r0 = item.pos0 + (ok0 ? po0 : 0), pos_r1 = item.pos0 + (ok1 ? po1 : 0);

    uint32_t qa[KSTEPS][4];
    {
        const __half* q0 = p.q + ((size_t)(item.row0 + (ok0 ? po0 : 0)) * p.n_q_heads + kvh * G + hh0) * HD + 2 * c;
        const __half* q1 = (F16 ? p.q : p.q_lo) + ((size_t)(item.row0 + (ok1 ? po1 : 0)) * p.n_q_heads + kvh * G + hh1) * HD + 2 * c;
#pragma unroll
        for (int ks = 0; ks < KSTEPS; ++ks) {
            qa[ks][0] = __ldcg(reinterpret_cast<const uint32_t*>(q0 + 16 * ks));
            qa[ks][1] = __ldcg(reinterpret_cast<const uint32_t*>(q1 + 16 * ks));
            qa[ks][2] = __ldcg(reinterpret_cast<const uint32_t*>(q0 + 16 * ks + 8));
            qa[ks][3] = __ldcg(reinterpret_cast<const uint32_t*>(q1 + 16 * ks + 8));
        }
    }
    float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
    float o[NT][4];
#pragma unroll
    for (int t = 0; t < NT; ++t) { o[t][0] = 0.f; o[t][1] = 0.f; o[t][2] = 0.f; o[t][3] = 0.f; }

    const int lr = lane & 7, lm = lane >> 3;
    const int k_tok = lr + 8 * (lm >> 1), k_chk = lm & 1;
    const int v_tok = lr + 8 * (lm & 1), v_chk = lm >> 1;
    const uint32_t k_row_off = (uint32_t)(k_tok * 128), v_row_off = (uint32_t)((16 + v_tok) * 128);

    for (int j = 0; j < n_blk; ++j) {
        const int s = j % APP_STAGES;
        const uint32_t base = ring + (uint32_t)(s * STAGE_BYTES);
        const bool landed = mbar_wait(smem_u32(&full_bar[s]), (uint32_t)(j / APP_STAGES) & 1u, abort_flag, p.status,
                                      STATUS_TIMEOUT_TMA);
        if (!__all_sync(0xffffffffu, landed)) break;
        const int npg = min(APP_BLK_PAGES, n_pg - APP_BLK_PAGES * j);
        const int key0 = j * APP_BLK_PAGES * ATTN_PAGE;
        // value rows of positions not written yet hold stale pool bytes (possibly NaN patterns): the
        // weights there are exactly zero, but 0 * NaN is not -- zero those rows (last page only).  Every
        // warp zeroes all of them itself before it reads any: the warps then need no barrier between
        // them (they store the same zeros), and this stage is not refilled afterwards.
        if (j == n_blk - 1 && item.kv_len < n_pg * ATTN_PAGE) {
            const int valid = item.kv_len - (n_pg - 1) * ATTN_PAGE;            // 1 .. 15 rows of the last page exist
            const uint32_t pbase = base + (uint32_t)((npg - 1) * PAGE_BYTES);
            for (int idx = lane; idx < (ATTN_PAGE - valid) * 8 * HALVES; idx += 32) {
                const int r = valid + idx / (8 * HALVES), rem = idx % (8 * HALVES);
                asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(pbase + (rem >> 3) * 4096 + (16 + r) * 128 +
                                                                           (rem & 7) * 16), "r"(0u) : "memory");
            }
            __syncwarp();
        }
        // ---- scores S[16 rows x 64 keys] = Q K^T (already in the log2 domain: q carries the scale) ----
        float sc[2 * APP_BLK_PAGES][4];
#pragma unroll
        for (int t = 0; t < 2 * APP_BLK_PAGES; ++t) { sc[t][0] = 0.f; sc[t][1] = 0.f; sc[t][2] = 0.f; sc[t][3] = 0.f; }
#pragma unroll
        for (int pgi = 0; pgi < APP_BLK_PAGES; ++pgi) {
            if (pgi < npg) {
                const uint32_t pb = base + (uint32_t)(pgi * PAGE_BYTES);
#pragma unroll
                for (int ks = 0; ks < KSTEPS; ++ks) {
                    const int h = ks >> 2, ch = 2 * (ks & 3) + k_chk;
                    uint32_t b0, b1, b2, b3;
                    ldmatrix_x4(pb + h * 4096 + k_row_off + (uint32_t)(((ch ^ (k_tok & 7)) << 4)), b0, b1, b2, b3);
                    mma_16816<F16>(sc[2 * pgi], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], b0, b1);
                    mma_16816<F16>(sc[2 * pgi + 1], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], b2, b3);
                }
            }
        }
        if (!F16) {                     // the row's score = high-part row + low-part row; both halves carry it from here
#pragma unroll
            for (int t = 0; t < 2 * APP_BLK_PAGES; ++t)
#pragma unroll
                for (int e = 0; e < 2; ++e) { sc[t][e] += sc[t][2 + e]; sc[t][2 + e] = sc[t][e]; }
        }
        // causal mask: the row at position P sees keys 0 .. P (also hides pages that were not loaded)
        if (key0 + APP_BLK_PAGES * ATTN_PAGE - 1 > item.pos0) {
#pragma unroll
            for (int t = 0; t < 2 * APP_BLK_PAGES; ++t)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int key = key0 + 8 * t + 2 * c + e;
                    if (key > pos_r0) sc[t][e] = -INFINITY;
                    if (key > pos_r1) sc[t][2 + e] = -INFINITY;
                }
        }
        float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
        for (int t = 0; t < 2 * APP_BLK_PAGES; ++t) {
            mx0 = fmaxf(mx0, fmaxf(sc[t][0], sc[t][1]));
            mx1 = fmaxf(mx1, fmaxf(sc[t][2], sc[t][3]));
        }
        mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
        mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
        mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
        mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
        // key 0 is visible to every row and lies in the first block: the running maxima are finite from there on
        const float mn0 = fmaxf(m0, mx0), mn1 = fmaxf(m1, mx1);
        const float al0 = fast_exp2(m0 - mn0), al1 = fast_exp2(m1 - mn1);
        float rs0 = 0.f, rs1 = 0.f;
#pragma unroll
        for (int t = 0; t < 2 * APP_BLK_PAGES; ++t) {
            sc[t][0] = fast_exp2(sc[t][0] - mn0); sc[t][1] = fast_exp2(sc[t][1] - mn0);
            sc[t][2] = fast_exp2(sc[t][2] - mn1); sc[t][3] = fast_exp2(sc[t][3] - mn1);
            rs0 += sc[t][0] + sc[t][1];
            rs1 += sc[t][2] + sc[t][3];
        }
        l0 = l0 * al0 + rs0;
        l1 = l1 * al1 + rs1;
        if (__any_sync(0xffffffffu, mn0 > m0 || mn1 > m1)) {      // a running maximum moved: rescale the accumulators
#pragma unroll
            for (int t = 0; t < NT; ++t) { o[t][0] *= al0; o[t][1] *= al0; o[t][2] *= al1; o[t][3] *= al1; }
        }
        m0 = mn0; m1 = mn1;
        // ---- O[16 x HD] += P[16 x 64 keys] V ----
#pragma unroll
        for (int pgi = 0; pgi < APP_BLK_PAGES; ++pgi) {
            if (pgi < npg) {
                const uint32_t pb = base + (uint32_t)(pgi * PAGE_BYTES);
                // weights lie in [0, 1]: plain round-to-nearest conversion, no saturation needed
                uint32_t a0, a1, a2, a3;
                if (F16) {
                    a0 = pack_unit_f16(sc[2 * pgi][0], sc[2 * pgi][1]); a1 = pack_unit_f16(sc[2 * pgi][2], sc[2 * pgi][3]);
                    a2 = pack_unit_f16(sc[2 * pgi + 1][0], sc[2 * pgi + 1][1]);
                    a3 = pack_unit_f16(sc[2 * pgi + 1][2], sc[2 * pgi + 1][3]);
                } else {
                    uint32_t h[4], lw[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) split2<false>(sc[2 * pgi + (k >> 1)][k & 1], h[k], lw[k]);
                    a0 = h[0] | (h[1] << 16); a1 = lw[0] | (lw[1] << 16);
                    a2 = h[2] | (h[3] << 16); a3 = lw[2] | (lw[3] << 16);
                }
#pragma unroll
                for (int np = 0; np < NT / 2; ++np) {
                    const int h = np >> 2, ch = 2 * (np & 3) + v_chk;
                    uint32_t b0, b1, b2, b3;
                    ldmatrix_x4_trans(pb + h * 4096 + v_row_off + (uint32_t)(((ch ^ (v_tok & 7)) << 4)), b0, b1, b2, b3);
                    mma_16816<F16>(o[2 * np], a0, a1, a2, a3, b0, b1);
                    mma_16816<F16>(o[2 * np + 1], a0, a1, a2, a3, b2, b3);
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&empty_bar[s]));
    }
    if (*abort_flag) return;
    l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
    l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
    const float i0 = 1.f / l0, i1 = 1.f / l1;
    __half* o0 = p.out + ((size_t)(item.row0 + po0) * p.n_q_heads + kvh * G + hh0) * HD + 2 * c;
    __half* o1 = p.out + ((size_t)(item.row0 + po1) * p.n_q_heads + kvh * G + hh1) * HD + 2 * c;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        if (!F16) {
            if (ok0) *reinterpret_cast<uint32_t*>(o0 + 8 * t) = pack_f16((o[t][0] + o[t][2]) * i0, (o[t][1] + o[t][3]) * i0);
            continue;
        }
        if (ok0) *reinterpret_cast<uint32_t*>(o0 + 8 * t) = pack_f16(o[t][0] * i0, o[t][1] * i0);
        if (ok1) *reinterpret_cast<uint32_t*>(o1 + 8 * t) = pack_f16(o[t][2] * i1, o[t][3] * i1);
    }
}

// ------------------------------------------------------------------------------------------------
// the same attention on the 5th-generation tensor cores
// ------------------------------------------------------------------------------------------------
// One CTA per (query block, KV head).  The block's query rows (positions x heads of the group) form
// two tiles of 128 rows = 128 TMEM lanes each, which share the keys and values streamed through
// shared memory.  Per block of 64 keys (4 pages) and tile:
//     S = Q K^T      tcgen05.mma M128 N64, Q and K K-major in shared memory        -> TMEM (two S buffers per tile)
//     P = 2^(S - m)  softmax warps, one thread per row (no shuffles), fp16          -> shared memory
//     O += P V       tcgen05.mma M128 N=HD, V as stored ([key][head_dim]: MN-major B), accumulated in TMEM
// m is the row maximum in use; it is only raised (and the row of O in TMEM and the running sum
// rescaled) when a block's maximum exceeds it by more than 2^8, so that P stays within fp16 range and
// the rescaling -- a read-modify-write of tensor memory -- is rare after the first blocks.
// Warp 0 streams K and V pages through a four-stage TMA ring (separate 16-row boxes so that the keys of
// a block are contiguous rows), warps 1 and 10 issue the MMAs of tile 0 and 1 (S of block j+1 is
// computed while the softmax of block j runs), warps 2..5 / 6..9 are the softmax threads of tile 0 / 1.
constexpr int APT_BN = 64;                       // keys per block
constexpr int APT_PAGES = APT_BN / ATTN_PAGE;
// TILES = 2: one CTA per SM holds two query tiles that share the streamed keys and values (four K/V stages).
// TILES = 1: one query tile per CTA, two CTAs per SM (two stages each): the keys and values are fetched
// once per tile, but one CTA's prologue and epilogue run under the other's main loop.
// TWO (with TILES = 1, one CTA per SM, four stages): the queries and the softmax weights are in two fp16 parts, high and
// low, each multiplied with the same keys and values into the same accumulator: products with a query and a weight of 22
// bits, as in the decode kernel.  It serves the appends that a decode-shaped step could hold (prefill_dense says which),
// so that they lose nothing against it: error of the logits against 64 bits, Qwen3-4B shape, 4 x 25 tokens behind 2000:
// step 2.98e-3, one part 3.50e-3, two parts 2.97e-3.
__host__ __device__ constexpr int apt_stages(int tiles, bool two) { return tiles == 1 && !two ? 2 : 4; }
__host__ __device__ constexpr int apt_threads(int tiles) { return tiles == 1 ? 192 : 352; }   // TMA warp, MMA warp (tile 0), 4 softmax warps per
                                                                          // tile, and for two tiles the MMA warp of tile 1
constexpr uint32_t APT_QSLAB = 128 * 128;        // 128 query rows of 128 bytes: one 64-element slab of a Q tile / one P tile
constexpr uint32_t APT_KSLAB = APT_BN * 128;     // 64 key rows of 128 bytes: one 64-element slab of a K or V tile
constexpr float APT_RESCALE_LOG2 = 8.f;
// Q tiles, P tiles, the K + V stages, and the slack to reach a 1024-byte boundary.  Two one-tile CTAs of
// head_dim 128 fill an SM to the byte (2 x (112 KB of tiles + 1 KB reserved + the barriers)): their slack is
// what is left, 864 bytes, which suffices where the dynamic region starts 160 bytes past a 1024-byte
// boundary, as it does behind the kernel's static shared memory; the kernel checks and refuses otherwise.
inline size_t apt_smem_bytes(int head_dim, int tiles, bool two) {
    const size_t slabs = head_dim / 64, parts = two ? 2 : 1;
    return tiles * parts * (slabs + 1) * APT_QSLAB + apt_stages(tiles, two) * 2 * slabs * APT_KSLAB +
           (tiles == 1 && !two && head_dim == 128 ? 864 : 1024);
}
inline int apt_positions_per_item(int group, int tiles) { return tiles * (128 / group); }

// Shared-memory descriptor of an MN-major operand tile with the 128-byte swizzle: rows are k (here: keys)
// of 128 bytes = 64 elements of the N dimension; 8-row groups are `sbo` bytes apart, the next 64 elements
// of N start `lbo` bytes further on.
__device__ __forceinline__ uint64_t smem_desc_sw128_mn(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3ffffu) >> 4);
    d |= (uint64_t)(lbo >> 4) << 16;
    d |= (uint64_t)(sbo >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// 16 consecutive fp32 columns of this warp's 32 TMEM lanes, written from registers
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Timing probe builds (-DAPT_PROBE) only: clock cycles one softmax warp of every CTA's first tile spends in each
// phase of a key block, summed over the launch.
#ifdef APT_PROBE
__device__ unsigned long long g_apt_probe[16];
#define APT_STAMP(i)                                                                         \
    do {                                                                                     \
        if (probe_on) {                                                                      \
            const long long now__ = clock64();                                               \
            atomicAdd(&g_apt_probe[i], (unsigned long long)(now__ - probe_t));               \
            probe_t = now__;                                                                 \
        }                                                                                    \
    } while (0)
#else
#define APT_STAMP(i) do { } while (0)
#endif

template <int HD, int TILES, bool TWO>
__global__ void __launch_bounds__(apt_threads(TILES), TILES == 1 && !TWO ? 2 : 1) attn_append_tc_kernel(const __grid_constant__ CUtensorMap tmKV16,
                                                                        AppendParams p) {
    constexpr int SLABS = HD / 64;
    constexpr uint32_t Q_TILE = SLABS * APT_QSLAB, P_TILE = APT_QSLAB, KV_BYTES = SLABS * APT_KSLAB;
    constexpr uint32_t STAGE_BYTES = 2 * KV_BYTES;
    constexpr int PARTS = TWO ? 2 : 1;                     // tile t: its high part, then (TWO) its low part, for Q and for P
    static_assert(!TWO || TILES == 1, "two parts: one query tile per CTA");
    constexpr int APT_STAGES = apt_stages(TILES, TWO), APT_THREADS = apt_threads(TILES);
    constexpr uint32_t TM_O = 2 * TILES * APT_BN;          // S: (2 tile + buffer) * 64 columns; O: TM_O + tile * HD
    constexpr uint32_t TM_COLS = TILES == 1 ? 256 : 512;
    constexpr uint32_t PAGE_ROWS_BYTES = ATTN_PAGE * 128;  // 16 rows of 128 bytes
    extern __shared__ uint8_t apt_smem_raw[];
    __shared__ __align__(8) uint64_t q_ready, kv_full[APT_STAGES], kv_empty[APT_STAGES], s_full[2][2], s_empty[2][2],
        p_full[2], p_empty[2], o_full[2];
    __shared__ uint32_t tmem_base_sm;
    __shared__ int abort_sm;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    grid_launch_dependents();
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&q_ready), 4 * TILES);
        for (int s = 0; s < APT_STAGES; ++s) { mbar_init(smem_u32(&kv_full[s]), 1); mbar_init(smem_u32(&kv_empty[s]), TILES); }
        for (int t = 0; t < 2; ++t) {
            for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&s_full[t][b]), 1); mbar_init(smem_u32(&s_empty[t][b]), 4); }
            mbar_init(smem_u32(&p_full[t]), 4); mbar_init(smem_u32(&p_empty[t]), 1); mbar_init(smem_u32(&o_full[t]), 1);
        }
        abort_sm = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tmap_prefetch(&tmKV16);
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_sm), TM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_sm;
    volatile int* abort_flag = &abort_sm;
    grid_dependency_wait();            // items, queries and the new keys/values come from earlier kernels / copies

    const AppendItem item = p.items[blockIdx.y];          // (all heads of the longest items come first)
    const int kvh = blockIdx.x;
    const int G = p.group;
    const int PT = 128 / G;                                       // positions per tile
    const int n_tiles = (TILES == 2 && item.n_pos > PT) ? 2 : 1;  // a second tile without rows to compute stays idle
    const int last_pos = item.pos0 + item.n_pos - 1;
    const int n_pg = last_pos / ATTN_PAGE + 1;
    const int b0 = item.blk0, n_blk = item.blk1 - b0;             // this CTA's key blocks
    const bool has_end = item.blk1 * APT_PAGES >= n_pg;           // ... include the last one
    const uint32_t base = (smem_u32(apt_smem_raw) + 1023u) & ~1023u;
    const uint32_t q_base = base, p_base = base + TILES * PARTS * Q_TILE, ring = p_base + TILES * PARTS * P_TILE;
    {
        uint32_t dyn_bytes;
        asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_bytes));
        if (ring + APT_STAGES * STAGE_BYTES > smem_u32(apt_smem_raw) + dyn_bytes) {       // CTA-uniform
            if (threadIdx.x == 0) record_status(p.status, STATUS_BAD_SMEM);
            tc_fence_before();
            __syncthreads();
            if (warp == 1) tmem_dealloc(tmem_base, TM_COLS);
            return;
        }
    }

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        int my_page = 0;
        for (int j = 0; j < n_blk; ++j) {
            if ((j & 7) == 0) {          // page ids of the next eight blocks, one per lane
                const int pg = APT_PAGES * (b0 + j) + lane;
                my_page = 0;
                if (pg < n_pg) {
                    my_page = __ldcg(p.block_table + (size_t)item.game * p.max_pages + pg);
                    if (my_page < 0 || my_page >= p.n_pages) {
                        record_status(p.status, STATUS_BAD_PAGE);
                        my_page = 0;
                    }
                }
            }
            const int s = j % APT_STAGES;
            bool ok = true;
            if (j >= APT_STAGES && lane == 0)
                ok = mbar_wait(smem_u32(&kv_empty[s]), (uint32_t)((j / APT_STAGES) - 1) & 1u, abort_flag, p.status,
                               STATUS_TIMEOUT_MMA);
            if (!__shfl_sync(0xffffffffu, ok ? 1 : 0, 0)) break;
            const int npg = min(APT_PAGES, n_pg - APT_PAGES * (b0 + j));
            const uint32_t stage = ring + (uint32_t)s * STAGE_BYTES;
            if (lane == 0) mbar_expect_tx(smem_u32(&kv_full[s]), (uint32_t)(npg * 2 * SLABS) * PAGE_ROWS_BYTES);
            __syncwarp();
            // lane k fetches page k of the block: its K rows and its V rows, one box per 64-element slab
            const int page = __shfl_sync(0xffffffffu, my_page, (j & 7) * APT_PAGES + (lane & (APT_PAGES - 1)));
            if (lane < npg) {
                const int y = (((p.layer * p.n_pages + page) * p.n_kv_heads) + kvh) * 32;      // K rows; V rows at y + 16
#pragma unroll
                for (int h = 0; h < SLABS; ++h) {
                    tma_load_2d_nohint(stage + h * APT_KSLAB + lane * PAGE_ROWS_BYTES, &tmKV16, 64 * h, y, smem_u32(&kv_full[s]));
                    tma_load_2d_nohint(stage + KV_BYTES + h * APT_KSLAB + lane * PAGE_ROWS_BYTES, &tmKV16, 64 * h, y + 16,
                                       smem_u32(&kv_full[s]));
                }
            }
        }
        if (*abort_flag && lane == 0) {        // the consumers gave up: bounded wait for the copies in flight
            for (int s = 0; s < APT_STAGES; ++s) {
                unsigned long long t0 = global_ns();
                while (!mbar_try(smem_u32(&kv_full[s]), 0) && !mbar_try(smem_u32(&kv_full[s]), 1) &&
                       global_ns() - t0 < TMA_WAIT_NS) {}
            }
        }
    } else if (warp == 1 || (TILES == 2 && warp == APT_THREADS / 32 - 1)) {
        // ---------------- MMA issuers: one warp per tile (the whole warp walks the loop, one elected lane issues) ----------------
        const int t = warp == 1 ? 0 : 1;
        if (t < n_tiles) {
            const uint32_t idesc_qk = tc_idesc_f16(APT_BN);
            const uint32_t idesc_pv = tc_idesc_f16(HD) | (1u << 16);          // B (V) is MN-major
#ifdef APT_PROBE
            const bool probe_on = t == 0 && lane == 0;
            long long probe_t = clock64();
#endif
            bool ok = mbar_wait_warp(smem_u32(&q_ready), 0u, abort_flag, p.status, STATUS_TIMEOUT_EPI);
            APT_STAMP(6);           // MMA warp: wait for Q
            const uint64_t da0 = smem_desc_sw128(q_base + (uint32_t)(t * PARTS) * Q_TILE);
            const uint64_t dp = smem_desc_sw128(p_base + (uint32_t)(t * PARTS) * P_TILE);
            auto issue_qk = [&](int j) -> bool {
                const int s = j % APT_STAGES, b = j & 1;
                if (!mbar_wait_warp(smem_u32(&kv_full[s]), (uint32_t)(j / APT_STAGES) & 1u, abort_flag, p.status, STATUS_TIMEOUT_TMA))
                    return false;
                APT_STAMP(7);       // MMA warp: wait for K/V
                if (j >= 2 && !mbar_wait_warp(smem_u32(&s_empty[t][b]), (uint32_t)((j >> 1) - 1) & 1u, abort_flag, p.status,
                                              STATUS_TIMEOUT_EPI))
                    return false;
                APT_STAMP(8);       // MMA warp: wait for the S buffer
                tc_fence_after();
                const uint64_t db0 = smem_desc_sw128(ring + (uint32_t)s * STAGE_BYTES);
                const uint32_t d_s = tmem_base + (uint32_t)((2 * t + b) * APT_BN);
                if (elect_one()) {
#pragma unroll
                    for (int part = 0; part < PARTS; ++part)
#pragma unroll
                        for (int h = 0; h < SLABS; ++h)
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                tc_mma_f16(d_s, da0 + (uint64_t)(part * (Q_TILE >> 4) + h * (APT_QSLAB >> 4) + 2 * k),
                                           db0 + (uint64_t)(h * (APT_KSLAB >> 4) + 2 * k), idesc_qk, (part > 0 || h > 0 || k > 0) ? 1u : 0u);
                    tc_commit(smem_u32(&s_full[t][b]));
                }
                __syncwarp();
                APT_STAMP(9);       // MMA warp: issue of Q.K
                return true;
            };
            ok = ok && issue_qk(0);
            for (int j = 0; ok && j < n_blk; ++j) {
                if (j + 1 < n_blk && !issue_qk(j + 1)) break;
                const int s = j % APT_STAGES;
                const int npg = min(APT_PAGES, n_pg - APT_PAGES * (b0 + j));
                const uint64_t dv = smem_desc_sw128_mn(ring + (uint32_t)s * STAGE_BYTES + KV_BYTES, APT_KSLAB, 1024u);
                if (!mbar_wait_warp(smem_u32(&p_full[t]), (uint32_t)j & 1u, abort_flag, p.status, STATUS_TIMEOUT_EPI)) break;
                tc_fence_after();
                APT_STAMP(10);      // MMA warp: wait for P
                if (elect_one()) {
                    const uint32_t d_o = tmem_base + TM_O + (uint32_t)(t * HD);
                    for (int ks = 0; ks < npg; ++ks)             // one page = 16 keys = one k step
#pragma unroll
                        for (int part = 0; part < PARTS; ++part)
                            tc_mma_f16(d_o, dp + (uint64_t)(part * (P_TILE >> 4) + 2 * ks), dv + (uint64_t)(ks * (PAGE_ROWS_BYTES >> 4)),
                                       idesc_pv, (j > 0 || ks > 0 || part > 0) ? 1u : 0u);
                    tc_commit(smem_u32(&o_full[t]));
                    tc_commit(smem_u32(&p_empty[t]));
                    // the stage is free once both tiles' MMAs on it have completed (one tile: it arrives for both)
                    tc_commit(smem_u32(&kv_empty[s]));
                    if (TILES == 2 && n_tiles == 1) tc_commit(smem_u32(&kv_empty[s]));
                }
                __syncwarp();
                APT_STAMP(11);      // MMA warp: issue of P.V
            }
        }
    } else {
        // ---------------- softmax: thread = query row = TMEM lane of its tile ----------------
        const int t = (warp - 2) >> 2;
        const int qd = warp & 3;
        const int r = 32 * qd + lane;
        const int po_l = r / G;
        const int po = t * PT + po_l;
        const bool row_ok = po_l < PT && po < item.n_pos;
        const int pos_r = item.pos0 + (row_ok ? po : 0);
        const int tile_pos0 = item.pos0 + t * PT;                 // no row of the tile sees less than keys 0 .. tile_pos0
#ifdef APT_PROBE
        const long long probe_t0 = clock64();
#endif
        constexpr int CPR = HD / 8;                 // 16-byte chunks per row
        constexpr int RPI = 32 / CPR;               // rows one warp-wide 16-byte access covers
        {
            // the warp's 32 rows of Q into the swizzled K-major tile, RPI rows per (coalesced) load
#pragma unroll
            for (int i = 0; i < CPR; ++i) {
                const int rr = 32 * qd + i * RPI + lane / CPR, c = lane % CPR;
                const int pl = rr / G, h2 = rr - pl * G;
                const int pp = t * PT + pl;
                const bool okr = pl < PT && pp < item.n_pos;
                const size_t row = ((size_t)(item.row0 + (okr ? pp : 0)) * p.n_q_heads + kvh * G + h2) * HD;
#pragma unroll
                for (int part = 0; part < PARTS; ++part) {
                    const uint4 v = __ldcg(reinterpret_cast<const uint4*>((part ? p.q_lo : p.q) + row) + c);
                    const uint32_t dst = q_base + (uint32_t)(t * PARTS + part) * Q_TILE + (uint32_t)(c >> 3) * APT_QSLAB + (uint32_t)rr * 128u +
                                         (uint32_t)(((c & 7) ^ (rr & 7)) << 4);
                    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&q_ready));
        }
        if (t < n_tiles) {
#ifdef APT_PROBE
            const bool probe_on = warp == 2 && lane == 0;
            long long probe_t = probe_t0;
            APT_STAMP(12);          // softmax warp: Q row into shared memory
#endif
            float m = -INFINITY, l = 0.f;
            const uint32_t t_lane = tmem_base + ((uint32_t)(qd * 32) << 16);
            const uint32_t t_o = t_lane + TM_O + (uint32_t)(t * HD);
            int done_blocks = 0;
            for (int j = 0; j < n_blk; ++j) {
                const int b = j & 1, s = j % APT_STAGES;
                if (!mbar_wait(smem_u32(&s_full[t][b]), (uint32_t)(j >> 1) & 1u, abort_flag, p.status, STATUS_TIMEOUT_MMA)) break;
                tc_fence_after();
                APT_STAMP(0);       // wait for S
                const uint32_t t_s = t_lane + (uint32_t)((2 * t + b) * APT_BN);
                const int key0 = (b0 + j) * APT_BN;
                const int vis = key0 + APT_BN - 1 > tile_pos0 ? pos_r - key0 : APT_BN;      // columns 0 .. vis are visible
                uint32_t v[4][16];
#pragma unroll
                for (int h = 0; h < 4; ++h) tmem_ld16_async(t_s + (uint32_t)(16 * h), v[h]);
                tmem_ld_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_empty[t][b]));         // the scores are in registers now
                APT_STAMP(1);       // S into registers
                // (four independent chains each for the maximum and the sum: the row is one thread's work)
                const bool all_vis = vis >= APT_BN - 1;
                float mxs[4];
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    mxs[h] = -INFINITY;
                    if (all_vis) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) mxs[h] = fmaxf(mxs[h], __uint_as_float(v[h][i]));
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (16 * h + i <= vis) mxs[h] = fmaxf(mxs[h], __uint_as_float(v[h][i]));
                    }
                }
                const float mx = fmaxf(fmaxf(mxs[0], mxs[1]), fmaxf(mxs[2], mxs[3]));
                if (j == 0) {
                    m = mx;                     // (a later part of an item may hold no key that the row sees: -inf, weights 0)
                } else {
                    const bool raise = mx > m + APT_RESCALE_LOG2;
                    if (__any_sync(0xffffffffu, raise)) {
                        // rescale this warp's rows of O: the previous block's P.V must have completed
                        if (!mbar_wait(smem_u32(&o_full[t]), (uint32_t)(j - 1) & 1u, abort_flag, p.status, STATUS_TIMEOUT_MMA))
                            break;
                        tc_fence_after();
                        const float alpha = raise ? fast_exp2(m - mx) : 1.f;
#pragma unroll 1
                        for (int c0 = 0; c0 < HD; c0 += 32) {
                            uint32_t w[2][16];
                            tmem_ld16_async(t_o + (uint32_t)c0, w[0]);
                            tmem_ld16_async(t_o + (uint32_t)(c0 + 16), w[1]);
                            tmem_ld_wait();
#pragma unroll
                            for (int h = 0; h < 2; ++h)
#pragma unroll
                                for (int i = 0; i < 16; ++i) w[h][i] = __float_as_uint(__uint_as_float(w[h][i]) * alpha);
                            tmem_st16(t_o + (uint32_t)c0, w[0]);
                            tmem_st16(t_o + (uint32_t)(c0 + 16), w[1]);
                        }
                        tmem_st_wait();
                        tc_fence_before();
                        if (raise) { l *= alpha; m = mx; }
                    }
                }
                APT_STAMP(2);       // maximum (and rescale)
                float sums[4];
                uint32_t w[4][8];               // the row of P as fp16 pairs, ready before the buffer is waited for
                uint32_t wl[TWO ? 4 : 1][8];    // what their rounding left
                auto keep = [&](int h, int i, float e0, float e1) {
                    w[h][i >> 1] = pack_unit_f16(e0, e1);
                    if (TWO) {
                        const float2 got = unpack_f16(w[h][i >> 1]);
                        wl[TWO ? h : 0][i >> 1] = pack_unit_f16(e0 - got.x, e1 - got.y);
                    }
                };
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    sums[h] = 0.f;
                    if (all_vis) {
#pragma unroll
                        for (int i = 0; i < 16; i += 2) {
                            const float e0 = fast_exp2(__uint_as_float(v[h][i]) - m);
                            const float e1 = fast_exp2(__uint_as_float(v[h][i + 1]) - m);
                            sums[h] += e0 + e1;
                            keep(h, i, e0, e1);
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; i += 2) {
                            const int col = 16 * h + i;
                            const float e0 = col <= vis ? fast_exp2(__uint_as_float(v[h][i]) - m) : 0.f;
                            const float e1 = col + 1 <= vis ? fast_exp2(__uint_as_float(v[h][i + 1]) - m) : 0.f;
                            sums[h] += e0 + e1;
                            keep(h, i, e0, e1);
                        }
                    }
                }
                const float rowsum = (sums[0] + sums[1]) + (sums[2] + sums[3]);
                APT_STAMP(3);       // exponentials
                if (j >= 1 && !mbar_wait(smem_u32(&p_empty[t]), (uint32_t)(j - 1) & 1u, abort_flag, p.status, STATUS_TIMEOUT_MMA))
                    break;
                APT_STAMP(4);       // wait for the P buffer
#pragma unroll
                for (int c = 0; c < 8; ++c) {           // 16-byte chunk (8 keys) of the row
                    const uint32_t dst = p_base + (uint32_t)(t * PARTS) * P_TILE + (uint32_t)r * 128u + (uint32_t)((c ^ (r & 7)) << 4);
                    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(w[c >> 1][4 * (c & 1)]),
                                 "r"(w[c >> 1][4 * (c & 1) + 1]), "r"(w[c >> 1][4 * (c & 1) + 2]), "r"(w[c >> 1][4 * (c & 1) + 3])
                                 : "memory");
                    if (TWO) {
                        const uint32_t(&x)[8] = wl[TWO ? c >> 1 : 0];
                        asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(dst + P_TILE), "r"(x[4 * (c & 1)]),
                                     "r"(x[4 * (c & 1) + 1]), "r"(x[4 * (c & 1) + 2]), "r"(x[4 * (c & 1) + 3]) : "memory");
                    }
                }
                // value rows of positions not written yet hold stale pool bytes (possibly NaN patterns): their
                // weights are exactly zero, but 0 * NaN is not -- zero them (they lie in the last page loaded).
                // Both tiles do it (the same zeros) before they release their P.V.
                if (j == n_blk - 1 && has_end && item.kv_len < n_pg * ATTN_PAGE) {
                    if (!mbar_wait(smem_u32(&kv_full[s]), (uint32_t)(j / APT_STAGES) & 1u, abort_flag, p.status, STATUS_TIMEOUT_TMA))
                        break;
                    const int npg = n_pg - APT_PAGES * (b0 + j);
                    const int valid = item.kv_len - (n_pg - 1) * ATTN_PAGE;            // rows of the last page that exist
                    const uint32_t vpage = ring + (uint32_t)s * STAGE_BYTES + KV_BYTES + (uint32_t)(npg - 1) * PAGE_ROWS_BYTES;
                    if (qd == 0 && lane < ATTN_PAGE && lane >= valid) {
#pragma unroll
                        for (int h = 0; h < SLABS; ++h)
#pragma unroll
                            for (int c = 0; c < 8; ++c)
                                asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(vpage + h * APT_KSLAB + lane * 128 + c * 16),
                                             "r"(0u) : "memory");
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&p_full[t]));
                APT_STAMP(5);       // P stores, fence, arrive
                l += rowsum;
                ++done_blocks;
                if (*abort_flag) break;
            }
            if (done_blocks == n_blk && !*abort_flag &&
                mbar_wait(smem_u32(&o_full[t]), (uint32_t)(n_blk - 1) & 1u, abort_flag, p.status, STATUS_TIMEOUT_MMA)) {
                tc_fence_after();
                const int hh = r - po_l * G;
                if (item.slot >= 0) {
                    const size_t prow = ((size_t)item.slot * p.n_kv_heads + kvh) * 256 + t * 128 + r;
                    uint4* part = reinterpret_cast<uint4*>(p.o_part + prow * HD);
                    if (row_ok) p.ml_part[prow] = make_float2(m, l);
#pragma unroll 1
                    for (int c0 = 0; c0 < HD; c0 += 32) {
                        uint32_t w[2][16];
                        tmem_ld16_async(t_o + (uint32_t)c0, w[0]);
                        tmem_ld16_async(t_o + (uint32_t)(c0 + 16), w[1]);
                        tmem_ld_wait();
                        if (row_ok) {
#pragma unroll
                            for (int h = 0; h < 2; ++h)
#pragma unroll
                                for (int q4 = 0; q4 < 4; ++q4)
                                    part[(c0 >> 2) + 4 * h + q4] = make_uint4(w[h][4 * q4], w[h][4 * q4 + 1], w[h][4 * q4 + 2], w[h][4 * q4 + 3]);
                        }
                    }
                } else {
                    const float inv = 1.f / l;
                    uint4* dst = reinterpret_cast<uint4*>(p.out + ((size_t)(item.row0 + po) * p.n_q_heads + kvh * G + hh) * HD);
#pragma unroll 1
                    for (int c0 = 0; c0 < HD; c0 += 32) {
                        uint32_t w[2][16];
                        tmem_ld16_async(t_o + (uint32_t)c0, w[0]);
                        tmem_ld16_async(t_o + (uint32_t)(c0 + 16), w[1]);
                        tmem_ld_wait();
                        if (row_ok) {
#pragma unroll
                            for (int h = 0; h < 2; ++h)
#pragma unroll
                                for (int q8 = 0; q8 < 2; ++q8) {
                                    uint4 o4;
                                    o4.x = pack_f16(__uint_as_float(w[h][8 * q8]) * inv, __uint_as_float(w[h][8 * q8 + 1]) * inv);
                                    o4.y = pack_f16(__uint_as_float(w[h][8 * q8 + 2]) * inv, __uint_as_float(w[h][8 * q8 + 3]) * inv);
                                    o4.z = pack_f16(__uint_as_float(w[h][8 * q8 + 4]) * inv, __uint_as_float(w[h][8 * q8 + 5]) * inv);
                                    o4.w = pack_f16(__uint_as_float(w[h][8 * q8 + 6]) * inv, __uint_as_float(w[h][8 * q8 + 7]) * inv);
                                    dst[(c0 >> 3) + 2 * h + q8] = o4;
                                }
                        }
                    }
                }
                tc_fence_before();
            }
            APT_STAMP(13);          // softmax warp: wait for the last P.V, normalise, store
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, TM_COLS);
}

// Adds up the parts of split items: one warp per query row (position x head of the group), all parts' loads in flight.
// Bound by L2 (4 bytes per element and part read, 2 per element written).
constexpr int APM_THREADS = 256, APM_MAX_PARTS = 8;
template <int HD>
__global__ void __launch_bounds__(APM_THREADS) attn_append_merge_kernel(const AppendMerge* __restrict__ merges, AppendParams p) {
    constexpr int EL = HD / 32;
    grid_launch_dependents();
    const int lane = threadIdx.x & 31, r = blockIdx.x * (APM_THREADS / 32) + (threadIdx.x >> 5);       // row of the two tiles
    const int kvh = blockIdx.y, G = p.group, PT = 128 / G;
    const AppendMerge mg = merges[blockIdx.z];                     // (uploaded before the pass's first kernel)
    const int po_l = (r & 127) / G, po = (r >> 7) * PT + po_l, hh = (r & 127) - po_l * G;
    if (po_l >= PT || po >= mg.n_pos) return;
    grid_dependency_wait();
    const size_t row0 = ((size_t)mg.slot * p.n_kv_heads + kvh) * 256 + r, step = (size_t)p.n_kv_heads * 256;
    float2 ml[APM_MAX_PARTS];
    float o[APM_MAX_PARTS][EL];
#pragma unroll
    for (int i = 0; i < APM_MAX_PARTS; ++i) {
        ml[i] = make_float2(-INFINITY, 0.f);
#pragma unroll
        for (int e = 0; e < EL; ++e) o[i][e] = 0.f;
        if (i < mg.parts) {
            ml[i] = __ldcg(p.ml_part + row0 + i * step);
            const float* src = p.o_part + (row0 + i * step) * HD + EL * lane;
#pragma unroll
            for (int e = 0; e < EL; e += 2) {
                const float2 v = __ldcg(reinterpret_cast<const float2*>(src + e));
                o[i][e] = v.x; o[i][e + 1] = v.y;
            }
        }
    }
    float M = -INFINITY, l = 0.f, acc[EL];
#pragma unroll
    for (int i = 0; i < APM_MAX_PARTS; ++i) M = fmaxf(M, ml[i].x);    // finite: key 0 is visible to every row
#pragma unroll
    for (int e = 0; e < EL; ++e) acc[e] = 0.f;
#pragma unroll
    for (int i = 0; i < APM_MAX_PARTS; ++i) {
        const float w = fast_exp2(ml[i].x - M);
        l += w * ml[i].y;
#pragma unroll
        for (int e = 0; e < EL; ++e) acc[e] += w * o[i][e];
    }
    const float inv = 1.f / l;
    __half* dst = p.out + ((size_t)(mg.row0 + po) * p.n_q_heads + kvh * G + hh) * HD + EL * lane;
#pragma unroll
    for (int e = 0; e < EL; e += 2) *reinterpret_cast<uint32_t*>(dst + e) = pack_f16(acc[e] * inv, acc[e + 1] * inv);
}

// How the query blocks of a pass are cut along the keys.  A CTA takes about 1.6 us per key block; a few query blocks leave
// most SMs idle for as long as the longest takes (100 tokens behind 2400: 16 CTAs of 40 blocks; 4967 -> 3767 us per call
// of the Qwen3-4B shape when cut).  Costs in key blocks: 3 a CTA (prologue, epilogue), 1 more for writing a partial, 5 for
// the merge; a cut has to win 15 %, since the SMs it fills are where the output projection would request its weights
// early (331 tokens behind 450: attention 25.8 -> 23.5 us, the call 0.7 % slower).  `blocks`: key blocks per query block;
// returns the most key blocks of a CTA.
inline int append_attn_cap(const std::vector<int>& blocks, int heads, int n_sm) {
    int longest = 0;
    for (int b : blocks) longest = std::max(longest, b);
    int best = longest;
    double best_cost = -1;
    for (int parts = 1; parts <= APM_MAX_PARTS; ++parts) {
        const int cap = (longest + parts - 1) / parts;
        if (parts > 1 && cap < 2) break;
        long long ctas = 0, sum = 0;
        for (int b : blocks) { const int n = (b + cap - 1) / cap; ctas += n; sum += b + n * (n > 1 ? 4 : 3); }
        if (parts > 1 && ctas * heads > 4 * n_sm) break;            // (bounds the partials' buffer, too)
        const double top = cap + (parts > 1 ? 4 : 3);
        const double cost = (ctas * heads <= n_sm ? top : (double)sum * heads / n_sm + 0.5 * top) + (parts > 1 ? 5 : 0);
        if (best_cost < 0 || cost < 0.85 * best_cost) { best_cost = cost; best = cap; }
    }
    return best;
}

}  // namespace spiral
