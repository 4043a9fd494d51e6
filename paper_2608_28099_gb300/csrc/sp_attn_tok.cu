// Split-KV attention of the k appended rows over [cached ; new] keys
// (Sec. 3.3, Eq. 1-3) on tcgen05 tensor cores with the tokens on the MMA's M
// side, for head_dim 128 and bf16 caches: the kernel for up to 32 query rows per kv
// head, and for up to 64 in larger batches (tok_wins below).
//
// The work list, its cuts and the partials are those of sp_attn_tc.cu: CTA
// (j, g) attends kv head g over share j of the 64-token tile list; a share's
// piece of one sequence is a segment.  What differs is the product's shape.  Per
// step of 128 tokens (two tiles of the list):
//   S^T  = K Q^T     M = 128 tokens (K straight from its ring slot), N = query
//                    rows padded to 16 (Q in shared memory as bf16 hi + lo, two
//                    MMAs per step, or plain, one)
//   softmax          one token per thread, the query rows split between two groups
//                    of four warps: the exponentials use all four SM sub-partitions
//                    whatever R is (with queries on the M side 32 rows keep one
//                    busy), and nothing is reduced over tokens: a row's running max
//                    only moves when some score exceeds it by 2^8 (a vote per step,
//                    then the rare path finds the row maxima and rescales O), row
//                    sums stay per thread until the segment ends
//   O^T += V^T P     M = 128 dims (V read in place as the transposed A operand),
//                    N = query rows, P as bf16 [token][row] in shared memory; on the
//                    first step of a segment of a short sequence as bf16 hi + lo, two
//                    MMAs (the lo plane in the free half of P's 128-byte lines up to 32
//                    rows, else over the step's K, which the scores are done with)
// Precision: a probability of 1, that of a row's maximum where it sets the running
// max, is the only one that bf16 holds exactly, and one maximum per 128 tokens leaves
// more to rounding than the queries-on-M kernel's one per 64.  Against that, the row
// sums (fp32) are over the probabilities as rounded: an error e of a token's weight
// then moves the output by e (v - o) instead of e v, never more on average over values of
// one distribution (sum w^2 - 2 sum w^3 + (sum w^2)^2 <= sum w^2); and sequences of two to
// eight tiles, up to 512 tokens, have the lo plane (two to four from 33 rows on, where
// holding the K slot costs 2-3 % of a call beyond).  Relative error of the output, 4 rows
// of 32 heads: 100 tokens 1.45e-3 (queries on M), 1.53e-3 (this kernel with neither),
// 1.00e-3 (now); 300 tokens 1.64e-3, 1.66e-3, 1.41e-3; 1000 tokens 1.66e-3, 1.67e-3,
// 1.63e-3; 4000 tokens 1.64e-3 in all.  The sums cost nothing that can be measured, the
// lo plane 0 to 4 % of the attention of a batch that has it (124 sequences of 92 to 155
// tokens, paged, 4 / 16 / 32 rows: 37.2 / 39.0 / 51.5 -> 38.7 / 39.2 / 51.4 us).
// An MMA costs the padded row count instead of 128 columns (40 cycles at 32 rows,
// shared-memory bandwidth of the token operand), and a step of 128 tokens takes
// 1.2-1.4 us while all SMs stream (1.2 GB at 6.0 TB/s, 0.89 of the copy rate, in the 8B
// paged call's kernel: HBM-bound) instead of the 1.5 us chain per 64 tokens of the
// queries-on-M kernel.  S^T is double-buffered in TMEM: the scores of step n + 1
// are ready when the softmax of step n ends.  The queries of the next segment are
// loaded by warps of their own into the other query buffer, so the pipeline does
// not drain at a segment boundary: it costs about 4 us (8-10 there).  What is left
// of the 4B call's 23 us (77 MB, 11.5 us at the copy rate): 5 us from launch to the
// first scores, 5 us from the last step to the merged output.
//
// K and V have rings of their own (a K slot is free once S^T is done), filled
// by two warps each: TMA for whole pages of a paged cache, cp.async for
// contiguous caches and partial pages, plain loads for the new rows.
// Warps 0-7: softmax, epilogue; 8-11: producers (even K, odd V); 12-14: queries;
// 15: MMA issue and TMEM.  Every wait is time-limited (SP_DEV_TIMEOUT).
#include <cudaTypedefs.h>
#include <string.h>

#include "sp_attn_plan.cuh"
#include "sp_common.cuh"
#include "sp_sm100.cuh"

namespace sp {

namespace {

constexpr int STEP = 128;                  // tokens per step: two tiles of the list
constexpr int SLOT = STEP * DH * 2;        // K or V of one step, 32 KB
constexpr int MAX_SLOTS = 4;
constexpr int SMEM_MAX = 227 * 1024;
constexpr int OFF_BAR = 0;                 // Bars
constexpr int OFF_ROW = 512;               // per-row tables and reductions
constexpr int ROW_WORDS = 11 * 128;
constexpr int OFF_CUT = OFF_ROW + ROW_WORDS * 4;
constexpr int OFF_TAB = OFF_CUT + (MAX_GRP + 4) * 4;  // prefix [B + 1], (sid, len) [B]
constexpr int THREADS = 512;
constexpr int PROD_WARP = 8, Q_WARP = 12, MMA_W = 15;
constexpr int SOFT_THREADS = 256, KV_THREADS = 64, Q_THREADS = 96;
constexpr int BAR_SOFT = 1, BAR_Q = 4;  // (BAR_SOFT + 1, + 2: one softmax group)

// Shared-memory plan of a launch (host): the queries and P sit in front of the
// rings, so that nothing the MMAs read past a buffer's rows leaves the window.
struct TokLayout {
    int r16;        // query rows padded to a multiple of 16
    int nk, nv;     // ring slots
    int off_q, q_bytes, off_p, off_k, off_v;
    int smem;
};

struct TokBars {
    uint64_t k_full[MAX_SLOTS], k_empty[MAX_SLOTS], v_full[MAX_SLOTS], v_empty[MAX_SLOTS];
    uint64_t s_full[2], q_full[2], q_empty[2], p_full, pv_done, fin;
    uint32_t tmem;
    int abort;
    int merge_now;
    int fm_merge, fm_b, fm_nseg;
    long long fm_slot0;
    int wsum[THREADS / 32];
};
static_assert(sizeof(TokBars) <= OFF_ROW, "barrier block");

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void soft_sync() {
    asm volatile("bar.sync %0, %1;" ::"n"(BAR_SOFT), "n"(SOFT_THREADS) : "memory");
}
__device__ __forceinline__ bool soft_any(bool x) {  // over the softmax warps
    int any;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.s32 q, %1, 0;\n\t"
        "barrier.cta.red.or.pred p, %2, %3, q;\n\t"
        "selp.s32 %0, 1, 0, p;\n\t}"
        : "=r"(any)
        : "r"((int)x), "n"(BAR_SOFT), "n"(SOFT_THREADS)
        : "memory");
    return any != 0;
}

struct OpMax {
    __device__ static float f(float a, float b) { return fmaxf(a, b); }
};
struct OpSum {
    __device__ static float f(float a, float b) { return a + b; }
};
// Reduce each of W values over the 32 lanes by halving exchanges (31 shuffles
// for W = 32): lane i ends with value i W / 32.
template <int W, typename Op>
__device__ __forceinline__ float lane_reduce(float (&v)[W], int lane) {
    static_assert(W == 8 || W == 16 || W == 32, "");
    int o = 16;
#pragma unroll
    for (int n = W; n > 1; o >>= 1, n >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int j = 0; j < n / 2; ++j) {
            const float send = up ? v[j] : v[j + n / 2], keep = up ? v[j + n / 2] : v[j];
            v[j] = Op::f(keep, __shfl_xor_sync(0xffffffffu, send, o));
        }
    }
#pragma unroll
    for (; o > 0; o >>= 1) v[0] = Op::f(v[0], __shfl_xor_sync(0xffffffffu, v[0], o));
    return v[0];
}

template <int W>
__device__ __forceinline__ void tmem_ldw(uint32_t addr, float (&v)[W]) {
    if constexpr (W == 32)
        tmem_ld32(addr, v);
    else if constexpr (W == 16)
        tmem_ld16(addr, v);
    else
        tmem_ld8(addr, v);
}
template <int W>
__device__ __forceinline__ void tmem_stw(uint32_t addr, const float (&v)[W]) {
    if constexpr (W == 32)
        tmem_st32(addr, v);
    else if constexpr (W == 16)
        tmem_st16(addr, v);
    else
        tmem_st8(addr, v);
}

// The steps of a CTA's share, in order.
struct Walk {
    const int *prefix;
    int B, x, x1;   // next tile of the list, the share's end
    Seg sg;
    int j, i, n;    // segment, step within it, steps of it
    __device__ __forceinline__ Walk(const int *p, int b, int x0, int xe) : prefix(p), B(b), x(x0), x1(xe), j(-1) { seg(); }
    __device__ __forceinline__ void seg() {
        ++j;
        i = 0;
        n = 0;
        if (x < x1) {
            sg = seg_at(prefix, B, x, x1);
            // the same in every lane, and known to be
            sg.n = __shfl_sync(0xffffffffu, sg.n, 0);
            x += sg.n;
            n = (sg.n + 1) / 2;
        }
    }
    __device__ __forceinline__ bool done() const { return n == 0; }
    __device__ __forceinline__ int tiles() const { return min(2, sg.n - 2 * i); }  // of this step
    __device__ __forceinline__ void next() {
        if (++i == n) seg();
    }
};

// Ring position: slot and the parity of its current use.
struct Ring {
    int n, slot = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ explicit Ring(int slots) : n(slots) {}
    __device__ __forceinline__ void next() {
        if (++slot == n) {
            slot = 0;
            ph ^= 1;
        }
    }
};

// Queries rr = hl k + r of sequence b for kv head g, scaled to log2 units, as bf16
// hi [and lo] in the K-major layout of the score MMA's B operand: [hi, lo][dim
// half][row][64 dims], 128-byte swizzle; rows past R are zero.  By threads t of n.
template <int NR>
__device__ __forceinline__ void load_queries(const AttnArgs &a, const int *ro_s, int b, int g, uint8_t *Q, int t,
                                             int n) {
    constexpr int U = 4;  // chunks of eight dims in flight per thread
#pragma unroll 1
    for (int i0 = t; i0 < NR * 16; i0 += U * n) {
        float4 v[U][2];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = i0 + u * n, rr = idx >> 4;
            v[u][0] = v[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (rr < a.R) {
                const float *src = a.q + ((size_t)b * a.k * a.Hq + g * a.G + ro_s[rr]) * DH + (idx & 15) * 8;
                v[u][0] = *(const float4 *)src;
                v[u][1] = *(const float4 *)(src + 4);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = i0 + u * n, rr = idx >> 4, c = idx & 15;
            if (rr >= NR) continue;
            const float x8[8] = {v[u][0].x, v[u][0].y, v[u][0].z, v[u][0].w,
                                 v[u][1].x, v[u][1].y, v[u][1].z, v[u][1].w};
            float h[8], l8[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float q = x8[e] * a.scale_log2;
                h[e] = __bfloat162float(__float2bfloat16_rn(q));
                l8[e] = q - h[e];
            }
            uint8_t *d = Q + (c >> 3) * (NR * 128) + (rr >> 3) * 1024 + (rr & 7) * 128 + (((c & 7) ^ (rr & 7)) << 4);
            st_shared_v4(d, pack_bf16(h[0], h[1]), pack_bf16(h[2], h[3]), pack_bf16(h[4], h[5]), pack_bf16(h[6], h[7]));
            if (!a.tc_q_plain)
                st_shared_v4(d + NR * 256, pack_bf16(l8[0], l8[1]), pack_bf16(l8[2], l8[3]), pack_bf16(l8[4], l8[5]),
                             pack_bf16(l8[6], l8[7]));
        }
    }
    fence_proxy_async();  // -> tensor-core reads
}

// NR: the query rows padded to a multiple of 16.
template <int NR>
__global__ void __launch_bounds__(THREADS, 1)
    attn_tok_kernel(const __grid_constant__ CUtensorMap map_k,
                    const __grid_constant__ CUtensorMap map_v, AttnArgs a, TokLayout lay) {
    constexpr int HC = NR / 2;                   // query rows of a softmax group
    constexpr int W = HC % 32 == 0 ? 32 : HC % 16 == 0 ? 16 : 8;  // columns per TMEM load
    constexpr int NC = HC / W;
    constexpr int EC = W < 16 ? W : 16;          // rows of an epilogue chunk
    constexpr uint32_t S_COLS = (NR + 31) / 32 * 32;  // TMEM columns of a score buffer
    constexpr uint32_t O_COL = 2 * S_COLS;
    constexpr uint32_t TMEM_COLS = NR <= 32 ? 128 : 256;
    static_assert(NR % 16 == 0 && NR <= 64, "query rows");
    constexpr bool LO_IN_LINE = NR <= 32;        // P's lo plane in P's lines, else in the K slot
    constexpr int LO_TILES = LO_IN_LINE ? 8 : 4; // tiles of the longest sequence that has one
    // (a sequence of one tile needs none: one maximum in either kernel)
    auto has_lo = [](const Seg &sg) { return sg.nt >= 2 && sg.nt <= LO_TILES; };
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    TokBars *bars = (TokBars *)(smem + OFF_BAR);
    float *m_s = (float *)(smem + OFF_ROW);      // running max of a row (-inf: nothing seen)
    float *mt_s = m_s + 128;                     // score above which it moves
    float *nm_s = mt_s + 128;                    // minus the max (0 for -inf), added to scores
    float *al_s = nm_s + 128;                    // rescale factor, or 1 / sum at the end
    float *red_s = al_s + 128;                   // [4][128] per-warp reductions
    int *rk_s = (int *)(red_s + 4 * 128);        // row % k
    int *lo_s = rk_s + 128;                      // first new row of the row's task
    int *ro_s = lo_s + 128;                      // (row % k) Hq + row / k: output row offset
    int *cuts = (int *)(smem + OFF_CUT);
    int *prefix = (int *)(smem + OFF_TAB);
    volatile int *abort = &bars->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int R = a.R, k = a.k, B = a.B, Hkv = a.Hkv;
    int2 *seqs = (int2 *)(prefix + ((B + 2) & ~1));
    const int kns = a.kn_stride ? a.kn_stride : k;  // rows per sequence of k_new / v_new
    const bool paged = a.kv.layout == SP_KV_PAGED;
    pdl_trigger();

    build_prefix<THREADS>(a, prefix, seqs, bars->wsum, blockIdx.x == 0 ? a.status : nullptr);
    const int T = prefix[B];
    const int n_grp = share_count((int)gridDim.x / Hkv, T, B, a.tc_min_tiles);
    const int grp = blockIdx.x / Hkv, g = blockIdx.x - grp * Hkv;
    if (grp >= n_grp) {  // uniform over the CTA: no tile for this one
        if (threadIdx.x == 0 && a.l2_next)
            prefetch_l2_share(a.l2_next, a.l2_next_bytes, blockIdx.x, gridDim.x);
        return;
    }
    if (threadIdx.x < PLAN_THREADS)  // (set-up is shared out over the warps)
        build_cuts(a, prefix, T, n_grp, cuts, bars->wsum);
    if (threadIdx.x >= 128 && threadIdx.x < 256) {
        const int rr = threadIdx.x - 128;
        const int rk = rr % k;
        rk_s[rr] = rk;
        lo_s[rr] = a.k_task ? (rk / a.k_task) * a.k_task : 0;
        ro_s[rr] = rk * a.Hq + rr / k;
    }
    if (threadIdx.x == PROD_WARP * 32) {
#pragma unroll 1
        for (int i = 0; i < lay.nk; ++i) {
            mbar_init(&bars->k_full[i], KV_THREADS);
            mbar_init(&bars->k_empty[i], 1);
        }
#pragma unroll 1
        for (int i = 0; i < lay.nv; ++i) {
            mbar_init(&bars->v_full[i], KV_THREADS);
            mbar_init(&bars->v_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars->s_full[i], 1);
            mbar_init(&bars->q_full[i], Q_THREADS);
            mbar_init(&bars->q_empty[i], 1);
        }
        mbar_init(&bars->p_full, SOFT_THREADS);
        mbar_init(&bars->pv_done, 1);
        mbar_init(&bars->fin, 1);
        bars->abort = 0;
        bars->merge_now = 0;
        bars->fm_merge = 0;
        fence_mbar_init();
        if (paged) {
            prefetch_tmap(&map_k);
            prefetch_tmap(&map_v);
        }
    }
    if (warp == MMA_W) {
        tmem_alloc(&bars->tmem, TMEM_COLS);
        tmem_relinquish();
    }
    // No griddepcontrol.wait here: the cache, page table and lengths belong to the
    // caller, so the producers start streaming while the previous kernel (which
    // writes the rotated queries and new keys) drains; the query warps, the
    // producers at a new row and the softmax warps wait before they touch its
    // output or write what an earlier kernel may still read.
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem;
    const int x0 = cuts[grp], x1 = cuts[grp + 1];

    if (warp >= PROD_WARP && warp < Q_WARP) {
        // ------------------------------------------------------------ producers
        const bool is_v = warp & 1;
        const int pidx = (warp - PROD_WARP) >> 1, ptid = pidx * 32 + lane;
        const bool lead = pidx == 0;
        uint64_t *full = is_v ? bars->v_full : bars->k_full, *empty = is_v ? bars->v_empty : bars->k_empty;
        uint8_t *ring = smem + (is_v ? lay.off_v : lay.off_k);
        const CUtensorMap *map = is_v ? &map_v : &map_k;
        const bf16 *pool = (const bf16 *)(is_v ? a.kv.v_pool : a.kv.k_pool);
        const float *fresh = is_v ? a.v_new : a.k_new;
        const uint64_t pol = policy_evict_first();
        const int P = a.kv.page_size;
        Ring rg(is_v ? lay.nv : lay.nk);
        int bad = 0, filled = 0;
        bool waited = false;
#pragma unroll 1
        for (Walk w(prefix, B, x0, x1); !w.done(); w.next()) {
            const int b = w.sg.b;
            const int2 sq = seqs[b];  // (cache id, length)
            const int L = sq.y, total = L + a.r0 + k;
            const int t0 = (w.sg.t_a + 2 * w.i) * TT, n_tok = w.tiles() * TT;
            const int n_cache = max(0, min(n_tok, L - t0));             // rows [0, n_cache)
            const int n_new = max(0, min(n_tok, total - t0)) - n_cache;  // then new rows
            const int n_pg = paged ? n_cache / P : 0;                   // whole pages: TMA
            // this step's page ids (up to eight), requested before the ring wait
            int page = -1;
            if (paged && lane * P < n_cache) {
                const int lp = t0 / P + lane;
                page = lp < a.kv.max_pages ? a.kv.page_table[(size_t)max(sq.x, 0) * a.kv.max_pages + lp] : -1;
                if (page < 0 || page >= a.kv.n_pages) {
                    page = -1;
                    bad = 1;
                } else if (lead && !is_v && a.gathered) {
                    a.gathered[(size_t)b * a.kv.max_pages + lp] = page;
                }
            }
            // warp-uniform verdict: the collectives below need every lane
            if (!__all_sync(0xffffffffu, mbar_wait(&empty[rg.slot], rg.ph ^ 1, abort))) break;
            uint8_t *dst = ring + rg.slot * SLOT;
            bool plain = false;  // this thread wrote shared memory or issued cp.async
            if (n_pg > 0 && lead) {
                // one TMA box per lane: the (page, head) block of P tokens; a page
                // outside the pool is zero-filled below
                const bool ok = lane < n_pg && page >= 0;
                const unsigned okm = __ballot_sync(0xffffffffu, ok);
                if (lane == 0 && okm) mbar_expect_tx(&full[rg.slot], (uint32_t)__popc(okm) * P * DH * 2u);
                __syncwarp();
                if (ok)  // the cache is read once: evict-first keeps queries and partials in L2
                    tma_load_4d_hint(dst + lane * P * 256, map, &full[rg.slot], 0, 0, 0, (page * Hkv + g) * (P / 8),
                                     pol);
#pragma unroll 1
                for (unsigned miss = ~okm & ((1u << n_pg) - 1u); miss; miss &= miss - 1) {
                    const int j = __ffs(miss) - 1;
#pragma unroll 1
                    for (int e = lane; e < P * 16; e += 32) st_shared_v4(dst + j * P * 256 + e * 16, 0, 0, 0, 0);
                    plain = true;
                }
            }
            const int r0_ = n_pg * (paged ? P : 0);  // first row not covered by TMA
            if (r0_ < n_tok) {
                plain = true;
                if (r0_ < n_cache) {
                    const bf16 *src = nullptr;
                    bool ok = true;
                    if (paged) {  // the last, partial page
                        const int pg = __shfl_sync(0xffffffffu, page, n_pg);
                        ok = pg >= 0;
                        if (ok) src = pool + ((size_t)pg * Hkv + g) * P * DH;
#pragma unroll 1
                        for (int idx = ptid; idx < (n_cache - r0_) * 16; idx += KV_THREADS) {
                            const int row = idx >> 4, c16 = idx & 15;
                            if (ok)
                                cp_async16(dst + kv_off(r0_ + row, c16), src + (size_t)row * DH + c16 * 8);
                            else
                                st_shared_v4(dst + kv_off(r0_ + row, c16), 0, 0, 0, 0);
                        }
                    } else {  // contiguous: token-major rows of 256 B, Hkv rows a token
                        src = (const bf16 *)(is_v ? a.kv.v_seq : a.kv.k_seq)[sq.x] + ((size_t)t0 * Hkv + g) * DH;
#pragma unroll 4
                        for (int idx = ptid; idx < n_cache * 16; idx += KV_THREADS) {
                            const int row = idx >> 4, c16 = idx & 15;
                            cp_async16(dst + kv_off(row, c16), src + (size_t)row * Hkv * DH + c16 * 8);
                        }
                    }
                }
                if (n_new > 0 && !waited) {
                    pdl_wait();  // the new rows come from the previous kernel
                    waited = true;
                }
                // new rows [B][k][Hkv][dh] fp32 -> bf16: two chunks per thread in flight
#pragma unroll 1
                for (int idx = ptid; idx < n_new * 16; idx += 2 * KV_THREADS) {
                    float4 f[2][2];
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int j = idx + u * KV_THREADS;
                        if (j < n_new * 16) {
                            const int rr = (t0 + n_cache + (j >> 4)) - L;
                            const float *o = fresh + (((size_t)b * kns + rr) * Hkv + g) * DH + (j & 15) * 8;
                            f[u][0] = *(const float4 *)o;
                            f[u][1] = *(const float4 *)(o + 4);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int j = idx + u * KV_THREADS;
                        if (j < n_new * 16)
                            st_shared_v4(dst + kv_off(n_cache + (j >> 4), j & 15), pack_bf16(f[u][0].x, f[u][0].y),
                                         pack_bf16(f[u][0].z, f[u][0].w), pack_bf16(f[u][1].x, f[u][1].y),
                                         pack_bf16(f[u][1].z, f[u][1].w));
                    }
                }
                const int n_fill = n_cache + n_new;
#pragma unroll 1
                for (int idx = ptid; idx < (n_tok - n_fill) * 16; idx += KV_THREADS)
                    st_shared_v4(dst + kv_off(n_fill + (idx >> 4), idx & 15), 0, 0, 0, 0);
            }
            if (plain) {
                fence_proxy_async();  // this thread's shared-memory stores
                cp_async_mbar_arrive(&full[rg.slot]);
            } else {
                mbar_arrive(&full[rg.slot]);
            }
            ++filled;
            rg.next();
        }
        asm volatile("cp.async.wait_all;" ::: "memory");  // nothing lands after the CTA is gone
        if (lead && lane == 0) {
            // drain TMA writes still in flight (only possible after an abort)
            Ring rd(rg.n);
#pragma unroll 1
            for (int j = 0; j < filled; ++j, rd.next())
                if (j + rg.n >= filled) mbar_wait_drain(&full[rd.slot], rd.ph);
        }
        bad = __any_sync(0xffffffffu, bad);
        if (bad && lane == 0 && a.status) atomicOr(a.status, SP_DEV_BAD_PAGE);
    } else if (warp >= Q_WARP && warp < MMA_W) {
        // ------------------------------------------------------------ queries
        // (the first segment's together with the softmax warps, which have nothing
        // else to do then)
        const int qt = threadIdx.x - Q_WARP * 32;
        pdl_wait();  // the rotated queries come from the previous kernel
        Ring rg(2);
        bool first = true;
#pragma unroll 1
        for (int x = x0; x < x1;) {
            const Seg sg = seg_at(prefix, B, x, x1);
            x += sg.n;
            if (!mbar_wait(&bars->q_empty[rg.slot], rg.ph ^ 1, abort)) break;
            load_queries<NR>(a, ro_s, sg.b, g, smem + lay.off_q + rg.slot * lay.q_bytes,
                             qt + (first ? SOFT_THREADS : 0), Q_THREADS + (first ? SOFT_THREADS : 0));
            if (first) asm volatile("bar.sync %0, %1;" ::"n"(BAR_Q), "n"(SOFT_THREADS + Q_THREADS) : "memory");
            first = false;
            mbar_arrive(&bars->q_full[rg.slot]);
            rg.next();
        }
    } else if (warp == MMA_W) {
        // ------------------------------------------------------------ MMA issue
        // S_0, S_1, then per step n: PV_n once softmax n has written P, and S_{n+2}
        // into the score buffer softmax n has read
        // (by the whole warp, the instructions under `lead`: see elect_one)
        const bool lead = elect_one();
        constexpr uint32_t idesc_s = idesc_bf16_f32(128, NR);
        constexpr uint32_t idesc_o = idesc_bf16_f32_bmn(128, NR) | (1u << 15);  // A MN-major too
        const uint64_t dk0 = sw128_kmajor_desc_sbo(smem + lay.off_k, GROUP_STRIDE);
        const uint64_t dq0 = sw128_kmajor_desc(smem + lay.off_q);
        const uint64_t dv0 = sw128_mnmajor_desc2(smem + lay.off_v, HALF_STRIDE, GROUP_STRIDE);
        const uint64_t dp0 = sw128_mnmajor_desc2(smem + lay.off_p, STEP * 128, 1024);
        const uint64_t dl0 = sw128_mnmajor_desc2(smem + lay.off_k, STEP * 128, 1024);
        const uint32_t q_step = (uint32_t)lay.q_bytes >> 4;
        const bool q_lo = !a.tc_q_plain;
        Walk ws(prefix, B, x0, x1);
        Ring rk(lay.nk), rv(lay.nv), rq(2);
        uint32_t sbuf = 0;
        bool ok = true;
        auto issue_s = [&]() {
            if (!ok || ws.done()) return;
            if (ws.i == 0) ok = mbar_wait_warp(&bars->q_full[rq.slot], rq.ph, abort);
            ok = ok && mbar_wait_warp(&bars->k_full[rk.slot], rk.ph, abort);
            if (!ok) return;
            tc_fence_after();
            fence_proxy_async();  // cp.async data -> tensor-core reads
            const uint64_t dk = dk0 + (uint32_t)(rk.slot * (SLOT >> 4));
            const uint64_t dq = dq0 + (uint32_t)rq.slot * q_step;
            const uint32_t d = tmem + sbuf * S_COLS;
            if (lead) {
#pragma unroll
                for (int kk = 0; kk < DH / 16; ++kk) {
                    // 16 dims = 32 B along a 128-byte row of dim half kk / 4
                    const uint64_t ak = dk + (uint64_t)((kk >> 2) * (HALF_STRIDE >> 4) + (kk & 3) * 2);
                    const uint64_t bq = dq + (uint64_t)((kk >> 2) * (NR * 128 >> 4) + (kk & 3) * 2);
                    mma_bf16(d, ak, bq, idesc_s, kk > 0 ? 1u : 0u);
                    if (q_lo) mma_bf16(d, ak, bq + (uint64_t)(NR * 256 >> 4), idesc_s, 1u);
                }
                if (LO_IN_LINE || ws.i > 0 || !has_lo(ws.sg)) mma_commit(&bars->k_empty[rk.slot]);
                mma_commit(&bars->s_full[sbuf]);
                if (ws.i == ws.n - 1) mma_commit(&bars->q_empty[rq.slot]);
            }
            if (ws.i == ws.n - 1) rq.next();
            rk.next();
            sbuf ^= 1;
            ws.next();
        };
        issue_s();
        issue_s();
        Ring rp(lay.nk);  // the step's K slot
        uint32_t ph = 0;
#pragma unroll 1
        for (Walk w(prefix, B, x0, x1); ok && !w.done(); w.next(), ph ^= 1) {
            const uint64_t dv = dv0 + (uint32_t)(rv.slot * (SLOT >> 4));
            const bool two = w.tiles() == 2;
            if (!mbar_wait_warp(&bars->v_full[rv.slot], rv.ph, abort)) break;
            fence_proxy_async();
            if (!mbar_wait_warp(&bars->p_full, ph, abort)) break;
            tc_fence_after();
            if (lead) {
#pragma unroll
                for (int kk = 0; kk < STEP / 16; ++kk)  // 16 tokens: two 8-token groups of V and of P
                    if (kk < TT / 16 || two)
                        mma_bf16(tmem + O_COL, dv + (uint64_t)(kk * (2 * GROUP_STRIDE >> 4)),
                                 dp0 + (uint64_t)(kk * (2048 >> 4)), idesc_o, (w.i > 0 || kk > 0) ? 1u : 0u);
                if (w.i == 0 && has_lo(w.sg)) {
                    const uint64_t dl = LO_IN_LINE ? dp0 + (64 >> 4) : dl0 + (uint32_t)(rp.slot * (SLOT >> 4));
#pragma unroll
                    for (int kk = 0; kk < STEP / 16; ++kk)
                        if (kk < TT / 16 || two)
                            mma_bf16(tmem + O_COL, dv + (uint64_t)(kk * (2 * GROUP_STRIDE >> 4)),
                                     dl + (uint64_t)(kk * (2048 >> 4)), idesc_o, 1u);
                    if (!LO_IN_LINE) mma_commit(&bars->k_empty[rp.slot]);
                }
                mma_commit(&bars->v_empty[rv.slot]);
                mma_commit(&bars->pv_done);
            }
            rv.next();
            rp.next();
            issue_s();
        }
        if (lead) mma_commit(&bars->fin);  // completes when every MMA is done
        __syncwarp();
    } else {
        // ------------------------------------------------------------ softmax + epilogue
        // Two groups of four warps, each all tokens of a step and half of the query
        // rows (columns of S^T and O^T): two warps per SM sub-partition hide each
        // other's latencies, and a thread's rows fit its registers.
        const int tok = threadIdx.x & 127;   // token of the step, later the output dim; == TMEM lane
        const int wq = warp & 3, cb = (warp >> 2) * HC;  // first query row of the group
        const uint32_t lane_base = tmem + ((uint32_t)(wq * 32) << 16) + (uint32_t)cb;
        pdl_wait();  // before writing what an earlier kernel may still be reading
        if (x0 < x1) {  // (an empty share has no queries: its query warps do not come either)
            load_queries<NR>(a, ro_s, seg_at(prefix, B, x0, x1).b, g, smem + lay.off_q, threadIdx.x,
                             SOFT_THREADS + Q_THREADS);
            asm volatile("bar.sync %0, %1;" ::"n"(BAR_Q), "n"(SOFT_THREADS + Q_THREADS) : "memory");
        }
        int n = 0;   // steps done
        bool ok = true;
        for (int x = x0; ok && x < x1;) {
            const Seg sg = seg_at(prefix, B, x, x1);
            x += sg.n;
            const int b = sg.b, n_steps = (sg.n + 1) / 2;
            // tokens relative to the segment: new rows start at new_rel, the
            // segment's tiles end at seg_end; row rr sees t < new_rel + r0 + rr % k + 1
            // but not the new rows of other tasks before its own
            const int new_rel = seqs[b].y - sg.t_a * TT, seg_end = sg.n * TT;
            const int j_first = group_of(cuts, n_grp, sg.xp);
            const int j_last = group_of(cuts, n_grp, sg.xp + sg.nt - 1);
            const bool whole = j_first == j_last;
            float l[HC];
#pragma unroll
            for (int j = 0; j < HC; ++j) l[j] = 0.f;
#pragma unroll 1
            for (int i = 0; i < n_steps; ++i, ++n) {
                const uint32_t s_col = (uint32_t)(n & 1) * S_COLS;
                // warp-uniform verdicts: the TMEM loads are warp-collective
                if (!__all_sync(0xffffffffu, mbar_wait(&bars->s_full[n & 1], (uint32_t)(n >> 1) & 1, abort)))
                    ok = false;
                tc_fence_after();
                const int t = i * STEP + tok;
                const bool masked = (i + 1) * STEP > min(new_rel, seg_end);  // uniform
                float sv[NC][W];
                auto scores = [&](int c, float (&s)[W]) {
                    tmem_ldw<W>(lane_base + s_col + c * W, s);
                    if (masked) {
#pragma unroll
                        for (int j = 0; j < W; ++j) {
                            const int rr = cb + c * W + j;
                            if (t >= seg_end || t >= new_rel + a.r0 + rk_s[rr] + 1 ||
                                (t >= new_rel && t < new_rel + lo_s[rr]))
                                s[j] = -INFINITY;
                        }
                    }
                };
#pragma unroll
                for (int c = 0; c < NC; ++c) scores(c, sv[c]);
                // does some row's max move?  (always on the segment's first step)
                bool grow = i == 0;
                if (i > 0) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        float(&s)[W] = sv[c];
#pragma unroll
                        for (int j4 = 0; j4 < W; j4 += 4) {
                            const float4 m4 = *(const float4 *)(mt_s + cb + c * W + j4);
                            grow = grow || s[j4] > m4.x || s[j4 + 1] > m4.y || s[j4 + 2] > m4.z || s[j4 + 3] > m4.w;
                        }
                    }
                }
                // one verdict for all warps; a timed-out one ends the segment for all
                const bool slow = soft_any(grow || !ok);
                bool pv_waited = false;
                if (slow) {
                    if (soft_any(!ok)) {
                        ok = false;
                        break;
                    }
                    // row maxima of the step; a row's max moves when it grows by more
                    // than RESCALE_LOG2 (or from nothing)
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        float s[W];
#pragma unroll
                        for (int j = 0; j < W; ++j) s[j] = sv[c][j];
                        const float v = lane_reduce<W, OpMax>(s, lane);
                        if (lane % (32 / W) == 0) red_s[wq * 128 + cb + c * W + lane / (32 / W)] = v;
                    }
                    soft_sync();
                    if (threadIdx.x < NR) {
                        const int rr = threadIdx.x;
                        const float mt = fmaxf(fmaxf(red_s[rr], red_s[128 + rr]), fmaxf(red_s[256 + rr], red_s[384 + rr]));
                        const float m = i == 0 ? -INFINITY : m_s[rr];
                        const bool up = mt > m + RESCALE_LOG2 || (m == -INFINITY && mt != -INFINITY);
                        const float mn = up ? mt : m;
                        al_s[rr] = up ? (m == -INFINITY ? 0.f : fast_exp2(m - mn)) : 1.f;
                        m_s[rr] = mn;
                        mt_s[rr] = mn + RESCALE_LOG2;
                        nm_s[rr] = mn == -INFINITY ? 0.f : -mn;
                    }
                    soft_sync();
                    if (i > 0) {
                        // O of the segment so far: complete once PV of the last step is
                        ok = __all_sync(0xffffffffu, mbar_wait(&bars->pv_done, (uint32_t)(n - 1) & 1, abort));
                        pv_waited = true;
                        tc_fence_after();
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            float o[W];
                            tmem_ldw<W>(lane_base + O_COL + c * W, o);
#pragma unroll
                            for (int j = 0; j < W; ++j) {
                                const float al = al_s[cb + c * W + j];
                                o[j] *= al;
                                l[c * W + j] *= al;
                            }
                            tmem_stw<W>(lane_base + O_COL + c * W, o);
                        }
                    }
                }
                // P of the previous step has been read
                if (n > 0 && !pv_waited)
                    ok = __all_sync(0xffffffffu, mbar_wait(&bars->pv_done, (uint32_t)(n - 1) & 1, abort));
                uint8_t *prow = smem + lay.off_p + (tok >> 3) * 1024 + (tok & 7) * 128;
                const bool with_lo = i == 0 && has_lo(sg);  // uniform
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    float(&s)[W] = sv[c];
#pragma unroll
                    for (int j8 = 0; j8 < W; j8 += 8) {
                        uint32_t pk[4], lo[4];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int j = j8 + 4 * h, cj = c * W + j;
                            const float4 m4 = *(const float4 *)(nm_s + cb + cj);
                            float p0, p1, p2, p3;
                            add2(p0, p1, s[j], s[j + 1], m4.x, m4.y);
                            add2(p2, p3, s[j + 2], s[j + 3], m4.z, m4.w);
                            p0 = fast_exp2(p0);
                            p1 = fast_exp2(p1);
                            p2 = fast_exp2(p2);
                            p3 = fast_exp2(p3);
                            const uint32_t u0 = pack_bf16(p0, p1), u1 = pack_bf16(p2, p3);
                            add2(l[cj], l[cj + 1], l[cj], l[cj + 1], __uint_as_float(u0 << 16),
                                 __uint_as_float(u0 & 0xffff0000u));
                            add2(l[cj + 2], l[cj + 3], l[cj + 2], l[cj + 3], __uint_as_float(u1 << 16),
                                 __uint_as_float(u1 & 0xffff0000u));
                            pk[2 * h] = u0;
                            pk[2 * h + 1] = u1;
                            if (LO_IN_LINE && with_lo) {
                                const float e0 = p0 - __uint_as_float(u0 << 16);
                                const float e1 = p1 - __uint_as_float(u0 & 0xffff0000u);
                                const float e2 = p2 - __uint_as_float(u1 << 16);
                                const float e3 = p3 - __uint_as_float(u1 & 0xffff0000u);
                                add2(l[cj], l[cj + 1], l[cj], l[cj + 1], e0, e1);
                                add2(l[cj + 2], l[cj + 3], l[cj + 2], l[cj + 3], e2, e3);
                                lo[2 * h] = pack_bf16(e0, e1);
                                lo[2 * h + 1] = pack_bf16(e2, e3);
                            }
                        }
                        const int c16 = (cb + c * W + j8) >> 3;  // 16-byte chunk of the line
                        st_shared_v4(prow + ((c16 ^ (tok & 7)) << 4), pk[0], pk[1], pk[2], pk[3]);
                        if (LO_IN_LINE && with_lo)
                            st_shared_v4(prow + (((c16 + 4) ^ (tok & 7)) << 4), lo[0], lo[1], lo[2], lo[3]);
                    }
                }
                if (!LO_IN_LINE && with_lo) {
                    // the lo plane in a pass of its own, in which the exponentials are formed
                    // again (in the one above its values do not fit the registers: 140 bytes
                    // of spills at 64 rows); every step takes the next of the nk K slots
                    uint8_t *lrow = prow + (lay.off_k - lay.off_p) + n % lay.nk * SLOT;
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
#pragma unroll
                        for (int j8 = 0; j8 < W; j8 += 8) {
                            const float *nm = nm_s + cb + c * W + j8;
                            float e[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const float p = fast_exp2(sv[c][j8 + j] + nm[j]);
                                e[j] = p - __bfloat162float(__float2bfloat16_rn(p));
                                l[c * W + j8 + j] += e[j];
                            }
                            const int c16 = (cb + c * W + j8) >> 3;
                            st_shared_v4(lrow + ((c16 ^ (tok & 7)) << 4), pack_bf16(e[0], e[1]), pack_bf16(e[2], e[3]),
                                         pack_bf16(e[4], e[5]), pack_bf16(e[6], e[7]));
                        }
                    }
                }
                fence_proxy_async();
                tc_fence_before();
                mbar_arrive(&bars->p_full);
            }
            if (soft_any(!ok)) {
                ok = false;
                break;
            }

            // ---- epilogue: row sums over the tokens, then O^T (thread = dim)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                float s[W];
#pragma unroll
                for (int j = 0; j < W; ++j) s[j] = l[c * W + j];
                const float v = lane_reduce<W, OpSum>(s, lane);
                if (lane % (32 / W) == 0) red_s[wq * 128 + cb + c * W + lane / (32 / W)] = v;
            }
            soft_sync();
            const size_t slot = ((size_t)grp + b) * Hkv + g;
            if (threadIdx.x < R) {
                const int rr = threadIdx.x;
                const float ls = (red_s[rr] + red_s[128 + rr]) + (red_s[256 + rr] + red_s[384 + rr]);
                al_s[rr] = whole ? (ls > 0.f ? 1.f / ls : 0.f) : 1.f;
                if (!whole) *(float2 *)(a.part_ml + (slot * R + rr) * 2) = make_float2(m_s[rr], ls);
            }
            ok = mbar_wait(&bars->pv_done, (uint32_t)(n - 1) & 1, abort);
            ok = !soft_any(!ok);  // (also orders al_s)
            if (!ok) break;
            tc_fence_after();
            // O^T through the idle P buffer, EC rows of each group at a time: a thread
            // then stores four consecutive dims, a warp one row.  (Rolled loops: this
            // code is cold at a segment's end, and each line of it that is not in the
            // instruction cache costs a round trip behind the K/V stream.)
            const size_t out0 = ((size_t)b * k * a.Hq + g * a.G) * DH;  // + ro_s[row] DH
            float *po = a.part_o + slot * R * DH;
            float *stage = (float *)(smem + lay.off_p) + (warp >> 2) * (EC * DH);
#pragma unroll 1
            for (int c0 = 0; c0 < HC; c0 += EC) {
                float o[EC];
                tmem_ldw<EC>(lane_base + O_COL + c0, o);
#pragma unroll
                for (int j = 0; j < EC; ++j) stage[j * DH + tok] = o[j];
                asm volatile("bar.sync %0, 128;" ::"r"(BAR_SOFT + 1 + (warp >> 2)) : "memory");
#pragma unroll 1
                for (int j = wq; j < EC; j += 4) {
                    const int rr = cb + c0 + j;
                    if (rr >= R) break;
                    const float4 v = *(const float4 *)(stage + j * DH + lane * 4);
                    const float w = al_s[rr];
                    if (whole)
                        act_store4(a.out, out0 + (size_t)ro_s[rr] * DH + lane * 4,
                                   make_float4(v.x * w, v.y * w, v.z * w, v.w * w));
                    else
                        *(float4 *)(po + (size_t)rr * DH + lane * 4) = v;
                }
                asm volatile("bar.sync %0, 128;" ::"r"(BAR_SOFT + 1 + (warp >> 2)) : "memory");
            }
            tc_fence_before();
            if (!whole && !a.tc_merge_kernel) {
                // count this segment; the one completing the pair merges all of its
                // partials, in segment order (the result does not depend on which
                // CTA finishes last)
                const int n_seg = j_last - j_first + 1;
                const int staged_max = min(kStagedSegs, (lay.off_v + lay.nv * SLOT - lay.off_q) / (R * (DH * 4 + 8)));
                soft_sync();  // the partial is written ...
                if (threadIdx.x == 0) {
                    __threadfence();  // ... and visible before it is counted
                    const int last = atomicAdd(a.counters + b * Hkv + g, 1) == n_seg - 1;
                    if (last) a.counters[b * Hkv + g] = 0;  // ready for the next launch
                    bars->merge_now = last;
                }
                soft_sync();
                const size_t slot0 = ((size_t)j_first + b) * Hkv + g;  // segment e: + e Hkv
                if (bars->merge_now && x >= x1 && n_seg <= staged_max) {
                    // the share's last segment: merged by the whole CTA once every
                    // role is done, through the idle shared memory
                    if (threadIdx.x == 0) {
                        bars->fm_b = b;
                        bars->fm_nseg = n_seg;
                        bars->fm_slot0 = (long long)slot0;
                        bars->fm_merge = 1;
                    }
                } else if (bars->merge_now) {
                    __threadfence();  // the other segments' partials are read after their count
#pragma unroll 1
                    for (int r0_ = 4 * (warp >> 2); r0_ < R; r0_ += 8) {  // the groups take rows in turn
                        float acc[4] = {0.f, 0.f, 0.f, 0.f}, ll[4] = {0.f, 0.f, 0.f, 0.f};
                        float mm[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll 1
                        for (int e0 = 0; e0 < n_seg; e0 += 2) {
                            float2 ml[2][4];
                            float ov[2][4];
#pragma unroll
                            for (int e = 0; e < 2; ++e)  // the loads of both segments in flight together
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    const bool in = e0 + e < n_seg && r0_ + q < R;
                                    const size_t at = (slot0 + (size_t)(e0 + e) * Hkv) * R + r0_ + q;
                                    ml[e][q] = in ? __ldcg((const float2 *)(a.part_ml + at * 2))
                                                  : make_float2(-INFINITY, 0.f);
                                    ov[e][q] = in ? __ldcg(a.part_o + at * DH + tok) : 0.f;
                                }
#pragma unroll
                            for (int e = 0; e < 2; ++e)
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    const float mn = fmaxf(mm[q], ml[e][q].x);
                                    if (mn == -INFINITY) continue;
                                    const float al = mm[q] == -INFINITY ? 0.f : exp2f(mm[q] - mn);
                                    const float wt = ml[e][q].x == -INFINITY ? 0.f : exp2f(ml[e][q].x - mn);
                                    ll[q] = ll[q] * al + wt * ml[e][q].y;
                                    acc[q] = acc[q] * al + wt * ov[e][q];
                                    mm[q] = mn;
                                }
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (r0_ + q < R)
                                act_store(a.out, out0 + (size_t)ro_s[r0_ + q] * DH + tok,
                                          acc[q] * (ll[q] > 0.f ? 1.f / ll[q] : 0.f));
                    }
                }
            }
        }
    }
    // every MMA must be finished before TMEM and shared memory go away
    mbar_wait_drain(&bars->fin, 0);
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort && a.status) atomicOr(a.status, SP_DEV_TIMEOUT);
    if (bars->fm_merge)
        staged_merge<THREADS>(a, smem + lay.off_q, bars->fm_b, g, bars->fm_nseg, (size_t)bars->fm_slot0, !*abort);
    // the cache stream of the slower CTAs leaves DRAM time for the next
    // projection's weights: this CTA's share goes to L2 (the K/V tiles were
    // loaded evict-first, so the weights stay)
    if (threadIdx.x == 0 && a.l2_next)
        prefetch_l2_share(a.l2_next, a.l2_next_bytes, blockIdx.x, gridDim.x);
    if (warp == MMA_W) tmem_dealloc(tmem, TMEM_COLS);
}

// Whether this kernel takes the call, and its shared memory: two query buffers, P,
// then the rings (K in front of V).
// Its cost grows with the query rows (scores a thread, the queries' and P's
// shared memory) where the queries-on-M kernel of sp_attn_tc.cu pays for 128 rows
// always, and most so for short sequences, whose steps are all first ones.  Lengths
// are known on the device only and max_seq_len may be far above them, so the rule
// uses the rows and the batch: it takes what no length makes more than 2 % slower.
// Whole calls of the 8B layer in us, that kernel -> this one, paged, per-sequence rows,
// 120 / 500 / 2000 / 4000 tokens (152 SMs, 8 kv heads):
//   up to 32 rows: everywhere (attention alone, B = 200, L = 100..300: 93 -> 56);
//   48 rows: B = 128 586 -> 583, 614 -> 593, 728 -> 705, 861 -> 847; B = 64 309 -> 311,
//     327 -> 317, 379 -> 361, 465 -> 442; but B = 16, 300 to 1700 tokens 174 -> 179;
//   64 rows: B = 128 715 -> 730, 747 -> 737, 854 -> 850, 990 -> 980; B = 64 378 -> 376,
//     397 -> 399, 442 -> 435, 510 -> 507; but B = 32 222 -> 227, 231 -> 236, 264 -> 263,
//     302 -> 297, and B = 16, 300 to 1700 tokens 170 -> 188; with hi + lo queries
//     B = 128 682 -> 670 at 60 tokens, 722 -> 711 at 300, 753 -> 746 at 1000;
//   80 rows: B = 128 968 -> 982, 1003 -> 1000, 1104 -> 1097, 1232 -> 1245.
bool tok_wins(const AttnArgs &a, int R16) {
    return R16 <= 32 || (R16 <= 64 && (long long)a.B * a.Hkv >= 3ll * a.tc_ctas);
}

bool tok_layout(const AttnArgs &a, TokLayout *lay) {
    const int R16 = (a.R + 15) / 16 * 16;
    if (!tok_wins(a, R16)) return false;
    const int tab = ((a.B + 2) & ~1) * 4 + a.B * 8;
    const int front = (OFF_TAB + tab + 1023) & ~1023;
    const int q = R16 * 256 * (a.tc_q_plain ? 1 : 2), p = STEP * 128;
    const int room = SMEM_MAX - 1024 - front - p;
    int slots = (room - 2 * q) / SLOT;
    if (slots < 4) return false;  // (more than 48 rows in batches with large tables)
    lay->r16 = R16;
    if (slots > 2 * MAX_SLOTS) slots = 2 * MAX_SLOTS;
    lay->nk = slots / 2;
    lay->nv = slots - lay->nk;
    lay->q_bytes = q;
    lay->off_q = front;
    lay->off_p = front + 2 * q;
    lay->off_k = lay->off_p + p;
    lay->off_v = lay->off_k + lay->nk * SLOT;
    lay->smem = lay->off_v + lay->nv * SLOT + 1024;
    return true;
}

template <int NR>
cudaError_t launch_tok(const AttnArgs &a, const TokLayout &lay, const CUtensorMap &mk, const CUtensorMap &mv,
                       cudaStream_t st) {
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(attn_tok_kernel<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             SMEM_MAX);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    return launch_k(attn_tok_kernel<NR>, dim3(a.tc_ctas), dim3(THREADS), (size_t)lay.smem, st, mk, mv, a, lay);
}

}  // namespace

bool attention_tok_supported(const AttnArgs &a) {
    TokLayout lay;
    return tok_layout(a, &lay);
}

cudaError_t launch_attention_tok(const AttnArgs &a, const CUtensorMap &map_k, const CUtensorMap &map_v,
                                 cudaStream_t st) {
    TokLayout lay;
    if (!tok_layout(a, &lay)) return cudaErrorInvalidValue;
    switch (lay.r16) {
    case 16: return launch_tok<16>(a, lay, map_k, map_v, st);
    case 32: return launch_tok<32>(a, lay, map_k, map_v, st);
    case 48: return launch_tok<48>(a, lay, map_k, map_v, st);
    case 64: return launch_tok<64>(a, lay, map_k, map_v, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace sp
