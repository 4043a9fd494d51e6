// Shared by the tensor-core attention kernels: the 64-token tile list, its cuts
// into per-CTA shares, the shared-memory tile layout and the merge of a pair's
// partials at a kernel's end.
#pragma once

#include "sp_common.cuh"
#include "sp_sm100.cuh"

namespace sp {

namespace {

using namespace sm100;

constexpr int DH = 128;
constexpr int TT = 64;                         // tokens per tile of the list
constexpr uint32_t GROUP_STRIDE = 2048;        // 8-token groups
constexpr uint32_t HALF_STRIDE = 1024;         // 64-dim halves within a group
constexpr int MAX_B = 2048;                    // sequences per launch (tile prefix in smem)
constexpr int MAX_GRP = 256;                   // groups (cuts table in smem)
constexpr float RESCALE_LOG2 = 8.f;            // tolerate p <= 2^8 before rescaling O
constexpr int kStagedSegs = 4;                 // most partials merged through the idle ring

// byte offset of 16-byte chunk c16 (0..15, 8 dims each) of token row `row` in a K or
// V slot (one tile of 64 rows, or a step of two: 0..127)
__device__ __forceinline__ uint32_t kv_off(int row, int c16) {
    return (uint32_t)((row >> 3) * GROUP_STRIDE + (c16 >> 3) * HALF_STRIDE + (row & 7) * 128 +
                      (((c16 & 7) ^ (row & 7)) << 4));
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&v);
}

__device__ __forceinline__ void named_sync(int id, int n) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// A CTA's piece of one sequence: tiles [t_a, t_a + n) of sequence b, which
// starts at tile xp of the list and has nt tiles.
struct Seg {
    int b, t_a, n, nt, xp;
};

// Segment holding tile x (x < x_end <= T), clipped at x_end.  prefix[b] is the
// first tile of sequence b; it grows strictly (every sequence has a tile for
// its new keys).
__device__ __forceinline__ Seg seg_at(const int *prefix, int B, int x, int x_end) {
    int lo = 0, hi = B - 1;
#pragma unroll 1
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= x) lo = mid;
        else hi = mid - 1;
    }
    Seg s;
    s.b = lo;
    s.xp = prefix[lo];
    s.nt = prefix[lo + 1] - s.xp;
    s.t_a = x - s.xp;
    s.n = min(s.nt - s.t_a, x_end - x);
    return s;
}

// The shares.  A segment (a share's piece of one sequence) costs the consumers a
// pipeline drain, the epilogue and the next queries' load, worth about `c` tiles
// of streaming, so the shares balance tiles + c per segment: every sequence b
// gets c virtual tiles in front of its own, the virtual list (T + c B long) is cut
// evenly, and a cut that lands in a sequence's virtual part moves to that
// sequence's first tile.  c falls back to 0 in that list when a share is shorter
// than c + 1 virtual tiles.  Two plans are made of those cuts:
//   near: a cut within min(share / 4, SNAP) tiles of a sequence start moves onto
//     it (a short piece of a sequence would pay a whole segment);
//   whole: a cut within half a virtual share of a sequence start moves onto it, so
//     that sequences shorter than a share are never split.
// and the one whose largest share is smaller is taken, counting its tiles, c per
// segment and MERGE_COST for each of its ends inside a sequence (a partial to write
// and to merge; nothing where a kernel of its own merges): near where sequences are
// longer or many more than the shares, whole where they are about as many.  The cuts
// never decrease; two may meet at a sequence start, and the share between them is
// then empty (every other one for four sequences of 15 tiles in eight shares).
// Attention step (8 kv heads, 152 SMs) with near alone -> the choice, paged, 96 query
// rows: 16 x 500 tokens 44.5 -> 22.3 us, 16 x 1000 47.4 -> 26.8; 16 rows, 16 x 1000:
// 20.2 -> 17.5.  MERGE_COST 0 and 4, 8 sequences of 60 to 203 tokens, 16 / 32 / 96
// rows: 23.6 / 29.7 / 42.0 and 19.5 / 21.5 / 29.7 us.  Of 2160 batches (6 to 32
// sequences of 36 to 6800 tokens, 16 to 128 rows) the choice took on average 4.4 % more
// than the better plan without it, 0.7 % with 4 (2: 1.4, 8: 0.9).
constexpr int SNAP = 4;
constexpr int MERGE_COST = 4;
constexpr int PLAN_THREADS = 128;
constexpr int PLAN_BAR = 15;  // named barrier of the planning warps

// Shares of T tiles in B sequences: none shorter than min_tiles on average, but
// one for each sequence as far as the groups go (4 x 200 tokens, 96 rows:
// 28.6 us in two shares, 16.1 in four).
__device__ __forceinline__ int share_count(int groups, int T, int B, int min_tiles) {
    return min(groups, max(ceil_div(T, max(1, min_tiles)), B));
}

// A cut: tile x of the list, in sequence s (B at the list's end).
struct Cut {
    int x, s;
};

__device__ __forceinline__ void share_cut(const int *prefix, int B, int T, int n, int j, int c, Cut *near, Cut *whole) {
    if (j <= 0 || j >= n) {
        near->x = whole->x = j <= 0 ? 0 : T;
        near->s = whole->s = j <= 0 ? 0 : B;
        return;
    }
    if ((long long)T + (long long)c * B < (long long)n * (c + 1)) c = 0;
    const unsigned V = (unsigned)T + c * B;  // < 2^31 + 2^21: c <= 1024, B <= MAX_B
    const unsigned share = V / n;
    const unsigned v = j * share + j * (V - share * n) / n;  // floor(j V / n)
    int lo = 0, hi = B - 1;  // last sequence whose virtual start vpre(b) = prefix[b] + c b is <= v
#pragma unroll 1
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((unsigned)prefix[mid] + c * mid <= v) lo = mid;
        else hi = mid - 1;
    }
    const int p0 = prefix[lo], p1 = prefix[lo + 1];
    const int off = (int)(v - p0 - c * lo);
    const int x = off < c ? p0 : min(p0 + off - c, p1 - 1);
    const int d0 = x - p0, d1 = p1 - x, delta = min(T / n / 4, SNAP);
    const bool to1 = d1 < d0;
    *near = (to1 ? d1 : d0) <= delta ? Cut{to1 ? p1 : p0, lo + to1} : Cut{x, lo};
    const int half = (int)((share + 1) / 2);
    const int e0 = max(off - c, 0), e1 = (int)((unsigned)p1 + c * (lo + 1) - v);
    *whole = e0 <= e1 && e0 <= half ? Cut{p0, lo} : e1 <= half ? Cut{p1, lo + 1} : Cut{x, lo};
}

// Tiles, segments and ends inside a sequence (m each) of the share [a, b).
__device__ __forceinline__ int share_cost(const int *prefix, Cut a, Cut b, int c, int m) {
    if (b.x <= a.x) return 0;
    const int cut_a = a.x != prefix[a.s], cut_b = b.x != prefix[b.s];
    return b.x - a.x + c * (b.s + cut_b - a.s) + m * (cut_a + cut_b);
}

// cuts[0 .. n] by the first PLAN_THREADS threads; worst: two ints per warp.  A
// warp's lane 31 holds the next warp's first cut.  The caller synchronises.
__device__ __forceinline__ void build_cuts(const AttnArgs &args, const int *prefix, int T, int n, int *cuts,
                                           int *worst) {
    constexpr int PER = 31 * (PLAN_THREADS / 32);
    const int B = args.B, c = args.tc_seg_cost, m = args.tc_merge_kernel ? 0 : MERGE_COST;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Cut near, whole;
    int m0 = 0, m1 = 0;
#pragma unroll 1
    for (int j0 = warp * 31; j0 < n; j0 += PER) {
        const int j = min(j0 + lane, n);
        share_cut(prefix, B, T, n, j, c, &near, &whole);
        Cut b0, b1;
        b0.x = __shfl_down_sync(0xffffffffu, near.x, 1);
        b0.s = __shfl_down_sync(0xffffffffu, near.s, 1);
        b1.x = __shfl_down_sync(0xffffffffu, whole.x, 1);
        b1.s = __shfl_down_sync(0xffffffffu, whole.s, 1);
        if (lane < 31 && j < n) {
            m0 = max(m0, share_cost(prefix, near, b0, c, m));
            m1 = max(m1, share_cost(prefix, whole, b1, c, m));
        }
    }
    m0 = __reduce_max_sync(0xffffffffu, m0);
    m1 = __reduce_max_sync(0xffffffffu, m1);
    if (n > 31) {  // (else the first warp has them all)
        if (lane == 0) {
            worst[2 * warp] = m0;
            worst[2 * warp + 1] = m1;
        }
        named_sync(PLAN_BAR, PLAN_THREADS);
#pragma unroll
        for (int w = 0; w < PLAN_THREADS / 32; ++w) {
            m0 = max(m0, worst[2 * w]);
            m1 = max(m1, worst[2 * w + 1]);
        }
    }
#pragma unroll 1
    for (int j0 = warp * 31; j0 < n; j0 += PER) {
        const int j = min(j0 + lane, n);
        if (n > PER) share_cut(prefix, B, T, n, j, c, &near, &whole);  // (else still in registers)
        cuts[j] = m1 < m0 ? whole.x : near.x;
    }
}

// Group whose share holds tile x (0 <= x < T): the largest j with cuts[j] <= x.
__device__ __forceinline__ int group_of(const int *cuts, int n, int x) {
    int lo = 0, hi = n - 1;
#pragma unroll 1
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cuts[mid] <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The tile list: prefix[b] = sum_{b' < b} ceil((L_b' + new rows) / TT), and each
// sequence's cache id and length, resolved once (seqs, when given).  By all
// THREADS threads; wsum holds one int per warp.
template <int THREADS>
__device__ __forceinline__ void build_prefix(const AttnArgs &a, int *prefix, int2 *seqs, int *wsum,
                                             int *status) {
    const int B = a.B, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int per = (B + THREADS - 1) / THREADS;
    const int b0 = min(B, (int)threadIdx.x * per), b1 = min(B, b0 + per);
    int sum = 0;
#pragma unroll 1
    for (int bb = b0; bb < b1; ++bb) {
        const SeqRef sq = resolve_seq(a.seq_ids, a.seq_lens, a.lens_by_batch, bb, a.kv.n_seqs,
                                      a.max_seq_len, status);
        if (seqs) seqs[bb] = make_int2(sq.sid, sq.len);
        const int v = ceil_div(sq.len + a.r0 + a.k, TT);
        prefix[bb] = v;
        sum += v;
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int run = incl - sum;
#pragma unroll 1
    for (int w = 0; w < warp; ++w) run += wsum[w];
#pragma unroll 1
    for (int bb = b0; bb < b1; ++bb) {
        const int v = prefix[bb];
        prefix[bb] = run;
        run += v;
    }
    if (threadIdx.x == 0) {
        int tot = 0;
#pragma unroll 1
        for (int w = 0; w < THREADS / 32; ++w) tot += wsum[w];
        prefix[B] = tot;
    }
    __syncthreads();
}

// Merge of the pair completed by this share's last segment, by the whole
// CTA: every partial of the pair lands in the idle K/V ring in one
// round of cp.async copies (O of segment e as [e][row][dh], then (max,
// sum) as [e][row]), then thread (row, c) combines 16-byte units c, c + 8,
// c + 16, c + 24 of its row in segment order, in the arithmetic of the attention
// kernels' own merge through registers, so the bits do not depend on which path ran.
// Shared-memory reads are conflict-free and eight lanes store 64
// contiguous bytes per plane.  Loads through registers would need a
// dependent round trip per two segments, each waiting behind the other
// SMs' cache streams.
// (Run by all THREADS threads; good: every wait of the kernel was served; uniform
// over the CTA.)
template <int THREADS>
__device__ __forceinline__ void staged_merge(const AttnArgs &a, uint8_t *stage, int b, int g, int n_seg,
                                             size_t slot0, bool good) {
    const int R = a.R, k = a.k, Hkv = a.Hkv;
    __threadfence();            // the other segments' partials are read after their count
    float2 *st_ml = (float2 *)(stage + (size_t)n_seg * R * DH * 4);
    const int units = R * (DH / 4);  // 16-byte units of one segment's O
#pragma unroll 4
    for (int idx = threadIdx.x; idx < n_seg * units; idx += THREADS) {
        const int e = idx / units, rem = idx - e * units;
        cp_async16(stage + (size_t)idx * 16, a.part_o + (slot0 + (size_t)e * Hkv) * R * DH + (size_t)rem * 4);
    }
#pragma unroll 1
    for (int idx = threadIdx.x; idx < n_seg * R; idx += THREADS) {
        const int e = idx / R, rr = idx - e * R;
        st_ml[idx] = __ldcg((const float2 *)(a.part_ml + ((slot0 + (size_t)e * Hkv) * R + rr) * 2));
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (good) {
#pragma unroll 1
        for (int item = threadIdx.x; item < R * 8; item += THREADS) {
            const int rr = item >> 3, c = item & 7;
            float2 ml[kStagedSegs];
            float4 ov[kStagedSegs][4];
#pragma unroll
            for (int e = 0; e < kStagedSegs; ++e) {
                const int ee = min(e, n_seg - 1);
                ml[e] = st_ml[ee * R + rr];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    ov[e][q] = ld_shared_v4f(stage + (((size_t)ee * R + rr) * (DH / 4) + c + 8 * q) * 16);
            }
            float acc[16], mm = -INFINITY, ll = 0.f;
#pragma unroll
            for (int j = 0; j < 16; ++j) acc[j] = 0.f;
#pragma unroll
            for (int e = 0; e < kStagedSegs; ++e) {
                if (e >= n_seg) break;
                const float mn = fmaxf(mm, ml[e].x);
                if (mn == -INFINITY) continue;
                const float al = mm == -INFINITY ? 0.f : exp2f(mm - mn);
                const float wt = ml[e].x == -INFINITY ? 0.f : exp2f(ml[e].x - mn);
                ll = ll * al + wt * ml[e].y;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    acc[4 * q] = acc[4 * q] * al + wt * ov[e][q].x;
                    acc[4 * q + 1] = acc[4 * q + 1] * al + wt * ov[e][q].y;
                    acc[4 * q + 2] = acc[4 * q + 2] * al + wt * ov[e][q].z;
                    acc[4 * q + 3] = acc[4 * q + 3] * al + wt * ov[e][q].w;
                }
                mm = mn;
            }
            const float il = ll > 0.f ? 1.f / ll : 0.f;
            const int hl = rr / k, r = rr - hl * k;
            const size_t o0 = (((size_t)b * k + r) * a.Hq + g * a.G + hl) * DH;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                act_store4(a.out, o0 + (size_t)(c + 8 * q) * 4,
                           make_float4(acc[4 * q] * il, acc[4 * q + 1] * il, acc[4 * q + 2] * il,
                                       acc[4 * q + 3] * il));
        }
    }
}

}  // namespace

}  // namespace sp
