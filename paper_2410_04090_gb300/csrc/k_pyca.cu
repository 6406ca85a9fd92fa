// Pyramidal Feature Aggregation, steps 3 and the aggregation (Sec. II-C-2).
//
// k_pfa_nms       one CTA per segment = (image, level, cell row), or one warp
//                 per segment (four per CTA) when every segment of the batch
//                 has at most 96 slots.  Each
//                 culled corner reads its own packed (K_l, K_r) and those of
//                 the q x q window around its s0 projection from the score map
//                 filled by the detection kernel, and is suppressed when a
//                 neighbour dominates it (sparse NMS: only occupied pixels are
//                 looked at).  Survivors are ranked by (y, x) inside the
//                 segment; segments of one level are already in y order.  A
//                 slot's coordinates, priority and rank go to the next kernel
//                 as one 16-byte record.
// k_pfa_finalize  a cluster of CTAs per image: prefix-sums the segment counts
//                 into canonical positions (level, y, x), clears the score map
//                 entries it used, applies the keypoint cap by a radix select
//                 on (K_l, K_r, response) with canonical order breaking ties,
//                 and writes the compacted keypoint list.
#include "jslam_internal.h"

namespace jslam {

// Candidate i of a segment with key `key`: its level coordinates, packed x |
// y << 13 | level << 26, and response (the key's upper half).
__device__ __forceinline__ uint32_t slot_pos(const SegRec &R, uint32_t key, int i, int k)
{
    const uint32_t inidx = 0xFFFFu - (key & 0xFFFFu);
    const uint32_t row = R.cdiv ? __umulhi(inidx, R.cdiv) : inidx;  // inidx / c
    const uint32_t x = (uint32_t)(k == 1 ? i : i / k) * (uint32_t)R.c + (inidx - row * (uint32_t)R.c);
    return x | (((uint32_t)R.y0 + row) << 13) | ((uint32_t)R.level << 26);
}
__device__ __forceinline__ uint32_t pos_x(uint32_t p) { return p & 0x1FFFu; }
__device__ __forceinline__ uint32_t pos_y(uint32_t p) { return (p >> 13) & 0x1FFFu; }
// Order of a segment's corners by (y, x): the position without its level, rows first.
__device__ __forceinline__ uint32_t pos_order(uint32_t p) { return (pos_y(p) << 13) | pos_x(p); }

// Whether a neighbour's packed (K_l, K_r) suppresses a corner's.
__device__ __forceinline__ bool dominates(uint32_t n, uint32_t own, int rule)
{
    const uint32_t ql = n >> 16, qr = n & 0xFFFFu, kl = own >> 16, kr = own & 0xFFFFu;
    return rule == 0 ? (ql > kl && qr > kr) : (ql > kl || (ql == kl && qr > kr));
}

// The finalisation's view of a slot: packed position, X | Y << 16, the cap
// priority K_l << 27 | K_r << 12 | response, and the rank in the segment.
__device__ __forceinline__ uint4 slot_info(uint32_t pos, int X, int Y, uint32_t own, uint32_t key, int rank)
{
    return make_uint4(pos, (uint32_t)X | ((uint32_t)Y << 16), ((own >> 16) << 27) | ((own & 0xFFFFu) << 12) | (key >> 16),
                      (uint32_t)rank);
}

__global__ void __launch_bounds__(kNmsThreads) k_pfa_nms(const __grid_constant__ Batch b)
{
    __shared__ uint32_t sk[kMaxSegment];
    __shared__ int alive_total;
    const int seg = blockIdx.x;
    const SegRec &R = b.seg_rec[seg];
    const int k = b.prm.k, rad = b.prm.nms_rad, rule = b.prm.rule;
    const int m = R.m, base = R.slot, W0 = R.W0, H0 = R.H0;
    let_next();
    after_previous();
    if (m > kMaxSegment) {
        for (int i = threadIdx.x; i < m; i += kNmsThreads)
            b.slot_info[base + i] = slot_info(0u, 0, 0, 0u, 0u, kSlotEmpty);
        if (threadIdx.x == 0) { atomicOr(b.err, kErrSegment); b.seg_count[seg] = 0; }
        return;
    }
    if (threadIdx.x == 0) alive_total = 0;
    __syncthreads();
    int my_alive = 0;
    for (int i = threadIdx.x; i < m; i += kNmsThreads) {
        const uint32_t key = b.slots[base + i];
        uint32_t v = 0xFFFFFFFFu;
        uint4 info = slot_info(0u, 0, 0, 0u, 0u, kSlotEmpty);
        if (key) {
            const uint32_t p = slot_pos(R, key, i, k);
            const int X = __ldg(R.projx + pos_x(p)), Y = __ldg(R.projy + pos_y(p));
            const uint32_t own = R.map[(size_t)Y * W0 + X];
            bool dom = false;
            for (int dy = -rad; dy <= rad; ++dy) {
                const int qy = Y + dy;
                if (qy < 0 || qy >= H0) continue;
                for (int dx = -rad; dx <= rad; ++dx) {
                    const int qx = X + dx;
                    if ((dx | dy) == 0 || qx < 0 || qx >= W0) continue;
                    const uint32_t w = R.map[(size_t)qy * W0 + qx];
                    if (w) dom |= dominates(w, own, rule);
                }
            }
            info = slot_info(p, X, Y, own, key, kSlotSuppressed);
            if (!dom) { v = pos_order(p); ++my_alive; }
        }
        b.slot_info[base + i] = info;
        sk[i] = v;
    }
    if (my_alive) atomicAdd(&alive_total, my_alive);
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += kNmsThreads) {
        const uint32_t v = sk[i];
        if (v == 0xFFFFFFFFu) continue;
        int rank = 0;
        for (int j = 0; j < m; ++j) rank += sk[j] < v;
        b.slot_info[base + i].w = (uint32_t)rank;
    }
    if (threadIdx.x == 0) b.seg_count[seg] = alive_total;
}

// The same per segment with one warp, for batches whose segments (cell rows:
// cells_x x k slots) all have at most 32 S slots: lane l takes slots l,
// l + 32, ..., and every step of their chains of dependent loads (slot ->
// projection -> own score and neighbours) is issued for all S slots before
// the next, so the chains overlap; a CTA of four warps takes four segments.
template <int S, int RAD>
__global__ void __launch_bounds__(kNmsThreads) k_pfa_nms_warp(const __grid_constant__ Batch b)
{
    __shared__ __align__(16) uint32_t sk[kNmsThreads / 32][32 * S];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int seg = blockIdx.x * (kNmsThreads / 32) + warp;
    let_next();
    if (seg >= b.n_segments) return;  // whole warps only
    const SegRec R = b.seg_rec[seg];
    const int k = b.prm.k, rule = b.prm.rule;
    const int m = R.m, base = R.slot, W0 = R.W0, H0 = R.H0;
    after_previous();
    if (m > 32 * S) {  // the host launches this kernel only when no segment is wider
        for (int i = lane; i < m; i += 32) b.slot_info[base + i] = slot_info(0u, 0, 0, 0u, 0u, kSlotEmpty);
        if (lane == 0) { atomicOr(b.err, kErrSegment); b.seg_count[seg] = 0; }
        return;
    }
    uint32_t key[S], own[S], pos[S];
    int X[S], Y[S];
    bool dom[S];
#pragma unroll
    for (int q = 0; q < S; ++q) key[q] = lane + 32 * q < m ? b.slots[base + lane + 32 * q] : 0u;
#pragma unroll
    for (int q = 0; q < S; ++q) {
        X[q] = Y[q] = 0;
        pos[q] = 0u;
        if (key[q]) {
            pos[q] = slot_pos(R, key[q], lane + 32 * q, k);
            X[q] = __ldg(R.projx + pos_x(pos[q]));
            Y[q] = __ldg(R.projy + pos_y(pos[q]));
        }
    }
#pragma unroll
    for (int q = 0; q < S; ++q) {
        own[q] = key[q] ? R.map[(size_t)Y[q] * W0 + X[q]] : 0u;
        dom[q] = false;
    }
    // a window row's loads (of all slots) are in flight together, for the
    // 3 x 3 window all eight neighbours'
    constexpr int kSide = 2 * RAD + 1, kRows = RAD == 1 ? 3 : 1;
#pragma unroll
    for (int dy0 = -RAD; dy0 <= RAD; dy0 += kRows) {
        uint32_t w[kRows][kSide][S];
#pragma unroll
        for (int r = 0; r < kRows; ++r)
#pragma unroll
            for (int c = 0; c < kSide; ++c)
#pragma unroll
                for (int q = 0; q < S; ++q) {
                    const int dx = c - RAD, dy = dy0 + r, qx = X[q] + dx, qy = Y[q] + dy;
                    w[r][c][q] = (dx | dy) != 0 && key[q] && qx >= 0 && qx < W0 && qy >= 0 && qy < H0
                                     ? R.map[(size_t)qy * W0 + qx] : 0u;
                }
#pragma unroll
        for (int r = 0; r < kRows; ++r)
#pragma unroll
            for (int c = 0; c < kSide; ++c)
#pragma unroll
                for (int q = 0; q < S; ++q)
                    if (w[r][c][q]) dom[q] |= dominates(w[r][c][q], own[q], rule);
    }
    uint32_t v[S];
    int rank[S], alive = 0;
#pragma unroll
    for (int q = 0; q < S; ++q) {
        v[q] = 0xFFFFFFFFu;
        rank[q] = key[q] ? kSlotSuppressed : kSlotEmpty;
        if (key[q] && !dom[q]) { v[q] = pos_order(pos[q]); rank[q] = 0; ++alive; }
        sk[warp][lane + 32 * q] = v[q];
    }
    __syncwarp();
    // entries past the segment are never below a corner
    for (int j = 0; j < m; j += 4) {
        const uint4 o = *reinterpret_cast<const uint4 *>(&sk[warp][j]);
#pragma unroll
        for (int q = 0; q < S; ++q)
            if (rank[q] >= 0) rank[q] += (o.x < v[q]) + (o.y < v[q]) + (o.z < v[q]) + (o.w < v[q]);
    }
#pragma unroll
    for (int q = 0; q < S; ++q)
        if (lane + 32 * q < m)
            b.slot_info[base + lane + 32 * q] = slot_info(pos[q], X[q], Y[q], own[q], key[q], rank[q]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) alive += __shfl_xor_sync(0xFFFFFFFFu, alive, off);
    if (lane == 0) b.seg_count[seg] = alive;
}

template <int RAD>
static cudaError_t launch_nms_warp(const Batch &b, cudaStream_t stream)
{
    constexpr int per = kNmsThreads / 32;
    const int grid = (b.n_segments + per - 1) / per;
    const bool early = start_early(b);
    if (b.max_segment <= 32) return launch_if(early, k_pfa_nms_warp<1, RAD>, dim3(grid), dim3(kNmsThreads), 0, stream, b);
    if (b.max_segment <= 64) return launch_if(early, k_pfa_nms_warp<2, RAD>, dim3(grid), dim3(kNmsThreads), 0, stream, b);
    return launch_if(early, k_pfa_nms_warp<3, RAD>, dim3(grid), dim3(kNmsThreads), 0, stream, b);
}

cudaError_t launch_pfa_nms(const Batch &b, cudaStream_t stream)
{
    if (b.n_segments == 0) return cudaSuccess;
    if (b.nms_kernel == 1 || b.max_segment > 96)
        return launch_if(start_early(b), k_pfa_nms, dim3(b.n_segments), dim3(kNmsThreads), 0, stream, b);
    switch (b.prm.nms_rad) {
    case 0: return launch_nms_warp<0>(b, stream);
    case 1: return launch_nms_warp<1>(b, stream);
    case 2: return launch_nms_warp<2>(b, stream);
    default: return launch_nms_warp<3>(b, stream);
    }
}

// Exclusive block-wide prefix sum of v; *total receives the block sum.  `ws`
// (a word a warp) may be used again once every thread has passed another
// barrier.
template <int NT>
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *ws, uint32_t *total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    // every warp sums the warps' totals for itself: those before it, and all
    const uint32_t t = lane < NT / 32 ? ws[lane] : 0u;
    *total = __reduce_add_sync(0xFFFFFFFFu, t);
    return __reduce_add_sync(0xFFFFFFFFu, lane < w ? t : 0u) + x - v;
}

// The finalisation of one image by a cluster of CTAs (one to eight, see
// launch_pfa_finalize): the candidate slots and then the canonical positions
// are shared out over its CTAs, the histograms of the cap's radix select are
// summed through distributed shared memory, and a cluster barrier ends each
// phase: the slots' and those of the select's three passes.  A thread that sums
// the others' histograms also keeps what the CTAs before its own have of it, so
// the place of a CTA's first keypoint needs no barrier more.
//
// What bounds it: latency -- a chain of barriers and dependent reads whose
// data lie in L2; the bytes are few.  One CTA of 1024 threads an image left
// the chip idle for small batches.  Stage times, before and now (us): one
// 1920x1080 pair (16 000 slots an image) 96 and 25, one 1241x376 pair 31 and
// 18, 16 mixed pairs 98 and 27, 100 pairs of 1241x376 47 and 33 (29, 22, 33 and
// 37 with two barriers more, one of them for the row index that
// k_orient_desc makes now).

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Barrier over the cluster; global and shared writes before it are seen after it.
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// 16 bytes at the address of `p` (a shared object of this CTA) in CTA `rank` of the cluster.
__device__ __forceinline__ uint4 ld_cluster(const void *p, uint32_t rank)
{
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    uint4 v;
    asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(r) : "memory");
    return v;
}

// Digits of the radix select over the cap priorities K_l << 27 | K_r << 12 |
// r (31 bits: K_l <= 8, K_r <= 8 x 4080, r <= 4080), high to low, of 11, 11
// and 9 bits: the first one reaches into K_r, since almost every K_l is 1 or 2.
constexpr int kSelPasses = 3, kSelBins = 2048;
constexpr int kFinSegs = 1024;   // segment offsets kept in shared memory (the rest in b.seg_off)
constexpr int kFinKeep = 4;      // positions of a thread in a round
constexpr int kFinCluster = 8;   // most CTAs of an image

__global__ void __launch_bounds__(kFinThreads, 3) k_pfa_finalize(const __grid_constant__ Batch b)
{
    __shared__ __align__(16) uint32_t hist[kSelPasses][kSelBins];
    __shared__ uint32_t ws[2][kFinThreads / 32];
    __shared__ uint32_t s_before[2];  // positions of the CTAs before: above the threshold, at it
    __shared__ uint32_t sh_digit[kSelPasses], sh_need[kSelPasses];
    __shared__ int lfirst[kMaxLevels + 1];
    __shared__ int s_off[kFinSegs];
    const int C = (int)cluster_size(), rank = (int)cluster_rank();
    const int lg = 31 - __clz(C);  // a power of two
    const int img = blockIdx.x >> lg;
    const ImageDesc &I = b.images[img];
    const int nl = I.levels, cap = I.max_feats, slot_base = I.slot_base;
    const int seg_base = I.seg_base, seg_count = I.seg_count;
    for (int i = threadIdx.x; i < kSelPasses * kSelBins; i += kFinThreads) (&hist[0][0])[i] = 0;
    if (threadIdx.x < 2) s_before[threadIdx.x] = 0u;
    let_next();
    after_previous();

    // Canonical offsets of the segments (level-major, then cell row), by
    // every CTA for itself (the same values).
    int S = 0;
    for (int base = 0, t = 0; base < seg_count; base += kFinThreads, t ^= 1) {
        const int i = base + threadIdx.x;
        const uint32_t v = i < seg_count ? (uint32_t)b.seg_count[seg_base + i] : 0u;
        uint32_t tot;
        const int ex = (int)block_excl_scan<kFinThreads>(v, ws[t], &tot);
        if (i < kFinSegs) s_off[i] = S + ex;
        else if (i < seg_count) b.seg_off[seg_base + i] = S + ex;
        S += (int)tot;
    }
    __syncthreads();
    // first canonical position of each level
    if (threadIdx.x <= kMaxLevels) {
        int first = S;
        if (threadIdx.x < nl) {
            const int i = b.levels[I.level_base + threadIdx.x].seg_base - seg_base;
            first = i < kFinSegs ? s_off[i] : b.seg_off[seg_base + i];
        }
        lfirst[threadIdx.x] = first;
    }

    // Canonical position of every survivor of this CTA's segments (a warp
    // each), its priority and coordinates written there; the map entries
    // cleared.
    uint32_t *const map = I.map;
    const int W0 = I.W0;
    for (int i = rank * (kFinThreads / 32) + ((int)threadIdx.x >> 5); i < seg_count; i += C * (kFinThreads / 32)) {
        const SegRec &R = b.seg_rec[seg_base + i];
        const int m = R.m, slot = R.slot, at = slot_base + (i < kFinSegs ? s_off[i] : b.seg_off[seg_base + i]);
        for (int j0 = threadIdx.x & 31; j0 < m; j0 += 96) {
            uint4 v[3];
#pragma unroll
            for (int q = 0; q < 3; ++q)
                v[q] = j0 + 32 * q < m ? b.slot_info[slot + j0 + 32 * q] : make_uint4(0u, 0u, 0u, (uint32_t)kSlotEmpty);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int r = (int)v[q].w;
                if (r == kSlotEmpty) continue;
                map[(size_t)(v[q].y >> 16) * W0 + (v[q].y & 0xFFFFu)] = 0;
                if (r >= 0) {
                    b.canon_prio[at + r] = v[q].z;
                    b.canon_pos[at + r] = make_uint2(v[q].x, v[q].y);
                }
            }
        }
    }
    cluster_sync();

    // This CTA's positions: [g0, g1), in rounds of kRound; a thread has
    // kFinKeep neighbouring ones of a round, those of the first round in
    // registers.
    constexpr int kRound = kFinKeep * kFinThreads;
    const uint32_t *prio = b.canon_prio + slot_base;
    const int g0 = (int)(((uint32_t)S * (uint32_t)rank) >> lg), g1 = (int)(((uint32_t)S * (uint32_t)(rank + 1)) >> lg);
    const int t0 = kFinKeep * (int)threadIdx.x;
    uint32_t mine[kFinKeep];
    const auto load = [&](int base) {
#pragma unroll
        for (int i = 0; i < kFinKeep; ++i) mine[i] = base + t0 + i < g1 ? prio[base + t0 + i] : 0u;
    };
    load(g0);

    // Cap: keep the max_feats largest priorities, ties at the threshold T
    // resolved in canonical order.
    const bool capped = S > cap;
    uint32_t T = 0, mask = 0;
    int quota = 0;
    // this thread's digits' share of the positions of the CTAs before this one:
    // with a prefix of T and a larger digit, and equal to T
    uint32_t before_up = 0, before_tie = 0;
    // f(priority) of every position of this thread
    const auto each = [&](auto f) {
        for (int base = g0; base < g1; base += kRound) {
            if (base != g0) load(base);
#pragma unroll
            for (int i = 0; i < kFinKeep; ++i)
                if (base + t0 + i < g1) f(mine[i]);
        }
        if (g1 - g0 > kRound) load(g0);
    };
    if (capped) {
        int need = cap;
#pragma unroll
        for (int pass = 0; pass < kSelPasses; ++pass) {
            const int sh = pass == 0 ? 20 : pass == 1 ? 9 : 0;
            each([&](uint32_t P) {
                if ((P & mask) == T) atomicAdd(&hist[pass][(P & ~mask) >> sh], 1u);
            });
            cluster_sync();
            // the largest digit whose count, added to the counts of the larger
            // digits, reaches `need` (which never exceeds the total): a thread
            // has four digits, from the largest down
            static_assert(kSelBins == 4 * kFinThreads, "four digits a thread");
            const int d0 = kSelBins - 4 - 4 * (int)threadIdx.x;
            uint4 n4 = make_uint4(0u, 0u, 0u, 0u), p4 = n4;
#pragma unroll
            for (int c = 0; c < kFinCluster; ++c)
                if (c < C) {
                    const uint4 h = ld_cluster(&hist[pass][d0], (uint32_t)c);
                    n4.x += h.x; n4.y += h.y; n4.z += h.z; n4.w += h.w;
                    if (c + 1 == rank) p4 = n4;
                }
            const int n[4] = { (int)n4.w, (int)n4.z, (int)n4.y, (int)n4.x };
            uint32_t tot;
            int cum = (int)block_excl_scan<kFinThreads>((uint32_t)(n[0] + n[1] + n[2] + n[3]), ws[pass & 1], &tot);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (cum < need && cum + n[j] >= need) {
                    sh_digit[pass] = (uint32_t)(d0 + 3 - j);
                    sh_need[pass] = (uint32_t)(need - cum);
                }
                cum += n[j];
            }
            __syncthreads();
            const int digit = (int)sh_digit[pass];
            const uint32_t p[4] = { p4.w, p4.z, p4.y, p4.x };
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                before_up += d0 + 3 - j > digit ? p[j] : 0u;
                if (pass == kSelPasses - 1) before_tie += d0 + 3 - j == digit ? p[j] : 0u;
            }
            T |= (uint32_t)digit << sh;
            mask = ~((1u << sh) - 1u);
            need = (int)sh_need[pass];
        }
        quota = need;
    }
    // this CTA has read the others' histograms (waited for at the end)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const int keep = capped ? cap : S;

    // Positions before this CTA's that are above the threshold and at it (not
    // capped: all are above)
    int carry_up = g0, carry_tie = 0;
    const auto counts = [&]() {  // of this thread's positions in the round in registers: above | at << 16
        uint32_t c = 0;
#pragma unroll
        for (int i = 0; i < kFinKeep; ++i) c += (mine[i] > T ? 1u : 0u) + (mine[i] == T ? 1u << 16 : 0u);
        return c;
    };
    static_assert(kRound < 65536, "a round's counts fit 16 bits");
    if (capped && C > 1) {
        before_up = __reduce_add_sync(0xFFFFFFFFu, before_up);
        before_tie = __reduce_add_sync(0xFFFFFFFFu, before_tie);
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&s_before[0], before_up);
            atomicAdd(&s_before[1], before_tie);
        }
        __syncthreads();
        carry_tie = (int)s_before[1];
    }
    if (capped) carry_up = (int)s_before[0];

    // the kept positions in order; position g is preceded by up + min(tie, quota) kept ones
    const KpOut &o = I.out;
    for (int base = g0, t = 0; base < g1; base += kRound, t ^= 1) {
        if (base != g0) load(base);
        uint2 at[kFinKeep];
#pragma unroll
        for (int i = 0; i < kFinKeep; ++i)
            at[i] = base + t0 + i < g1 ? b.canon_pos[slot_base + base + t0 + i] : make_uint2(0u, 0u);
        int up = carry_up + t0, tie = 0;
        uint32_t tot = kRound;
        if (capped) {
            const uint32_t ex = block_excl_scan<kFinThreads>(counts(), ws[t], &tot);
            up = carry_up + (int)(ex & 0xFFFFu);
            tie = carry_tie + (int)(ex >> 16);
        }
#pragma unroll
        for (int i = 0; i < kFinKeep; ++i) {
            const int g = base + t0 + i;
            if (g >= g1) break;
            const uint32_t P = mine[i];
            const int oi = up + min(tie, quota);
            const bool is_up = !capped || P > T, is_tie = capped && P == T;
            const int l = (int)(at[i].x >> 26);
            // level starts: of this level and of the empty ones before it
            for (int m = l; m >= 0 && lfirst[m] == g; --m) I.level_start[m] = oi;
            if (is_up || (is_tie && tie < quota)) {
                o.x[oi] = (uint16_t)pos_x(at[i].x);
                o.y[oi] = (uint16_t)pos_y(at[i].x);
                o.X[oi] = (uint16_t)(at[i].y & 0xFFFFu);
                o.Y[oi] = (uint16_t)(at[i].y >> 16);
                o.level[oi] = (uint8_t)l;
                o.response[oi] = (uint16_t)(P & 0xFFFu);
                o.k_levels[oi] = (uint8_t)(P >> 27);
                o.k_resp[oi] = (P >> 12) & 0x7FFFu;
            }
            up += is_up;
            tie += is_tie;
        }
        carry_up += (int)(tot & 0xFFFFu);
        carry_tie += (int)(tot >> 16);
    }
    if (rank == 0 && threadIdx.x <= kMaxLevels) {
        if (lfirst[threadIdx.x] == S) I.level_start[threadIdx.x] = keep;  // no position of this level or a later one
        if (threadIdx.x == 0) {
            *I.count = keep;
            *I.count_hdr = keep;
        }
    }
    // no CTA ends while another may read its histograms
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// CTAs per image.  More of them shorten the chains of a small batch, each
// costs the cluster's barriers, and in a large batch the images fill the
// chip: at least 700 slots a CTA, and no more CTAs than SMs -- two an image
// also when all of them run at once (three CTAs fit an SM).  Measured with 1 /
// 2 / 4 / 8 (us, finalisation stage before the last rounds of tuning): one
// 1920x1080 pair (16 000 slots an image) 84 / 51 / 37 / 31, one 1241x376 pair
// (3 900) 34 / 24 / 23 / 24, 16 mixed pairs (to 16 000) 86 / 53 / 39 / 41, 12
// of 752x480 (2 900) 29 / 23 / 21 / 35, 25 of 1241x376 35 / 27 / 27 / 45, 100 of
// 1241x376 45 / 37 / 61 / 158.
static int finalize_ctas(const Batch &b)
{
    int c = 1;
    while (c < kFinCluster && b.max_slots / (2 * c) >= 700 &&
           (b.n_images * 2 * c <= b.n_sm || (c == 1 && b.n_images * 2 <= 3 * b.n_sm)))
        c *= 2;
    return c;
}

cudaError_t launch_pfa_finalize(const Batch &b, cudaStream_t stream)
{
    if (b.n_images == 0) return cudaSuccess;
    const int C = finalize_ctas(b);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(b.n_images * C);
    cfg.blockDim = dim3(kFinThreads);
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_after
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = start_early(b) ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, k_pfa_finalize, b);
}

}  // namespace jslam
