// ORB extraction for all scales at once and stereo row matching (Sec. III:
// streamlined multiscale detection and extraction; middle-end stereo
// matching by descriptor-distance minimisation).
//
// k_orient_desc  one warp per keypoint (and turn) of any image and level.  The
//                tensor unit brings the keypoint's box of the raw level (the
//                radius-15 disk) and of the blurred one (the 27 x 27 patch the
//                BRIEF pattern reaches) to shared memory, those of the next
//                keypoint while this one is computed.  The lanes read the disk
//                as words and accumulate the intensity moments m10, m01 with
//                byte dot products over the bytes inside the disk; lanes 0..29
//                each test one sector boundary (float with an error margin,
//                IEEE double with explicit rounding inside it, so the sector
//                equals the one the host-side definition gives); the 256 BRIEF
//                comparisons read the patch 32 at a time and are packed into
//                words by a ballot.  The row index of the canonical list that the
//                matching reads is written here too.
// k_match        half a warp per left keypoint: for each right level within one
//                of the keypoint's level, takes the s0 row band of the
//                canonical (level, y, x) list (Y is non-decreasing in y) from
//                the row index (two independent loads per level), scans the
//                band with the lanes, and keeps the smallest (Hamming
//                distance, disparity, index) by a min-reduction.
#include <algorithm>

#include <cuda.h>

#include "jslam_internal.h"

namespace jslam {

constexpr int kDiskWords = 9;             // aligned words covering the 31 disk columns of a row
constexpr int kOrbWarps = 4;              // warps per CTA
constexpr int kOrbMaxTurns = 32;          // keypoints a warp takes, at most (a lane keeps each one's moments)
static_assert(kDiskRows * 3 > 2 * kDiskR + 1 && 3 * kDiskWords <= 32, "a lane's rows cover the disk");
constexpr int kOrbRaw = (kOrbBoxW * kOrbRawH + 127) / 128 * 128, kOrbBlur = (kOrbBoxW * kOrbBlurH + 127) / 128 * 128;

// A keypoint's boxes: rows of 48 bytes from the 16-byte boundary at or before
// the disk's (the patch's) first column.
struct __align__(128) OrbBuf {
    uint8_t raw[kOrbRaw];
    uint8_t blur[kOrbBlur];
};
constexpr int kOrbSmem = 2 * kOrbWarps * (int)sizeof(OrbBuf);  // two boxes a warp

__device__ __forceinline__ uint32_t orb_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Wait for the mbarrier phase `parity`, giving up after about a second.
__device__ __forceinline__ bool orb_wait(uint32_t bar, uint32_t parity)
{
    const long long start = clock64();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
        if (clock64() - start > (1ll << 31)) return false;
    }
}

// One box of a keypoint by TMA; x is a multiple of 16 and the box starts
// inside the level (it may end past its right edge: those bytes are zero and
// unused).
__device__ __forceinline__ void orb_box(const CUtensorMap *map, const uint8_t *to, int x, int y, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(orb_smem(to)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar) : "memory");
}

// What bounds it: shared-memory and load latency (the dependent chain box ->
// moments -> sector -> pattern -> patch, 32 warps an SM).  Reading disk and
// patch with plain loads touches a line per row, 75 of the 170 load
// wavefronts a keypoint took, and those bounded it: 400 000 keypoints 0.260 ms
// with one warp each and 563 instructions a keypoint; 0.211 ms now, with 345
// (0.205 and 328 without the row index, which the finalisation wrote then).
// A warp takes keypoints i, i + stride, ... of its image.
__global__ void __launch_bounds__(32 * kOrbWarps) k_orient_desc(const __grid_constant__ Batch b)
{
    extern __shared__ __align__(128) uint8_t orb_mem[];
    __shared__ __align__(8) uint64_t s_bar[kOrbWarps][2];
    const ImageDesc &I = b.images[blockIdx.y];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t bar = orb_smem(s_bar[warp]);
    if (lane < 2) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar + 8 * lane) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    // lane < 27 of the disk: word column w, rows r0, r0 + 3, ...
    const int w = lane % kDiskWords, r0 = lane / kDiskWords;
    const float cosf_l = lane < kBins ? __ldg(b.bin_cosf + lane) : 0.0f;
    const float sinf_l = lane < kBins ? __ldg(b.bin_sinf + lane) : 0.0f;
    let_next();
    after_previous();
    const int count = *I.count, stride = gridDim.x * kOrbWarps;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        // the host's mirror of the counts and of the error word (what this
        // kernel adds goes into a word of its own, so that neither store
        // replaces the other)
        b.host_counts[blockIdx.y] = count;
        if (blockIdx.y == 0) {
            const uint32_t err = *b.err;
            if (err) *reinterpret_cast<volatile uint32_t *>(b.host_err) = err;
        }
    }
    const KpOut &o = I.out;
    // The row index of the canonical list, for the stereo matching: entry v of
    // level l's table is the first index of the level whose Y is >= v, else
    // the level's end, for v = 0 .. H0.  Keypoint j owns the entries (Y[j - 1],
    // Y[j]] when it is not the level's first (below); a CTA fills a level's
    // entries up to the first keypoint's Y (the level's start) and after the
    // last one's (its end).  Here and not at the end of the finalisation, where
    // it took one more barrier of the cluster.
    const int rows = I.H0 + 1;
    for (int l = blockIdx.x; l < I.levels; l += gridDim.x) {
        const int s = I.level_start[l], e = I.level_start[l + 1];
        if (s == e) continue;
        const int ys = o.Y[s], ye = o.Y[e - 1];
        int32_t *const rf = I.row_first + (size_t)l * rows;
        for (int v = threadIdx.x; v < rows; v += 32 * kOrbWarps) {
            if (v <= ys) rf[v] = s;
            else if (v > ye) rf[v] = e;
        }
    }
    const int first = blockIdx.x * kOrbWarps + warp;
    if (first >= count) return;
    const CUtensorMap *const maps = b.orb_maps + 2 * I.level_base;
    OrbBuf *const buf = reinterpret_cast<OrbBuf *>(orb_mem) + 2 * warp;
    const uint16_t *const xs = o.x, *const ys = o.y;
    const uint8_t *const lv = o.level;
    // the boxes of the keypoint at (x, y) into buffer k.  The keypoint is at
    // least `border` (>= 16) from every edge, so the 31 x 31 square of the
    // moment disk and the 27 x 27 patch are inside the level.
    const auto issue = [&](int x, int y, int level, int k) {
        if (lane == 0) {
            const CUtensorMap *map = maps + 2 * level;
            const uint32_t bk = bar + 8 * k;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bk),
                         "r"((uint32_t)(kOrbBoxW * (kOrbRawH + kOrbBlurH))) : "memory");
            orb_box(map, buf[k].raw, (x - kDiskR) & ~15, y - kDiskR, bk);
            orb_box(map + 1, buf[k].blur, (x - kPatR) & ~15, y - kPatR, bk);
        }
    };
    int x = xs[first], y = ys[first], level = lv[first];
    issue(x, y, level, 0);
    // the row-index entries of this warp's keypoints, a lane each (a warp has
    // at most kOrbMaxTurns)
    if (const int j = first + lane * stride; j < count) {
        const int l = lv[j], Yj = o.Y[j], Yp = j > 0 ? (int)o.Y[j - 1] : 0;
        if (j != I.level_start[l]) {
            int32_t *const rf = I.row_first + (size_t)l * rows;
            for (int v = Yp + 1; v <= Yj; ++v) rf[v] = j;
        }
    }
    __syncwarp();
    int nx = 0, ny = 0, nlev = 0;
    if (first + stride < count) { nx = xs[first + stride]; ny = ys[first + stride]; nlev = lv[first + stride]; }
    uint32_t *const desc = o.desc;
    int my10 = 0, my01 = 0;  // the moments of the keypoint of turn `lane`

    int turn = 0;
    for (int i = first; i < count; i += stride, ++turn) {
        const int k2 = turn & 1;
        if (i + stride < count) issue(nx, ny, nlev, k2 ^ 1);
        int n2x = 0, n2y = 0, n2l = 0;
        if (i + 2 * stride < count) { n2x = xs[i + 2 * stride]; n2y = ys[i + 2 * stride]; n2l = lv[i + 2 * stride]; }
        // Disk moments: 31 rows x 9 words from the word that holds column x -
        // 15; a lane has one word column and every third row.  Per word the
        // bytes inside the disk are kept (a table's masks, by the alignment)
        // and two byte dot products add to the sum S of the pixels and to that
        // of (dx + 18) I; U sums S after every row, so that the sum of k I_k is
        // 11 S - U for the lane's row number k, row dy = r0 + 3 k - 15.
        const int al = (x - kDiskR) & 3;
        uint32_t mask[kDiskRows];
#pragma unroll
        for (int k = 0; k < kDiskRows; ++k) mask[k] = __ldg(b.disk_mask + (al * kDiskRows + k) * 32 + lane);
        if (!orb_wait(bar + 8 * k2, (turn >> 1) & 1)) {
            // flag it, and wait once more, with the same limit, for the copies
            // in flight, so that none lands in the memory of a CTA that ended
            if (lane == 0) {
                atomicOr(b.err, kErrTimeout);
                *reinterpret_cast<volatile uint32_t *>(b.host_err + kHostErrOrb) = kErrTimeout;
            }
            orb_wait(bar + 8 * k2, (turn >> 1) & 1);
            if (i + stride < count) orb_wait(bar + 8 * (k2 ^ 1), ((turn + 1) >> 1) & 1);
            return;
        }
        const uint32_t *src = reinterpret_cast<const uint32_t *>(buf[k2].raw) + r0 * (kOrbBoxW / 4) +
                              (((x - kDiskR) & 15) >> 2) + w;
        const uint32_t wdx = (uint32_t)(4 * w + 3 - al) * 0x01010101u + 0x03020100u;  // dx + 18 of the word's bytes
        uint32_t Sm = 0, U = 0, Sw = 0;
#pragma unroll
        for (int k = 0; k < kDiskRows; ++k) {
            const uint32_t v = src[k * 3 * (kOrbBoxW / 4)] & mask[k];
            Sm = __dp4a(v, 0x01010101u, Sm);
            Sw = __dp4a(v, wdx, Sw);
            U += Sm;
        }
        const int m10 = __reduce_add_sync(0xFFFFFFFFu, (int)Sw - 18 * (int)Sm);
        const int m01 = __reduce_add_sync(0xFFFFFFFFu, (r0 - kDiskR + 3 * kDiskRows) * (int)Sm - 3 * (int)U);

        // Sector b is the one whose lower boundary has the moment vector on its
        // left (m01 cos - m10 sin >= 0 in IEEE double) and whose upper boundary
        // does not.  The test runs in float first: |m| < 2^24 is exact, and the
        // float result is within (|m01| + |m10|) 2^-22 of the exact value with
        // the double table entries, so outside 2^-20 times that its sign is the
        // double test's; lanes inside the margin (rare) take the double test.
        bool left_of = false;
        if (lane < kBins) {
            const float fa = (float)m01, fb = (float)m10;
            const float t = __fsub_rn(__fmul_rn(fa, cosf_l), __fmul_rn(fb, sinf_l));
            const float margin = (fabsf(fa) + fabsf(fb)) * 0x1p-20f;
            if (fabsf(t) > margin) {
                left_of = t > 0.0f;
            } else {
                const double t1 = __dmul_rn((double)m01, b.bin_cos[lane]);
                const double t2 = __dmul_rn((double)m10, b.bin_sin[lane]);
                left_of = __dsub_rn(t1, t2) >= 0.0;
            }
        }
        const uint32_t Lt = __ballot_sync(0xFFFFFFFFu, left_of) & ((1u << kBins) - 1u);
        const uint32_t next = (Lt >> 1) | ((Lt & 1u) << (kBins - 1));
        const uint32_t T = Lt & ~next & ((1u << kBins) - 1u);
        const bool zero = (m10 == 0 && m01 == 0);
        const int bin = (zero || T == 0) ? 0 : __ffs(T) - 1;

        // shared addresses of p (low half) and q of a pair: offsets from the
        // patch's corner, and its place
        const uint32_t *pat = b.pattern_off + (size_t)bin * kPairs + lane;
        const uint32_t at = (orb_smem(buf[k2].blur) + (uint32_t)((x - kPatR) & 15)) * 0x00010001u;
        uint32_t myword = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t pq = __ldg(pat + 32 * k) + at;
            uint32_t p8, q8;
            asm volatile("ld.shared.u8 %0, [%1];" : "=r"(p8) : "r"(pq & 0xFFFFu));
            asm volatile("ld.shared.u8 %0, [%1];" : "=r"(q8) : "r"(pq >> 16));
            const uint32_t word = __ballot_sync(0xFFFFFFFFu, p8 < q8);
            if (lane == k) myword = word;
        }
        if (lane < 8) desc[(size_t)i * 8 + lane] = myword;
        if (lane == 0) o.angle_bin[i] = (uint8_t)bin;
        if (lane == turn) { my10 = m10; my01 = m01; }
        x = nx; y = ny; level = nlev;
        nx = n2x; ny = n2y; nlev = n2l;
        __syncwarp();  // the buffer has been read
    }
    // the angles of all turns at once
    if (lane < turn) o.angle[first + lane * stride] = my10 == 0 && my01 == 0 ? 0.0f : atan2f((float)my01, (float)my10);
}

// Keypoints per warp: as many as leave two rounds of resident warps (32 an
// SM), so that a warp brings the next boxes while it computes and shares what
// it does once (its tables, the angles); one in small batches.  1 / 2 / 4 / 8 /
// 16 (us): 100 pairs of 1241x376 340 / 256 / 217 / 210 / 205, 16 mixed pairs 59
// / 52 / 47 / 45 / 45, one pair of 1241x376 10 / 12 / 13 / 16 / 24.
static int orb_turns(const Batch &b)
{
    const long long keypoints = (long long)b.max_capacity * b.n_images;
    return (int)std::min<long long>(std::max<long long>(keypoints / (64 * b.n_sm), 1), 16);
}

cudaError_t configure_orb()
{
    return cudaFuncSetAttribute(k_orient_desc, cudaFuncAttributeMaxDynamicSharedMemorySize, kOrbSmem);
}

cudaError_t launch_orient_desc(const Batch &b, cudaStream_t stream)
{
    if (b.n_images == 0 || b.max_capacity == 0) return cudaSuccess;
    const int turns = orb_turns(b);
    static_assert(16 <= kOrbMaxTurns, "a lane keeps each turn's moments");
    dim3 grid((b.max_capacity + kOrbWarps * turns - 1) / (kOrbWarps * turns), b.n_images);
    return launch_after(k_orient_desc, grid, dim3(32 * kOrbWarps), kOrbSmem, stream, b);
}

// Half a warp per left keypoint: its band holds a few dozen candidates at
// most, of which a good part lies outside the search range.  What bounds it:
// the chain of gathers from L2 (keypoint -> row index -> X -> descriptor);
// eight CTAs an SM hide most of it.  200 000 left keypoints: 0.121 ms with a
// warp each, 0.068 now (six CTAs an SM cost 8 % more).
__global__ void __launch_bounds__(256, 8) k_match(const __grid_constant__ Batch b)
{
    const PairDesc &P = b.pairs[blockIdx.y];
    const int l16 = threadIdx.x & 15;
    const ImageDesc &Il = b.images[P.left];
    const ImageDesc &Ir = b.images[P.right];
    let_next();
    after_previous();
    const int count = *Il.count;
    int i = blockIdx.x * 16 + (threadIdx.x >> 4);
    if ((i & ~1) >= count) return;  // whole warps only
    const bool valid = i < count;
    i = min(i, count - 1);
    const KpOut &ol = Il.out, &orr = Ir.out;
    const int n = ol.level[i];
    const int X = ol.X[i], Y = ol.Y[i];
    const int band = b.levels[Il.level_base + n].band;
    const uint4 *dp = reinterpret_cast<const uint4 *>(ol.desc + (size_t)i * 8);
    const uint4 l0 = dp[0], l1 = dp[1];

    const int m_lo = max(0, n - 1), m_hi = min(Ir.levels - 1, n + 1);
    // the band [Y - band, Y + band] of each level: lower bounds of Y - band
    // and Y + band + 1 from the row index (rows clamped to [0, H0]; a level
    // without keypoints has an empty band and an unwritten table)
    const int va = min(max(Y - band, 0), Ir.H0), vz = min(max(Y + band + 1, 0), Ir.H0);
    int ra[3], rz[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int m = m_lo + q;
        ra[q] = rz[q] = 0;
        if (m <= m_hi) {
            const int s = Ir.level_start[m], e = Ir.level_start[m + 1];
            const int32_t *rf = Ir.row_first + (size_t)m * (Ir.H0 + 1);
            ra[q] = e > s ? rf[va] : s;
            rz[q] = e > s ? rf[vz] : s;
        }
    }
    // the three bands as one run of candidates over the lanes (a band of a
    // level outside the frame, or of an empty level, is empty), so a few
    // dozen candidates take one or two passes of loads, not one per level
    const int c0 = rz[0] - ra[0], c01 = c0 + (rz[1] - ra[1]), T = c01 + (rz[2] - ra[2]);
    const uint16_t *const Xr = orr.X;
    const uint32_t *const descr = orr.desc;
    // smallest (distance, disparity), then index: a lane's candidates come in
    // index order
    uint32_t best = 0xFFFFFFFFu, best_j = 0xFFFFFFFFu;
    for (int t = l16; t < T; t += 16) {
        const int j = t < c0 ? ra[0] + t : (t < c01 ? ra[1] + (t - c0) : ra[2] + (t - c01));
        const int disp = X - (int)Xr[j];
        if ((uint32_t)disp > (uint32_t)b.prm.max_disp) continue;
        const uint4 *dr = reinterpret_cast<const uint4 *>(descr + (size_t)j * 8);
        const uint4 r0 = dr[0], r1 = dr[1];
        const uint32_t d = __popc(l0.x ^ r0.x) + __popc(l0.y ^ r0.y) + __popc(l0.z ^ r0.z) + __popc(l0.w ^ r0.w) +
                           __popc(l1.x ^ r1.x) + __popc(l1.y ^ r1.y) + __popc(l1.z ^ r1.z) + __popc(l1.w ^ r1.w);
        const uint32_t key = (d << 16) | (uint32_t)disp;
        if (key < best) { best = key; best_j = (uint32_t)j; }
    }
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) {
        const uint32_t k2 = __shfl_xor_sync(0xFFFFFFFFu, best, off), j2 = __shfl_xor_sync(0xFFFFFFFFu, best_j, off);
        if (k2 < best || (k2 == best && j2 < best_j)) { best = k2; best_j = j2; }
    }
    if (l16 == 0 && valid) {
        const int d = (int)(best >> 16);  // 0xFFFF: no candidate
        const bool ok = d <= b.prm.max_dist && best != 0xFFFFFFFFu;
        P.match_idx[i] = ok ? (int)best_j : -1;
        P.disparity[i] = ok ? (int16_t)(best & 0xFFFFu) : (int16_t)0;
        P.dist[i] = (uint16_t)d;
    }
}

// Feature tracking by projection (middle-end): one warp per query.  For each
// level of the band the row index narrows the frame's canonical list to a
// conservative Y range; lanes take the exact float window test and the
// Hamming distance, and a warp reduction keeps the smallest (distance,
// index) and the second-smallest distance.
__global__ void __launch_bounds__(256) k_track(const __grid_constant__ Batch b, const __grid_constant__ TrackArgs a)
{
    const int lane = threadIdx.x & 31;
    const int q = blockIdx.x * 8 + (threadIdx.x >> 5);
    let_next();
    after_previous();
    if (q >= a.n) return;
    const ImageDesc &I = b.images[a.image];
    const int lv = a.level[q];
    unsigned long long best = ~0ull;   // distance << 32 | index
    uint32_t second = 0xFFFFFFFFu;
    // the band lv - 1 .. lv + 1 clipped to the frame's levels: a query one
    // level past the deepest meets that level (its window scaled by
    // zeta^lv), a deeper one meets none
    if (lv <= kMaxLevels) {
        const float u = a.u[q], v = a.v[q];
        const float r = __fmul_rn(a.radius, a.zeta_f[lv]);
        uint32_t dq[8];
#pragma unroll
        for (int w = 0; w < 8; ++w) dq[w] = a.desc[(size_t)q * 8 + w];
        const KpOut &o = I.out;
        const int m_lo = max(0, lv - 1), m_hi = min(I.levels - 1, lv + 1);
        const int ylo = (int)floorf(v - r) - 1, yhi = (int)ceilf(v + r) + 1;  // covers every Y that can pass
        // rows of the row index, clamped to [0, H0] (64-bit: yhi may be INT_MAX)
        const int va = (int)min(max((long long)ylo, 0ll), (long long)I.H0);
        const int vz = (int)min(max((long long)yhi + 1, 0ll), (long long)I.H0);
        for (int m = m_lo; m <= m_hi; ++m) {
            const int s = I.level_start[m], e = I.level_start[m + 1];
            const int32_t *rf = I.row_first + (size_t)m * (I.H0 + 1);
            const int z0 = e > s ? rf[va] : s;
            const int z1 = e > s ? max(rf[vz], z0) : s;
            for (int j = z0 + lane; j < z1; j += 32) {
                const float dx = __fsub_rn((float)o.X[j], u), dy = __fsub_rn((float)o.Y[j], v);
                if (fabsf(dx) > r || fabsf(dy) > r) continue;
                const uint4 *dr = reinterpret_cast<const uint4 *>(o.desc + (size_t)j * 8);
                const uint4 r0 = dr[0], r1 = dr[1];
                const uint32_t d = __popc(dq[0] ^ r0.x) + __popc(dq[1] ^ r0.y) + __popc(dq[2] ^ r0.z) +
                                   __popc(dq[3] ^ r0.w) + __popc(dq[4] ^ r1.x) + __popc(dq[5] ^ r1.y) +
                                   __popc(dq[6] ^ r1.z) + __popc(dq[7] ^ r1.w);
                const unsigned long long key = ((unsigned long long)d << 32) | (unsigned)j;
                if (key < best) {
                    second = min(second, (uint32_t)(best >> 32));
                    best = key;
                } else {
                    second = min(second, d);
                }
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long ob = __shfl_xor_sync(0xFFFFFFFFu, best, off);
            const uint32_t os = __shfl_xor_sync(0xFFFFFFFFu, second, off);
            const unsigned long long lo = ob < best ? ob : best, hi = ob < best ? best : ob;
            second = min(min(second, os), (uint32_t)(hi >> 32));
            best = lo;
        }
    }
    if (lane == 0) {
        if (best == ~0ull) {
            a.out_idx[q] = -1;
            a.out_dist[q] = 0xFFFF;
        } else {
            const uint32_t d = (uint32_t)(best >> 32);
            const bool ok = (int)d <= a.max_dist && (second == 0xFFFFFFFFu || 10u * d <= 9u * second);
            a.out_idx[q] = ok ? (int)(best & 0xFFFFFFFFu) : -1;
            a.out_dist[q] = (uint16_t)d;
        }
    }
}

cudaError_t launch_track(const Batch &b, const TrackArgs &a, cudaStream_t stream)
{
    if (a.n == 0) return cudaSuccess;
    return launch_after(k_track, dim3((a.n + 7) / 8), dim3(256), 0, stream, b, a);
}

cudaError_t launch_match(const Batch &b, cudaStream_t stream)
{
    if (b.n_pairs == 0 || b.max_capacity == 0) return cudaSuccess;
    dim3 grid((b.max_capacity + 15) / 16, b.n_pairs);
    return launch_after(k_match, grid, dim3(256), 0, stream, b);
}

}  // namespace jslam
