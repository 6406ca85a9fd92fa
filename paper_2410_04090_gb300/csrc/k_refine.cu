// Correlation minimisation of the stereo matches (Sec. III, middle-end
// stereo matching): sub-pixel disparity and depth of every accepted
// descriptor match.
//
// k_refine5        the default window (w = 5): half a warp per left keypoint.
//                  Window and strip are staged in shared memory as words; lane
//                  k sums the centre-normalised absolute differences of shift
//                  k, two pixels to an operation: with v = left + 1024 - cc -
//                  right in 16-bit lanes (cc the difference of the centres),
//                  |left - right - cc| = 2 max(v, 1024) - v - 1024, and the
//                  sums of max(v, 1024) and of right are dot products.
// k_refine         any half-size: one warp per left keypoint, bytes staged,
//                  lanes 0..2(2L+1)-1 each sum one shift over half of the rows
//                  (20 pairs of 1241x376, L = 5, with the median: 64 us at w =
//                  3, 121 at w = 8, where k_refine5 takes 31 with stage events).
//                  In both a warp minimum picks the first minimum shift, and
//                  one lane takes the decisions in integers and computes
//                  delta, disparity and depth in float (the host-side
//                  definition's doubles to a few float ulps; the FP64 pipe is
//                  a small fraction of the FP32 rate here).
// k_refine_median  one CTA per pair: the median SAD of the surviving matches
//                  by a radix select of two 9-bit digits, then the matches
//                  above 2.1 times it are rejected.
#include "jslam_internal.h"

namespace jslam {

constexpr int kRefW = kRefineMaxW, kRefL = kRefineMaxL;
constexpr int kRefLeft = (2 * kRefW + 1) * (2 * kRefW + 1);
constexpr int kRefRight = (2 * kRefW + 1) * (2 * kRefW + 2 * kRefL + 1);

// xr0 = floor(X / s + 0.5): in float, |X / s - q| < 2^-10 for X < 2^13, so a q
// more than 2^-8 away from a half-integer rounds as the double does; closer
// ones (rare) take the double computation.
__device__ __forceinline__ int right_column(const LevelDesc &A, int X)
{
    const float q = __fmul_rn((float)X, A.zeta_inv_f);
    const float fr = q - floorf(q);
    int xr0 = (int)floorf(q + 0.5f);
    if (fabsf(fr - 0.5f) < 0x1p-8f) xr0 = (int)floor(__dadd_rn(__ddiv_rn((double)X, A.zeta), 0.5));
    return xr0;
}

// Sub-pixel disparity and depth from the SADs d1, d2, d3 of the shifts ts - 1,
// ts, ts + 1 (d2 the first minimum, ts inside the search range); nothing is
// written for a rejected match.
__device__ __forceinline__ void sub_pixel(const LevelDesc &A, int xi, int xr0, int ts, int d1, int d2, int d3,
                                          int max_disp, double bf, float *disp_out, float *depth_out)
{
    const long long num = d1 - d3, den = 2ll * (d1 + d3 - 2 * d2);
    // disparity >= 0 <=> q den >= num; <= max_disp <=> s (q den - num) <= max_disp den
    const long long qi = (long long)xi - xr0 - ts;
    bool ok = den != 0 && (num < 0 ? -num : num) <= den && qi * den >= num;
    if (ok) {
        // s (q den - num) <= max_disp den, in float unless within a
        // relative 2^-18 of equality (float error < 2^-21 relative)
        const float lhs = __fmul_rn(A.zeta_f, (float)(qi * den - num));
        const float rhs = __fmul_rn((float)max_disp, (float)den);
        if (lhs > rhs * (1.0f + 0x1p-18f)) ok = false;
        else if (!(lhs < rhs * (1.0f - 0x1p-18f)))
            ok = !(__dmul_rn(A.zeta, (double)(qi * den - num)) > (double)max_disp * (double)den);
    }
    if (ok) {
        const float delta = __fdiv_rn((float)num, (float)den);
        const float disp = __fmul_rn(A.zeta_f, __fsub_rn((float)qi, delta));
        *disp_out = disp;
        *depth_out = bf > 0.0 ? __fdiv_rn((float)bf, fmaxf(disp, 0.01f)) : 0.0f;
    }
}

constexpr int kR5 = 5, kR5Side = 2 * kR5 + 1;  // the default window

// What bounds it: instruction issue, the absolute differences (1331 a
// keypoint at L = 5).  20 pairs of 1241x376 (40 000 left keypoints), both
// kernels of the refinement: 86 us with a warp per keypoint and a difference
// per operation (and the median's digits searched by one thread), 27 now; one
// pair 27 and 12 us.
__global__ void __launch_bounds__(256) k_refine5(const __grid_constant__ Batch b, int L, double bf)
{
    // per half warp: right strip rows of 8 words, left rows of 4 (as loaded),
    // the left window's pixels in 16-bit pairs (0, 2), (1, 3), ... (8, 10), (9, none)
    __shared__ __align__(16) uint32_t s_right[16][kR5Side][8];
    __shared__ __align__(16) uint32_t s_left[16][kR5Side][4];
    __shared__ __align__(16) uint32_t s_pair[16][kR5Side][8];
    const int hw = threadIdx.x >> 4, l16 = threadIdx.x & 15;
    const PairDesc &P = b.pairs[blockIdx.y];
    const ImageDesc &Il = b.images[P.left];
    const ImageDesc &Ir = b.images[P.right];
    let_next();
    after_previous();
    const int count = *Il.count;
    int i = blockIdx.x * 16 + hw;
    if ((i & ~1) >= count) return;  // whole warps only
    const bool valid = i < count;
    i = min(i, count - 1);
    const int j = P.match_idx[i];
    const int n = Il.out.level[i], xi = Il.out.x[i], yi = Il.out.y[i];
    const LevelDesc &A = b.levels[Il.level_base + n];
    const LevelDesc &B = b.levels[Ir.level_base + n];
    const int W = A.W, H = A.H, pitch = A.pitch;
    const int xr0 = j >= 0 ? right_column(A, Ir.out.X[max(j, 0)]) : 0;
    const bool in = j >= 0 && xi - kR5 >= 0 && xi + kR5 < W && yi - kR5 >= 0 && yi + kR5 < H && xr0 - L - kR5 >= 0 &&
                    xr0 + L + kR5 < W;
    float disp_out = -1.0f, depth_out = 0.0f;
    uint32_t sad_out = 0xFFFFFFFFu;
    if (__any_sync(0xFFFFFFFFu, in)) {
        // rows as aligned words (both levels have one pitch): the strip's 2 (5
        // + L) + 1 <= 25 bytes lie in 7 words, the window's 11 in 4; a word
        // past them may reach into the row's pitch or the buffer's slack
        const int xl = xi - kR5, xr = xr0 - L - kR5, y0 = yi - kR5;
        if (in) {
            const uint32_t *lsrc = reinterpret_cast<const uint32_t *>(A.raw + (size_t)y0 * pitch) + (xl >> 2);
            const uint32_t *rsrc = reinterpret_cast<const uint32_t *>(B.raw + (size_t)y0 * pitch) + (xr >> 2);
            // all loads before the stores, which may write to what is loaded for
            // all the compiler knows (the call below 32.3 us with a store after
            // each load, 26.8 so)
            uint32_t rw[6], lw[3];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const int r = 2 * k + (l16 >> 3);
                rw[k] = r < kR5Side ? rsrc[(size_t)r * (pitch >> 2) + (l16 & 7)] : 0u;
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int r = 4 * k + (l16 >> 2);
                lw[k] = r < kR5Side ? lsrc[(size_t)r * (pitch >> 2) + (l16 & 3)] : 0u;
            }
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const int r = 2 * k + (l16 >> 3);
                if (r < kR5Side) s_right[hw][r][l16 & 7] = rw[k];
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int r = 4 * k + (l16 >> 2);
                if (r < kR5Side) s_left[hw][r][l16 & 3] = lw[k];
            }
        }
        __syncwarp();
        // lane r: row r of the window, aligned and spread to 16 bits, and its sum
        uint32_t suml = 0;
        if (in && l16 < kR5Side) {
            const uint4 v = *reinterpret_cast<const uint4 *>(s_left[hw][l16]);
            const uint32_t sh = (uint32_t)xl << 3;  // modulo 32
            const uint32_t w0 = __funnelshift_r(v.x, v.y, sh), w1 = __funnelshift_r(v.y, v.z, sh),
                           w2 = __funnelshift_r(v.z, v.w, sh) & 0x00FFFFFFu;
            *reinterpret_cast<uint4 *>(&s_pair[hw][l16][0]) =
                make_uint4(w0 & 0x00FF00FFu, (w0 >> 8) & 0x00FF00FFu, w1 & 0x00FF00FFu, (w1 >> 8) & 0x00FF00FFu);
            *reinterpret_cast<uint2 *>(&s_pair[hw][l16][4]) = make_uint2(w2 & 0x00FF00FFu, (w2 >> 8) & 0x00FF00FFu);
            suml = __dp4a(w0, 0x01010101u, __dp4a(w1, 0x01010101u, __dp4a(w2, 0x01010101u, 0u)));
        }
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) suml += __shfl_xor_sync(0xFFFFFFFFu, suml, off);
        __syncwarp();
        const int nsh = 2 * L + 1;
        uint32_t key = 0xFFFFFFFFu;
        int sad = 0;
        if (in && l16 < nsh) {
            const uint8_t *lb = reinterpret_cast<const uint8_t *>(s_left[hw][kR5]) + (xl & 3) + kR5;
            const int at = (xr & 3) + l16;  // first byte of the shifted window in a strip row
            const uint8_t *rb = reinterpret_cast<const uint8_t *>(s_right[hw][kR5]) + at + kR5;
            const int cc = (int)*lb - (int)*rb;
            const uint32_t K = (uint32_t)(1024 - cc), K2 = K * 0x00010001u;
            const uint32_t sh = (uint32_t)at << 3;
            uint32_t sum_max = 0, sum_r = 0;
#pragma unroll
            for (int r = 0; r < kR5Side; ++r) {
                const uint32_t *q = &s_right[hw][r][at >> 2];
                const uint32_t q1 = q[1], q2 = q[2];
                const uint32_t w0 = __funnelshift_r(q[0], q1, sh), w1 = __funnelshift_r(q1, q2, sh),
                               w2 = __funnelshift_r(q2, q[3], sh) & 0x00FFFFFFu;
                const uint4 pa = *reinterpret_cast<const uint4 *>(&s_pair[hw][r][0]);
                const uint2 pb = *reinterpret_cast<const uint2 *>(&s_pair[hw][r][4]);
                const auto add = [&](uint32_t l, uint32_t rr) {
                    sum_max = __dp2a_lo(__vmaxu2(l + K2 - rr, 0x04000400u), 0x0101u, sum_max);
                };
                add(pa.x, w0 & 0x00FF00FFu);
                add(pa.y, (w0 >> 8) & 0x00FF00FFu);
                add(pa.z, w1 & 0x00FF00FFu);
                add(pa.w, (w1 >> 8) & 0x00FF00FFu);
                add(pb.x, w2 & 0x00FF00FFu);
                add(pb.y, (w2 >> 8) & 0x00FF00FFu);
                sum_r = __dp4a(w0, 0x01010101u, __dp4a(w1, 0x01010101u, __dp4a(w2, 0x01010101u, sum_r)));
            }
            // the twelfth pixel of a row is 0 on both sides: v = K there
            constexpr int kPix = kR5Side * kR5Side;
            const int a = (int)sum_max - kR5Side * max((int)K, 1024);
            sad = 2 * a - ((int)suml + kPix * (int)K - (int)sum_r) - kPix * 1024;
            key = ((uint32_t)sad << 4) | (uint32_t)l16;
        }
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) key = min(key, __shfl_xor_sync(0xFFFFFFFFu, key, off));
        const int kb = (int)(key & 15u);
        const int d1 = __shfl_sync(0xFFFFFFFFu, sad, max(kb - 1, 0), 16);
        const int d3 = __shfl_sync(0xFFFFFFFFu, sad, min(kb + 1, nsh - 1), 16);
        if (in && l16 == 0) {
            sad_out = key >> 4;
            const int ts = kb - L;
            if (ts != -L && ts != L)
                sub_pixel(A, xi, xr0, ts, d1, (int)sad_out, d3, b.prm.max_disp, bf, &disp_out, &depth_out);
        }
    }
    if (l16 == 0 && valid) {
        P.sub_disp[i] = disp_out;
        P.depth[i] = depth_out;
        P.corr[i] = sad_out;
    }
}

__global__ void __launch_bounds__(256) k_refine(const __grid_constant__ Batch b, int w, int L, double bf)
{
    __shared__ uint8_t s_left[8][kRefLeft];
    __shared__ uint8_t s_right[8][kRefRight];
    const int pair = blockIdx.y;
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int i = blockIdx.x * 8 + wi;
    const PairDesc &P = b.pairs[pair];
    const ImageDesc &Il = b.images[P.left];
    const ImageDesc &Ir = b.images[P.right];
    let_next();
    after_previous();
    if (i >= *Il.count) return;
    const int j = P.match_idx[i];
    float disp_out = -1.0f, depth_out = 0.0f;
    uint32_t sad_out = 0xFFFFFFFFu;
    if (j >= 0) {
        const int n = Il.out.level[i], xi = Il.out.x[i], yi = Il.out.y[i];
        const LevelDesc &A = b.levels[Il.level_base + n];
        const LevelDesc &B = b.levels[Ir.level_base + n];
        const int xr0 = right_column(A, Ir.out.X[j]);
        const int W = A.W, H = A.H;
        if (xi - w >= 0 && xi + w < W && yi - w >= 0 && yi + w < H && xr0 - L - w >= 0 && xr0 + L + w < W) {
            const int pw = 2 * w + 1, rw = 2 * (w + L) + 1;
            uint8_t *lp = s_left[wi], *rp = s_right[wi];
            const uint8_t *la0 = A.raw + (size_t)(yi - w) * A.pitch + (xi - w);
            const uint8_t *rb0 = B.raw + (size_t)(yi - w) * B.pitch + (xr0 - L - w);
            for (int r = 0; r < pw; ++r) {
                if (lane < pw) lp[r * pw + lane] = la0[(size_t)r * A.pitch + lane];
                for (int c = lane; c < rw; c += 32) rp[r * rw + c] = rb0[(size_t)r * B.pitch + c];
            }
            __syncwarp();
            const int nsh = 2 * L + 1;
            int part = 0;
            if (lane < 2 * nsh) {
                const int k = lane % nsh, half = lane / nsh;  // shift t = k - L
                const int lc = lp[w * pw + w], rc = rp[w * rw + k + w];
                const int r0 = half == 0 ? 0 : w, r1 = half == 0 ? w : pw;  // rows [0, w) and [w, 2w + 1)
                const int cc = lc - rc;  // |(l - lc) - (r - rc)| = |(l - r) - cc|
                for (int r = r0; r < r1; ++r) {
                    const uint8_t *la = lp + r * pw, *ra = rp + r * rw + k;
                    for (int c = 0; c < pw; ++c) part += abs((int)la[c] - (int)ra[c] - cc);
                }
            }
            const int other = __shfl_down_sync(0xFFFFFFFFu, part, nsh);
            const int sad = part + other;  // valid in lanes 0..nsh-1
            unsigned long long key = lane < nsh ? ((unsigned long long)sad << 8) | (unsigned)lane : ~0ull;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const unsigned long long o = __shfl_xor_sync(0xFFFFFFFFu, key, off);
                key = o < key ? o : key;
            }
            const int kb = (int)(key & 0xFFu);
            const int d1 = __shfl_sync(0xFFFFFFFFu, sad, max(kb - 1, 0));
            const int d3 = __shfl_sync(0xFFFFFFFFu, sad, min(kb + 1, nsh - 1));
            sad_out = (uint32_t)(key >> 8);
            const int ts = kb - L;
            if (ts != -L && ts != L)
                sub_pixel(A, xi, xr0, ts, d1, (int)sad_out, d3, b.prm.max_disp, bf, &disp_out, &depth_out);
        }
    }
    if (lane == 0) {
        P.sub_disp[i] = disp_out;
        P.depth[i] = depth_out;
        P.corr[i] = sad_out;
    }
}

constexpr int kMedThreads = 512, kMedKeep = 4;  // SADs a thread keeps in registers (the rest read again)

__global__ void __launch_bounds__(kMedThreads) k_refine_median(const __grid_constant__ Batch b)
{
    __shared__ uint32_t hist[2][kMedThreads];
    __shared__ uint32_t ws[kMedThreads / 32];
    __shared__ uint32_t s_digit[2], s_rank[2];
    const PairDesc &P = b.pairs[blockIdx.x];
    hist[0][threadIdx.x] = hist[1][threadIdx.x] = 0u;
    let_next();
    after_previous();
    const int n = *b.images[P.left].count;
    // SADs of the surviving matches (0xFFFFFFFF for the others: a SAD is at
    // most 441 x 510 < 2^18)
    const auto load = [&](int i) { return i < n && P.sub_disp[i] >= 0.0f ? P.corr[i] : 0xFFFFFFFFu; };
    uint32_t mine[kMedKeep];
#pragma unroll
    for (int q = 0; q < kMedKeep; ++q) mine[q] = load((int)threadIdx.x + q * kMedThreads);
    const auto each = [&](auto f) {
#pragma unroll
        for (int q = 0; q < kMedKeep; ++q)
            if (mine[q] != 0xFFFFFFFFu) f((int)threadIdx.x + q * kMedThreads, mine[q]);
        for (int i = threadIdx.x + kMedKeep * kMedThreads; i < n; i += kMedThreads) {
            const uint32_t v = load(i);
            if (v != 0xFFFFFFFFu) f(i, v);
        }
    };
    __syncthreads();
    uint32_t high = 0, rank = 0;
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
        each([&](int, uint32_t v) {
            if (pass == 0) atomicAdd(&hist[0][v >> 9], 1u);
            else if (v >> 9 == high) atomicAdd(&hist[1][v & 511u], 1u);
        });
        __syncthreads();
        // the digit of the element of rank `rank` in ascending order (pass 0:
        // the median is element total / 2 of the list)
        const uint32_t h = hist[pass][threadIdx.x];
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        uint32_t x = h;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) ws[w] = x;
        __syncthreads();
        const uint32_t t = lane < kMedThreads / 32 ? ws[lane] : 0u;
        const uint32_t before = __reduce_add_sync(0xFFFFFFFFu, lane < w ? t : 0u) + x - h;
        if (pass == 0) {
            const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, t);
            if (total == 0) return;  // by every thread
            rank = total / 2;
        }
        if (before <= rank && rank < before + h) { s_digit[pass] = threadIdx.x; s_rank[pass] = rank - before; }
        __syncthreads();
        if (pass == 0) { high = s_digit[0]; rank = s_rank[0]; }
    }
    const unsigned long long median = (high << 9) | s_digit[1];
    each([&](int i, uint32_t v) {
        if (10ull * v > 21ull * median) {
            P.sub_disp[i] = -1.0f;
            P.depth[i] = 0.0f;
        }
    });
}

cudaError_t launch_refine(const Batch &b, int w, int L, double bf, cudaStream_t stream)
{
    if (b.n_pairs == 0 || b.max_capacity == 0) return cudaSuccess;
    const cudaError_t e =
        w == kR5 ? launch_after(k_refine5, dim3((b.max_capacity + 15) / 16, b.n_pairs), dim3(256), 0, stream, b, L, bf)
                 : launch_after(k_refine, dim3((b.max_capacity + 7) / 8, b.n_pairs), dim3(256), 0, stream, b, w, L, bf);
    if (e != cudaSuccess) return e;
    return launch_after(k_refine_median, dim3(b.n_pairs), dim3(kMedThreads), 0, stream, b);
}

}  // namespace jslam
