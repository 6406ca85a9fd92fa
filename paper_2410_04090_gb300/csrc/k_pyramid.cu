// Image pyramid with Gaussian filtering (Sec. III, streamlined multiscale
// detection and extraction: Gaussian filtering before ORB).
//
// k_pyramid   one warp per strip of any (image, level): resamples the level
//             from level 0 (bilinear, Q8 taps from host tables), writes it
//             (level 0: an aligned copy of the input), and writes its 7-tap
//             Gaussian.
//
// A strip has kPyrCols output columns and the level's pyr_rows output rows.  A
// lane owns four adjacent columns (one 32-bit word of the level) and walks
// down the rows with everything in registers; a warp never waits for another.
//   source    the strip's bytes of the source rows it needs, each once, are
//             brought into the warp's ring in shared memory by asynchronous
//             copies, a 16-byte unit a lane (the units that hold a byte of the
//             row's range), several rows ahead.
//   raw row   level 0: the input's four bytes.  Deeper levels are resampled
//             from level 0 separably and exactly: a source row's samples
//             (256 - a) p0 + a p1 are one two-way byte dot product each, over
//             the two source bytes that a byte permute picks from the eight
//             bytes at the lane's first tap; two rows' samples give four
//             rounded pixels.  A source row that two level rows need is
//             interpolated once.
//   Gaussian  7 taps, vertically first: a column's last four rows are the
//             bytes of one word, so its sum is two four-way dot products, over
//             that word and the one of four rows before; then horizontally on
//             the 16-bit column sums, the neighbours' by shuffles: each output
//             is four two-way dot products; one rounding at the end.
// The first and the last lane only supply the horizontal neighbours, so a
// strip is 30 lanes x 4 columns wide; a strip computes six rows more than it
// writes, three above and three below (see pyramid_strip_rows for how tall).
//
// What bounds it: instruction issue (77 % of the slots, 110 instructions per
// strip row; DRAM at 31 %, a pixel of the pyramid being two bytes written).
// For 100 pairs of 1241x376 with 8 levels it takes 0.333 ms; a CTA per
// 128 x 32 tile, with byte gathers and three shared-memory stages between
// barriers, executed 72 instructions per pixel and took 0.740 ms.  One pair
// (10 rows a strip): 16.2 us, before 19.6.
#include <cuda.h>

#include "jslam_internal.h"

namespace jslam {

// The blur weights w0 .. w6 as bytes for dot products: {0, w0, w1, w2},
// {w3, w4, w5, w6}, {w0, w1, w2, w3}, {w4, w5, w6, 0} (byte 0 first; every
// weight is below 256).
__constant__ uint32_t c_blur_pk[4];

cudaError_t set_blur_weights(const int32_t w[7])
{
    const auto B = [](int b0, int b1, int b2, int b3) {
        return (uint32_t)b0 | ((uint32_t)b1 << 8) | ((uint32_t)b2 << 16) | ((uint32_t)b3 << 24);
    };
    const uint32_t pk[4] = { B(0, w[0], w[1], w[2]), B(w[3], w[4], w[5], w[6]), B(w[0], w[1], w[2], w[3]),
                             B(w[4], w[5], w[6], 0) };
    return cudaMemcpyToSymbol(c_blur_pk, pk, sizeof(pk));
}

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint32_t ld_shared(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}

// Where a lane's four columns come from in a source row.
//   kPyrCopy   level 0: four bytes from one word window
//   kPyrOne    the four taps' bytes lie in eight bytes (up to 2 source
//              columns an output column)
//   kPyrTwo    the first two taps' in eight bytes, the last two's in another
//              eight (up to 6)
//   kPyrBytes  any scale: two byte loads a column, from global memory
template <int MODE> struct PyrTaps {
    static constexpr int kWin = MODE == kPyrTwo ? 2 : 1;         // windows
    uint32_t off[MODE == kPyrBytes ? 8 : kWin];  // first column of each window (of each byte: kPyrBytes)
    uint32_t sel[MODE == kPyrBytes ? 1 : 4];     // byte selectors: the two taps of a column (kPyrCopy: sel[0], all four)
    uint32_t wgt[4];                             // 256 - a | a << 16

    // the lane's columns gx .. gx + 3, clamped to the level; W0 >= 8
    __device__ __forceinline__ void init(const LevelDesc &L, int W0, int gx)
    {
        if constexpr (MODE == kPyrCopy) {
            const int xs = min(max(gx, 0), W0 - 4);
            uint32_t s = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) s |= (uint32_t)(min(max(gx + k, 0), W0 - 1) - xs) << (4 * k);
            off[0] = (uint32_t)xs;
            sel[0] = s;
        } else {
            int xa[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t t = __ldg(L.tapx + min(max(gx + k, 0), L.W - 1));
                xa[k] = (int)(t & 0xFFFFu);
                wgt[k] = (256u - (t >> 16)) | (t & 0xFFFF0000u);
            }
            if constexpr (MODE == kPyrBytes) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    off[2 * k] = (uint32_t)xa[k];
                    off[2 * k + 1] = (uint32_t)min(xa[k] + 1, W0 - 1);
                }
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    // a window of eight bytes inside the row
                    const int first = min(MODE == kPyrTwo && k >= 2 ? xa[2] : xa[0], W0 - 8);
                    off[MODE == kPyrTwo ? k >> 1 : 0] = (uint32_t)first;
                    sel[k] = (uint32_t)(xa[k] - first) | ((uint32_t)(min(xa[k] + 1, W0 - 1) - first) << 4);
                }
            }
        }
    }

    // eight (kPyrCopy: four) bytes at shared address o
    static __device__ __forceinline__ void window(uint32_t o, uint32_t &a, uint32_t &z)
    {
        const uint32_t p = o & ~3u, w1 = ld_shared(p + 4);
        a = __funnelshift_r(ld_shared(p), w1, o << 3);  // takes the shift modulo 32
        if (MODE != kPyrCopy) z = __funnelshift_r(w1, ld_shared(p + 8), o << 3);
    }

    // the four horizontal samples of a source row whose range lies at shared
    // address at (kPyrBytes: of the row `row` in global memory)
    __device__ __forceinline__ void samples(uint32_t at, const uint8_t *row, uint32_t (&h)[4]) const
    {
        if constexpr (MODE == kPyrBytes) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                h[k] = (wgt[k] & 0xFFFFu) * row[off[2 * k]] + (wgt[k] >> 16) * row[off[2 * k + 1]];
        } else {
            uint32_t a[kWin], z[kWin];
#pragma unroll
            for (int i = 0; i < kWin; ++i) window(at + off[i], a[i], z[i]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = MODE == kPyrTwo ? k >> 1 : 0;
                h[k] = __dp2a_lo(wgt[k], __byte_perm(a[i], z[i], sel[k]), 0u);
            }
        }
    }
};

// A warp's shared memory: the source ring, and per row of the strip (and a
// few past its end) the source rows to copy and the ones to use.
//   bring  for its first and second source row: offset of the 16-byte unit
//          that holds the range's first byte; shared address | bytes from that
//          unit to the range's end << 20 (0 bytes: nothing to copy)
//   use    where the ranges of the two source rows lie (shared addresses;
//          kPyrBytes: the source rows), the vertical weight, whether the first
//          one is new
struct __align__(16) PyrShared {
    uint8_t ring[kPyrRing];
    uint4 bring[kPyrMaxRows + 18];
    uint4 use[kPyrMaxRows + 10];
};

__device__ __forceinline__ void st_global_if(bool p, uint8_t *to, uint32_t v)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %0, 0;\n @p st.global.u32 [%1], %2;\n}"
                 ::"r"((uint32_t)p), "l"(to), "r"(v) : "memory");
}

__device__ __forceinline__ void copy16_if(bool p, uint32_t to, const uint8_t *from)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %0, 0;\n @p cp.async.cg.shared.global [%1], [%2], 16;\n}"
                 ::"r"((uint32_t)p), "r"(to), "l"(from) : "memory");
}

template <int MODE>
__device__ __forceinline__ void pyramid_strip(const Batch &b, const LevelDesc &L, PyrShared &S, const uint8_t *base,
                                              int pitch0, int W0, int H0, int x0, int y0)
{
    constexpr int kAhead = MODE == kPyrTwo ? kPyrAheadTwo : kPyrAhead;  // rows ahead that are being copied
    const int lane = threadIdx.x;
    const int W = L.W, H = L.H, pitch = L.pitch;
    const int n = min(L.pyr_rows, H - y0) + 6;  // rows y0 - 3 .. of the level, clamped
    const int gx = x0 - 4 + 4 * lane;
    const bool writes = lane >= 1 && lane <= 30 && gx < W;
    PyrTaps<MODE> T;
    T.init(L, W0, gx);

    // The source rows' common byte range: whole windows, clamped at the edges.
    // A row is copied from the 16-byte boundary at or before its first byte.
    uint32_t c_first = 0, c_bytes = 0, stride = 0, slots = 1;
    const uint32_t ring = smem_u32(S.ring);
    if constexpr (MODE != kPyrBytes) {
        c_first = __shfl_sync(0xFFFFFFFFu, T.off[0], 0);
        c_bytes = __shfl_sync(0xFFFFFFFFu, T.off[PyrTaps<MODE>::kWin - 1], 31) + (MODE == kPyrCopy ? 4 : 8) - c_first;
        stride = (c_bytes + 15u + 15u) & ~15u;
        slots = (uint32_t)kPyrRing / stride;
#pragma unroll
        for (int i = 0; i < PyrTaps<MODE>::kWin; ++i) T.off[i] -= c_first;
    }
    const uintptr_t from = reinterpret_cast<uintptr_t>(base) + c_first;
    const uint32_t lead0 = (uint32_t)(from & 15u);

    // What each row needs: its second source row, and its first one unless
    // the row before has it as its second.  A row above the level's first or
    // below its last repeats the row before and uses the same source rows.
    uint32_t n_src = 0;
    for (int q0 = 0; q0 < n + 12; q0 += 32) {
        const int q = q0 + lane, y = y0 - 3 + q;
        int r[2][2];  // first and second source row of the row before and of this one
        uint32_t w = 0;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int cy = min(max(y - 1 + i, 0), H - 1);
            const uint32_t t = MODE == kPyrCopy ? (uint32_t)cy : __ldg(L.tapy + cy);
            r[i][0] = (int)(t & 0xFFFFu);
            r[i][1] = MODE == kPyrCopy ? r[i][0] : min(r[i][0] + 1, H0 - 1);
            w = t >> 16;
        }
        const bool fresh = q < n && (q == 0 || (y > 0 && y < H));
        const bool first = MODE != kPyrCopy && fresh && (q == 0 || r[1][0] != r[0][1]);
        const uint32_t bf = __ballot_sync(0xFFFFFFFFu, fresh), b1 = __ballot_sync(0xFFFFFFFFu, first);
        const uint32_t below = (1u << lane) - 1u;
        // its second source row, counting the new ones (the first one is the one before)
        const uint32_t m = n_src + __popc(bf & below) + __popc(b1 & below) + (first ? 1u : 0u) - (fresh ? 0u : 1u);
        const uint32_t oa = lead0 + (uint32_t)r[1][0] * (uint32_t)pitch0, ob = lead0 + (uint32_t)r[1][1] * (uint32_t)pitch0;
        const uint32_t ta = ring + (m - 1u) % slots * stride, tb = ring + m % slots * stride;
        if (q < n + 12)
            S.bring[q] = make_uint4(oa & ~15u, first ? ta | ((oa & 15u) + c_bytes) << 20 : 0u, ob & ~15u,
                                    fresh ? tb | ((ob & 15u) + c_bytes) << 20 : 0u);
        if (q < n + 3)
            S.use[q] = make_uint4(MODE == kPyrBytes ? (uint32_t)r[1][0] : ta + (oa & 15u),
                                  MODE == kPyrBytes ? (uint32_t)r[1][1] : tb + (ob & 15u), w,
                                  MODE != kPyrOne || first || !fresh ? 1u : 0u);
        n_src += __popc(bf) + __popc(b1);
    }
    __syncwarp();

    // Rows q and q + 1: a lane copies one 16-byte unit of a source row.  Level
    // 0 has one source row per row; kPyrOne rows have up to 16 units, so the
    // warp's halves take the two source rows.
    const uint32_t unit = 16u * (uint32_t)(MODE == kPyrOne ? lane & 15 : lane);
    const uint8_t *const from_l = reinterpret_cast<const uint8_t *>(from & ~static_cast<uintptr_t>(15)) + unit;
    const auto bring = [&](int q) {
        if constexpr (MODE != kPyrBytes) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = MODE == kPyrTwo ? 0 : 1; j < 2; ++j) {
                    const uint2 c = reinterpret_cast<const uint2 *>(S.bring + q + i)[MODE == kPyrOne ? lane >> 4 : j];
                    copy16_if(unit < c.y >> 20, (c.y & 0xFFFFFu) + unit, from_l + c.x);
                }
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
    };
    for (int q = 0; q < kAhead; q += 2) bring(q);

    // rows y0 - 3 + q of this lane's word, as far down as the loop is
    uint8_t *raw_p = L.raw_w + ((ptrdiff_t)(y0 - 3) * pitch + gx);
    const ptrdiff_t to_blur = L.blur - L.raw_w - 3 * (ptrdiff_t)pitch;
    const uint32_t A = c_blur_pk[0], Bw = c_blur_pk[1], Cw = c_blur_pk[2], Dw = c_blur_pk[3];
    uint32_t hb[4] = {};
    // column k's bytes of rows q - 3 .. q, newest in byte 3, kept for four
    // rows in slots that rotate with the row (the loop is unrolled over them)
    uint32_t col[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k) col[j][k] = 0;

    for (int q0 = 0; q0 < n; q0 += 4) {  // the rows past n - 1 write nothing
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = q0 + u;
            if (MODE != kPyrBytes && (u & 1) == 0) {
                asm volatile("cp.async.wait_group %0;" ::"n"(kAhead / 2 - 1) : "memory");
                __syncwarp();  // every lane's units of the two rows are there; every lane is done with the rows before
                bring(q + kAhead);
            }
            const uint4 use = S.use[q];
            uint32_t word;  // the raw word of the row
            if constexpr (MODE == kPyrCopy) {
                uint32_t a, z;
                PyrTaps<MODE>::window(use.y + T.off[0], a, z);
                word = __byte_perm(a, 0u, T.sel[0]);
            } else {
                uint32_t ha[4];
                if (MODE != kPyrOne || __any_sync(0xFFFFFFFFu, use.w)) {
                    T.samples(use.x, base + (size_t)use.x * pitch0, ha);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) ha[k] = hb[k];
                }
                T.samples(use.y, base + (size_t)use.y * pitch0, hb);
                // rounded sums below 2^24: the pixel is byte 2 of each
                const uint32_t w1 = use.z, w0 = 256u - w1;
                uint32_t v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) v[k] = w0 * ha[k] + (w1 * hb[k] + 32768u);
                word = __byte_perm(__byte_perm(v[0], v[1], 0x0062), __byte_perm(v[2], v[3], 0x0062), 0x5410);
            }
            st_global_if(writes && (uint32_t)(q - 3) < (uint32_t)(n - 6), raw_p, word);
            uint32_t v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t older = col[u][k];
                // newest byte in, the oldest out
                col[u][k] = __byte_perm(col[(u + 3) & 3][k], word, 0x4321u + (uint32_t)(k << 12));
                // rows q - 6 .. q - 4 against {0, w0, w1, w2}, q - 3 .. q against {w3, w4, w5, w6}
                v[k] = __dp4a(col[u][k], Bw, __dp4a(older, A, 0u));
            }
            if (q0 > 0) {  // output row y0 + q - 6
                // column sums, two to a word: columns -4 .. 7 of the lane's word
                uint32_t c[6];
                c[2] = __byte_perm(v[0], v[1], 0x5410);
                c[3] = __byte_perm(v[2], v[3], 0x5410);
                c[0] = __shfl_up_sync(0xFFFFFFFFu, c[2], 1);
                c[1] = __shfl_up_sync(0xFFFFFFFFu, c[3], 1);
                c[4] = __shfl_down_sync(0xFFFFFFFFu, c[2], 1);
                c[5] = __shfl_down_sync(0xFFFFFFFFu, c[3], 1);
                // words i .. i + 3 against the weight words P (first two) and Q
                // (last two); the rounding term starts each sum, the sums stay
                // below 2^24, so each result is byte 2 of its sum
                const auto dot7 = [&](int i, uint32_t P, uint32_t Q) {
                    const uint32_t lo = __dp2a_hi(c[i + 1], P, __dp2a_lo(c[i], P, 32768u));
                    return __dp2a_hi(c[i + 3], Q, __dp2a_lo(c[i + 2], Q, lo));
                };
                const uint32_t s0 = dot7(0, A, Bw), s1 = dot7(1, Cw, Dw), s2 = dot7(1, A, Bw), s3 = dot7(2, Cw, Dw);
                st_global_if(writes && (uint32_t)(q - 6) < (uint32_t)(n - 6), raw_p + to_blur,
                             __byte_perm(__byte_perm(s0, s1, 0x0062), __byte_perm(s2, s3, 0x0062), 0x5410));
            }
            raw_p += pitch;
        }
    }
}

// One warp per CTA: every branch on a strip's rows is uniform for the compiler.
__global__ void __launch_bounds__(32, kPyrWarpsPerSm) k_pyramid(const __grid_constant__ Batch b,
                                                                 const __grid_constant__ Inputs in)
{
    __shared__ PyrShared S;
    after_previous();
    let_next();
    if (blockIdx.x == 0 && threadIdx.x == 0) *b.tile_next = 0u;  // for the detection launch that follows
    const PyrRec R = b.pyr_rec[b.pyr_first + blockIdx.x];
    const LevelDesc &L = b.levels[R.level];
    const ImageDesc &I = b.images[L.image];
    const int x0 = R.x0, y0 = R.y0;
    // level 0 reads the input; deeper levels resample the input, or in the
    // cascaded pyramid the level above (complete: an earlier launch)
    const uint8_t *base = L.src ? L.src : in.ptr[L.image];
    const int W0 = L.src ? L.src_W : I.W0, H0 = L.src ? L.src_H : I.H0;
    const int pitch0 = L.src ? L.src_pitch : in.pitch[L.image];
    switch (L.pyr_mode) {
    case kPyrCopy: pyramid_strip<kPyrCopy>(b, L, S, base, pitch0, W0, H0, x0, y0); break;
    case kPyrOne: pyramid_strip<kPyrOne>(b, L, S, base, pitch0, W0, H0, x0, y0); break;
    case kPyrTwo: pyramid_strip<kPyrTwo>(b, L, S, base, pitch0, W0, H0, x0, y0); break;
    default: pyramid_strip<kPyrBytes>(b, L, S, base, pitch0, W0, H0, x0, y0); break;
    }
}

const void *pyramid_kernel() { return reinterpret_cast<const void *>(k_pyramid); }

// The launch may start while the call before ends where its strips are more
// than two rounds of those that run at once, and in a cascaded pyramid.  With
// fewer, the strips that start early are not spread evenly, and the last ones
// wait for them.  us a call, early or not: 100 pairs of 640x480 230 / 233, 16
// mixed pairs 363 / 366, 16 of 800x602 cascaded 321 / 324; 12 of 752x480 with
// the learned skip (1.4 rounds) 218 / 212, 24 of 647x363 240 / 239.
cudaError_t launch_pyramid_strips(const Batch &b, const Inputs &in, int first, int count, cudaStream_t stream)
{
    if (count == 0) return cudaSuccess;
    Batch bn = b;
    bn.pyr_first = first;
    const bool early = b.pyr_cascaded || count > 2 * b.n_sm * kPyrWarpsPerSm;
    return launch_if(early, k_pyramid, dim3(count), dim3(32), 0, stream, bn, in);
}

cudaError_t launch_pyramid(const Batch &b, const Inputs &in, cudaStream_t stream)
{
    if (!b.pyr_cascaded) return launch_pyramid_strips(b, in, 0, b.pyr_tiles, stream);
    // cascaded: level number n after n - 1, each launch over every image
    for (int n = 0; n < kMaxLevels; ++n) {
        const int first = b.pyr_pass_first[n];
        const cudaError_t e = launch_pyramid_strips(b, in, first, b.pyr_pass_first[n + 1] - first, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace jslam
