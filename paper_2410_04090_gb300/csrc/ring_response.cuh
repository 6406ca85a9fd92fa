// The arc response: the alternative reading of the corner response of
// Sec. III ("sum of absolute differences over the circle", read as over the
// arc that makes the pixel a corner).  For each polarity whose longest
// circular run N of Eq. 1 labels satisfies Eq. 3 (P_min <= N <= P_max), the
// sum of (|d_k| - eps) over the ring positions that lie on a circular run of
// that polarity of length N; the response is the larger of the two sums.
// Every term is at least 1 (the labels are strict), so a corner's response
// lies in [P_min, 16 x 254]; it fits the 16-bit response field and the key
// response << 16 of the culling.
//
// The ring is walked in this library's order (position 0 below the centre,
// image y down); another start or direction around the circle keeps every
// circular run, so the sums are those of any other ordering of the ring.
#pragma once

#include <cstdint>

namespace jslam {

// What bounds it: instructions (a lane a corner), so no step loops or branches
// by its data: ring flags are shifted in by their sign bits, runs and the
// positions on them come by doubling, and the sum over the positions is four
// byte dot products.  Detection of 24 pairs of 647x363 with three keypoints a
// cell and this response: 201 us by walking the ring's bits, 100 so (86 with
// the whole ring's response).

// Longest circular run of set bits of a 16-bit mask (16 for 0xFFFF), and the
// positions lying on a run of that length.
__device__ __forceinline__ uint32_t ring_arc_positions(uint32_t m, int *len)
{
    // x_k, bit i: a run of k from position i on (bit i is position i mod 16)
    const uint32_t x1 = m | (m << 16), x2 = x1 & (x1 >> 1), x4 = x2 & (x2 >> 2), x8 = x4 & (x4 >> 4);
    uint32_t starts = 0xFFFFu, t;  // of the runs of n or more
    int n = 0;
    t = starts & x8;
    if (t) { starts = t; n = 8; }
    t = starts & (x4 >> n);
    if (t) { starts = t; n += 4; }
    t = starts & (x2 >> n);
    if (t) { starts = t; n += 2; }
    t = starts & (x1 >> n);
    if (t) { starts = t; n += 1; }
    if (m == 0xFFFFu) { starts = m; n = 16; }
    *len = n;
    // every start's n positions: windows of the largest power of two, twice
    uint32_t on = starts;
    int w = 1;
    if (n >= 2) { on |= on << 1; w = 2; }
    if (n >= 4) { on |= on << 2; w = 4; }
    if (n >= 8) { on |= on << 4; w = 8; }
    if (n > 0) on |= on << (n - w);  // a full ring's starts are all positions
    return n > 0 ? (on | (on >> 16)) & 0xFFFFu : 0u;
}

// Arc response of the pixel at p (rows rowb bytes apart) for threshold eps
// and run bounds [p_min, p_max]; 0 when neither polarity qualifies.
__device__ __forceinline__ int ring_arc(const uint8_t *p, int rowb, int eps, int p_min, int p_max)
{
    constexpr int DX[16] = { 0, 1, 2, 3, 3, 3, 2, 1, 0, -1, -2, -3, -3, -3, -2, -1 };
    constexpr int DY[16] = { 3, 3, 2, 1, 0, -1, -2, -3, -3, -3, -2, -1, 0, 1, 2, 3 };
    const int hi = (int)p[0] + eps, lo = (int)p[0] - eps;
    uint32_t v[16], mb = 0, md = 0;
#pragma unroll
    for (int k = 15; k >= 0; --k) {
        v[k] = p[DY[k] * rowb + DX[k]];
        mb = __funnelshift_l((uint32_t)(hi - (int)v[k]), mb, 1);
        md = __funnelshift_l((uint32_t)((int)v[k] - lo), md, 1);
    }
    uint32_t ring[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        ring[i] = v[4 * i] + (v[4 * i + 1] << 8) + ((v[4 * i + 2] << 16) + (v[4 * i + 3] << 24));
    int best = 0;
    const auto polarity = [&](bool bright) {
        int n;
        const uint32_t on = ring_arc_positions(bright ? mb : md, &n);
        uint32_t sum = 0;  // of the pixels on the runs
#pragma unroll
        for (int i = 0; i < 4; ++i)  // four bits to the low bits of four bytes
            sum = __dp4a(ring[i], (((on >> (4 * i)) & 0xFu) * 0x00204081u) & 0x01010101u, sum);
        const int c = __popc(on);
        const int r = bright ? (int)sum - c * hi : c * lo - (int)sum;
        if (n >= p_min && n <= p_max) best = max(best, r);
    };
    // nine of the sixteen positions: one polarity at most
    if (p_min >= 9) {
        polarity(__popc(mb) > __popc(md));
    } else {
        polarity(true);
        polarity(false);
    }
    return best;
}

}  // namespace jslam
