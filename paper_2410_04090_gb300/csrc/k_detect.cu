// Detection stage: FAST with Bounded Rectification, per-cell culling and the
// scatter half of PFA.
//
// k_fast_bits persistent CTAs over blocks of culling cells of any (image,
//             level): stage the raw tile plus its halo in shared memory (TMA),
//             evaluate the 16-pixel ring of every pixel (Sec. II-A, Eq. 1 labels, Eq. 3
//             bounded run length; Sec. III bit masks and SAD response), keep
//             the top-k corners of each cell (Sec. II-C-1, Feature Culling)
//             and add each survivor to the s0 score map (Sec. II-C-2, PFA
//             steps 1-2: K_l and K_r accumulate in one packed word).  The tile
//             is transposed into bit-planes and each thread tests 32 pixels
//             of a row at once with bitwise arithmetic (carry-chain compares,
//             run windows), scoring its corners in place; tiles come with
//             host-made records staged by bulk copies.
#include <algorithm>
#include <type_traits>

#include <cuda.h>

#include "jslam_internal.h"
#include "ring_response.cuh"

namespace jslam {

// ---------------------------------------------------------------- FAST + FC
//
// One persistent CTA loops over detection tiles (a block of whole culling
// cells of any image and level).  The raw tile plus its halo is fetched by
// TMA (one 2-D tensor map per level) into one of two shared-memory buffers
// while the CTA works on the other, with an mbarrier per buffer.  Per tile:
//   1. the tile's bytes become bit-planes, 32 pixels of a row to a word;
//   2. primary threshold: a thread compares the 16 ring positions of 32 pixels
//      at a time and tests the circular runs of the flags (Eq. 3, P_min and
//      P_max) with word operations;
//   3. each corner's response is computed and the cell's top-k is kept by
//      atomicMax on the key response << 16 | (0xFFFF - index in cell)
//      (strongest first, then smaller y, then smaller x);
//   4. fallback threshold, only for pixels of cells left without a corner
//      (cells with no pixel inside the border never ask for it);
//   5. slots are written and every survivor is added to the s0 score map
//      (PFA steps 1-2: K_l << 16 | K_r in one word).

// Majority of three words, bitwise: the carry out of a + b with carry in c.
__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a | b)); }

__host__ __device__ inline int fast_align(int v, int a) { return (v + a - 1) / a * a; }

// Dynamic shared memory of the kernel: the two tile boxes, the
// box's bit-planes (max_planes bytes: box rows of (chunks + 1) x 8 words and
// a 16-byte pad, see bs_row_units), cell states and selections of two tiles
// (by tile parity) and the work list of a pass (16-bit item indices; a tile
// has at most kFastMaxTile rows of 4 items).  The fixed-size parts (corner
// windows, tile records, staged projections, mbarriers) are static arrays of
// the kernel.
constexpr int kBitsWin = 128;
constexpr int kBitsMaxItems = kFastMaxTile * (kFastMaxTile / 32);
struct BitsLayout {
    int buf0, buf1, planes, has_hi, sel, wlist, total;
};
__host__ __device__ inline BitsLayout bits_layout(int max_box, int max_cells, int k, int max_planes)
{
    BitsLayout l;
    int o = 0;
    l.buf0 = o;   o += fast_align(max_box, 128);
    l.buf1 = o;   o += fast_align(max_box, 128);
    l.planes = o; o += fast_align(max_planes, 16);
    l.has_hi = o; o += 2 * fast_align(max_cells, 16);
    l.sel = o;    o += 2 * fast_align(max_cells * k * 4, 16);
    l.wlist = o;  o += kBitsMaxItems * 2;
    l.total = o;
    return l;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Whether the mbarrier phase `parity` is complete (waits a bounded time itself).
__device__ __forceinline__ bool try_tile(uint64_t *bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return done != 0;
}

// Wait for the mbarrier phase `parity`, giving up after about a second.
__device__ __forceinline__ bool wait_tile(uint64_t *bar, uint32_t parity)
{
    if (try_tile(bar, parity)) return true;
    const long long start = clock64();
    while (clock64() - start <= (1ll << 31))
        if (try_tile(bar, parity)) return true;
    return false;
}

// Failure-detection self-test: a tile wait on an mbarrier that nothing
// arrives on runs out after its limit, sets kErrTimeout and returns, as the
// detection kernels do when a tile load does not complete.
__global__ void k_wait_selftest(uint32_t *err)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (!wait_tile(&bar, 0u) && threadIdx.x == 0) atomicOr(err, kErrTimeout);
}

cudaError_t launch_wait_selftest(uint32_t *err, cudaStream_t stream)
{
    k_wait_selftest<<<1, 32, 0, stream>>>(err);
    return cudaGetLastError();
}

// ---- bit-sliced ring test: 32 pixels per word, bit j of word i = bit i of
// pixel j's byte.  a > b for 8-bit numbers: the carry out of a + ~b, one
// majority per bit; c + e: a ripple adder against the constant's bit masks.

// Bit-planes of a 32-byte chunk (bytes j of words a, z in memory order):
// output word i, bit j = bit i of byte j.  The bytes are gathered so that byte
// b of word w is byte 8 b + w of the chunk; each byte lane of the eight words
// is then an 8 x 8 bit matrix (row = word, column = bit), transposed by three
// rounds of exchanges between words 4, 2 and 1 apart.
__device__ __forceinline__ void bs_transpose(uint4 a, uint4 z, uint4 *dst)
{
    uint32_t w[8];
    const uint32_t v[2][4] = { { a.x, a.z, z.x, z.z }, { a.y, a.w, z.y, z.w } };
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t t0 = __byte_perm(v[h][0], v[h][1], 0x5140), t1 = __byte_perm(v[h][0], v[h][1], 0x7362);
        const uint32_t u0 = __byte_perm(v[h][2], v[h][3], 0x5140), u1 = __byte_perm(v[h][2], v[h][3], 0x7362);
        w[4 * h + 0] = __byte_perm(t0, u0, 0x5410);
        w[4 * h + 1] = __byte_perm(t0, u0, 0x7632);
        w[4 * h + 2] = __byte_perm(t1, u1, 0x5410);
        w[4 * h + 3] = __byte_perm(t1, u1, 0x7632);
    }
#pragma unroll
    for (int s = 4; s > 0; s >>= 1) {
        const uint32_t m = s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (i & s) continue;
            const uint32_t lo = w[i], hi = w[i + s];
            w[i] = (lo & m) | ((hi << s) & ~m);
            w[i + s] = ((lo >> s) & m) | (hi & ~m);
        }
    }
    dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
    dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
}

__device__ __forceinline__ uint32_t bs_greater(const uint32_t (&a)[8], const uint32_t (&b)[8])
{
    uint32_t c = a[0] & ~b[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) c = maj3(a[i], ~b[i], c);
    return c;
}

// Longest circular run of the 16 flag words in [9, 13]: A3 = windows of 3, A9
// = three A3 end to end, a run of 14 = an A9 and the one five positions on.
__device__ __forceinline__ uint32_t bs_run_9_13(const uint32_t (&F)[16])
{
    uint32_t A3[16], A9[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) A3[q] = F[q] & F[(q + 1) & 15] & F[(q + 2) & 15];
#pragma unroll
    for (int q = 0; q < 16; ++q) A9[q] = A3[q] & A3[(q + 3) & 15] & A3[(q + 6) & 15];
    uint32_t r9 = A9[0] | A9[1], r14 = A9[0] & A9[5];
#pragma unroll
    for (int q = 2; q < 16; q += 2) r9 |= A9[q] | A9[q + 1];
#pragma unroll
    for (int q = 1; q < 16; ++q) r14 |= A9[q] & A9[(q + 5) & 15];
    return r9 & ~r14;
}

// Whether one of the 16 words A and the one `off` (0..kTop) positions on are
// both set, per bit.  off is the same in all threads.
template <int kTop>
__device__ __forceinline__ uint32_t bs_both_any(const uint32_t (&A)[16], int off)
{
    const auto at = [&](int o) {
        uint32_t x = 0, y = 0;
#pragma unroll
        for (int q = 0; q < 16; q += 2) {
            x |= A[q] & A[(q + o) & 15];
            y |= A[q + 1] & A[(q + 1 + o) & 15];
        }
        return x | y;
    };
    if (kTop == 0) return at(0);
    if (kTop == 1) return off ? at(1) : at(0);
    if (kTop == 3) {
        switch (off) {
        case 0: return at(0);
        case 1: return at(1);
        case 2: return at(2);
        default: return at(3);
        }
    }
    switch (off) {
    case 0: return at(0);
    case 1: return at(1);
    case 2: return at(2);
    case 3: return at(3);
    case 4: return at(4);
    case 5: return at(5);
    case 6: return at(6);
    case 7: return at(7);
    default: return at(8);
    }
}

// Windows of W flags to windows of 2 W.
template <int W>
__device__ __forceinline__ void bs_double(uint32_t (&A)[16])
{
    uint32_t B[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) B[q] = A[q] & A[(q + W) & 15];
#pragma unroll
    for (int q = 0; q < 16; ++q) A[q] = B[q];
}

// Whether the longest circular run of the 16 flag words of either polarity is
// in [p_min, p_max]; the words of F are spent.  A run of n or more is two
// windows of w flags, w the largest power of two (up to 8) that is not above
// n, n - w positions apart; p_max = 16 has no upper test.  Loops, since four
// copies of the switch cost more (178 -> 198 us).
__device__ __forceinline__ uint32_t bs_run_any(uint32_t (&F)[2][16], uint32_t nb, uint32_t nd, int p_min, int p_max)
{
    uint32_t bits = 0, never = nb;
    const int over = p_max + 1;
#pragma unroll 1
    for (int p = 0; p < 2; ++p) {
        uint32_t least = 0, more = 0;
        const auto test = [&](auto top, int w) {
#pragma unroll 1
            for (int t = 0; t < 2; ++t) {
                const int off = (t ? over : p_min) - w;
                if ((unsigned)off > (unsigned)decltype(top)::value) continue;
                const uint32_t r = bs_both_any<decltype(top)::value>(F[0], off);
                if (t) more = r;
                else least = r;
            }
        };
        if (p_min < 8) test(std::integral_constant<int, 0>{}, 1);
        bs_double<1>(F[0]);
        if (p_min < 8) test(std::integral_constant<int, 1>{}, 2);
        bs_double<2>(F[0]);
        if (p_min < 8) test(std::integral_constant<int, 3>{}, 4);
        bs_double<4>(F[0]);
        test(std::integral_constant<int, 8>{}, 8);
        bits |= least & ~more & ~never;
        never = nd;
#pragma unroll
        for (int q = 0; q < 16; ++q) F[0][q] = F[1][q];
    }
    return bits;
}

// Bounded-rectification response of the pixel at p (rows rowb bytes apart):
// the sum of |ring pixel - centre| over the 16 ring positions, the ring
// bytes packed four to a word (rows +-3: dx = -1, 0, 1; rows +-2: dx = +-2;
// rows +-1 and 0: dx = +-3) and summed by byte-SIMD absolute differences.
__device__ __forceinline__ int ring_sad(const uint8_t *p, int rowb)
{
    const uint8_t *u3 = p + 3 * rowb, *d3 = p - 3 * rowb, *u2 = p + 2 * rowb, *d2 = p - 2 * rowb;
    const uint8_t *u1 = p + rowb, *d1 = p - rowb;
    const uint32_t w0 = (uint32_t)u3[-1] | ((uint32_t)u3[0] << 8) | ((uint32_t)u3[1] << 16) | ((uint32_t)d3[-1] << 24);
    const uint32_t w1 = (uint32_t)d3[0] | ((uint32_t)d3[1] << 8) | ((uint32_t)u2[-2] << 16) | ((uint32_t)u2[2] << 24);
    const uint32_t w2 = (uint32_t)d2[-2] | ((uint32_t)d2[2] << 8) | ((uint32_t)u1[-3] << 16) | ((uint32_t)u1[3] << 24);
    const uint32_t w3 = (uint32_t)d1[-3] | ((uint32_t)d1[3] << 8) | ((uint32_t)p[-3] << 16) | ((uint32_t)p[3] << 24);
    const uint32_t cc = (uint32_t)p[0] * 0x01010101u;
    return (int)(__vsadu4(w0, cc) + __vsadu4(w1, cc) + __vsadu4(w2, cc) + __vsadu4(w3, cc));
}

// Corner bits of the 32 pixels of tile row py, chunk m (pixels 32 m + j).
// `planes`: box rows of `ru` 16-byte units, chunk m at unit 2 m; tile pixel 0
// sits at box column sb, so pixel 32 m + j + dx is bit sb + dx + j of chunks
// (m, m + 1).  kAny: any run bounds, else 9 and 13.
template <bool kAny>
__device__ __forceinline__ uint32_t bs_corners(const uint32_t *planes, int ru, int py, int m, int sb,
                                               const uint32_t (&eps)[8], int p_min, int p_max)
{
    constexpr int RDX[16] = { 0, 1, 2, 3, 3, 3, 2, 1, 0, -1, -2, -3, -3, -3, -2, -1 };
    constexpr int RDY[16] = { 3, 3, 2, 1, 0, -1, -2, -3, -3, -3, -2, -1, 0, 1, 2, 3 };
    uint32_t C[8], Tb[8], Td[8];
    {
        const uint4 *r = reinterpret_cast<const uint4 *>(planes) + (py + 3) * ru + 2 * m;
        const uint4 l0 = r[0], l1 = r[1], h0 = r[2], h1 = r[3];
        const uint32_t lo[8] = { l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w };
        const uint32_t hi[8] = { h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w };
#pragma unroll
        for (int i = 0; i < 8; ++i) C[i] = __funnelshift_r(lo[i], hi[i], sb);
    }
    // thresholds C + eps and C - eps = ~(~C + eps), eps as a word mask for each
    // of its bits; a centre whose sum wraps (nb: C + eps >= 256, nd: C < eps)
    // is never brighter (darker), its flags are dropped at the end
    uint32_t nb = 0, nd = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        Tb[i] = C[i] ^ eps[i] ^ nb;
        Td[i] = C[i] ^ eps[i] ^ nd;
        nb = maj3(C[i], eps[i], nb);
        nd = maj3(~C[i], eps[i], nd);
    }
    uint32_t F[2][16];  // brighter, darker
#pragma unroll
    for (int dy = 3; dy >= -3; --dy) {
        const uint4 *r = reinterpret_cast<const uint4 *>(planes) + (py + 3 + dy) * ru + 2 * m;
        const uint4 l0 = r[0], l1 = r[1], h0 = r[2], h1 = r[3];
        const uint32_t lo[8] = { l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w };
        const uint32_t hi[8] = { h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w };
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            if (RDY[q] != dy) continue;
            uint32_t P[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) P[i] = __funnelshift_r(lo[i], hi[i], sb + RDX[q]);
            F[0][q] = bs_greater(P, Tb);
            F[1][q] = bs_greater(Td, P);
        }
    }
    if (kAny) return bs_run_any(F, nb, nd, p_min, p_max);
    return (bs_run_9_13(F[0]) & ~nb) | (bs_run_9_13(F[1]) & ~nd);
}

// Bits j of the 32 pixels of tile row chunk px0..px0+31 whose cell state
// (row of states `st`, cells of c pixels) satisfies keep(state).
template <typename Keep>
__device__ __forceinline__ uint32_t cell_bits(const uint8_t *st, int px0, int tw, int c, uint32_t cinv, Keep keep)
{
    const int x_last = min(px0 + 31, tw - 1);
    const int c0 = (int)(((uint32_t)px0 * cinv) >> 16), c1 = (int)(((uint32_t)x_last * cinv) >> 16);
    uint32_t bits = 0;
    for (int cx = c0; cx <= c1; ++cx) {
        if (!keep(st[cx])) continue;
        const int a = max(cx * c - px0, 0), z = min((cx + 1) * c - px0, 32);
        bits |= (z >= 32 ? 0xFFFFFFFFu : ((1u << z) - 1u)) & (0xFFFFFFFFu << a);
    }
    return bits;
}

// floor(v / c) for 0 <= v < 128 and 1 <= c <= 128 with cinv = ceil(2^16 / c):
// exact because v * c < 2^16 (as for the tile's items, v < 2^11 and c <= 5).
__device__ __forceinline__ int div_small(int v, uint32_t cinv) { return (int)(((uint32_t)v * cinv) >> 16); }

// v / d by d's reciprocal (recip_of; 0 stands for d = 1).
__device__ __forceinline__ int div_recip(int v, uint32_t recip) { return recip ? (int)__umulhi((uint32_t)v, recip) : v; }

// Bits j of the 32 pixels px0 + j of a tile row that lie inside the level's
// evaluated columns [plo, phi) (tile coordinates).
__device__ __forceinline__ uint32_t border_bits(int px0, int plo, int phi)
{
    const int lo = min(max(plo - px0, 0), 32), hi = min(max(phi - px0, 0), 32);
    return (hi >= 32 ? 0xFFFFFFFFu : ((1u << hi) - 1u)) & (lo >= 32 ? 0u : (0xFFFFFFFFu << lo));
}

// Work list of a pass of k_fast_bits: appends to wlist (count in *n) every
// item (row r0 + itm / nch, chunk itm % nch) holding an evaluated pixel whose
// cell state satisfies keep(state), so that the pass runs full warps over
// those items only.  Warp-uniform loop; one atomic per warp and round.
template <typename Keep>
__device__ __forceinline__ void list_items(uint16_t *wlist, int *n, int items, int nch, uint32_t nchinv, int r0,
                                           int plo, int phi, const uint8_t *has_hi, int ncx, int tw, int c,
                                           uint32_t cinv, int lane, int warp, Keep keep)
{
    for (int base = warp * 32; base < items; base += kFastThreads) {
        const int itm = base + lane;
        bool need = false;
        if (itm < items) {
            const int rr = div_small(itm, nchinv), px0 = 32 * (itm - rr * nch);
            const uint32_t v = border_bits(px0, plo, phi);
            need = v && (v & cell_bits(has_hi + div_small(r0 + rr, cinv) * ncx, px0, tw, c, cinv, keep));
        }
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, need);
        int at = 0;
        if (lane == 0 && bal) at = atomicAdd(n, __popc(bal));
        at = __shfl_sync(0xFFFFFFFFu, at, 0);
        if (need) wlist[at + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)itm;
    }
}

// Bulk copy of tile record t into shared memory, completing on `bar`.
__device__ __forceinline__ void fetch_rec(const Batch &b, int t, TileRec *dst, uint64_t *bar)
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"((uint32_t)sizeof(TileRec)) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(b.tile_rec + t)),
                 "r"((uint32_t)sizeof(TileRec)), "r"(smem_u32(bar)) : "memory");
}

// The tile box (TMA) and the tile's projection ranges (bulk copies) of record
// R, all completing on `bar`.
__device__ __forceinline__ void issue_rec_tile(const TileRec &R, uint8_t *buf, uint8_t *prj, uint64_t *bar)
{
    const uint32_t box = (uint32_t)(R.box_w * R.box_h);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(box + (uint32_t)(R.prj_bytes_x + R.prj_bytes_y)) : "memory");
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_u32(buf)), "l"(reinterpret_cast<uint64_t>(R.tmap)), "r"(R.xs), "r"(R.ys), "r"(smem_u32(bar))
        : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(prj)), "l"(reinterpret_cast<uint64_t>(R.prj_src_x)), "r"((uint32_t)R.prj_bytes_x),
                 "r"(smem_u32(bar)) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(prj + kPrjBytes)), "l"(reinterpret_cast<uint64_t>(R.prj_src_y)),
                 "r"((uint32_t)R.prj_bytes_y), "r"(smem_u32(bar)) : "memory");
}

// Thread 0 of k_fast_bits after a tile's box did not arrive in time: wait
// once more, with the same limit, for the copies it still has in flight (this
// box and, if there is one, the next tile's record), so that none lands in the
// shared memory of a CTA that has ended.  rph bit s is the parity of the next
// completion of record barrier 2 + s, phases bit p that of box barrier p.
__device__ __forceinline__ void drain_bits(uint64_t *bars, bool more, int cur, int s3, uint32_t phases, uint32_t rph)
{
    wait_tile(&bars[cur], (phases >> cur) & 1u);
    const int sn = s3 == 2 ? 0 : s3 + 1;
    if (more) wait_tile(&bars[2 + sn], (rph >> sn) & 1u);
}

// Tiles come with host-made records; from its fourth tile on a
// CTA takes the next one from a counter (cleared by the pyramid launch
// before), which evens out what their corners cost (100 pairs of 1241x376:
// 0.692 -> 0.596 ms).  Per tile: tile wait, cell states, bit-planes, a barrier;
// thread 0 then issues the next tile's box and projection ranges, fetches the
// record after it and asks for the number of the one after that; each threshold pass
// classifies 32 pixels of a row per thread, and every warp scores its own
// corners right away through a window of entries in shared memory, keeping
// each cell's k best by atomic maxima; a barrier ends each pass, and the slots
// are written.  Cell states, selections and counters are kept by tile parity,
// so that no barrier ends a tile: a warp may start the next one while others
// write this one's slots (what the next tile's first phase overwrites -- the
// planes, the other set -- was last read before the barrier that ended this
// tile's passes, and what thread 0 refills, before the next one's first).
// What bounds it: the ALU pipe (LOP3 and shifts, half rate: 69 % busy) and the
// barriers and dependent steps between.  Four warps a CTA, five CTAs an SM (96
// registers): with eight warps and three CTAs a barrier stopped more of the
// SM.  For 100 pairs of 1241x376 the kernel executed 1750 instructions per
// 1024 pixels and took 0.965 ms; now 1420 and 0.577 ms (threads and barriers
// 0.965 -> 0.82, run test and registers -> 0.765, host-made tile numbers,
// reciprocals and whole-word clears -> 0.729, blocks of cells that fill the
// warps -> 0.692, tiles from a counter -> 0.596, largest first -> 0.585).
// Compile-time variants: kAny, run bounds other than 9 and 13 (the same kernel
// with a run test that takes them at run time: 16 pairs of 800x602 on six
// levels 178 us, 229 by byte lanes with a cardinal pre-test and a table of
// corner masks, 131 with the default bounds); kArc, the corner response (the
// arc's, an opt-in reading, or the whole ring's SAD); kSkip, the learned
// cell-skip mode; kTop1, one keypoint per cell (k = 1, the default) or several.
template <bool kAny, bool kArc, bool kSkip, bool kTop1>
__global__ void __launch_bounds__(kFastThreads, kFastCtasPerSm) k_fast_bits(const __grid_constant__ Batch b)
{
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ int s_skipped[2];  // skipped cells, by tile parity
    __shared__ int s_more[2];     // whether another tile follows, by tile parity
    __shared__ int s_nlist[2];  // work-list lengths of pass 0 (cells skipped) and pass 1
    __shared__ int s_abort;
    __shared__ uint32_t s_rph;  // thread 0: parity of the next completion of each record barrier (bit s)
    __shared__ __align__(16) uint16_t s_wbuf[kFastThreads / 32][kBitsWin];
    __shared__ __align__(16) TileRec recs[3];
    __shared__ __align__(16) uint8_t s_prj[2][2 * kPrjBytes];  // per box: x range, y range
    __shared__ __align__(8) uint64_t bars[5];                   // [0..1] boxes, [2..4] records
    const int k = kTop1 ? 1 : b.prm.k, border = b.prm.border;
    const BitsLayout lay = bits_layout(b.fast_max_box, b.fast_max_cells, k, b.fast_max_planes);
    uint8_t *const buf0 = smem + lay.buf0, *const buf1 = smem + lay.buf1;
    uint32_t *planes = reinterpret_cast<uint32_t *>(smem + lay.planes);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint16_t *wbuf = s_wbuf[warp];
    uint16_t *wlist = reinterpret_cast<uint16_t *>(smem + lay.wlist);

    if ((smem_u32(buf0) | smem_u32(buf1)) & 127u) {
        if (threadIdx.x == 0) atomicOr(b.err, kErrDecode);
        return;
    }
    // thread 0: the next tile and the one after it
    const int tiles = b.fast_tiles;
    int t1 = tiles, t2 = tiles;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 5; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bars[i])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
        // the grid is no larger than the number of tiles
        fetch_rec(b, blockIdx.x, &recs[0], &bars[2]);
        t1 = (int)(blockIdx.x + gridDim.x);
        t2 = t1 + (int)gridDim.x;
        if (t1 < tiles) fetch_rec(b, t1, &recs[1], &bars[3]);
    }
    after_previous();
    if (threadIdx.x == 0) {
        if (wait_tile(&bars[2], 0u)) issue_rec_tile(recs[0], buf0, s_prj[0], &bars[0]);
        else {
            // give up, after waiting once more (same limit) for both
            // record copies, so that none lands after the CTA has ended
            atomicOr(b.err, kErrTimeout);
            s_abort = 1;
            wait_tile(&bars[2], 0u);
            if (t1 < tiles) wait_tile(&bars[3], 0u);
        }
        s_rph = 1u;
    }
    if (threadIdx.x < 2) s_skipped[threadIdx.x] = 0;
    __syncthreads();
    if (s_abort) return;
    uint32_t phases = 0u;  // bit p: parity of the next completion of box barrier p

    for (int it = 0;; ++it) {
        const int cur = it & 1, s3 = it % 3;
        const TileRec &R = recs[s3];
        const uint16_t *prj = reinterpret_cast<const uint16_t *>(s_prj[cur]);
        uint8_t *const has_hi = smem + lay.has_hi + cur * fast_align(b.fast_max_cells, 16);
        uint32_t *const sel =
            reinterpret_cast<uint32_t *>(smem + lay.sel + cur * fast_align(b.fast_max_cells * k * 4, 16));
        if (threadIdx.x == 0) {
            // read last before the barrier that ended the previous tile's passes
            s_skipped[cur ^ 1] = 0;
            s_nlist[0] = s_nlist[1] = 0;
            s_more[cur] = t1 < tiles;
        }
        uint8_t *const tb = cur ? buf1 : buf0;
        // the box and the projections
        if (!wait_tile(&bars[cur], (phases >> cur) & 1u)) {
            if (threadIdx.x == 0) {
                atomicOr(b.err, kErrTimeout);
                drain_bits(bars, t1 < tiles, cur, s3, phases, s_rph);
            }
            return;
        }
        phases ^= 1u << cur;
        bool all_skipped;
        {
        // record fields are read where needed (shared memory): values read
        // before a barrier are not carried across it
        const int c = R.c, W = R.W, Hh = R.H, x0 = R.x0, y0 = R.y0, rowb = R.box_w;
        const int ncx = R.ncx, cells = ncx * R.ncy;
        // learned skip: the image's proposal skipped at least one cell (an
        // image with none takes the exact path: no per-cell flags, no extra
        // barrier)
        const bool tskip = kSkip && R.skip != nullptr && b.skip_any[R.image] != 0;
        // cell states and cleared selections.  State: 0 no corner yet, 1
        // primary-threshold corner, 2 skipped by the learned proposal (its
        // centre projects into a skipped s0 cell), 3 no pixel inside the
        // evaluation border (never holds a corner, so it neither calls for the
        // fallback pass nor joins it)
        int my_skipped = 0;
        if (R.all_open && !tskip) {
            for (int i = threadIdx.x; i < (cells + 3) >> 2; i += kFastThreads) reinterpret_cast<uint32_t *>(has_hi)[i] = 0u;
        } else {
            for (int i = threadIdx.x; i < cells; i += kFastThreads) {
                const int lcy = i / ncx, lcx = i - lcy * ncx;
                const int cx0 = (R.ccx0 + lcx) * c, cy0 = (R.ccy0 + lcy) * c;
                const bool evaluated = cx0 + c > border && cx0 < W - border && cy0 + c > border && cy0 < Hh - border;
                uint8_t st = evaluated ? 0 : 3;
                if (tskip && evaluated) {
                    const int px = min(cx0 + c / 2, W - 1), py = min(cy0 + c / 2, Hh - 1);
                    const int X = prj[R.prj_off_x + px - x0], Y = prj[kPrjBytes / 2 + R.prj_off_y + py - y0];
                    st = R.skip[(Y / R.skip_c0) * R.skip_cells_x + X / R.skip_c0] ? 2 : 0;
                }
                if (tskip && st != 0) { st = 2; ++my_skipped; }
                has_hi[i] = st;
            }
        }
        for (int i = threadIdx.x; i < (cells * k + 3) >> 2; i += kFastThreads)
            reinterpret_cast<uint4 *>(sel)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (my_skipped) atomicAdd(&s_skipped[cur], my_skipped);
        // in skip mode the cell states and the skipped count are complete
        // before the planes
        if (tskip) __syncthreads();
        all_skipped = tskip && s_skipped[cur] == cells;

        // bit-planes of the box rows [r0, r1 + 6) that the evaluated rows
        // [r0, r1) read, chunks 0..nch (an item of chunk m reads m and m + 1),
        // one 32-byte chunk per thread
        const int r0 = R.r0, nch = R.nch, ru = bs_row_units(nch);
        if (!all_skipped) {
            const int chunks = R.items > 0 ? (R.r1 - r0 + 6) * (nch + 1) : 0;
            const uint32_t row_inv = R.row_inv;
            for (int ci = threadIdx.x; ci < chunks; ci += kFastThreads) {
                const int rr = div_small(ci, row_inv), kc = ci - rr * (nch + 1), r = r0 + rr;
                const uint4 *src = reinterpret_cast<const uint4 *>(tb + r * rowb + 32 * kc);
                bs_transpose(src[0], src[1], reinterpret_cast<uint4 *>(planes) + r * ru + 2 * kc);
            }
            // cells skipped by the proposal: pass 0 runs over the items that
            // hold a pixel of a cell that is not (states are complete: skip
            // mode has a barrier after them)
            if (tskip && s_skipped[cur] > 0) {
                list_items(wlist, &s_nlist[0], R.items, nch, R.nch_inv, r0, R.plo, R.phi, has_hi, ncx, R.tw, c,
                           (uint32_t)R.cinv, lane, warp,
                           [](uint8_t st) { return st != 2; });
            }
        }
        }
        __syncthreads();
        const bool more = s_more[cur] != 0;
        if (!more) let_next();  // this CTA's last tile
        if (threadIdx.x == 0 && more) {
            // the next tile's record was fetched one tile ago; the slot of the
            // record after it, the other box and its projections were last
            // read before the barrier above (after a record wait runs out
            // nothing more is issued; the CTA stops after this tile's passes)
            const int sn = s3 == 2 ? 0 : s3 + 1;
            if (wait_tile(&bars[2 + sn], (s_rph >> sn) & 1u)) {
                issue_rec_tile(recs[sn], cur ? buf0 : buf1, s_prj[cur ^ 1], &bars[cur ^ 1]);
                s_rph ^= 1u << sn;
                t1 = t2;
                if (t1 < tiles) {
                    const int sa = s3 == 0 ? 2 : s3 - 1;
                    fetch_rec(b, t1, &recs[sa], &bars[2 + sa]);
                    t2 = 3 * (int)gridDim.x + (int)atomicAdd(b.tile_next, 1u);  // used one tile on
                }
            } else { atomicOr(b.err, kErrTimeout); s_abort = 1; }
        }
        const bool some_skipped = kSkip && s_skipped[cur] > 0;  // constant false outside skip mode

        {
        const int c = R.c, tw = R.tw, rowb = R.box_w, ncx = R.ncx;
        const uint32_t cinv = (uint32_t)R.cinv;
        const int plo = R.plo, phi = R.phi, r0 = R.r0;
        const int nch = R.nch, sb = R.delta + 4, ru = bs_row_units(nch), items = R.items;
        const uint32_t nchinv = R.nch_inv;  // item / nch by a multiply (item < 2^9)
        const uint8_t *tbytes = tb + R.delta;  // pixel (x, y) at (y - y0 + 3) * rowb + (x - x0 + 4)
        for (int pass = 0; pass < 2 && !all_skipped; ++pass) {
            const int eps = pass == 0 ? R.eps_hi : R.eps_lo;
            if (pass == 1) {
                // fallback pass only while a cell that is open got no corner
                // (selections are final after pass 0's barrier): every warp
                // looks for itself and marks the cells that have one
                if (eps <= 0) break;
                bool open = false;
                for (int i = lane; i < ncx * R.ncy; i += 32) {
                    if (has_hi[i] != 0) continue;
                    if (sel[i * k]) has_hi[i] = 1;
                    else open = true;
                }
                if (!__any_sync(0xFFFFFFFFu, open)) break;
                __syncwarp();  // this warp's marks
            }
            // pass 0 covers every item, or the listed ones when cells are
            // skipped; pass 1 lists the items holding a pixel of a cell still
            // without a corner
            const bool listed = pass == 1 || some_skipped;
            if (pass == 1) {
                list_items(wlist, &s_nlist[1], items, nch, nchinv, r0, plo, phi, has_hi, ncx, tw, c, cinv, lane, warp,
                           [](uint8_t st) { return st == 0; });
                __syncthreads();
            }
            const int n_work = listed ? s_nlist[pass] : items;
            uint32_t eps_mask[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) eps_mask[i] = 0u - (((uint32_t)eps >> i) & 1u);
            for (int base = warp * 32; base < n_work; base += kFastThreads) {
                const int w = base + lane;
                uint32_t bits = 0;
                int py = 0, px0 = 0;
                if (w < n_work) {
                    const int itm = listed ? (int)wlist[w] : w;
                    const int rr = div_small(itm, nchinv), m = itm - rr * nch;
                    py = r0 + rr;
                    px0 = 32 * m;
                    uint32_t valid = border_bits(px0, plo, phi);
                    if (listed && valid) {
                        const uint8_t *strow = has_hi + div_small(py, cinv) * ncx;
                        // pass 1: only cells without a corner (and not skipped); pass 0: not in a
                        // skipped cell.  One copy of the loop for both spills less in the skip mode
                        // (12 pairs of 752x480 213.0 -> 211.4 us).
                        valid &= cell_bits(strow, px0, tw, c, cinv,
                                           [=](uint8_t st) { return pass == 1 ? st == 0 : st != 2; });
                    }
                    if (valid) bits = bs_corners<kAny>(planes, ru, py, m, sb, eps_mask, b.prm.p_min, b.prm.p_max) & valid;
                }
                // the warp's corners in order, scored through windows of kBitsWin entries
                const int nb = __popc(bits);
                int incl = nb;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= o) incl += y;
                }
                const int total = __shfl_sync(0xFFFFFFFFu, incl, 31);
                const int ebase = (py << 7) | px0;  // entry of pixel px0 + j: ebase + j
                for (int w0 = 0; w0 < total; w0 += kBitsWin) {
                    // this lane's corners from the highest (the order does not matter)
                    uint32_t bb = bits;
                    if (total <= kBitsWin) {
                        for (uint16_t *to = wbuf + (incl - nb); bb; ++to) {
                            const int j = 31 - __clz(bb);
                            bb ^= 1u << j;
                            *to = (uint16_t)(ebase + j);
                        }
                    } else {
                        for (int id = incl - nb; bb && id < w0 + kBitsWin; ++id) {
                            const int j = 31 - __clz(bb);
                            bb ^= 1u << j;
                            if (id >= w0) wbuf[id - w0] = (uint16_t)(ebase + j);
                        }
                    }
                    __syncwarp();
                    const int n = min(total - w0, kBitsWin);
                    for (int i = lane; i < n; i += 32) {
                        const int e = wbuf[i];
                        const int cy_ = e >> 7, cx_ = e & 127;
                        const uint8_t *pp = tbytes + (cy_ + 3) * rowb + (cx_ + 4);
                        const int r = kArc ? ring_arc(pp, rowb, eps, b.prm.p_min, b.prm.p_max)
                                                     : ring_sad(pp, rowb);
                        const int ccy = div_small(cy_, cinv), ccx = div_small(cx_, cinv);
                        const uint32_t inidx = (uint32_t)((cy_ - ccy * c) * c + (cx_ - ccx * c));
                        const uint32_t key = ((uint32_t)r << 16) | (0xFFFFu - inidx);
                        if (kTop1) {
                            atomicMax(&sel[ccy * ncx + ccx], key);
                        } else {
                            // the cell's k largest keys in falling order: each
                            // entry keeps the larger and passes the smaller on
                            // (a key below the last entry, which only grows,
                            // cannot be among them)
                            uint32_t *const top = sel + (ccy * ncx + ccx) * k;
                            if (key > *reinterpret_cast<volatile uint32_t *>(top + k - 1)) {
                                uint32_t v = key;
                                for (int j = 0; j < k && v; ++j) v = min(v, atomicMax(top + j, v));
                            }
                        }
                    }
                    __syncwarp();
                }
            }
            __syncthreads();  // the selections of this pass are complete
        }
        }
        if (s_abort) {  // thread 0 could not start the next tile
            if (threadIdx.x == 0) {
                const int sn = s3 == 2 ? 0 : s3 + 1;
                wait_tile(&bars[2 + sn], (s_rph >> sn) & 1u);  // the record copy that did not complete
            }
            return;
        }

        // slots and the s0 score map, projections from
        // the staged ranges
        const int c = R.c, ncx = R.ncx, cells = ncx * R.ncy;
        for (int e = threadIdx.x; e < cells * k; e += kFastThreads) {
            const int cell = kTop1 ? e : e / k, j = e - cell * k;
            const int lcy = div_recip(cell, R.ncx_div);
            const int gcx = R.ccx0 + cell - lcy * ncx, gcy = R.ccy0 + lcy;
            const uint32_t key = sel[e];
            b.slots[R.slot_base + (gcy * R.cells_x + gcx) * k + j] = key;
            if (key) {
                const int inidx = 0xFFFF - (int)(key & 0xFFFFu), row = div_recip(inidx, R.cdiv);
                const int x = gcx * c + inidx - row * c, y = gcy * c + row;
                if (x >= R.W || y >= R.H) { atomicOr(b.err, kErrDecode); continue; }
                const int X = prj[R.prj_off_x + x - R.x0], Y = prj[kPrjBytes / 2 + R.prj_off_y + y - R.y0];
                atomicAdd(R.map + (size_t)Y * R.W0 + X, (1u << 16) + (key >> 16));
            }
        }
        if (!more) break;
    }
}

int fast_smem_bytes(int max_box, int max_cells, int k, int max_planes)
{
    return bits_layout(max_box, max_cells, k, max_planes).total;
}

// The detection kernel of a batch: by its run bounds, response, skip mode and
// keypoints per cell (index kAny * 8 + kArc * 4 + kSkip * 2 + kTop1).
static const void *const kFastBitsVariants[16] = {
    reinterpret_cast<const void *>(k_fast_bits<false, false, false, false>),
    reinterpret_cast<const void *>(k_fast_bits<false, false, false, true>),
    reinterpret_cast<const void *>(k_fast_bits<false, false, true, false>),
    reinterpret_cast<const void *>(k_fast_bits<false, false, true, true>),
    reinterpret_cast<const void *>(k_fast_bits<false, true, false, false>),
    reinterpret_cast<const void *>(k_fast_bits<false, true, false, true>),
    reinterpret_cast<const void *>(k_fast_bits<false, true, true, false>),
    reinterpret_cast<const void *>(k_fast_bits<false, true, true, true>),
    reinterpret_cast<const void *>(k_fast_bits<true, false, false, false>),
    reinterpret_cast<const void *>(k_fast_bits<true, false, false, true>),
    reinterpret_cast<const void *>(k_fast_bits<true, false, true, false>),
    reinterpret_cast<const void *>(k_fast_bits<true, false, true, true>),
    reinterpret_cast<const void *>(k_fast_bits<true, true, false, false>),
    reinterpret_cast<const void *>(k_fast_bits<true, true, false, true>),
    reinterpret_cast<const void *>(k_fast_bits<true, true, true, false>),
    reinterpret_cast<const void *>(k_fast_bits<true, true, true, true>),
};

static const void *detect_kernel_of(const Batch &b)
{
    const bool any = b.prm.p_min != 9 || b.prm.p_max != 13;
    return kFastBitsVariants[(any ? 8 : 0) + (b.prm.resp_arc ? 4 : 0) + (b.skip_any ? 2 : 0) + (b.prm.k == 1 ? 1 : 0)];
}

cudaError_t launch_detect(const Batch &b, cudaStream_t stream)
{
    if (b.fast_tiles == 0) return cudaSuccess;
    static int cached_smem = -1, cached_blocks = 0, n_sm = 0;
    static const void *cached_fn = nullptr;
    cudaError_t e;
    if (n_sm == 0) {
        int dev = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    }
    const void *fn = detect_kernel_of(b);
    if (cached_smem != b.fast_smem || cached_fn != fn) {
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&cached_blocks, fn, kFastThreads, b.fast_smem)) !=
            cudaSuccess)
            return e;
        cached_smem = b.fast_smem;
        cached_fn = fn;
    }
    int per_sm = std::max(1, cached_blocks);
    if (b.fast_ctas_per_sm > 0) per_sm = std::min(per_sm, b.fast_ctas_per_sm);
    const int grid = std::min(b.fast_tiles, per_sm * n_sm);
    void *args[] = { const_cast<Batch *>(&b) };
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kFastThreads);
    cfg.dynamicSmemBytes = (size_t)b.fast_smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];  // as launch_after
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = start_early(b) ? 1 : 0;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

// Detection CTAs of this batch's launch that fit on one SM at once.
cudaError_t detect_ctas_that_fit(const Batch &b, int *per_sm)
{
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, detect_kernel_of(b), kFastThreads, b.fast_smem);
}

cudaError_t configure_kernels()
{
    cudaError_t e = cudaSuccess;
    for (const void *fn : kFastBitsVariants)
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    return e;
}

}  // namespace jslam
