// Internal types shared by the host code and the kernels of libjslam.
//
// The whole batch (every image of every stereo pair, every pyramid level) is
// described by three device tables built on the host:
//   ImageDesc[2 * pairs]   one per image (pair p: left = 2p, right = 2p + 1)
//   LevelDesc[sum levels]  one per (image, level), image-major
//   PairDesc[pairs]        stereo matching outputs
// and each kernel's grid is a flat list of work units mapped onto these
// tables through small prefix arrays (tiles per level, segments per level),
// so a batch of mixed image sizes and pyramid depths runs in one launch per
// stage.
#pragma once

#include <cstdint>
#include <utility>
#include <cuda.h>
#include <cuda_runtime.h>

#include "tile_plan.h"

namespace jslam {

constexpr int kBins = 30;        // orientation sectors of 12 degrees
constexpr int kPairs = 256;      // BRIEF point pairs
constexpr int kDiskR = 15;       // intensity-centroid disk radius
constexpr int kPatR = 13;        // rotated BRIEF offsets lie in [-13, 13]
constexpr int kDiskRows = 11;    // disk rows of a lane: every third of the 31 (and past the last)
constexpr int kOrbBoxW = 48, kOrbRawH = 31, kOrbBlurH = 27;  // a keypoint's boxes of the raw and the blurred level
constexpr int kPatPitch = kOrbBoxW;  // row pitch of the staged 27 x 27 BRIEF patch
constexpr int kMaxSegment = 4096;  // candidate slots per (level, cell row)
constexpr int kMaxImages = 256;    // images per batch (two per stereo pair)

// Pyramid strip: output columns per warp (30 lanes x 4 pixels), and how a
// lane reads its source columns (see k_pyramid).
constexpr int kPyrCols = 120, kPyrMinRows = 6, kPyrMaxRows = 58;
constexpr int kPyrWarpsPerSm = 22;  // strips that run on an SM at once
// Parts of a batch of host frames, each uploaded while the pyramid of the part
// before is made, and the bytes a part has at least.
constexpr int kUploadParts = 4;
constexpr size_t kUploadPartBytes = (size_t)4 << 20;
// The ring of a strip's source rows: two source rows per row, for the two
// rows in use and the rows ahead that are being copied, and the source row
// before them; rows of up to 16 (kPyrOne) and 32 (kPyrTwo) 16-byte units.
constexpr int kPyrRing = 6656, kPyrAhead = 6, kPyrAheadTwo = 4;
constexpr int kPyrMaxOne = 256, kPyrMaxTwo = 512;
static_assert((2 * (kPyrAhead + 2) + 1) * kPyrMaxOne <= kPyrRing, "ring");
static_assert((2 * (kPyrAheadTwo + 2) + 1) * kPyrMaxTwo <= kPyrRing, "ring");
enum { kPyrCopy = 0, kPyrOne = 1, kPyrTwo = 2, kPyrBytes = 3 };
constexpr int kLutWords = 2048;            // 2^16-entry corner bit table
constexpr int kSkipC = 16;                 // channels of the learned cell-skip net
constexpr int kSkipTileW = 26, kSkipTileH = 12;  // its logits per CTA (grid pitch 26 + 6 = 32)
constexpr int kRefineMaxW = 10, kRefineMaxL = 7;  // correlation window half-size and search radius limits
constexpr int kNmsThreads = 128;
constexpr int kFinThreads = 512;

// Of the host's words after the counts: 0 mirrors the error word, this one has
// the descriptor kernel's own errors.
constexpr int kHostErrOrb = 2;

// Device error bits (OR-ed into the context's error word).
constexpr uint32_t kErrSegment = 1u << 0;  // a segment was larger than kMaxSegment
constexpr uint32_t kErrDecode = 1u << 1;   // a candidate decoded outside its level
constexpr uint32_t kErrTimeout = 1u << 2;  // a bounded wait for a tile load gave up

struct KpOut {
    uint16_t *x, *y, *X, *Y, *response;
    uint8_t *level, *angle_bin, *k_levels;
    uint32_t *k_resp;
    float *angle;
    uint32_t *desc;  // capacity x 8
    int32_t capacity;
};

struct LevelDesc {
    const uint8_t *raw;      // raw level (level 0: aligned copy of the input)
    uint8_t *raw_w;          // the same buffer, written by the pyramid kernel
    uint8_t *blur;           // blurred level
    const uint32_t *tapx;    // bilinear taps: src index | weight << 16 (levels >= 1)
    const uint32_t *tapy;
    const uint16_t *projx;   // s0 projection of each x / y of the level
    const uint16_t *projy;
    // source of the resampling: nullptr = level 0 (the input image); in the
    // cascaded pyramid the raw level n - 1 (taps then use one factor zeta)
    const uint8_t *src;
    int32_t src_W, src_H, src_pitch;
    int32_t pyr_mode;        // how the pyramid kernel reads the source columns (kPyr...)
    int32_t pyr_rows;        // output rows of its strips
    int32_t W, H, pitch;     // pitch of raw: width rounded up to 128
    int32_t blur_pitch;
    int32_t c, cells_x, cells_y;
    int32_t bx, by;          // cells per detection tile
    int32_t cinv;            // ceil(2^16 / c): exact division by c for values < 128
    const CUtensorMap *tmap; // TMA map of the raw level
    int32_t box_w, box_h;    // detection tile box: bytes per row (multiple of 16) and rows
    int32_t slot_base;       // first candidate slot of the level
    int32_t seg_base;        // first segment (cell row) of the level
    int32_t image, level;
    int32_t band;            // stereo row band for keypoints of this level
    double zeta;             // zeta^n (repeated multiplication in double)
    float zeta_f, zeta_inv_f; // zeta^n and 1 / zeta^n rounded to float
};

struct ImageDesc {
    int32_t W0, H0;
    int32_t levels, level_base;
    int32_t eps_hi, eps_lo;  // eps_lo <= 0: no fallback
    int32_t max_feats;
    int32_t slot_base, slot_count;
    int32_t seg_base, seg_count;
    uint32_t *map;           // W0 * H0 packed (K_l << 16 | K_r); all zero between runs
    int32_t *count;          // keypoint count written by finalisation
    int32_t *count_hdr;      // the same count in the header of the pair's result block
    int32_t *level_start;    // kMaxLevels + 1 entries
    // row index of the canonical list, per level H0 + 1 entries: entry v is
    // the first index of the level whose Y is >= v (the level's end if none);
    // written by k_orient_desc for levels with keypoints, read by k_match
    int32_t *row_first;
    KpOut out;
    // learned cell-skip (skip == nullptr: exact mode)
    float *skip_logits;      // skip_h8 x skip_w8 logits at 1/8 scale
    uint8_t *skip;           // per s0 culling cell: 1 = skipped
    int32_t skip_w8, skip_h8, skip_cells_x, skip_cells_y, skip_c0;
};

// Device copy of the skip net: BF16 weights, FP32 biases.
struct SkipModelDev {
    const uint16_t *w1, *w2, *w3;  // [16][9], [16][16][9], [16][9]
    const float *b1, *b2;          // [16], [16]
    float b3;
};

struct PairDesc {
    int32_t left, right;
    int32_t *match_idx;
    int16_t *disparity;
    uint16_t *dist;
    float *sub_disp;         // correlation minimisation: sub-pixel disparity (-1 rejected)
    float *depth;            //   depth bf / disparity (0 rejected)
    uint32_t *corr;          //   SAD at the best shift (0xFFFFFFFF: none computed)
};

// Parameters fixed for a context.
struct Params {
    int32_t p_min, p_max, k, nms_rad, border, rule;
    int32_t max_disp, max_dist;
    int32_t resp_arc;        // 1: arc response (see ring_response.cuh); 0: sum over the whole circle
};

// Level-0 pixels of every image of the call.  Passed by value as a kernel
// parameter so that a plan (which depends only on the shapes) is reused
// across calls whose input buffers differ.
struct Inputs {
    const uint8_t *ptr[kMaxImages];
    int32_t pitch[kMaxImages];
};

// One detection tile, prepared on the host: the
// tile's place in its level, the level's and image's scalars, and the
// 16-byte-aligned ranges of the level's s0 projection tables that cover the
// tile's columns and rows.  The kernel copies it into shared memory with a
// bulk copy, so no chain of descriptor loads precedes a tile.
constexpr int kPrjBytes = 288;  // staged projection bytes per axis: 2 x 128 + alignment slack, rounded to 16
struct __align__(16) TileRec {
    int32_t ccx0, ccy0, ncx, ncy, x0, y0, tw, th, xs, ys, delta;
    int32_t c, cells_x, W, H, cinv, box_w, box_h, slot_base;
    int32_t eps_hi, eps_lo, W0, skip_c0, skip_cells_x;
    int32_t prj_bytes_x, prj_bytes_y;  // bulk copy sizes (multiples of 16)
    int32_t prj_off_x, prj_off_y;      // element offset of x0 / y0 in the staged copies
    int32_t image;                     // the tile's image
    int32_t r0, r1, plo, phi;          // evaluated rows and columns of the tile
    int32_t nch, items;                // 32-pixel chunks of a row; (evaluated row, chunk) items
    uint32_t nch_inv, row_inv;         // ceil(2^16 / nch), ceil(2^16 / (nch + 1))
    uint32_t cdiv, ncx_div;            // reciprocals of c and ncx (see div_recip)
    int32_t all_open;                  // every cell has evaluated pixels
    const CUtensorMap *tmap;
    const uint16_t *prj_src_x, *prj_src_y;
    uint32_t *map;
    const uint8_t *skip;
};
static_assert(sizeof(TileRec) % 16 == 0, "bulk copies move multiples of 16 bytes");

// Reciprocal for div_recip: v / d for v * d below 2^32.
inline uint32_t recip_of(int d) { return d == 1 ? 0u : (uint32_t)(((1ull << 32) + (uint64_t)d - 1) / (uint64_t)d); }

// One segment (cell row of a level): where its candidate slots lie and what
// turns a slot into coordinates and score-map entries.
struct __align__(16) SegRec {
    const uint16_t *projx, *projy;
    uint32_t *map;
    int32_t slot, m;         // first slot, slots (cells_x x k)
    int32_t c, y0;           // cell size, first row
    uint32_t cdiv;           // reciprocal of c (see recip_of)
    int32_t W0, H0, level;
};
// One pyramid strip: its level and first output column and row.
struct __align__(16) PyrRec {
    int32_t level, x0, y0, pad;
};
// Rank of a slot that is no survivor (SlotInfo's w): no corner, suppressed.
constexpr int kSlotEmpty = -2, kSlotSuppressed = -1;

// Everything the kernels of one extraction need.
struct Batch {
    const ImageDesc *images;
    const LevelDesc *levels;
    const CUtensorMap *orb_maps;    // per level: keypoint boxes of the raw and of the blurred level
    const PairDesc *pairs;
    const PyrRec *pyr_rec;          // pyramid strips, ordered by level number
    int32_t pyr_pass_first[kMaxLevels + 1];  // cascaded: first strip of each level number
    int32_t pyr_cascaded;           // a launch per level number instead of one over every strip
    int32_t pyr_first;              // first strip of a launch
    const SegRec *seg_rec;          // one per segment
    int32_t n_images, n_levels, n_pairs, n_segments;
    int32_t max_segment;            // largest segment (cells_x x k slots) of the batch
    int32_t pyr_tiles, fast_tiles;  // pyramid strips, detection tiles
    int32_t max_capacity;           // largest keypoint capacity of any image
    int32_t fast_smem;              // dynamic shared memory of the detection kernel
    int32_t fast_max_box, fast_max_cells;  // its tile layout maxima
    int32_t fast_max_planes;        // bit-plane bytes of the largest tile box
    const TileRec *tile_rec;        // one per detection tile
    uint32_t *tile_next;            // detection tiles taken beyond each CTA's first three (zero before the launch)
    const uint32_t *corner_lut;     // bit m: P_min <= longest circular run of m <= P_max
    uint32_t *slots;                // candidate keys per slot
    uint4 *slot_info;               // per slot: position, X | Y << 16, cap priority, rank in its segment
    int32_t *seg_count;             // survivors per segment
    int32_t *seg_off;               // exclusive prefix of seg_count per image
    uint32_t *canon_prio;           // cap priority of each canonical position
    uint2 *canon_pos;               // its x | y << 13 | level << 26, X | Y << 16
    int32_t max_slots;              // most candidate slots of an image
    int32_t n_sm;                   // streaming multiprocessors of the device
    const int8_t *pattern;          // kBins x kPairs x 4
    const uint32_t *pattern_off;    // kBins x kPairs: patch offsets of p | of q << 16 (pitch kPatPitch, from the corner)
    const uint32_t *disk_mask;      // 4 alignments x kDiskRows x 32 lanes: bytes of a word inside the moment disk
    const double *bin_cos, *bin_sin;
    const float *bin_cosf, *bin_sinf;  // the same tables rounded to float (fast sector test)
    uint32_t *err;
    Params prm;
    int32_t skip_max_tiles, skip_max_cells;  // learned cell-skip launch shape
    int32_t *skip_any;              // learned skip: per image, nonzero once its proposal skipped a cell
    int32_t nms_kernel;             // 0: a warp per segment where segments allow, 1: a CTA per segment
    int32_t fast_ctas_per_sm;       // persistent detection CTAs per SM (0: as many as fit)
    int32_t *host_counts;           // pinned host memory: keypoint count per image
    uint32_t *host_err;             // pinned host memory: the error word as the last kernel of an extraction saw it
};

// Kernel launchers (one per stage), all on `stream`.
cudaError_t launch_pyramid(const Batch &b, const Inputs &in, cudaStream_t stream);
cudaError_t launch_pyramid_strips(const Batch &b, const Inputs &in, int first, int count, cudaStream_t stream);
cudaError_t launch_detect(const Batch &b, cudaStream_t stream);
cudaError_t launch_wait_selftest(uint32_t *err, cudaStream_t stream);
cudaError_t launch_pfa_nms(const Batch &b, cudaStream_t stream);
cudaError_t launch_pfa_finalize(const Batch &b, cudaStream_t stream);
cudaError_t launch_orient_desc(const Batch &b, cudaStream_t stream);
cudaError_t launch_match(const Batch &b, cudaStream_t stream);
cudaError_t launch_refine(const Batch &b, int w, int L, double bf, cudaStream_t stream);

// Feature tracking by projection: caller-projected queries against one image's keypoints.
struct TrackArgs {
    int32_t image, n, max_dist;
    float radius;
    float zeta_f[kMaxLevels + 1];  // zeta^n rounded to float, n = 0..kMaxLevels
    const float *u, *v;
    const uint8_t *level;
    const uint32_t *desc;
    int32_t *out_idx;
    uint16_t *out_dist;
};
cudaError_t launch_track(const Batch &b, const TrackArgs &a, cudaStream_t stream);
cudaError_t launch_fc_ablation(const Batch &b, uint16_t *crf, const uint64_t *off, uint32_t *keys,
                               const int *level_blocks, int max_pixels, int max_levels, const int *level_cells_y,
                               const int *level_c, int n_max, cudaStream_t stream, cudaEvent_t mid);
cudaError_t launch_skipnet(const Batch &b, const SkipModelDev &m, float thresh, cudaStream_t stream);
cudaError_t set_blur_weights(const int32_t w[7]);
cudaError_t configure_kernels();
cudaError_t configure_skipnet();
cudaError_t configure_orb();
int skipnet_smem_bytes();

#ifdef __CUDACC__
// Programmatic dependent launch along an extraction's kernels: a kernel
// launched with launch_after may start while the one before it on the stream
// still runs, does what needs none of its results (plan tables, barriers), and
// waits for its completion in after_previous(); let_next() in a kernel says
// that all its CTAs have started, so that the next one may.  Every kernel of
// the chain waits before it reads or writes anything that another one touches,
// so each sees the results of all before it.  Without a predecessor on the
// stream that allows it, a launch is an ordinary one.  What other kernels (or a
// user's kernel before the first one) write is read with ordinary loads: a
// read-only one (__ldg) may be served from before the wait, since its data has
// to be constant while the kernel is resident.  Tables of the plan and of the
// context are.
//
// Descriptors, matching and what follows always start so, the pyramid by a rule
// of its own (launch_pyramid_strips), detection, NMS and finalisation only while the detection tiles all run at once (start_early).
// Beyond that the CTAs that sit and wait take the slots of the kernel before,
// and persistent ones are spread over the SMs by where that one ended first: us
// per call with none / with descriptors and matching / with all: one pair of
// 320x240 76 / 69 / 66, of 1241x376 with refinement and tracking 126 / 115 /
// 105, of 1920x1080 143 / 142 / 142; 100 of 1241x376 1251 / 1258 / 1348, 16
// streams of four sizes 375 / 368 / 415, 24 pairs of 647x363 343 / 338 / 381, 16
// of 800x602 on a cascaded pyramid 390 / 373 / 502 (before detection of the last
// two became faster; they take 239 and 325 now).
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

static inline bool start_early(const Batch &b) { return b.fast_tiles <= kFastCtasPerSm * b.n_sm; }

template <class... P, class... A>
cudaError_t launch_if(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A &&...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

template <class... P, class... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A &&...args)
{
    return launch_if(true, kernel, grid, block, smem, stream, std::forward<A>(args)...);
}
#endif

}  // namespace jslam
