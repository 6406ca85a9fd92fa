// Choice of the detection tiles (see tile_plan.h).
#include "tile_plan.h"

#include <algorithm>

namespace jslam {
namespace {

// Shared memory of a detection tile's two boxes and planes.
int tile_bytes(int tw, int th)
{
    int bw, bh;
    detect_box(tw, th, &bw, &bh);
    return bh * (2 * bw + 16 * bs_row_units((tw + 31) / 32));
}

// Issue slots of a detection tile with `rows` evaluated rows of
// nch 32-pixel chunks: measured on the 1241x376 sequence, about 1000 a warp's
// round of ring tests and responses, 115 a round of transposed chunks, 300 a
// tile.
double tile_cost(int rows, int nch)
{
    const int rounds = (rows * nch + kFastThreads - 1) / kFastThreads;
    const int chunks = rows ? ((rows + 6) * (nch + 1) + kFastThreads - 1) / kFastThreads : 0;
    return 1000.0 * rounds + 115.0 * chunks + 300.0;
}

// One column of a level's tiles, h rows and nch chunks each: their cost, and
// that of the dearest one.  A tile's evaluated rows are those of [y0, y0 + h)
// in [border, H - border), so all are full or empty but the ones that hold
// either bound.
constexpr int kMaxChunks = kFastMaxTile / 32;
struct Column {
    double cost[kMaxChunks + 1], tile[kMaxChunks + 1];
};
Column tile_column(int H, int border, int h)
{
    const int tiles = (H + h - 1) / h, lo = border, hi = std::max(H - border, border);
    int rows[4], count[4], n = 0, others = tiles;
    const auto add = [&](int r, int c) {
        if (c <= 0) return;
        rows[n] = r;
        count[n++] = c;
        others -= c;
    };
    add(h, hi / h - (lo + h - 1) / h);  // the full ones
    const bool cut_lo = hi > lo && lo % h != 0, cut_hi = hi > lo && hi % h != 0;
    if (cut_lo) add(std::min(lo / h * h + h, hi) - lo, 1);
    if (cut_hi && !(cut_lo && hi / h == lo / h)) add(hi - std::max(hi / h * h, lo), 1);
    add(0, others);
    Column col{};
    for (int nch = 1; nch <= kMaxChunks; ++nch)
        for (int i = 0; i < n; ++i) {
            const double one = tile_cost(rows[i], nch);
            col.cost[nch] += count[i] * one;
            col.tile[nch] = std::max(col.tile[nch], one);
        }
    return col;
}

constexpr int kHeights[] = { 96, 64, 48, 32, 24, 16 };
constexpr int kNumHeights = 6;

// A level's best block for each of the heights allowed: cells, cost of the
// level's tiles, of its dearest one.
struct Choice {
    int bx, by;
    double cost, tile;
};

// Cells per detection tile of a level.  A tile's evaluated
// rows x 32-pixel chunks are items, a lane each, so cells whose size divides
// neither 32 nor the CTA leave lanes and warps idle: with about 128 x 64
// pixels, 22-pixel cells made 132 items for 128 threads.  Of the blocks at
// most max_w x max_h pixels (one cell at least) whose two boxes and planes
// take at most `budget` bytes of shared memory, the one whose tiles over the
// level cost least, for every max_h at once.  A level has two widths of tiles
// and few numbers of evaluated rows, so a block's cost takes two additions
// however many tiles there are.  The blocks of a pair of eight levels (one
// host core), by adding up the tiles of every block for every height, and so:
// 1241x376 with cells of 32 pixels 1.1 and 0.06 ms, 1920x1080 of 32 / 16 / 8 / 4
// pixels 6.9 / 24 / 182 / 1750 and 0.05 / 0.10 / 0.29 / 0.83 ms.
long long level_choices(int W, int H, int c, int k, int border, int max_w, const int *max_h, int n_h, int budget,
                        Choice *best)
{
    const int cells_x = (W + c - 1) / c, cells_y = (H + c - 1) / c;
    const int tallest = std::min(cells_y, std::max(max_h[0] / c, 1));  // heights fall
    std::vector<Column> columns;
    columns.reserve(tallest);
    long long compared = 0;
    for (int i = 0; i < n_h; ++i) best[i] = { 1, 1, -1.0, 0.0 };
    for (int x = 1; x <= cells_x && (x == 1 || x * c <= max_w); ++x) {
        const int wide = std::min(x * c, W), cols = (cells_x + x - 1) / x;
        const int last = (W - (cols - 1) * x * c + 31) / 32, nch = cols > 1 ? (wide + 31) / 32 : last;
        for (int y = 1; y <= tallest; ++y) {
            if (x * y > 1 && (x * y * k > kFastMaxCellsPerCta || tile_bytes(wide, std::min(y * c, H)) > budget)) break;
            if ((int)columns.size() < y) columns.push_back(tile_column(H, border, y * c));
            const Column &C = columns[y - 1];
            const double cost = (cols - 1) * C.cost[nch] + C.cost[last], tile = std::max(C.tile[nch], C.tile[last]);
            ++compared;
            for (int i = 0; i < n_h && (y == 1 || y * c <= max_h[i]); ++i)
                if (best[i].cost < 0.0 || cost < best[i].cost) best[i] = { x, y, cost, tile };
        }
    }
    return compared;
}

bool same(const Geometry &a, const Geometry &b)
{
    bool eq = a.levels == b.levels;
    for (int l = 0; eq && l < a.levels; ++l) eq = a.W[l] == b.W[l] && a.H[l] == b.H[l] && a.c[l] == b.c[l];
    return eq;
}

}  // namespace

// Detection tiles of every level of a batch (pairs of one shape share them).
// A chosen tile size is about what the tiles get (up to half as tall again
// where that fits).  By default the tallest tiles whose launch takes least
// time: large tiles waste less on their halo, but a launch of few tiles ends
// with most CTAs idle, so the estimate adds the dearest tile to the tiles'
// cost shared out over the CTAs that run at once (five an SM fit the budget
// of a 128 x 74 tile).  Detection of 100 pairs of 1241x376: 0.729 ms with the
// largest blocks of 128 x 64 pixels whose width is a multiple of 4, 0.692 with
// these.  Heights up to 96 / 64 / 48 / 32 / 24 (us): those 100 pairs 585 / 596 /
// 680 / 748 / 783 (default 585), one pair of 320x240 14.2 / 14.2 / 14.2 / 13.0 /
// 12.3 (12.6).
long long detect_blocks(const std::vector<Geometry> &geo, int k, int border, int tile_w, int tile_h, bool chosen,
                        int n_sm, std::vector<LevelBlocks> &blocks)
{
    struct Shape {
        const Geometry *geo;
        Choice level[kMaxLevels][kNumHeights];
        int pairs;
    };
    const int chosen_h = std::min(tile_h * 3 / 2, kFastMaxTile);
    const int *const heights = chosen ? &chosen_h : kHeights;
    const int n_h = chosen ? 1 : kNumHeights;
    const int budget = tile_bytes(tile_w, tile_h * 23 / 20);
    std::vector<Shape> shapes;
    std::vector<int> shape_of(geo.size());
    long long compared = 0;
    for (size_t p = 0; p < geo.size(); ++p) {
        size_t s = p > 0 && same(geo[p], geo[p - 1]) ? (size_t)shape_of[p - 1] : 0;
        while (s < shapes.size() && !same(geo[p], *shapes[s].geo)) ++s;
        if (s == shapes.size()) {
            shapes.push_back({});
            Shape &S = shapes.back();
            S.geo = &geo[p];
            for (int l = 0; l < geo[p].levels; ++l)
                compared += level_choices(geo[p].W[l], geo[p].H[l], geo[p].c[l], k, border, tile_w, heights, n_h,
                                          budget, S.level[l]);
        }
        ++shapes[s].pairs;
        shape_of[p] = (int)s;
    }
    int pick = 0;
    double best = -1.0;
    for (int i = 0; i < n_h; ++i) {
        double sum = 0.0, tile = 0.0;
        for (const Shape &S : shapes)
            for (int l = 0; l < S.geo->levels; ++l) {
                sum += 2.0 * S.pairs * S.level[l][i].cost;
                tile = std::max(tile, S.level[l][i].tile);
            }
        const double time = sum / ((double)kFastCtasPerSm * n_sm) + tile;
        if (best < 0.0 || time < best) { best = time; pick = i; }
    }
    blocks.resize(geo.size());
    for (size_t p = 0; p < geo.size(); ++p) {
        const Shape &S = shapes[(size_t)shape_of[p]];
        for (int l = 0; l < S.geo->levels; ++l) blocks[p][l] = { S.level[l][pick].bx, S.level[l][pick].by };
    }
    return compared;
}

}  // namespace jslam
