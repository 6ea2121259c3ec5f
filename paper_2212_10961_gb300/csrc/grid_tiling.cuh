// Tiling of one grid synthesis on the tensor cores: tile and chunk sizes, the
// patch of (y, z) cells, the shared-memory rings and the workspace tables.
// Evaluated on the host for a grid of cells and on the device for the node
// lattice of the band path, whose size the device chooses (band.cuh).
#pragma once

#include <cstdint>

#include "grid_common.cuh"

namespace grf {
namespace gridt {

constexpr int kGM = 128;                    // x cells per tile (TMEM lanes)
constexpr int kGN = 128;                    // (y, z) cells per tile (accumulator columns)
constexpr int kGModes = 32;                 // modes per chunk
constexpr int kGK = 2 * kGModes;            // K elements per chunk (re, im)
constexpr int kGOpBytes = kGM * kGK * 2;    // one FP16 operand tile (128 x 64): 16 KB
constexpr int kGPair = 2 * kGOpBytes;       // hi and lo tiles of one operand
constexpr int kGRowBytes = kGModes * 8 + 16;  // one table row of a chunk: 32 float2 + 16 bytes of padding
                                              // (consecutive rows start in different shared-memory banks)
constexpr int kGMaxSA = 4;
constexpr int kGSB = 3;                     // formed B stages (3-D)
constexpr int kGEpiWarps = 16;
constexpr int kGThreads = 32 * (kGEpiWarps + 2);
constexpr int kGColsPerWarp = kGN / (kGEpiWarps / 4);    // TMEM columns a warp folds (4 lane quarters)
// B formation: thread t forms one 4-mode group (t / 64) of two columns that
// share a y cell (z cells 2 q and 2 q + 1 of the patch, pair t mod 64), so the
// y row is read once for both
constexpr int kGFormPairs = kGN / 2;
static_assert(kGColsPerWarp % 32 == 0 && 32 * kGEpiWarps == kGFormPairs * (kGModes / 4), "epilogue warp layout");
constexpr uint32_t kGSbo = 1024;            // 8-row groups of a tile: one 128-byte-swizzle atom apart
constexpr uint32_t kGKStep = 32;            // bytes of 16 K elements inside an atom row
constexpr uint32_t kGTmemCols = 512;
constexpr uint32_t kGCorrCol = 256;         // hi.lo + lo.hi accumulator of the tile
constexpr uint32_t kGSumCol = 384;          // running FP32 sum of the folded hi.hi intervals
constexpr int kGBarBytes = 256;
constexpr int kGAlignPad = 1024;            // room to start the stages on a 1024-byte boundary
constexpr int kGSmemMax = gridc::kSmemMax;
constexpr int kGBandSmem = kGSmemMax - 2048;  // beside the descriptor in static shared memory
static_assert(kGM == 128 && kGN == 128, "tile shape is fixed by the TMEM layout");

__host__ __device__ constexpr int min2(int a, int b) { return a < b ? a : b; }
__host__ __device__ constexpr int64_t align_up256(int64_t v) { return (v + 255) & ~int64_t(255); }

// Layout of one grid synthesis: mode, patch, tiles, shared-memory rings and
// workspace tables.
struct GridPlan {
    bool form;
    int pk_log2, n_mt, n_kt, n_lt, nc, sa, a_stage, off_b, off_bar, smem;
    int max_split;  // mode splits for grids of few tiles (the launch takes at most one per fold interval)
    int64_t n_tiles, a_bytes, y_bytes, w_bytes, b_bytes, part_bytes;
};

// Grids of at most 64 tiles split each tile's modes over up to 8 CTAs, so
// that about 128 work items fill the GPU.
constexpr int kGMaxSplit = 8;
constexpr int64_t kGSplitItems = 128;

__host__ __device__ inline GridPlan grid_plan(int32_t nx, int32_t ny, int32_t nz, int32_t nc) {
    GridPlan g{};
    g.form = nz > 1;
    g.nc = nc;
    g.n_mt = (nx + kGM - 1) / kGM;
    if (g.form) {
        // patch 2^p y-cells by 128 / 2^p z-cells (p = 2 .. 6): fewest wasted
        // columns and staged table rows; 64 x 2 patches stage 66 rows, which
        // leaves two copy stages instead of three (the loads no longer hide
        // behind the products: 2.9 against 1.1 us per chunk)
        float best = 3.0e38f;
        for (int pk = 2; pk <= 6; ++pk) {
            const int PK = 1 << pk, PL = kGN / PK;
            const float cols = float((ny + PK - 1) / PK * PK) * float((nz + PL - 1) / PL * PL);
            const float w = cols / (float(ny) * float(nz)) + 1e-3f * float(PK + PL) + (pk == 6 ? 0.25f : 0.0f);
            if (w < best) {
                best = w;
                g.pk_log2 = pk;
            }
        }
        const int tb = ((1 << g.pk_log2) + (kGN >> g.pk_log2)) * kGRowBytes;
        g.a_stage = (kGPair + tb + 1023) / 1024 * 1024;  // swizzle atoms start on 1024-byte boundaries
        g.sa = min2(kGMaxSA, (kGBandSmem - kGAlignPad - kGBarBytes - kGSB * kGPair) / g.a_stage);
        g.off_b = g.sa * g.a_stage;
        g.off_bar = g.off_b + kGSB * kGPair;
    } else {
        g.pk_log2 = 7;
        g.a_stage = 2 * kGPair;
        g.sa = min2(kGMaxSA, (kGBandSmem - kGAlignPad - kGBarBytes) / g.a_stage);
        g.off_b = g.sa * g.a_stage;
        g.off_bar = g.off_b;
    }
    g.smem = g.off_bar + kGBarBytes + kGAlignPad;
    g.n_kt = (ny + (1 << g.pk_log2) - 1) >> g.pk_log2;
    const int PL = kGN >> g.pk_log2;
    g.n_lt = (nz + PL - 1) / PL;
    g.n_tiles = int64_t(g.n_mt) * g.n_kt * g.n_lt;
    g.max_split = g.n_tiles >= kGSplitItems ? 1 : min2(kGMaxSplit, static_cast<int>(kGSplitItems / g.n_tiles));
    g.part_bytes = g.max_split > 1 ? align_up256(int64_t(g.max_split) * nx * ny * nz * 4) : 0;
    g.a_bytes = align_up256(int64_t(g.n_mt) * g.nc * kGPair);
    if (g.form) {
        g.y_bytes = align_up256(int64_t(g.nc) * ny * kGRowBytes);
        g.w_bytes = align_up256(int64_t(g.nc) * nz * kGRowBytes);
    } else {
        g.b_bytes = align_up256(int64_t(g.n_kt) * g.nc * kGPair);
    }
    return g;
}

// fold: chunks per fold interval (the last one of a tile may be shorter).
__host__ __device__ inline void set_tiling(GridTiling& d, const GridPlan& g, int32_t nx, int32_t ny, int32_t nz,
                                           int32_t fold) {
    d.nx = nx;
    d.ny = ny;
    d.nz = nz;
    d.nc = g.nc;
    d.fc = min2(fold, g.nc);
    d.n_mt = g.n_mt;
    d.n_kt = g.n_kt;
    d.n_lt = g.n_lt;
    d.pk_log2 = g.pk_log2;
    d.n_tiles = g.n_tiles;
    d.n_split = min2(g.max_split, (g.nc + d.fc - 1) / d.fc);  // whole fold intervals per split
    d.n_items = d.n_tiles * d.n_split;
    d.xn = nx;
    d.lz = nz;
    d.zn = nz;
    d.form = g.form ? 1 : 0;
    d.sa = g.sa;
    d.a_stage = g.a_stage;
    d.off_b = g.off_b;
    d.off_bar = g.off_bar;
}

}  // namespace gridt
}  // namespace grf
