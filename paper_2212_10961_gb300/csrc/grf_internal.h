// Internal layout shared by the host code and the CUDA kernels of the
// spectral Gaussian-random-field library.  Not part of the public ABI.
#pragma once

#include <cstddef>
#include <cstdint>

#include <vector_types.h>

#include "grf.h"

#ifndef GRF_CHECKED
#define GRF_CHECKED 0  // 1 in the checked build (libgrf_checked.so)
#endif

namespace grf {

// ---------------------------------------------------------------------------
// Device mode table (built on the host by grf_pack_table).
//
// Modes are stored in decreasing order of h_j = sum_c |a_jc| (turns per unit
// length) and padded with zero-amplitude modes to a multiple of kChunk, so the
// chunked loops need no tail.  Sections (byte offsets from the table start,
// all 256-byte aligned):
//   hot  : float4[n_pad]   (2 pi a_x, 2 pi a_y, 2 pi a_z, A)  -- radians/unit
//   cold : float4[2*n_pad] (ah_x, al_x, ah_y, al_y), (ah_z, al_z, psi_h, psi_l)
//          a = ah + al and psi = psi_h + psi_l as FP32 pairs (turns)
//   order: int32[n_pad]    original mode index j (-1 for padding)
//   kpref: int32[kBuckets] kpref[b] = #{j : h_j * 2^((b - bias)/4) > 1}, the
//          length of the prefix of modes whose phase span over a box of
//          half-extent E exceeds tau turns is read at bucket(E / tau)
//   kappa: double[3*n_pad] standardised wave-vector of the mode in the slot
//          (zeros beyond dim and for padding); filled when the modes were
//          packed with their kappa (header has_kappa = 1).  Only the adjoint
//          reads it: the chain rule to l and R needs u = kappa / (2 pi l),
//          which a periodic axis's rounded frequency no longer determines.
// Every mode at an odd sorted position is stored in the equivalent form
// (-A, psi + 1/2): A cos(2 pi (a.x + psi)) = -A cos(2 pi (a.x + psi + 1/2)).
// Half of the terms then evaluate the hardware cosine half a turn away with
// the opposite sign, so a mean offset of its error over the phases cancels
// between the two halves instead of adding up over all N terms (it would
// otherwise grow like c * sum_j A_j ~ sqrt(N)).  Only the adjoint's dA_j
// changes sign with the form (dpsi, da and the chain rule are invariant).
// ---------------------------------------------------------------------------
constexpr int kChunk = 128;          // modes per shared-memory chunk
constexpr int kBuckets = 160;        // extent buckets
constexpr int kBucketBias = 100;     // E_b = 2^((b - kBucketBias) / 4)
constexpr float kTauLight = 8.0f;    // warp-origin path iff h_j * E_warp <= tau1 (turns)
constexpr float kTauMedium = 16.0f;  // lane-origin path iff h_j * E_lane <= tau2 (turns)
constexpr uint32_t kTableMagic = 0x54465247u;  // "GRFT"

// Sorted position s holds its mode in the form (-A, psi + 1/2).
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr bool mode_flipped(int64_t s) { return (s & 1) != 0; }
// Largest |a_c| (turns per unit length) accepted: with |x| < 2^16 the exact
// phase split needs |a x| < 2^46.
constexpr double kMaxFrequency = 1073741824.0;  // 2^30

struct TableHeader {
    uint32_t magic;
    int32_t n_modes;
    int32_t n_pad;
    int32_t dim;
    float tau;
    int32_t n_buckets;
    int32_t bucket_bias;
    int32_t has_kappa;  // 1: the kappa section holds the modes' kappa
    int64_t off_hot;
    int64_t off_cold;
    int64_t off_order;
    int64_t off_kpref;
    int64_t total_bytes;
    int64_t off_kappa;
    float amp_max;      // largest |A_j| as stored (FP32): the grid path's operand scale
    int32_t pad_;
    int64_t reserved[5];
};
static_assert(sizeof(TableHeader) <= 256, "table header must fit in 256 bytes");

inline int64_t align256(int64_t v) { return (v + 255) & ~int64_t(255); }
inline int64_t pad_modes(int64_t n) { return (n + kChunk - 1) / kChunk * kChunk; }

struct TableLayout {
    int64_t n_pad, off_hot, off_cold, off_order, off_kpref, off_kappa, total;
};

inline TableLayout table_layout(int64_t n_modes) {
    TableLayout L;
    L.n_pad = pad_modes(n_modes);
    L.off_hot = 256;
    L.off_cold = L.off_hot + align256(L.n_pad * 16);
    L.off_order = L.off_cold + align256(L.n_pad * 32);
    L.off_kpref = L.off_order + align256(L.n_pad * 4);
    L.off_kappa = L.off_kpref + align256(kBuckets * 4);
    L.total = L.off_kappa + align256(L.n_pad * 24);
    return L;
}

// ---------------------------------------------------------------------------
// Cell plan (device buffer built by grf_plan_cells).
//   header  : PlanHeader (256 B)
//   segs    : SegInfo[n_segments]
//   xs,ys,zs: float[n_cells] sorted coordinates
//   perm    : int32[n_cells] original (plan-global) index of sorted cell i
//   keys_in, keys_out : uint32[n_cells]   (planning scratch)
//   vals_in           : int32[n_cells]    (planning scratch)
//   sort_tmp          : radix-sort temporary storage
// ---------------------------------------------------------------------------
constexpr uint32_t kPlanMagic = 0x4E4C5047u;  // "GPLN"

struct GridCheck {
    unsigned long long c1;  // min {n >= 1 : (y_n, z_n) != (y_0, z_0)}, n_cells if none
    unsigned long long c2;  // min {n >= 1 : z_n != z_0}, n_cells if none (3-D)
    int32_t bad;            // some cell is not at (X_i, Y_k, Z_l) of its index
    int32_t pad_;
    uint64_t tag;           // host-assigned plan number
    float lo[3], hi[3];     // bounds of the cells
};
constexpr int kMortonBits = 10;                // quantised coordinate bits per axis

struct PlanHeader {
    uint32_t magic;
    int32_t status;       // device-side error bits
    int32_t dim;
    int32_t n_segments;
    int64_t n_cells;
    int64_t off_segs, off_xs, off_ys, off_zs, off_perm, off_keys_in, off_keys_out, off_vals_in,
        off_sort_tmp, sort_tmp_bytes, total_bytes;
    // Cartesian-grid check of a single-segment 2-D / 3-D plan (GridCheck):
    // the first index whose (y, z) differs from cell 0's (= nx), the first
    // whose z differs (= nx ny), a mismatch flag, and the plan's tag.  The
    // axes X (nx), Y (ny), Z (nz) are written over the keys_in scratch.
    GridCheck grid;
    int64_t reserved[7];
};
static_assert(sizeof(PlanHeader) <= 256, "plan header must fit in 256 bytes");

struct SegInfo {
    int64_t begin;        // first cell (global index)
    int64_t count;
    float lo[3];          // bounding box (float bits ordered as ints during the reduction)
    float hi[3];
    float inv_brick[3];   // quantisation levels per unit length (same on every axis)
    int32_t nb[3];        // quantisation levels per axis (<= 2^kMortonBits)
    int32_t pad;
};

struct PlanLayout {
    int64_t off_segs, off_xs, off_ys, off_zs, off_perm, off_keys_in, off_keys_out, off_vals_in,
        off_sort_tmp, sort_tmp_bytes, total;
};

size_t radix_sort_temp_bytes(int64_t n_cells);  // defined in plan.cu

inline PlanLayout plan_layout(int64_t n_cells, int32_t n_segments) {
    PlanLayout L;
    L.off_segs = 256;
    L.off_xs = L.off_segs + align256(int64_t(n_segments) * int64_t(sizeof(SegInfo)));
    L.off_ys = L.off_xs + align256(n_cells * 4);
    L.off_zs = L.off_ys + align256(n_cells * 4);
    L.off_perm = L.off_zs + align256(n_cells * 4);
    L.off_keys_in = L.off_perm + align256(n_cells * 4);
    L.off_keys_out = L.off_keys_in + align256(n_cells * 4);
    L.off_vals_in = L.off_keys_out + align256(n_cells * 4);
    L.off_sort_tmp = L.off_vals_in + align256(n_cells * 4);
    L.sort_tmp_bytes = int64_t(radix_sort_temp_bytes(n_cells));
    L.total = L.off_sort_tmp + align256(L.sort_tmp_bytes);
    return L;
}

// ---------------------------------------------------------------------------
// Map parameters as the kernels see them.
// ---------------------------------------------------------------------------
// Internal map bit, outside the public grf_map_bits: the field-mismatch loss
// of the calibration step and its gradient (grf_synth_mismatch), fused into
// the synthesis epilogue.
constexpr int32_t kMapMismatch = 1 << 16;

struct MapDev {
    int32_t bits;
    int32_t n_thr;
    float thr[GRF_MAX_THRESHOLDS];
    float values[GRF_MAX_THRESHOLDS + 1];
    float k_ref, phi0, phi1, phi_min, phi_max;
    float mu, sigma_inv;
    float* Y;
    float* K;
    uint8_t* F;
    float* P;
    // kMapMismatch: K = exp(Y), gY = g_scale (K - T) K, and per-unit sums of
    // (K - T)^2 in lpart (one entry per warp tile, or per block of the
    // split finalize), reduced afterwards into *loss / n_mean
    const float* T;
    float* G;
    double* lpart;
    double* loss;
    double inv_n_mean;
    float g_scale;        // 2 / n_mean (FP32, as the standalone loss kernel forms it)
    int32_t pad_;
};

struct BandDesc;

// One realisation as the forward kernel sees it.
struct FwdDesc {
    const float4* hot;
    const float4* cold;
    const int32_t* kpref;
    int32_t n_pad;
    int32_t dim;
    float inv_tau1;       // 1 / (span limit of the light class, turns)
    float inv_tau2;       // 1 / (span limit of the medium class, turns)
    const float* xs;      // sorted coordinates of this realisation's segment
    const float* ys;
    const float* zs;
    const int32_t* perm;  // original (plan-global) index of each sorted cell
    int64_t perm_base;    // first plan-global index of the segment
    int64_t n_cells;
    // band path (band.cuh): the table holds the band->nh direct modes, in
    // band->n_splits mode splits, and add[sorted cell] the light modes' sum
    const BandDesc* band;
    const float* add;
    MapDev map;
};

struct SegInfo;

// Most bytes of a call's tables and partial sums beside the direct sums' own:
// 1 GB, or 64 bytes per cell where that is more.
inline int64_t ws_most(int64_t n_cells) {
    return n_cells > (int64_t(1) << 24) ? 64 * n_cells : int64_t(1) << 30;
}

// Cartesian grid of a plan: cell n = i + nx (k + ny l) at (X_i, Y_k, Z_l).
struct GridGeom {
    int32_t nx, ny, nz;
    const float* X;
    const float* Y;
    const float* Z;
    const SegInfo* seg;  // bounds of the cells
};

// Coordinates of one axis of a grid synthesis: cell i at p[i], or, on the node
// lattice of the band path (band.cuh; p null), node i at (n0 + i) h.
struct AxisSrc {
    const float* p;
    float h;
    int32_t n0;
};

// Tables of one grid synthesis (workspace) as the prep kernel fills them.
struct GridPrep {
    const TableHeader* thdr;
    const float4* hot;
    const float4* cold;
    const int32_t* idx;  // table slots of the modes summed (-1: none), null for all in order
    AxisSrc ax[3];
    float gain_h[3];       // node spacings of the axes whose window gain multiplies the amplitudes (0: none)
    float scale;           // amplitude scale (0: from the table's largest amplitude)
    int32_t xn;            // x cells of a row block (GridDesc); rows beyond the first block are
    float zstep;           // shifted by this z distance per block
    int32_t nx, ny, nz, nc, n_mt, n_kt, dim;
    int32_t form;          // 1: 3-D (B formed from ytab, wztab), 0: B tabulated in btab
    unsigned char* atab;   // x phasors: FP16 hi/lo tiles [n_mt][nc][2][128 x 64]
    unsigned char* btab;   // 2-D: B tiles [n_kt][nc][2][128 x 64]
    float2* ytab;          // 3-D: [nc][ny][32] y phasors
    float2* wztab;         // 3-D: [nc][nz][32] (amplitude, psi, z) phasors
};

// Sizes of one grid synthesis (grid_tiling.cuh).
struct GridTiling {
    int64_t n_tiles;
    int64_t n_items;  // tiles x splits
    float scale;      // amplitude scale (0: from the table's largest amplitude)
    int32_t nx, ny, nz;
    int32_t nc;       // chunks of 32 modes
    int32_t fc;       // chunks per fold interval
    int32_t n_mt, n_kt, n_lt;
    int32_t pk_log2;  // (y, z) patch: 2^pk_log2 along y, 128 / 2^pk_log2 along z
    int32_t form;     // 1: B formed in shared memory from the staged table rows
    int32_t sa;       // stages of the copy ring
    int32_t a_stage;  // bytes per copy stage
    int32_t off_b;    // formed B ring (form)
    int32_t off_bar;  // barriers
    int32_t n_split;  // mode splits per tile (whole fold intervals each)
    // rows of a tile: x cell i mod xn in z block i / xn of lz layers (cells:
    // one block; node lattices of few x nodes fill the 128 rows with several)
    int32_t xn, lz, zn;
    // band path, at the cells: the light modes as nl further chunks before the
    // others, B from light[(l ny + k) lp + node] * l_inv
    int32_t nl, lp;
    float l_inv;
};

// One grid synthesis as the tensor-core kernel sees it.
struct GridDesc {
    const unsigned char* atab;
    const unsigned char* btab;
    const float2* ytab;
    const float2* wztab;
    const TableHeader* thdr;
    float* part;      // [n_split][xn ny zn] partial fields, summed by the finalize kernel
    int32_t quiet;    // 1: the tiles are not counted (nodes are not cells)
    // light chunks: A tiles latab[n_mt][nl] (x weights), first node of an x
    // tile lstart[n_mt], the rows of x nodes
    const unsigned char* latab;
    const int32_t* lstart;
    const float* light;
    GridTiling t;
    MapDev map;
};

// Band path (band.cuh) of one call, chosen on the device by band_select_kernel.
struct BandAxis {
    float h, inv_h;  // node spacing (0 with ident)
    int32_t n0, m;   // nodes (n0 + k) h, k < m
    int32_t ident;   // 1: not interpolated, the nodes are the axis's cells
};
struct BandDesc {
    int32_t nh;        // modes summed at the cells
    int32_t n_light;   // modes summed at the nodes (0: band path not taken)
    int32_t n_splits;  // mode splits whose partials the finalize kernel adds (0: none)
    int32_t finalize;  // 1: band_finalize_kernel writes the cells
    int64_t loss_nb;   // loss partials written
    int32_t lp;        // floats per row of x nodes
    float lw;          // factor of the x weights' operand tiles: lw l_inv = 1 / (amplitude scale)
    BandAxis ax[3];
    GridTiling nodes;  // light modes on the node lattice
    GridTiling cells;  // direct modes at the cells of a grid
};

// What the host knows of a band-path call: the table, the cells' axes or
// bounds, the limits of the workspace and the measured rates.
struct BandSelect {
    const float4* hot;
    const float4* cold;
    int32_t n_modes, dim;
    int32_t* idx_h;         // [n_modes padded to 32] table slots of the modes summed at the cells,
    int32_t* idx_l;         // and of those summed at the nodes, in table order, then -1
    const SegInfo* seg;     // bounds of the cells
    const int32_t* status;  // the plan's: bit 1 for cells that are not finite
    int32_t n[3];           // grid: cells per axis (0 without a grid)
    const float* X;         // grid: the x axis
    float us_mode;           // time of one mode summed directly, us
    float us_node;           // time of one mode at one node, us
    float us_fixed;          // time of the lattice's own kernels, us
    float us_heavy;          // time of the direct sum's kernels beside the modes', us
    int64_t cap_nodes;       // most nodes
    int64_t cap_part;        // floats of the nodes' partial sums
    int64_t cap_mid;         // most (x, y) nodes x z cells
    int32_t cap_mt;          // most 128-row tiles of the nodes' x operand
    int32_t cap_nl;          // most light chunks of an x tile
    int32_t cap_ax[3];       // most nodes of an axis (grids: at most its cells besides)
    int32_t fold;
    int32_t n_mt;            // x tiles of the cells
    int32_t* lstart;         // [n_mt] first x node of a tile (written here; null: no light chunks)
    int32_t chunk;           // the direct sum takes whole chunks of this many modes
    int32_t max_split;       // mode splits of the direct sum (1: unsplit)
    int32_t split_cells;     // 1: the direct sum leaves partial sums to the finalize kernel
    int64_t loss_nb_tiles;   // loss partials of an unsplit direct sum, and of the finalize kernel
    int64_t loss_nb_finalize;
    const TableHeader* thdr;
    GridTiling cells;        // the cells' tiling (all modes)
};

// Room of a band-path call's workspace for the lattice's tables, next to what
// the selection accepts (grf_debug_lattice_room).
struct LatticeRoom {
    int64_t limit[3];  // most nodes of an axis that the selection accepts
    int64_t held[3];   // nodes of an axis that the tables hold
    int64_t nodes, nodes_held;
    int64_t bytes;     // the lattice's part of the workspace (0: not offered)
    int64_t base;      // a grid path's own part; 0 at any cells
};

// Adjoint on the band path (band_bwd.cu): one axis of a grid's transposed
// interpolation, the phasor tables at the nodes, and the split of the sums.
struct BandAxisTab {
    float* w;        // [cells][8] weights
    int32_t* start;  // [cells] first node
    int2* range;     // [nodes] first and last cell of a node, counted as ord says
    float* wt;       // [cells of a node][nodes] the same weights by node, from the node's first cell
    int32_t* most;   // [2] most cells of a node, or 0 where wt does not hold them; 1 where ord counts
    int32_t* ord;    // [cells] axes in no order: the cells in the order of their nodes
    int32_t* pos;    // [nodes] scratch of that order
};
// Floats of BandAxisTab::wt: a node of an axis in order has about 8 cells /
// nodes cells.
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int64_t band_wt_floats(int64_t cells) { return 16 * cells + 1024; }
struct BandPhasors {
    float2* ph[3];   // [nodes][light modes padded to 128]
    float* off[3];   // [nodes] coordinate from the axis's first node
    double* gain;    // [4][light modes padded to 128]: the window's gain, and per axis
                     // (d ln gain / d a_c) / (2 pi)
    int32_t* rank;   // [table slots] light mode of the slot, or ~ direct mode
};
struct BandNodes {
    int32_t n_mt, n_xc, groups;  // mode tiles, x chunks, groups of lines
};
#ifdef __CUDACC__
__host__ __device__
#endif
inline BandNodes band_nodes_split(int32_t n_light, int32_t mx, int32_t lines, int32_t blocks) {
    BandNodes s;
    s.n_mt = (n_light + 127) / 128;
    s.n_xc = (mx + 63) / 64;
    const int32_t batches = (lines + 15) / 16, want = blocks / (s.n_mt * s.n_xc);
    s.groups = want < 1 ? 1 : want > batches ? batches : want;
    return s;
}
// Groups of a grid adjoint's units: one CTA per SM (mode tiles x groups <=
// SMs), at most kAdjMaxCtas of them.
constexpr int kAdjMaxCtas = 256;
#ifdef __CUDACC__
__host__ __device__
#endif
inline int32_t grid_adjoint_groups(int32_t n_mt, int64_t units, int32_t sms) {
    int64_t g = n_mt > 0 ? sms / n_mt : 1;
    if (g > units) g = units;
    const int64_t room = n_mt > 0 && kAdjMaxCtas / n_mt > 1 ? kAdjMaxCtas / n_mt : 1;
    if (g > room) g = room;
    return g < 1 ? 1 : static_cast<int32_t>(g);
}
// Splits of the cells of band_direct_kernel (blocks for each tile of 128 modes).
#ifdef __CUDACC__
__host__ __device__
#endif
inline int32_t band_direct_splits(int32_t nh, int32_t blocks) {
    const int32_t tiles = (nh + 127) / 128;
    return tiles < 1 ? 1 : blocks / tiles > 1 ? blocks / tiles : 1;
}
// The band path's part of the adjoint's reduction (null: all modes from part).
struct BandReduce {
    const BandDesc* b;
    const int32_t* rank;
    const double* gain;
    const double* part;    // light modes' sums over the nodes
    int32_t blocks;        // as in band_nodes_split
    int32_t direct_units;  // > 0: direct sums of the grid adjoint (units, SMs);
    int32_t direct_sms;    // 0: of band_direct_kernel (its blocks)
};

// Work tile of the batched launch: realisation r, tile index t inside it.
struct WorkItem {
    int32_t r;
    int32_t t;
};

// Batched workspace layout.
struct BatchHeader {
    uint32_t magic;
    int32_t n_items;
    int32_t n_work;
    int32_t tile_cells;
    int32_t cfg;          // kernel configuration index
    int32_t dim_max;
    int64_t off_desc, off_work, off_counter, total_bytes;
    int64_t reserved[24];
};
constexpr uint32_t kBatchMagic = 0x48435442u;  // "BTCH"

// ---------------------------------------------------------------------------
// Kernel launchers (defined in the .cu files), all asynchronous on `stream`.
// Return cudaError_t as int.
// ---------------------------------------------------------------------------
// seg: the segment's bounds, to take the band path with the first
// cells_band_ws_bytes of the workspace; null: all modes directly.  few: few
// modes are expected to be left for the direct sum.
struct CellsBand {
    const SegInfo* seg = nullptr;
    bool few = false;
};
int launch_synth_fwd(const FwdDesc& d, const void* table, int64_t n_modes, const CellsBand& band, void* workspace,
                     size_t ws_bytes, int32_t* status, void* stream);
// Entries of MapDev::lpart a launch of n cells may write (kMapMismatch).
int64_t mismatch_partials(int64_t n_cells);
// loss = (sum of the nb partials, fixed order) * inv_n, one block.
// nb_dev, if not null, holds the count on the device instead of nb.
int launch_loss_sum(const double* part, int64_t nb, const int64_t* nb_dev, double inv_n, double* out, void* stream);

// Checked builds (-DGRF_CHECKED=1): device accesses skipped since the last
// call because an index read from device memory was out of range, per
// translation unit, then reset; ~0 if the counter cannot be read; always 0
// in release builds.
unsigned long long take_index_faults_fwd();
unsigned long long take_index_faults_bwd();
unsigned long long take_index_faults_plan();
// Warp tiles of single-field synthesis launches that took the general and the
// lattice path since the last call, then reset (synchronous); cudaError_t.
int take_path_counts(unsigned long long* general, unsigned long long* lattice);
// The same for the 3-D adjoint's warp tiles (synth_bwd.cu).
int take_bwd_path_counts(unsigned long long* general, unsigned long long* lattice);
size_t synth_workspace_bytes(int64_t n_cells);
int launch_synth_batched(const void* workspace, const BatchHeader& h, int32_t* status,
                         int32_t* counter, void* stream);
int fwd_tile_cells(int cfg);
int launch_map(const MapDev& m, int64_t n, const float* Y, void* stream);
int launch_bimap(const grf_bimap& m, int64_t n, const float* Y1, const float* Y2, uint8_t* F, float* P,
                 void* stream);
// tag: host-assigned plan number, stored with the grid check (GridCheck::tag)
int launch_plan(int32_t dim, int32_t n_segments, const int64_t* seg_offsets_host, const float* x,
                const float* y, const float* z, void* plan, const PlanLayout& L, uint64_t tag, void* stream);
// band: the segment's bounds, to take the band path, whose workspace
// (cells_adjoint_band_ws_bytes) follows bwd_workspace_bytes; null: all modes directly.
// periodic_mask: bit c set when axis c is periodic (its frequency is rounded,
// so its dL/da reaches neither kappa, l nor R).
int launch_synth_bwd(const void* table, int64_t n_modes, int32_t dim, double sigma,
                     const double* ell, const double* rot, int32_t periodic_mask, const float* xs,
                     const float* ys, const float* zs,
                     const int32_t* perm, int64_t perm_base, int64_t n_cells, const float* gY,
                     const grf_grads& g, const SegInfo* band, void* workspace, int32_t* status, void* stream);
size_t bwd_workspace_bytes(int64_t n_cells, int64_t n_modes, int32_t dim);
// Per-mode terms of the scalar gradients the adjoint's reduction writes
// (contrib rows: (A / sigma) dA, three l terms, nine R terms).
constexpr int kBwdContrib = 13;
// The adjoint's reduction and chain rule from per-mode partial sums:
// part[s][slot][5] = (sum g cos, sum g sin, sum g x sin, sum g y sin,
// sum g z sin) for s < splits (summed in increasing s), gpart[0 .. n_gpart)
// partial sums of g, contrib: kBwdContrib x n_pad doubles of scratch.
int launch_bwd_reduce(const void* table, int64_t n_modes, int32_t dim, double sigma, const double* ell,
                      const double* rot, int32_t periodic_mask, const grf_grads& g, double* part, int32_t splits,
                      double* gpart, int32_t n_gpart, double* contrib, const BandReduce& band, void* stream);
// Tensor-core adjoint on a Cartesian grid in x-fastest order (synth_grid_bwd.cu):
// workspace bytes, the launch (scan, prep, tensor-core kernel, reduction) and
// the units computed since the last call (synchronous).
size_t bwd_grid_ws_bytes(int32_t nx, int32_t ny, int32_t nz, int64_t n_pad);
int launch_synth_bwd_grid(const void* table, int64_t n_modes, int32_t dim, const GridGeom& gg, const float* gY,
                          double sigma, const double* ell, const double* rot, int32_t periodic_mask,
                          const grf_grads& g, void* ws, bool band, int32_t* status, void* stream);
// Measured times of the band path (us): one mode at one node (tensor cores,
// whole 128 x 128 tiles), the kernels that the lattice adds, and the kernels
// that a call pays for when the device finds no lattice worth while.
constexpr double kBandNodeUs = 1.0 / 22.0e6, kBandFixedUs = 15.0, kBandTryUs = 14.0;
// band: the band path, whose workspace (bwd_grid_band_ws_bytes) follows.
size_t bwd_grid_band_ws_bytes(int32_t nx, int32_t ny, int32_t nz, int64_t n_pad);
double grid_adjoint_us_per_mode(int32_t nx, int32_t ny, int32_t nz);
// Measured times of the adjoint's band path (us): one mode at one node, and the
// kernels that the lattice adds.
constexpr double kBandNodeAdjUs = 1.0 / 6.0e6;
double grid_adjoint_band_us(int32_t nx, int32_t ny, int32_t nz);
// The same as a forecast of whole calls: a mode as products, the other kernels
// of a call with all of them so, what those and the lattice's chain take
// beside grid_adjoint_band_us, and the kernels of modes left for the products.
double grid_adjoint_call_us_per_mode(int32_t nx, int32_t ny, int32_t nz);
constexpr double kAdjCallUs = 35.0, kAdjBandCallUs = 40.0 + kBandTryUs;
double grid_adjoint_heavy_us(int64_t n_cells);
size_t cells_adjoint_band_ws_bytes(int64_t n_cells, int64_t n_modes, int32_t dim);
LatticeRoom cells_adjoint_room(int64_t n_cells, int64_t n_modes, int32_t dim);
LatticeRoom cells_room(int64_t n_cells, int64_t n_modes, int32_t dim);
LatticeRoom grid_room(int32_t nx, int32_t ny, int32_t nz, int64_t n_pad);
LatticeRoom grid_adjoint_room(int32_t nx, int32_t ny, int32_t nz, int64_t n_pad);
double cells_adjoint_us_per_mode(int64_t n_cells);
double cells_adjoint_band_us(int64_t n_cells, int32_t dim);
// max |g| (inf if some g is not finite) and compensated sums of g, per block of
// a fixed partition of n values into adj_scan_blocks().
int launch_adj_scan(const float* g, int64_t n, const float* X, int32_t nx, float* gmax, double* gsum, float* xmax,
                    void* stream);
int adj_scan_blocks();
// Kernels of band_bwd.cu.
int launch_band_grid_spread(const BandDesc* b, const GridGeom& gg, const float* g, const BandAxisTab* tab, float* h1,
                            float* h2, float* nodes, int sms, void* stream);
int launch_band_spread(const BandDesc* b, int32_t dim, const float* xs, const float* ys, const float* zs,
                       const int32_t* perm, int64_t perm_base, int64_t n, const float* g, const float* gmax,
                       int n_gmax, unsigned long long* lattice, float* nodes, int sms, void* stream);
int launch_band_direct(const BandDesc* b, int32_t dim, const float4* cold, const int32_t* idx, const float* xs,
                       const float* ys, const float* zs, const int32_t* perm, int64_t perm_base, int64_t n,
                       const float* g, double* part, int blocks, void* stream);
int launch_band_nodes(const BandDesc* b, const float4* cold, const int32_t* idx_l, const int32_t* idx_h,
                      const GridGeom& gg, int32_t dim, const float* nodes, const BandPhasors& t, double* part, int sms,
                      void* stream);
int take_grid_adj_units(unsigned long long* units);
int launch_mismatch(int64_t n, const float* K, const float* T, float* gY, double* loss, void* ws,
                    void* stream);
size_t mismatch_workspace_bytes(int64_t n);
int launch_mufu_probe(int32_t blocks, int32_t iters, float* sink, void* stream);
// Grid path (synth_grid.cu): workspace bytes of the tables, the launch (prep
// + tensor-core kernel), tiles computed since the last call (synchronous),
// and the MMA self-test.
size_t grid_ws_bytes(int32_t nx, int32_t ny, int32_t nz, int64_t n_pad);
// Loss partials (kMapMismatch) the grid path writes: one per epilogue warp per tile.
int64_t grid_loss_partials(int32_t nx, int32_t ny, int32_t nz);
// Tiles of 128 x 128 cells of a grid.
int64_t grid_tiles(int32_t nx, int32_t ny, int32_t nz);
// band: the band path (band.cuh), whose workspace follows (ws_bytes >=
// grid_ws_bytes + grid_band_ws_bytes).
int launch_synth_grid(const void* table, int64_t n_modes, int32_t dim, const GridGeom& gg, const MapDev& map,
                      void* ws, bool band, int32_t fc, int32_t* status, void* stream);
// Time of one mode summed at the cells of a grid by the grid path, us.
double grid_us_per_mode(int32_t nx, int32_t ny, int32_t nz);
// Whether the grid path splits the modes of this grid's tiles over several CTAs.
bool grid_splits(int32_t nx, int32_t ny, int32_t nz);
// Further workspace of the band path on a grid (0: not taken at these sizes).
size_t grid_band_ws_bytes(int32_t nx, int32_t ny, int32_t nz, int64_t n_pad);
// Band path kernels (band.cu).
int launch_band_select(const BandSelect& p, BandDesc* out, void* stream);
int launch_band_lines(const BandDesc* b, float* part, const GridGeom& gg, float* mid, float* rows, int sms,
                      void* stream);
int launch_band_finalize(const BandDesc* b, const float* mid, const float* part, const GridGeom& gg,
                         const MapDev& map, unsigned long long* tiles, int sms, void* stream);
int64_t band_finalize_blocks(const GridGeom& gg);
// Band path at the cells of any plan (synth_grid.cu): workspace bytes (0: not
// taken at these sizes) and the launch up to the light modes' sums at the
// sorted cells; `d` gets the direct modes' table, `add` and `band`.
size_t cells_band_ws_bytes(int64_t n_cells, int64_t n_modes, int32_t dim);
int launch_cells_band(const void* table, int64_t n_modes, FwdDesc& d, const SegInfo* seg, void* ws,
                      int32_t max_split, int64_t loss_tiles, int64_t loss_finalize, int32_t* status, void* stream);
// Time of one mode summed at n cells of a plan that is not a grid, and of the
// interpolation to them, us.
double cells_us_per_mode(int64_t n_cells);
int64_t cells_band_cap(int64_t n_cells);
double cells_band_us(int64_t n_cells, int32_t dim);
int launch_band_cells(const BandDesc* b, const float* nodes, int32_t dim, const float* xs, const float* ys,
                      const float* zs, int64_t n, float* out, void* stream);
int take_grid_tiles(unsigned long long* tiles);
int launch_mma_probe(const uint16_t* A, const uint16_t* B, int32_t k_chunks, float* D, int32_t* status,
                     void* stream);
int launch_grid_check(int32_t dim, int64_t n, const float* x, const float* y, const float* z, void* plan,
                      const PlanLayout& L, void* stream);
int launch_selftest_wait(uint64_t limit_ns, int32_t* status, void* stream);
void count_launches(int64_t n);
// Record `message` as the calling thread's last error and return `code`.
int set_error(int code, const char* message);
// Allocation point of the host code: throws std::bad_alloc while injected
// failures remain (grf_debug_inject_alloc_failures); ABI entry points turn
// it into GRF_ENOMEM.
void alloc_point();

}  // namespace grf
