// Adjoint on the band-limited path (band.cuh): dL/dY is carried to the node
// lattice with the interpolation's weights transposed, and the light modes'
// sums are taken over the nodes.
//
// With G the gradient at the nodes and gain_j the window's gain,
//     E_j = sum_i g_i e^{i theta_ij} = gain_j sum_n G_n e^{2 pi i (a_j . X_n + psi_j)},
// and S_c = sum_i g_i x_ic sin theta_ij is the derivative of E_j in a_jc: with
// the nodes' own sums S~_c (of G, X_n) it is
//     S_c = gain_j S~_c - (d ln gain_j / d a_jc) / (2 pi) Re E_j,
// applied in FP64 by the reduction (bwd_reduce_kernel), which also applies the
// chain rule as on the other paths.
//
// Kernels, between the selection (band.cu) and the reduction (synth_bwd.cu):
//   grid:  band_axis_kernel      per axis: weights, first nodes, cells of a node
//          band_tx_kernel        x: g -> (x nodes) x (y, z cells)
//          band_tline_kernel     y, then z
//   cells: band_spread_kernel    groups of cells -> fixed-point node sums
//          band_unfix_kernel     fixed point -> FP32
//   both:  band_phasor_kernel    phasors of the light modes at the nodes' axes
//          band_nodes_kernel     the sums over the nodes
//   cells: band_direct_kernel    the direct modes' sums at the cells
#include <cuda_runtime.h>

#include <algorithm>

#include "band.cuh"
#include "device_common.cuh"
#include "grid_tiling.cuh"
#include "launch.cuh"

namespace grf {

namespace {

using band::kW;

// ---------------------------------------------------------------------------
// Grid: transposed interpolation axis by axis
// ---------------------------------------------------------------------------

// Block c: the cells' weights of axis c, their first nodes, for every node the
// first and last of the cells that read it, and the weights by node.  The
// cells are counted in the axis's own order where it runs one way; on an axis
// in no order by their first nodes (`ord`, a counting sort), so that a node's
// cells are neighbours there too: read as they come, a node takes the whole
// axis (2048 x 128 x 64 cells of a rough field, all axes in random order: 1363
// us a call, 680 so).  Where the cells crowd at few nodes that order would take long
// and wt may not hold the weights: the sums then run over all cells between
// the first and the last, skipping those that do not read the node.
constexpr int kCrowd = 64;  // most cells with the same first node that are put in order
__global__ void __launch_bounds__(1024) band_axis_kernel(const BandDesc* b, GridGeom gg, BandAxisTab tx, BandAxisTab ty,
                                                         BandAxisTab tz) {
    __shared__ int most, ups, downs, crowd, warps[32];
    pdl_wait();
    if (b->n_light == 0) return;
    const int c = blockIdx.x;
    const BandAxis ax = b->ax[c];
    const float* X = c == 0 ? gg.X : c == 1 ? gg.Y : gg.Z;
    const int n = c == 0 ? gg.nx : c == 1 ? gg.ny : gg.nz;
    const BandAxisTab t = c == 0 ? tx : c == 1 ? ty : tz;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) most = ups = downs = crowd = 0;
    for (int k = threadIdx.x; k < ax.m; k += blockDim.x) t.range[k] = make_int2(INT_MAX, -1);
    __syncthreads();
    const int nt = band::taps(ax);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        float w[kW];
        const float x = __ldg(X + i), before = __ldg(X + max(i - 1, 0));
        const int s = band::cell_weights(ax, x, i, w);
        if (!ax.ident && x > before) ups = 1;
        if (!ax.ident && x < before) downs = 1;
        t.start[i] = s;
#pragma unroll
        for (int k = 0; k < kW; ++k) w[k] = k < nt ? w[k] : 0.0f;
        float4* o = reinterpret_cast<float4*>(t.w + static_cast<int64_t>(i) * kW);
        o[0] = make_float4(w[0], w[1], w[2], w[3]);
        o[1] = make_float4(w[4], w[5], w[6], w[7]);
    }
    __syncthreads();
    bool sorted = ups != 0 && downs != 0;
    if (sorted) {
        // cells per first node, then of the nodes before it
        for (int k = threadIdx.x; k < ax.m; k += blockDim.x) t.pos[k] = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += blockDim.x) atomicAdd(&t.pos[t.start[i]], 1);
        __syncthreads();
        int carry = 0;
        for (int k0 = 0; k0 < ax.m; k0 += blockDim.x) {
            const int k = k0 + threadIdx.x, own = k < ax.m ? t.pos[k] : 0;
            if (own > kCrowd) crowd = 1;
            int v = own;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, v, off);
                if (lane >= off) v += o;
            }
            if (lane == 31) warps[warp] = v;
            __syncthreads();
            int sum = warps[lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, sum, off);
                if (lane >= off) sum += o;
            }
            const int until = __shfl_sync(0xffffffffu, sum, max(warp - 1, 0));
            if (k < ax.m) t.pos[k] = carry + (warp > 0 ? until : 0) + v - own;
            carry += __shfl_sync(0xffffffffu, sum, 31);
            __syncthreads();
        }
        sorted = crowd == 0;
    }
    if (sorted) {
        for (int i = threadIdx.x; i < n; i += blockDim.x) t.ord[atomicAdd(&t.pos[t.start[i]], 1)] = i;
        __syncthreads();
        // pos[k] is now the end of node k's cells; they get a fixed order
        for (int k = threadIdx.x; k < ax.m; k += blockDim.x) {
            const int p0 = k > 0 ? t.pos[k - 1] : 0, p1 = t.pos[k];
            for (int p = p0 + 1; p < p1; ++p) {
                const int v = t.ord[p];
                int q = p;
                for (; q > p0 && t.ord[q - 1] > v; --q) t.ord[q] = t.ord[q - 1];
                t.ord[q] = v;
            }
            // read by the cells whose first node is k - 7 to k
            t.range[k] = make_int2(k >= kW ? t.pos[k - kW] : 0, p1 - 1);
        }
    } else {
        for (int i0 = 0; i0 < n; i0 += blockDim.x) {
            const int i = i0 + threadIdx.x;
            const int s = i < n ? t.start[i] : -1;
            // of neighbours with the same nodes the first and the last count
            const int prev = __shfl_up_sync(0xffffffffu, s, 1), next = __shfl_down_sync(0xffffffffu, s, 1);
            const bool low = lane == 0 || prev != s, high = lane == 31 || next != s;
            if (i >= n) continue;  // the last round
            for (int k = 0; k < nt; ++k) {
                if (low) atomicMin(&t.range[s + k].x, i);
                if (high) atomicMax(&t.range[s + k].y, i);
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < ax.m; k += blockDim.x)
        if (t.range[k].x <= t.range[k].y) atomicMax(&most, t.range[k].y - t.range[k].x + 1);
    __syncthreads();
    // nodes that no cell reads: an empty range
    for (int k = threadIdx.x; k < ax.m; k += blockDim.x)
        if (t.range[k].x > t.range[k].y) t.range[k] = make_int2(0, -1);
    const bool fits = static_cast<int64_t>(most) * ax.m <= band_wt_floats(n);
    if (threadIdx.x == 0) {
        t.most[0] = fits ? most : 0;
        t.most[1] = sorted ? 1 : 0;
    }
    if (!fits) return;
    __syncthreads();
    constexpr int kAt = 4;  // values in flight of a thread: each is a chain of loads
    const int all = most * ax.m;
    for (int u0 = threadIdx.x; u0 < all; u0 += kAt * blockDim.x) {
        float w[kAt];
#pragma unroll
        for (int e = 0; e < kAt; ++e) {
            const int u = min(u0 + e * static_cast<int>(blockDim.x), all - 1);
            const int q = u / ax.m, node = u - q * ax.m;
            const int2 r = t.range[node];
            const int p = min(r.x + q, n - 1), i = sorted ? t.ord[p] : p;
            const unsigned k = static_cast<unsigned>(node - t.start[i]);
            w[e] = q <= r.y - r.x && k < kW ? t.w[static_cast<int64_t>(i) * kW + (k & (kW - 1))] : 0.0f;
        }
#pragma unroll
        for (int e = 0; e < kAt; ++e)
            if (u0 + e * static_cast<int>(blockDim.x) < all) t.wt[u0 + e * static_cast<int>(blockDim.x)] = w[e];
    }
}

// x: out[row][node] = sum over the node's cells of w g[row][cell].  A block
// takes kTxRows rows of cells, staged in shared memory in pieces of kTxCells:
// lanes are nodes, warps groups of rows, a thread kTxPer rows of one node (a
// weight is read once for them).  Of a row of more than one piece, 32 nodes
// take only the cells that they weigh: staged whole for each 32 nodes, a row of
// 16 384 cells and 520 nodes was read 17 times.  Bound by the read of g and by
// latency.
constexpr int kTxRows = 32, kTxPer = 4, kTxCells = 256;
__global__ void __launch_bounds__(256) band_tx_kernel(const BandDesc* b, const float* g, int nx, int64_t n_rows,
                                                      BandAxisTab tab, float* __restrict__ out) {
    __shared__ float gs[kTxRows / kTxPer][kTxCells][kTxPer];
    pdl_wait();
    if (b->n_light == 0) return;
    const int mx = b->ax[0].m, most = tab.most[0];
    const int32_t* ord = tab.most[1] ? tab.ord : nullptr;  // cells in the order of their nodes
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // a row of one piece stays for all its nodes; of a longer one a unit takes
    // 32 nodes
    const bool whole = nx <= kTxCells;
    const int passes = whole ? 1 : (mx + 31) / 32;
    const int64_t units = (n_rows + kTxRows - 1) / kTxRows * passes;
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
        const int64_t r0 = u / passes * kTxRows;
        const int first = static_cast<int>(u % passes) * 32, last = whole ? mx : min(first + 32, mx);
        const int nr = static_cast<int>(min(static_cast<int64_t>(kTxRows), n_rows - r0));
        for (int n0 = first; n0 < last; n0 += 32) {
            const int node = n0 + lane;
            const int2 range = node < mx ? tab.range[node] : make_int2(0, -1);
            float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            // the cells of the row that these nodes need (the same in every warp)
            int lo = 0, hi = nx - 1;
            if (!whole) {
                lo = __reduce_min_sync(0xffffffffu, range.y < range.x ? INT_MAX : range.x) & ~31;
                hi = __reduce_max_sync(0xffffffffu, range.y);
            }
            for (int c0 = lo; c0 <= hi; c0 += kTxCells) {
                const int nc = min(kTxCells, hi + 1 - c0);
                if (n0 == 0 || !whole) {
                    __syncthreads();
                    if (ord == nullptr) {
                        for (int r = warp; r < kTxRows; r += 8)
#pragma unroll 4
                            for (int i = lane; i < nc; i += 32)
                                gs[r / kTxPer][i][r % kTxPer] = r < nr ? g[(r0 + r) * nx + c0 + i] : 0.0f;
                    } else {
                        for (int i = lane; i < nc; i += 32) {
                            const int cell = ord[c0 + i];
                            for (int r = warp; r < kTxRows; r += 8)
                                gs[r / kTxPer][i][r % kTxPer] = r < nr ? g[(r0 + r) * nx + cell] : 0.0f;
                        }
                    }
                    __syncthreads();
                }
                const int ca = max(range.x, c0), cb = min(range.y, c0 + nc - 1);
                auto add = [&](float w, int i) {
                    const float4 v = *reinterpret_cast<const float4*>(gs[warp][i - c0]);
                    acc.x = fmaf(w, v.x, acc.x);
                    acc.y = fmaf(w, v.y, acc.y);
                    acc.z = fmaf(w, v.z, acc.z);
                    acc.w = fmaf(w, v.w, acc.w);
                };
                if (most > 0) {
                    const float* wt = tab.wt + (ca - range.x) * mx + node;
#pragma unroll 8
                    for (int i = ca; i <= cb; ++i, wt += mx) add(*wt, i);
                } else {
                    for (int i = ca; i <= cb; ++i) {
                        const int cell = ord != nullptr ? ord[i] : i;
                        const unsigned k = static_cast<unsigned>(node - tab.start[cell]);
                        if (k < kW) add(tab.w[static_cast<int64_t>(cell) * kW + k], i);
                    }
                }
            }
            if (node < mx) {
                const float v[kTxPer] = {acc.x, acc.y, acc.z, acc.w};
#pragma unroll
                for (int q = 0; q < kTxPer; ++q) {
                    const int r = warp * kTxPer + q;
                    if (r < nr) out[(r0 + r) * mx + node] = v[q];
                }
            }
        }
        __syncthreads();
    }
}

// y (kY) and z: out[node][column] = sum over the node's cells of w in[cell][column].
// y: columns are the x nodes of every layer l, in[(l ny + cell) m_x + i] ->
// out[(l m_y + node) m_x + i]; z: columns are the (x, y) nodes.  One thread per
// value, contiguous over the columns; all loads of a value are independent.
template <bool kY>
__global__ void __launch_bounds__(256) band_tline_kernel(const BandDesc* b, const float* in, int n, int nz,
                                                         BandAxisTab tab, float* __restrict__ out) {
    pdl_wait();
    if (b->n_light == 0) return;
    const int mx = b->ax[0].m, m = kY ? b->ax[1].m : b->ax[2].m, most = tab.most[0];
    const int32_t* ord = tab.most[1] ? tab.ord : nullptr;  // cells in the order of their nodes
    const int64_t plane = static_cast<int64_t>(mx) * b->ax[1].m;
    const int64_t all = kY ? plane * nz : plane * m;
    const int64_t stride = kY ? mx : plane;
    for (int64_t u = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; u < all;
         u += static_cast<int64_t>(gridDim.x) * 256) {
        int node;
        const float* src;
        if (kY) {
            const int64_t l = u / plane;
            const int p = static_cast<int>(u - l * plane);
            node = p / mx;
            src = in + l * n * mx + (p - node * mx);
        } else {
            node = static_cast<int>(u / plane);
            src = in + (u - node * plane);
        }
        const int2 range = tab.range[node];
        float acc = 0.0f;
        if (most > 0 && ord == nullptr) {
#pragma unroll 8
            for (int i = range.x; i <= range.y; ++i)
                acc = fmaf(tab.wt[(i - range.x) * m + node], src[i * stride], acc);
        } else if (most > 0) {
#pragma unroll 8
            for (int i = range.x; i <= range.y; ++i)
                acc = fmaf(tab.wt[(i - range.x) * m + node], src[ord[i] * stride], acc);
        } else {
            for (int i = range.x; i <= range.y; ++i) {
                const int cell = ord != nullptr ? ord[i] : i;
                const unsigned k = static_cast<unsigned>(node - tab.start[cell]);
                if (k < kW) acc = fmaf(tab.w[static_cast<int64_t>(cell) * kW + k], src[cell * stride], acc);
            }
        }
        out[u] = acc;
    }
}

// ---------------------------------------------------------------------------
// Cells of any plan: spread to fixed-point node sums
// ---------------------------------------------------------------------------

// Two powers of two: `first` brings max |g| below 1 before the weights (a tiny
// g would lose its weights' tails to underflow), `second` then the sum of any
// cells' |g| below 2^61 (weights are below 1/2 and at most one in sum): sums
// of integers do not depend on their order, so the atomics leave the result
// deterministic.  The grain is 2^-61 of n max |g| or less.
struct FixedScale {
    float first, second;
};
constexpr float kFiniteMax = 3.402823466e38f;
__device__ __forceinline__ FixedScale fixed_scale(const float* gmax, int n_gmax, int64_t n) {
    float m = 0.0f;
    for (int k = threadIdx.x & 31; k < n_gmax; k += 32) m = fmaxf(m, gmax[k]);
    m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
    if (!(m > 0.0f) || !(m <= kFiniteMax)) return FixedScale{1.0f, 1.0f};
    int e = 0, c = 0;
    frexpf(m, &e);
    frexpf(static_cast<float>(n), &c);
    return FixedScale{ldexpf(1.0f, min(126, -e)), ldexpf(1.0f, 61 - c)};  // -e >= -128; below 2^-126 g is subnormal
}

__device__ __forceinline__ bool gmax_finite(const float* gmax, int n_gmax) {
    bool ok = true;
    for (int k = threadIdx.x & 31; k < n_gmax; k += 32) ok = ok && gmax[k] <= kFiniteMax;
    return __all_sync(0xffffffffu, ok);
}

// A warp takes up to kSpreadCells consecutive sorted cells and adds them, one
// after the other, to a box of nodes of its own in shared memory: the lanes
// hold eight x nodes of four y rows, 16 nodes each.  The cells are first put in
// the order of their first nodes (a stable counting sort: the order of the sums
// is fixed), so that cells with the same nodes, about (node spacing / cell
// spacing)^3 of them, add up in registers and the box is read and written once
// for them: added cell by cell, the box took 133 instructions per cell and 637
// us for 2M cells.  Then the box goes to the lattice by integer atomics.
// A group whose box does not fit (one across a jump of the cells' order) is
// taken in quarters, down to 32 cells, which then send their values straight to
// the lattice, 512 atomics a cell: sent so as a whole, the few groups that jump
// made two thirds of the atomics.  Bound by latency (warps active 15 %, issue
// 47 %), hence the small box, which lets 14 warps stay on an SM, and the next
// cell's weights loaded ahead: 579 -> 397 us for 2M cells.
constexpr int kSpreadCells = 256, kSpreadWarps = 2, kSpreadFloats = 2048, kSpreadBins = 512;
struct SpreadSmem {
    float box[kSpreadFloats];
    float wts[32][28];  // a round's weights: x (times g), y, z; 16-byte aligned rows
    int at[32];
    int bins[kSpreadBins];
    short order[kSpreadCells];
};
template <int DIM>
__global__ void __launch_bounds__(32 * kSpreadWarps) band_spread_kernel(
    const BandDesc* b, const float* __restrict__ xs, const float* __restrict__ ys, const float* __restrict__ zs,
    const int32_t* __restrict__ perm, int64_t perm_base, int64_t n, const float* g, const float* gmax, int n_gmax,
    int cells, unsigned long long* lattice) {
    __shared__ __align__(16) SpreadSmem smem[kSpreadWarps];
    pdl_wait();
    if (b->n_light == 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    SpreadSmem& sm = smem[warp];
    const FixedScale scale = fixed_scale(gmax, n_gmax, n);
    BandAxis ax[DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c) ax[c] = b->ax[c];
    const int mx = ax[0].m;
    const int64_t plane = static_cast<int64_t>(mx) * ax[1].m;
    const int64_t first = (static_cast<int64_t>(blockIdx.x) * kSpreadWarps + warp) * cells;
    if (first >= n) return;  // no block-wide barrier below
    const int all = static_cast<int>(min(static_cast<int64_t>(cells), n - first));
    int part = all;
    for (int at = 0; at < all;) {
        const int64_t c0 = first + at;
        const int nc = min(part, all - at);
        const float* src[3] = {xs + c0, ys + c0, zs + c0};
        // ---- the cells' first nodes and the group's box
        constexpr int kPer = kSpreadCells / 32;
        int s[kPer][DIM];
        int f0[3] = {0, 0, 0}, nb[3] = {1, 1, 1};
#pragma unroll
        for (int c = 0; c < DIM; ++c) {
            int lo = INT_MAX, hi = 0;
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                float v;
                s[q][c] = band::locate(ax[c], __ldg(src[c] + min(q * 32 + lane, nc - 1)), v);
                lo = min(lo, s[q][c]);
                hi = max(hi, s[q][c]);
            }
            f0[c] = __reduce_min_sync(0xffffffffu, lo);
            nb[c] = __reduce_max_sync(0xffffffffu, hi) + kW - f0[c];
        }
        const int pitch = (nb[0] + 3) & ~3;
        const int slab = pitch * nb[1];
        const bool staged = static_cast<int64_t>(slab) * nb[2] <= kSpreadFloats;
        if (!staged && nc > 32) {  // a group across a jump of the order: its quarters
            part = (nc + 127) / 128 * 32;
            continue;
        }
        __syncwarp();
        const int sx = nb[0] - kW + 1, sy = nb[1] - kW + 1, sz = DIM > 2 ? nb[2] - kW + 1 : 1;
        const bool sorted = staged && static_cast<int64_t>(sx) * sy * sz <= kSpreadBins;
        if (staged)
            for (int k = lane; k < slab * nb[2]; k += 32) sm.box[k] = 0.0f;
        // ---- order of the cells
        if (sorted) {
            for (int k = lane; k < kSpreadBins; k += 32) sm.bins[k] = 0;
            __syncwarp();
            int rank[kPer], key[kPer];
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                const bool in = q * 32 + lane < nc;
                key[q] = ((DIM > 2 ? s[q][DIM - 1] - f0[2] : 0) * sy + s[q][1] - f0[1]) * sx + s[q][0] - f0[0];
                const unsigned same = __match_any_sync(0xffffffffu, in ? key[q] : -1);
                rank[q] = in ? sm.bins[key[q]] + __popc(same & ((1u << lane) - 1u)) : 0;
                __syncwarp();
                if (in && (same >> lane) == 1u) sm.bins[key[q]] = rank[q] + 1;  // the last lane of the bin
                __syncwarp();
            }
            int run = 0;
            for (int k = 0; k < kSpreadBins; k += 32) {
                const int own = sm.bins[k + lane];
                int v = own;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int o = __shfl_up_sync(0xffffffffu, v, off);
                    if (lane >= off) v += o;
                }
                sm.bins[k + lane] = run + v - own;
                run += __shfl_sync(0xffffffffu, v, 31);
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < kPer; ++q)
                if (q * 32 + lane < nc) sm.order[sm.bins[key[q]] + rank[q]] = static_cast<short>(q * 32 + lane);
        } else {
            for (int i = lane; i < nc; i += 32) sm.order[i] = static_cast<short>(i);
        }
        const int lx = lane & 7, ly = lane >> 3;
        constexpr int kz = DIM > 2 ? kW : 1;
        float acc[kz][2];
#pragma unroll
        for (int z = 0; z < kz; ++z) acc[z][0] = acc[z][1] = 0.0f;
        int cur = -1;
        auto flush = [&]() {
            float* p = sm.box + cur + ly * pitch + lx;
            float old[kz][2];
#pragma unroll
            for (int z = 0; z < kz; ++z) {
                old[z][0] = p[z * slab];
                old[z][1] = p[z * slab + 4 * pitch];
            }
#pragma unroll
            for (int z = 0; z < kz; ++z) {
                p[z * slab] = old[z][0] + acc[z][0];
                p[z * slab + 4 * pitch] = old[z][1] + acc[z][1];
                acc[z][0] = acc[z][1] = 0.0f;
            }
            __syncwarp();
        };
        for (int i0 = 0; i0 < nc; i0 += 32) {
            const int m = min(32, nc - i0);
            __syncwarp();
            if (lane < m) {
                const int i = sm.order[i0 + lane];
                const int64_t o = static_cast<int64_t>(__ldg(perm + c0 + i)) - perm_base;
                const float gv = index_ok(o, n) ? g[o] * scale.first * scale.second : 0.0f;
                float w[kW], v;
                const int px = band::locate(ax[0], __ldg(src[0] + i), v);
                band::weights(v, w);
                float4* out = reinterpret_cast<float4*>(sm.wts[lane]);
                out[0] = make_float4(w[0] * gv, w[1] * gv, w[2] * gv, w[3] * gv);
                out[1] = make_float4(w[4] * gv, w[5] * gv, w[6] * gv, w[7] * gv);
                const int py = band::locate(ax[1], __ldg(src[1] + i), v);
                band::weights(v, w);
                out[2] = make_float4(w[0], w[1], w[2], w[3]);
                out[3] = make_float4(w[4], w[5], w[6], w[7]);
                int pz = 0;
                if (DIM > 2) {
                    pz = band::locate(ax[DIM - 1], __ldg(src[2] + i), v);
                    band::weights(v, w);
                    out[4] = make_float4(w[0], w[1], w[2], w[3]);
                    out[5] = make_float4(w[4], w[5], w[6], w[7]);
                }
                sm.at[lane] = staged ? (pz - f0[2]) * slab + (py - f0[1]) * pitch + (px - f0[0])
                                     : static_cast<int>(pz * plane + static_cast<int64_t>(py) * mx + px);
            }
            __syncwarp();
            // the next cell's weights are loaded before the current one is added
            float wx, wa, wb, wn[kz];
            int next;
            auto load = [&](int q) {
                const float* w = sm.wts[q];
                wx = w[lx];
                wa = w[kW + ly];
                wb = w[kW + 4 + ly];
                if (DIM > 2) {
                    const float4 a = *reinterpret_cast<const float4*>(w + 2 * kW);
                    const float4 c = *reinterpret_cast<const float4*>(w + 2 * kW + 4);
                    wn[0] = a.x; wn[1 % kz] = a.y; wn[2 % kz] = a.z; wn[3 % kz] = a.w;
                    wn[4 % kz] = c.x; wn[5 % kz] = c.y; wn[6 % kz] = c.z; wn[7 % kz] = c.w;
                } else {
                    wn[0] = 1.0f;
                }
                next = sm.at[q];
            };
            load(0);
#pragma unroll 2
            for (int q = 0; q < m; ++q) {
                const float w0 = wx * wa, w1 = wx * wb;
                float wz[kz];
#pragma unroll
                for (int z = 0; z < kz; ++z) wz[z] = wn[z];
                const int to = next;
                load(min(q + 1, m - 1));
                if (staged) {
                    if (to != cur) {  // uniform over the warp
                        if (cur >= 0) flush();
                        cur = to;
                    }
#pragma unroll
                    for (int z = 0; z < kz; ++z) {
                        acc[z][0] = fmaf(wz[z], w0, acc[z][0]);
                        acc[z][1] = fmaf(wz[z], w1, acc[z][1]);
                    }
                } else {
                    unsigned long long* p = lattice + to + ly * mx + lx;
#pragma unroll
                    for (int z = 0; z < kz; ++z) {
                        atomicAdd(p + z * plane, static_cast<unsigned long long>(__float2ll_rn(wz[z] * w0)));
                        atomicAdd(p + z * plane + 4 * mx, static_cast<unsigned long long>(__float2ll_rn(wz[z] * w1)));
                    }
                }
            }
        }
        at += nc;
        if (!staged) continue;
        if (cur >= 0) flush();
        const int rows = nb[1] * nb[2];
        // four rows of up to eight nodes, or one of up to 32, at a time
        const int per = nb[0] <= 8 ? 4 : nb[0] <= 16 ? 2 : 1, wide = 32 / per;
        for (int r = lane / wide; r < rows; r += per) {
            const int z = r / nb[1], y = r - z * nb[1];
            unsigned long long* p = lattice + (f0[2] + z) * plane + static_cast<int64_t>(f0[1] + y) * mx + f0[0];
            for (int x = lane % wide; x < nb[0]; x += wide) {
                const long long v = __float2ll_rn(sm.box[z * slab + y * pitch + x]);
                if (v != 0) atomicAdd(p + x, static_cast<unsigned long long>(v));
            }
        }
    }
}

// Clears the fixed-point lattice the selection has chosen.
__global__ void __launch_bounds__(256) band_clear_kernel(const BandDesc* b, unsigned long long* lattice) {
    pdl_wait();
    if (b->n_light == 0) return;
    const int64_t n = static_cast<int64_t>(b->ax[0].m) * b->ax[1].m * b->ax[2].m;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * 256)
        lattice[i] = 0ull;
}

__global__ void __launch_bounds__(256) band_unfix_kernel(const BandDesc* b, const unsigned long long* lattice,
                                                         const float* gmax, int n_gmax, int64_t n_cells, float* out) {
    pdl_wait();
    if (b->n_light == 0) return;
    const FixedScale scale = fixed_scale(gmax, n_gmax, n_cells);
    // a g that is not finite: so are all sums
    const double inv = gmax_finite(gmax, n_gmax)
                           ? 1.0 / (static_cast<double>(scale.first) * static_cast<double>(scale.second))
                           : __longlong_as_double(0x7ff8000000000000ll);
    const int64_t n = static_cast<int64_t>(b->ax[0].m) * b->ax[1].m * b->ax[2].m;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * 256)
        out[i] = static_cast<float>(static_cast<double>(static_cast<long long>(lattice[i])) * inv);
}

// ---------------------------------------------------------------------------
// Sums over the nodes
// ---------------------------------------------------------------------------

// Tables of one call: per axis the phasors ph[node][mode] of the light modes
// (z: with psi) and the coordinates off[node] relative to the axis's first
// node; and rank[slot], the light mode of a table slot or ~ the direct one.
__global__ void __launch_bounds__(256) band_phasor_kernel(const BandDesc* b, const float4* __restrict__ cold,
                                                          const int32_t* idx_l, const int32_t* idx_h, GridGeom gg, int dim,
                                                          BandPhasors t) {
    pdl_wait();
    const int nl = b->n_light, nh = b->nh;
    const int step = gridDim.x * blockDim.x, u0 = blockIdx.x * blockDim.x + threadIdx.x;
    for (int u = u0; u < nl + nh; u += step) {
        if (u < nl)
            t.rank[idx_l[u]] = u;
        else
            t.rank[idx_h[u - nl]] = ~(u - nl);
    }
    if (nl == 0) return;
    const unsigned np = static_cast<unsigned>((nl + 127) / 128 * 128);
    const unsigned m[3] = {static_cast<unsigned>(b->ax[0].m), static_cast<unsigned>(b->ax[1].m),
                           static_cast<unsigned>(b->ax[2].m)};
    const float* cells[3] = {gg.X, gg.Y, gg.Z};
    // gain and slopes (FP64: the gains multiply the gradients)
    for (unsigned j = u0; j < static_cast<unsigned>(nl); j += step) {
        const int s = idx_l[j];
        const float4 c0 = __ldg(cold + 2 * s), c1 = __ldg(cold + 2 * s + 1);
        const double a[3] = {static_cast<double>(c0.x) + static_cast<double>(c0.y),
                             static_cast<double>(c0.z) + static_cast<double>(c0.w),
                             static_cast<double>(c1.x) + static_cast<double>(c1.y)};
        double lg = 0.0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const BandAxis ax = b->ax[c];
            double slope = 0.0;
            if (c < dim && !ax.ident) {
                const double xi = a[c] * static_cast<double>(ax.h);
                lg += band::log_gain(xi);
                slope = band::log_gain_slope(xi) * static_cast<double>(ax.h) * 0.15915494309189535;
            }
            t.gain[(1 + c) * static_cast<int64_t>(np) + j] = slope;
        }
        t.gain[j] = exp(lg);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const BandAxis ax = b->ax[c];
        const bool has = c < dim;
        const AxisSrc src = ax.ident ? AxisSrc{cells[c], 0.0f, 0} : AxisSrc{nullptr, ax.h, ax.n0};
        for (unsigned u = u0; u < m[c]; u += step)
            t.off[c][u] = has ? band::axis_at(src, u) - band::axis_at(src, 0) : 0.0f;
        for (unsigned u = u0; u < m[c] * np; u += step) {
            const unsigned node = u / np, j = u - node * np;
            float cs = 0.0f, sn = 0.0f;
            const int s = idx_l[j];
            if (s >= 0) {
                const float4 c0 = __ldg(cold + 2 * s), c1 = __ldg(cold + 2 * s + 1);
                float turns = 0.0f;
                if (c == 0) turns = turns_axis(c0.x, c0.y, band::axis_at(src, node));
                if (c == 1) turns = turns_axis(c0.z, c0.w, band::axis_at(src, node));
                if (c == 2) {
                    if (has) turns = turns_axis(c1.x, c1.y, band::axis_at(src, node));
                    turns = frac_turn(frac_turn(turns + c1.z) + c1.w);
                }
                sincospif(2.0f * turns, &sn, &cs);
            }
            t.ph[c][u] = make_float2(cs, sn);
        }
    }
}

// part[split][light mode][5] = (sum G cos, sum G sin, sum G X_c sin) over the
// split's share of the lattice (FP64).  A thread owns a mode; its x phasors of
// 64 nodes stay in shared memory while the block walks lines of nodes along x,
// 16 at a time, their G broadcast: per node and line four FFMA (the product
// with the phasor and with its x-weighted copy), then per line the product
// with the y and z phasors.  FP32 within a line, two-float sums over the
// lines.  Bound by FFMA issue (66 per 6 shared-memory wavefronts); G is read
// once per mode tile from L2.
constexpr int kNLines = 16, kNX = 64, kNModes = 128;
constexpr int kNSmem = kNX * kNModes * 8 + kNX * kNLines * 4 + kNX * 4;
__global__ void __launch_bounds__(kNModes, 3) band_nodes_kernel(const BandDesc* b, const float* G,
                                                                BandPhasors t, int dim, GridGeom gg, int blocks,
                                                                double* part) {
    extern __shared__ __align__(16) unsigned char nsm[];
    float2* xp = reinterpret_cast<float2*>(nsm);                        // [kNX][kNModes]
    float* gs = reinterpret_cast<float*>(nsm + kNX * kNModes * 8);      // [kNX][kNLines]
    float* xw = gs + kNX * kNLines;                                     // [kNX]
    pdl_wait();
    const int nl = b->n_light;
    if (nl == 0) return;
    const int np = (nl + kNModes - 1) / kNModes * kNModes;
    const int mx = b->ax[0].m, my = b->ax[1].m;
    const int lines = my * b->ax[2].m;
    const BandNodes S = band_nodes_split(nl, mx, lines, blocks);
    const int tid = threadIdx.x;
    for (int u = blockIdx.x; u < S.n_mt * S.n_xc * S.groups; u += gridDim.x) {
        const int mt = u % S.n_mt, rest = u / S.n_mt;
        const int xc = rest % S.n_xc, grp = rest / S.n_xc;
        const int m = mt * kNModes + tid;
        const int i0 = xc * kNX, ni = min(kNX, mx - i0);
        __syncthreads();
#pragma unroll 8
        for (int i = 0; i < ni; ++i) xp[i * kNModes + tid] = t.ph[0][static_cast<int64_t>(i0 + i) * np + m];
        if (tid < kNX) xw[tid] = tid < ni ? t.off[0][i0 + tid] : 0.0f;
        float hi[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, lo[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        const int nb = (lines + kNLines - 1) / kNLines;
        const int b0 = static_cast<int>(static_cast<int64_t>(nb) * grp / S.groups);
        const int b1 = static_cast<int>(static_cast<int64_t>(nb) * (grp + 1) / S.groups);
        for (int bt = b0; bt < b1; ++bt) {
            const int l0 = bt * kNLines, nr = min(kNLines, lines - l0);
            __syncthreads();
#pragma unroll
            for (int e = tid; e < kNX * kNLines; e += kNModes) {
                const int r = e / kNX, i = e - r * kNX;
                if (i < ni) gs[i * kNLines + r] = r < nr ? G[static_cast<int64_t>(l0 + r) * mx + i0 + i] : 0.0f;
            }
            __syncthreads();
            float dr[kNLines], di[kNLines], er[kNLines], ei[kNLines];
#pragma unroll
            for (int r = 0; r < kNLines; ++r) dr[r] = di[r] = er[r] = ei[r] = 0.0f;
            for (int i = 0; i < ni; ++i) {
                const float2 p = xp[i * kNModes + tid];
                const float w = xw[i], wr = w * p.x, wi = w * p.y;
#pragma unroll
                for (int q = 0; q < kNLines / 4; ++q) {
                    const float4 v = *reinterpret_cast<const float4*>(gs + i * kNLines + 4 * q);
                    const float gv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        dr[4 * q + e] = fmaf(p.x, gv[e], dr[4 * q + e]);
                        di[4 * q + e] = fmaf(p.y, gv[e], di[4 * q + e]);
                        er[4 * q + e] = fmaf(wr, gv[e], er[4 * q + e]);
                        ei[4 * q + e] = fmaf(wi, gv[e], ei[4 * q + e]);
                    }
                }
            }
            float s[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
            int l = l0 / my, k = l0 - l * my;
#pragma unroll
            for (int r = 0; r < kNLines; ++r) {
                if (r < nr) {
                    const float2 y = t.ph[1][static_cast<int64_t>(k) * np + m];
                    const float2 z = t.ph[2][static_cast<int64_t>(l) * np + m];
                    const float pr = fmaf(y.x, z.x, -y.y * z.y), pi = fmaf(y.x, z.y, y.y * z.x);
                    const float im = fmaf(dr[r], pi, di[r] * pr);
                    s[0] += fmaf(dr[r], pr, -di[r] * pi);
                    s[1] += im;
                    s[2] += fmaf(er[r], pi, ei[r] * pr);
                    s[3] = fmaf(t.off[1][k], im, s[3]);
                    s[4] = fmaf(t.off[2][l], im, s[4]);
                    if (++k == my) {
                        k = 0;
                        ++l;
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 5; ++q) two_sum_acc(hi[q], lo[q], s[q]);
        }
        double* o = part + (static_cast<int64_t>(xc * S.groups + grp) * np + m) * 5;
        const double ssin = static_cast<double>(hi[1]) + static_cast<double>(lo[1]);
        o[0] = static_cast<double>(hi[0]) + static_cast<double>(lo[0]);
        o[1] = ssin;
        const float* cells[3] = {gg.X, gg.Y, gg.Z};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            // the offsets are from the axis's first node
            const BandAxis ax = b->ax[c];
            const double x0 = c >= dim  ? 0.0
                              : ax.ident ? static_cast<double>(__ldg(cells[c]))
                                         : static_cast<double>(ax.n0) * static_cast<double>(ax.h);
            o[2 + c] = static_cast<double>(hi[2 + c]) + static_cast<double>(lo[2 + c]) + x0 * ssin;
        }
    }
}

// The modes left for the direct sum, at the cells of any plan: part[split][direct
// mode][5] over the split's groups of cells.  A warp holds 256 cells in
// registers (8 per lane) and walks the modes; a lane sums its cells and the
// warp adds the lanes (a fixed butterfly).  These are the table's fastest
// modes, so the phase is reduced exactly at every cell unless the group is
// compact enough for the mode; compared with the mode-stationary kernel no
// slot is spent on padding and a handful of modes fills the GPU (89 modes at
// 2M cells: 4.4 ms there).  Bound by instruction issue.
constexpr int kDirCells = 256, kDirModes = 128, kDirWarps = 4;
template <int DIM>
__global__ void __launch_bounds__(32 * kDirWarps, 4) band_direct_kernel(
    const BandDesc* b, const float4* __restrict__ cold, const int32_t* idx, const float* __restrict__ xs,
    const float* __restrict__ ys, const float* __restrict__ zs, const int32_t* __restrict__ perm, int64_t perm_base,
    int64_t n, const float* g, double* part) {
    __shared__ float4 mode[kDirModes][2];
    __shared__ float2 acc[kDirWarps][kDirModes][5];
    pdl_wait();
    const int nh = b->nh;
    if (nh == 0) return;
    const int tiles = (nh + kDirModes - 1) / kDirModes, splits = band_direct_splits(nh, gridDim.x);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t groups = (n + kDirCells - 1) / kDirCells;
    for (int u = blockIdx.x; u < tiles * splits; u += gridDim.x) {
        const int mt = u % tiles, sp = u / tiles;
        const int nm = min(kDirModes, nh - mt * kDirModes);
        __syncthreads();
        for (int k = threadIdx.x; k < nm; k += blockDim.x) {
            const int s = idx[mt * kDirModes + k];
            mode[k][0] = __ldg(cold + 2 * s);
            mode[k][1] = __ldg(cold + 2 * s + 1);
        }
        for (int k = lane; k < kDirModes * 5; k += 32) (&acc[warp][0][0])[k] = make_float2(0.0f, 0.0f);
        __syncthreads();
        for (int64_t gr = static_cast<int64_t>(sp) * kDirWarps + warp; gr < groups;
             gr += static_cast<int64_t>(splits) * kDirWarps) {
            constexpr int kPer = kDirCells / 32;
            const int64_t c0 = gr * kDirCells;
            float x[kPer][DIM], gv[kPer], x0[DIM];
            const float* src[3] = {xs, ys, zs};
            float E = 0.0f;
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                const int64_t i = c0 + q * 32 + lane;
                const int64_t o = i < n ? static_cast<int64_t>(__ldg(perm + i)) - perm_base : 0;
                gv[q] = i < n && index_ok(o, n) ? g[o] : 0.0f;
#pragma unroll
                for (int c = 0; c < DIM; ++c) x[q][c] = __ldg(src[c] + (i < n ? i : c0));
            }
#pragma unroll
            for (int c = 0; c < DIM; ++c) {
                float lo = x[0][c], hi = x[0][c];
#pragma unroll
                for (int q = 1; q < kPer; ++q) {
                    lo = fminf(lo, x[q][c]);
                    hi = fmaxf(hi, x[q][c]);
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
                    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, off));
                    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, off));
                }
                x0[c] = 0.5f * lo + 0.5f * hi;
                E = fmaxf(E, fmaxf(hi - x0[c], x0[c] - lo));
            }
            for (int k = 0; k < nm; ++k) {
                const float4 m0 = mode[k][0], m1 = mode[k][1];
                float s[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
                const float span = (fabsf(m0.x) + fabsf(m0.z) + fabsf(m1.x)) * E;
                // a group that the phase spans by at most 8 turns: the exact phase at
                // its origin and FP32 offsets (uniform over the warp)
                const bool near = span <= kTauLight;
                const float t0 = near ? phase_exact_turns<DIM>(x0, m0, m1) : 0.0f;
#pragma unroll
                for (int q = 0; q < kPer; ++q) {
                    float turns;
                    if (near) {
                        turns = fmaf(m0.x, x[q][0] - x0[0], t0);
                        if (DIM > 1) turns = fmaf(m0.z, x[q][1 % DIM] - x0[1 % DIM], turns);
                        if (DIM > 2) turns = fmaf(m1.x, x[q][2 % DIM] - x0[2 % DIM], turns);
                        turns = frac_turn(turns);
                    } else {
                        turns = phase_exact_turns<DIM>(x[q], m0, m1);
                    }
                    const float th = kTwoPiF * turns;
                    const float gs = gv[q] * hw_sin(th);
                    s[0] = fmaf(gv[q], hw_cos(th), s[0]);
                    s[1] += gs;
                    // coordinates relative to the group's origin: small weights
#pragma unroll
                    for (int c = 0; c < DIM; ++c) s[2 + c] = fmaf(gs, x[q][c] - x0[c], s[2 + c]);
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1)
#pragma unroll
                    for (int q = 0; q < 2 + DIM; ++q) s[q] += __shfl_xor_sync(0xffffffffu, s[q], off);
                if (lane < 2 + DIM) {
                    float v = s[0];
#pragma unroll
                    for (int q = 1; q < 2 + DIM; ++q) v = lane == q ? s[q] : v;
                    float2 a = acc[warp][k][lane];
                    two_sum_acc(a.x, a.y, v);
                    if (lane >= 2) {
                        // the origin's part, its product exact
                        float xc = x0[0];
#pragma unroll
                        for (int c = 1; c < DIM; ++c) xc = lane == 2 + c ? x0[c] : xc;
                        const float p = xc * s[1];
                        two_sum_acc(a.x, a.y, p);
                        a.y += fmaf(xc, s[1], -p);
                    }
                    acc[warp][k][lane] = a;
                }
            }
        }
        __syncthreads();
        for (int k = threadIdx.x; k < nm * 5; k += blockDim.x) {
            double v = 0.0;
            for (int w = 0; w < kDirWarps; ++w) {
                const float2 a = (&acc[w][0][0])[k];
                v += static_cast<double>(a.x) + static_cast<double>(a.y);
            }
            part[(static_cast<int64_t>(sp) * tiles * kDirModes + mt * kDirModes) * 5 + k] = v;
        }
    }
}

}  // namespace

int launch_band_direct(const BandDesc* b, int32_t dim, const float4* cold, const int32_t* idx, const float* xs,
                       const float* ys, const float* zs, const int32_t* perm, int64_t perm_base, int64_t n,
                       const float* g, double* part, int blocks, void* stream) {
    return launch_chained(dim > 2 ? band_direct_kernel<3> : band_direct_kernel<2>, blocks, 32 * kDirWarps, 0,
                          static_cast<cudaStream_t>(stream), b, cold, idx, xs, ys, zs, perm, perm_base, n, g, part);
}

int launch_band_grid_spread(const BandDesc* b, const GridGeom& gg, const float* g, const BandAxisTab* tab, float* h1,
                            float* h2, float* nodes, int sms, void* stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t rows = int64_t(gg.ny) * gg.nz;
    cudaError_t e = launch_chained(band_axis_kernel, gg.nz > 1 ? 3 : 2, 1024, 0, st, b, gg, tab[0], tab[1], tab[2]);
    if (e == cudaSuccess)
        // long rows: a unit per 32 nodes, of which there are at most as many as cells
        e = launch_chained(band_tx_kernel,
                           static_cast<unsigned>(std::min<int64_t>(
                               (rows + kTxRows - 1) / kTxRows * (gg.nx > kTxCells ? (gg.nx + 31) / 32 : 1),
                               gg.nx > kTxCells ? sms * 7 : sms * 64)),
                           256, 0, st, b, g, gg.nx, rows, tab[0], h1);
    if (e == cudaSuccess)
        e = launch_chained(band_tline_kernel<true>, sms * 16, 256, 0, st, b, h1, gg.ny, gg.nz, tab[1],
                           gg.nz > 1 ? h2 : nodes);
    if (e == cudaSuccess && gg.nz > 1)
        e = launch_chained(band_tline_kernel<false>, sms * 16, 256, 0, st, b, h2, gg.nz, gg.nz, tab[2], nodes);
    return e;
}

int launch_band_spread(const BandDesc* b, int32_t dim, const float* xs, const float* ys, const float* zs,
                       const int32_t* perm, int64_t perm_base, int64_t n, const float* g, const float* gmax,
                       int n_gmax, unsigned long long* lattice, float* nodes, int sms, void* stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // a warp's group is a chain of sort, sum and write-out: smaller groups where
    // the warps would not fill the GPU twice (262k cells x 1024 modes: 168 us a
    // call with 256 cells to a warp, 150 with 64)
    int cells = kSpreadCells;
    while (cells > 64 && n / cells < int64_t(sms) * 14 * 2) cells /= 2;
    const int64_t groups = (n + cells - 1) / cells;
    const unsigned grid = static_cast<unsigned>((groups + kSpreadWarps - 1) / kSpreadWarps);
    cudaError_t e = launch_chained(band_clear_kernel, sms * 4, 256, 0, st, b, lattice);
    if (e == cudaSuccess)
        e = launch_chained(dim > 2 ? band_spread_kernel<3> : band_spread_kernel<2>, grid, 32 * kSpreadWarps, 0, st, b,
                           xs, ys, zs, perm, perm_base, n, g, gmax, n_gmax, cells, lattice);
    if (e == cudaSuccess)
        e = launch_chained(band_unfix_kernel, sms * 4, 256, 0, st, b, lattice, gmax, n_gmax, n, nodes);
    return e;
}

int launch_band_nodes(const BandDesc* b, const float4* cold, const int32_t* idx_l, const int32_t* idx_h,
                      const GridGeom& gg, int32_t dim, const float* nodes, const BandPhasors& t, double* part, int sms,
                      void* stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e =
        cudaFuncSetAttribute(band_nodes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kNSmem);
    if (e == cudaSuccess)
        e = launch_chained(band_phasor_kernel, sms * 8, 256, 0, st, b, cold, idx_l, idx_h, gg, dim, t);
    if (e == cudaSuccess)
        e = launch_chained(band_nodes_kernel, sms * 3, kNModes, kNSmem, st, b, nodes, t, dim, gg, sms * 3, part);
    return e;
}

}  // namespace grf
