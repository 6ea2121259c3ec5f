// The band-limited path of large spectral sums (band.cuh): choice of the node
// lattice on the device, interpolation from the nodes to the cells.
//
// Kernels of one forward call on a Cartesian grid, in order:
//   band_select_kernel   (1 block) modes to sum directly, node spacings, tilings
//   band_prep_kernel     tables of both sums (synth_grid.cu)
//   grid_band_kernel     light modes at the nodes, tensor cores (synth_grid.cu)
//   band_sum_kernel      adds the mode splits' partial sums
//   band_line_kernel     z: nodes -> (x, y) nodes at the cell layers; where
//                        the direct sum's product takes the light modes, also
//                        y: -> rows of x nodes at the (y, z) cells
//   grid_band_kernel     direct modes at the cells; large 3-D grids add the
//                        light modes' chunks and write the maps
//   band_finalize_kernel y and x interpolation and maps where the previous
//                        kernel left partial sums or had no modes
// At the cells of any plan: the first four, then band_cells_kernel (the light
// modes' sum at the sorted cells) and synth_fwd_kernel (synth_fwd.cu) for the
// direct modes, which adds it.
// Kernels that find nothing to do return at once; all are launched chained.
#include <cuda_runtime.h>

#include <algorithm>

#include "band.cuh"
#include "device_common.cuh"
#include "grid_tiling.cuh"
#include "launch.cuh"

namespace grf {

namespace {

using band::kW;

constexpr int kSelThreads = 1024;
constexpr int kKeep = 8;  // modes a selecting thread keeps in registers
constexpr int kNodeSplits = 32;     // most mode splits of a node tile
constexpr int64_t kNodeItems = 152;  // (tile, mode split) items of the nodes' sum
// Modes are binned by the largest of their frequencies relative to the axes'
// typical ones, eight bins per octave from 2^-8 to 2^8.
constexpr int kBins = 128, kBinsPerOctave = 8, kBinBias = 64;

// Node axis for modes of at most `a` turns per unit length over [lo, hi].
// n > 0: a grid axis of n cells, left alone where the lattice would not be
// coarser.  h is rounded down to 8 significant bits, so that n h is exact for
// |n| < 2^16; returns false where the coordinates need more.
__device__ __forceinline__ bool node_axis(float a, float lo, float hi, int n, BandAxis& ax) {
    ax.ident = 0;
    // at least one node spacing per extent, whatever the frequencies
    const float cap = hi > lo ? hi - lo : fmaxf(1.0f, fabsf(lo));
    const float h = a * cap > band::kXi ? band::kXi / a : cap;
    ax.h = __int_as_float(__float_as_int(h) & 0x7fff0000);
    ax.inv_h = 1.0f / ax.h;
    const float f0 = floorf(lo * ax.inv_h), f1 = floorf(hi * ax.inv_h);
    const bool ok = ax.h > 1e-30f && isfinite(hi - lo) && fmaxf(fabsf(f0), fabsf(f1)) < static_cast<float>(band::kMaxNode - 2 * kW);
    const int m = ok ? static_cast<int>(f1) - static_cast<int>(f0) + kW : INT_MAX;
    if (n > 0 && m >= n) {
        ax = BandAxis{0.0f, 0.0f, 0, n, 1};
        return true;
    }
    ax.n0 = ok ? static_cast<int>(f0) - (kW / 2 - 1) : 0;
    ax.m = m;
    return ok;
}

// z blocks of a node lattice's tile rows (GridDesc): the number with the
// fewest 128 x 128 tiles, by one warp (lane = blocks - 1).
__device__ __forceinline__ int z_blocks(const BandAxis (&ax)[3], int cap_mt) {
    const int lane = threadIdx.x & 31, nb = lane + 1;
    unsigned best = ~0u;
    const int lz = (ax[2].m + nb - 1) / nb;
    const int rt = (ax[0].m * nb + gridt::kGM - 1) / gridt::kGM;
    if (nb == 1 || (!ax[2].ident && lz >= 2 && rt <= cap_mt)) {
        int ct = INT_MAX;
        for (int pk = 2; pk <= 6; ++pk) {
            const int PK = 1 << pk, PL = gridt::kGN >> pk;
            const int cols = ((ax[1].m + PK - 1) / PK) * ((lz + PL - 1) / PL);
            ct = min(ct, pk == 6 ? cols + cols / 4 : cols);  // as grid_plan
        }
        best = static_cast<unsigned>(min(static_cast<int64_t>(rt) * ct, static_cast<int64_t>(0x3ffffff))) << 5 | lane;
    }
    return static_cast<int>(__reduce_min_sync(0xffffffffu, best) & 31u) + 1;
}

// |a_x|, |a_y|, |a_z| and |A| of table slot j.
__device__ __forceinline__ float4 mode_of(const BandSelect& p, int j) {
    const float4 c0 = __ldg(p.cold + 2 * j), c1 = __ldg(p.cold + 2 * j + 1);
    return make_float4(fabsf(c0.x), fabsf(c0.z), fabsf(c1.x), fabsf(__ldg(&p.hot[j].w)));
}

// Whether the workspace holds a lattice of mx x my x mz nodes.
__device__ __forceinline__ bool lattice_fits(const BandSelect& p, int mx, int my, int mz) {
    if (max(mx, max(my, mz)) >= 1 << 20) return false;  // the products below fit
    const int64_t plane = static_cast<int64_t>(mx) * my;
    return mx <= p.cap_ax[0] && my <= p.cap_ax[1] && mz <= p.cap_ax[2] && plane * mz <= p.cap_nodes &&
           (p.n[2] <= 1 || plane * p.n[2] <= p.cap_mid);
}

// Estimated time of summing `light` modes at mx x my x mz nodes (whole
// tensor-core tiles of 128 x 128) and `heavy` directly; 3e38 where the
// lattice does not fit the workspace.
__device__ float candidate_time(const BandSelect& p, int heavy, int light, int mx, int my, int mz) {
    const float direct = p.us_mode * static_cast<float>((heavy + p.chunk - 1) / p.chunk * p.chunk) +
                         (heavy > 0 ? p.us_heavy : 0.0f);
    if (light == 0) return direct;
    if (max(mx, max(my, mz)) >= 1 << 20) return 3.0e38f;  // the products below fit
    // one node more per axis than estimated: the light modes' own largest
    // frequencies, at most the bin's edge, may place the nodes less favourably
    const int64_t plane = static_cast<int64_t>(mx + 1) * (my + 1);
    if (plane * (mz + 1) > p.cap_nodes || (p.n[2] > 1 && plane * p.n[2] > p.cap_mid)) return 3.0e38f;
    if (mx >= p.cap_ax[0] || my >= p.cap_ax[1] || mz >= p.cap_ax[2]) return 3.0e38f;
    const int64_t tile = gridt::kGM * gridt::kGN;
    const float nodes = static_cast<float>((static_cast<int64_t>(mx) * my * mz + tile - 1) / tile * tile);
    return direct + p.us_node * nodes * static_cast<float>(light) + p.us_fixed;
}

__device__ __forceinline__ float approx_sqrt(float v) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// band::gain(xi) or a little more (below 2^-16 of it), for the amplitude
// scale; 1 with xi = 0 (axes that are not interpolated have h = 0).
__device__ __forceinline__ float gain_bound(float xi) {
    const float q2 = band::kPiW * band::kPiW * xi * xi;
    const float r = __fdividef(q2, band::kBeta + approx_sqrt(fmaxf(band::kBeta * band::kBeta - q2, 0.0f)));
    return __expf(r) * (1.00001f - r * (1.0f / band::kBeta));
}

// Sum over the block of one value per thread and axis, in a fixed order.
__device__ __forceinline__ void block_sum3(float (&v)[3], float (*sh)[32], float (&out)[3]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v[c] += __shfl_xor_sync(0xffffffffu, v[c], off);
        if (lane == 0) sh[c][warp] = v[c];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float t = sh[c][lane];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        out[c] = t;
    }
}

// Which modes to sum at the nodes, and on which lattice.  The modes are
// ordered by r = max_c |a_c| / s_c, s_c the axis's typical frequency (the
// square of the mean of sqrt |a_c|: defined for the heavy-tailed spectra too),
// because the lattice is a box in frequency: the light modes are those of the
// bins up to one, the one of least estimated time.
// One block; latency-bound (a few barriers' worth of dependent steps on a few
// thousand modes), so the steps run on as many threads as they have items and
// the code is kept short: its instructions are fetched once.
__global__ void __launch_bounds__(kSelThreads, 1) band_select_kernel(const __grid_constant__ BandSelect p,
                                                                      BandDesc* out) {
    __shared__ int count[kBins];  // modes per bin, then of the bins up to it
    __shared__ int amax[3];       // largest |a_c| of the light modes (bits)
    __shared__ int m[3][kBins];
    __shared__ float red[3][32];
    __shared__ BandAxis axs[3];
    __shared__ float lo[3], hi[3];
    __shared__ int ranks[kKeep][32];  // light modes of each warp of a pass, then of those before it
    __shared__ int bad, gmax, width;
    __shared__ unsigned long long best;
    pdl_wait();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int n = p.n_modes, dim = p.dim;
    if (t < kBins) count[t] = 0;
    if (t < 3) {
        amax[t] = 0;
        lo[t] = p.seg->lo[t];
        hi[t] = p.seg->hi[t];
    }
    if (t == 0) {
        bad = *p.status & 1;
        gmax = 0;
        width = 0;
        best = ~0ull;
    }
    // the first kKeep modes of a thread stay in registers, with their bins
    float4 mine[kKeep];
    int bin[kKeep];
    float sums[3] = {0.0f, 0.0f, 0.0f}, total[3];
    auto add_roots = [&](const float4& a) {
        sums[0] += approx_sqrt(a.x);
        sums[1] += approx_sqrt(a.y);
        sums[2] += approx_sqrt(a.z);
    };
#pragma unroll
    for (int q = 0; q < kKeep; ++q) {
        const int j = q * kSelThreads + t;
        mine[q] = j < n ? mode_of(p, j) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
#pragma unroll
    for (int q = 0; q < kKeep; ++q) add_roots(mine[q]);
    for (int j = kKeep * kSelThreads + t; j < n; j += kSelThreads) add_roots(mode_of(p, j));
    block_sum3(sums, red, total);
    float s[3], inv_s[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float mean = total[c] / static_cast<float>(n);
        s[c] = mean * mean;
        inv_s[c] = s[c] > 0.0f ? 1.0f / s[c] : 0.0f;
    }
    auto bin_of = [&](const float4& a) {
        const float r = fmaxf(a.x * inv_s[0], fmaxf(a.y * inv_s[1], a.z * inv_s[2]));
        // r = 0 gives -inf, which converts to the least integer
        const int k = static_cast<int>(floorf(kBinsPerOctave * __log2f(r))) + kBinBias;
        return max(0, min(k, kBins - 1));
    };
    // ---- modes per bin, then of the bins up to it
#pragma unroll
    for (int q = 0; q < kKeep; ++q) {
        bin[q] = kBins;
        if (q * kSelThreads + t < n) {
            bin[q] = bin_of(mine[q]);
            atomicAdd(&count[bin[q]], 1);
        }
    }
    for (int j = kKeep * kSelThreads + t; j < n; j += kSelThreads) atomicAdd(&count[bin_of(mode_of(p, j))], 1);
    // ---- nodes per axis of every candidate, the modes of the bins up to k,
    // from the bins' upper edges (the last bin has none: nothing lies beyond)
    if (t < 3 * kBins) {
        const int c = t / kBins, k = t % kBins;
        BandAxis ax;
        int nodes = 1;
        if (c < dim)
            nodes = !bad && node_axis(s[c] * exp2f(static_cast<float>(k + 1 - kBinBias) / kBinsPerOctave), lo[c], hi[c],
                                      p.n[c], ax)
                        ? ax.m
                        : INT_MAX;
        m[c][k] = nodes;
    }
    __syncthreads();
    if (warp == 0) {
        int carry = 0;
        for (int b = 0; b < kBins / 32; ++b) {
            int v = count[32 * b + lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, v, off);
                if (lane >= off) v += o;
            }
            v += carry;
            count[32 * b + lane] = v;
            carry = __shfl_sync(0xffffffffu, v, 31);
        }
    }
    __syncthreads();
    // ---- the cheapest (candidate kBins: all modes directly)
    if (t < kBins + 32) {
        const int k = min(t, kBins);
        // the last bin holds the modes beyond every edge too
        const float cost = k == kBins - 1 ? 3.0e38f
                           : k < kBins ? candidate_time(p, n - count[k], count[k], m[0][k], m[1][k], m[2][k])
                                     : candidate_time(p, n, 0, 0, 0, 0);
        unsigned long long c = static_cast<unsigned long long>(__float_as_uint(cost)) << 32 | static_cast<unsigned>(k);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) c = min(c, __shfl_xor_sync(0xffffffffu, c, off));
        if (lane == 0) atomicMin(&best, c);
    }
    __syncthreads();
    const int pick = static_cast<int>(best & 0xffffffffu);
    int n_light = pick < kBins ? count[pick] : 0;
    // the light modes' own largest frequencies, at most the bin's edges
    if (n_light > 0) {
        float a[3] = {0.0f, 0.0f, 0.0f};
        auto widen = [&](const float4& f, bool light) {
            a[0] = fmaxf(a[0], light ? f.x : 0.0f);
            a[1] = fmaxf(a[1], light ? f.y : 0.0f);
            a[2] = fmaxf(a[2], light ? f.z : 0.0f);
        };
#pragma unroll
        for (int q = 0; q < kKeep; ++q) widen(mine[q], bin[q] <= pick);
        for (int j = kKeep * kSelThreads + t; j < n; j += kSelThreads) {
            const float4 f = mode_of(p, j);
            widen(f, bin_of(f) <= pick);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {  // non-negative floats order as their bits
            const unsigned v = __reduce_max_sync(0xffffffffu, __float_as_uint(a[c]));
            if (lane == 0) atomicMax(&amax[c], static_cast<int>(v));
        }
    }
    __syncthreads();
    if (t < 3) {
        BandAxis ax{0.0f, 0.0f, 0, 1, 1};
        if (n_light > 0 && t < dim) node_axis(__int_as_float(amax[t]), lo[t], hi[t], p.n[t], ax);
        axs[t] = ax;
    }
    __syncthreads();
    // The candidates' sizes come from the bins' edges, which a mode at an edge
    // may pass by a rounding, and from typical frequencies that underflow where
    // all are tiny: what is taken is what fits with the modes' own frequencies.
    if (n_light > 0 && !lattice_fits(p, axs[0].m, axs[1].m, axs[2].m)) n_light = 0;
    // ---- light chunks: first x node of every tile, a multiple of 4 (16-byte
    // loads of the rows), and the most nodes of a tile
    if (p.lstart != nullptr && n_light > 0 && n_light < n) {
        const BandAxis ax = axs[0];
        for (int mt = warp; mt < p.n_mt; mt += kSelThreads / 32) {
            int s0 = INT_MAX, s1 = 0;
            for (int i = mt * gridt::kGM + lane; i < min((mt + 1) * gridt::kGM, p.n[0]); i += 32) {
                float v;
                const int s = ax.ident ? max(0, min(i, ax.m - kW)) : band::locate(ax, __ldg(p.X + i), v);
                s0 = min(s0, s);
                s1 = max(s1, s);
            }
            s0 = __reduce_min_sync(0xffffffffu, s0) & ~3;
            s1 = __reduce_max_sync(0xffffffffu, s1);
            if (lane == 0) {
                p.lstart[mt] = s0;
                atomicMax(&width, s1 + kW - s0);
            }
        }
        __syncthreads();
        if (width > p.cap_nl * gridt::kGK) n_light = 0;  // an axis in no order may need more than there is room for
    }
    const int nh = n - n_light;
    const BandAxis none{0.0f, 0.0f, 0, 0, 1};
    const BandAxis ax[3] = {n_light > 0 ? axs[0] : none, n_light > 0 ? axs[1] : none, n_light > 0 ? axs[2] : none};
    if (t < 3) out->ax[t] = n_light > 0 ? axs[t] : none;
    // ---- slots of the light and the other modes, in table order, and a bound
    // of the light ones' amplitudes with their gains
    float top = 0.0f;
    int before = 0;  // light modes of the passes before
    for (int j0 = 0; j0 < n; j0 += kKeep * kSelThreads) {
        unsigned light = 0;
#pragma unroll
        for (int q = 0; q < kKeep; ++q) {
            const int j = j0 + q * kSelThreads + t;
            float4 a = mine[q];
            bool is = n_light > 0 && bin[q] <= pick;
            if (j0 > 0) {
                a = j < n ? mode_of(p, j) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                is = n_light > 0 && j < n && bin_of(a) <= pick;
            }
            if (is) top = fmaxf(top, a.w * (gain_bound(a.x * ax[0].h) * gain_bound(a.y * ax[1].h)) * gain_bound(a.z * ax[2].h));
            const unsigned vote = __ballot_sync(0xffffffffu, is);
            light |= is ? 1u << q : 0u;
            if (lane == 0) ranks[q][warp] = __popc(vote);
        }
        __syncthreads();
        if (warp == 0) {
            int carry = before;
#pragma unroll
            for (int q = 0; q < kKeep; ++q) {
                const int own = ranks[q][lane];
                int v = own;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int o = __shfl_up_sync(0xffffffffu, v, off);
                    if (lane >= off) v += o;
                }
                ranks[q][lane] = carry + v - own;
                carry += __shfl_sync(0xffffffffu, v, 31);
            }
            if (lane == 0) count[0] = carry;  // the bins' counts are no longer needed
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kKeep; ++q) {
            const int j = j0 + q * kSelThreads + t;
            const bool is = light >> q & 1u;
            const unsigned vote = __ballot_sync(0xffffffffu, is);
            const int rank = ranks[q][warp] + __popc(vote & ((1u << lane) - 1u));
            if (j < n) (is ? p.idx_l[rank] : p.idx_h[j - rank]) = j;
        }
        before = count[0];
        __syncthreads();
    }
    if (t < 128) {  // whole chunks (of 32 modes; the cells' kernels without a grid take 128)
        if (n_light + t < (n_light + 127) / 128 * 128) p.idx_l[n_light + t] = -1;
        if (nh + t < (nh + 127) / 128 * 128) p.idx_h[nh + t] = -1;
    }
    {
        const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(top));
        if (lane == 0) atomicMax(&gmax, static_cast<int>(w));
    }
    __syncthreads();
    if (warp == 0) {
        // the light modes' sum at the nodes
        const int nb = n_light > 0 && ax[2].m > 1 ? z_blocks(ax, p.cap_mt) : 1;
        if (lane == 0) {
            GridTiling o{};
            int e = 0;
            const float a = __int_as_float(gmax);
            if (a > 0.0f) frexpf(a, &e);
            if (n_light > 0) {
                const int lz = (ax[2].m + nb - 1) / nb;
                gridt::GridPlan gp = gridt::grid_plan(ax[0].m * nb, ax[1].m, lz, (n_light + gridt::kGModes - 1) / gridt::kGModes);
                // few tiles: enough mode splits to fill the GPU; two chunks per fold
                // (the accumulator's truncation grows with the interval)
                gp.max_split = gp.n_tiles >= kNodeItems ? 1 : gridt::min2(kNodeSplits, static_cast<int>(kNodeItems) / static_cast<int>(gp.n_tiles));
                gridt::set_tiling(o, gp, ax[0].m * nb, ax[1].m, lz, min(p.fold, 2));
                o.xn = ax[0].m;
                o.zn = ax[2].m;
                const int64_t nodes = static_cast<int64_t>(ax[0].m) * ax[1].m * ax[2].m;
                if (o.n_split * nodes > p.cap_part) {  // one copy always fits (cap_nodes <= cap_part)
                    o.n_split = static_cast<int>(p.cap_part / nodes);
                    o.n_items = o.n_tiles * o.n_split;
                }
            }
            o.scale = ldexpf(1.0f, e);
            out->nodes = o;
        }
    } else if (warp == 1 && lane == 0) {
        // direct modes at the cells of a grid: the host's tiling with fewer chunks
        GridTiling q = p.cells;
        q.nc = (nh + p.chunk - 1) / p.chunk;
        q.fc = max(1, min(p.fold, q.nc));
        q.n_split = max(1, gridt::min2(p.max_split, (q.nc + q.fc - 1) / q.fc));
        q.n_items = nh > 0 ? q.n_tiles * q.n_split : 0;
        q.nl = p.lstart != nullptr && n_light > 0 && nh > 0 ? (width + gridt::kGK - 1) / gridt::kGK : 0;
        q.lp = (ax[0].m + 3) & ~3;
        // rows / S is at most (light modes) x gain^3, which may pass FP16's
        // range: the excess goes to the weights
        int e = 0, k = 0;
        const float a = p.thdr->amp_max;
        if (a > 0.0f) frexpf(a, &e);
        frexpf(static_cast<float>(n_light) * 22.0f, &k);
        k = max(0, k - 15);
        q.l_inv = ldexpf(1.0f, -e - k);
        const int fin = p.n[0] > 0 ? nh == 0 || p.split_cells : q.n_split > 1;
        out->nh = nh;
        out->n_light = n_light;
        out->n_splits = p.n[0] > 0 && !(nh > 0 && fin) ? 0 : q.n_split;
        out->finalize = fin;
        out->loss_nb = fin ? p.loss_nb_finalize : p.loss_nb_tiles;
        out->lp = q.lp;
        out->lw = ldexpf(1.0f, k);
        out->cells = q;
    }
}

// The nodes' partial sums of the mode splits, added in split order and
// compensated, as the cells' are, into the first one's place (bound by the read).
__global__ void __launch_bounds__(256) band_sum_kernel(const BandDesc* b, float* part) {
    pdl_wait();
    const int n_split = b->nodes.n_split;
    if (b->n_light == 0 || n_split == 1) return;
    const int64_t all = static_cast<int64_t>(b->ax[0].m) * b->ax[1].m * b->ax[2].m;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; i < all;
         i += static_cast<int64_t>(gridDim.x) * 256) {
        float x[kNodeSplits];  // all loads in flight: summed as they come, 1024 x 512 cells took 5 us more
#pragma unroll
        for (int q = 0; q < kNodeSplits; ++q) x[q] = q < n_split ? part[q * all + i] : 0.0f;
        float v = x[0], e = 0.0f;
#pragma unroll
        for (int q = 1; q < kNodeSplits; ++q) two_sum_acc(v, e, x[q]);
        part[i] = v + e;
    }
}

// Interpolation along one axis.  kY = false (z): mid[l][y node][x node] from
// the nodes; kY = true (3-D): rows[(l ny + k) lp + x node] from mid, zero for
// the x nodes up to lp (a multiple of 4).
// A block takes 64 columns (the values of one axis position, contiguous in
// memory) and a run of cells of the axis: the run's nodes go to shared memory,
// each read once per block, and the cells' weights, shared by the columns;
// then every cell takes its eight nodes.  An
// axis in no order may need more nodes than fit; its cells read them from
// memory.
constexpr int kCols = 64, kLineNodes = 96, kLineRun = 64;
template <bool kY>
__global__ void __launch_bounds__(256) band_line_kernel(const BandDesc* b, const float* src, const float* cells,
                                                        int n, int nz, float* __restrict__ out) {
    __shared__ float nodes[kLineNodes][kCols];
    __shared__ __align__(16) float wts[kLineRun][kW];
    __shared__ int start[kLineRun];
    __shared__ int first, last;
    pdl_wait();
    if (b->n_light == 0 || (kY && b->finalize)) return;
    const BandAxis ax = kY ? b->ax[1] : b->ax[2];
    const int mx = b->ax[0].m, lp = b->lp;
    const int64_t plane = static_cast<int64_t>(mx) * b->ax[1].m;
    const int64_t stride = kY ? mx : plane;                      // node to node
    const int columns = kY ? nz * lp : static_cast<int>(plane);
    const int cb = (columns + kCols - 1) / kCols, nt = band::taps(ax);
    // cells per block: for about four blocks per SM of 152
    const int run = max(8, min(kLineRun, static_cast<int>(static_cast<int64_t>(cb) * n / (4 * 152))));
    const int runs = (n + run - 1) / run;
    const int lane = threadIdx.x & (kCols - 1), row = threadIdx.x / kCols;
    for (int u = blockIdx.x; u < cb * runs; u += gridDim.x) {
        const int k0 = u / cb * run, nk = min(run, n - k0);
        __syncthreads();  // the previous run's tables are no longer read
        if (threadIdx.x == 0) {
            first = INT_MAX;
            last = 0;
        }
        __syncthreads();
        if (threadIdx.x < nk) {
            float w[kW];
            const int k = k0 + threadIdx.x;
            const int s = band::cell_weights(ax, __ldg(cells + k), k, w);
            start[threadIdx.x] = s;
#pragma unroll
            for (int q = 0; q < kW; ++q) wts[threadIdx.x][q] = q < nt ? w[q] : 0.0f;
            atomicMin(&first, s);
            atomicMax(&last, s + nt);
        }
        // the column's values: node 0 of it, and its place in the output
        const int c = (u % cb) * kCols + lane;
        const float* col = src;
        float* o = out;
        bool zero = false;  // a column that pads the rows
        if (c < columns) {
            if (kY) {
                const int l = c / lp, i = c - l * lp;
                zero = i >= mx;
                col += l * plane + i;
                o += static_cast<int64_t>(l) * n * lp + i;
            } else {
                col += c;
                o += c;
            }
        }
        const int64_t ostride = kY ? lp : plane;
        __syncthreads();
        const int n0 = first, nn = last - first;
        const bool staged = nn <= kLineNodes;
        if (staged && c < columns) {
#pragma unroll 8
            for (int q = row; q < nn; q += 256 / kCols) nodes[q][lane] = zero ? 0.0f : col[(n0 + q) * stride];
        }
        __syncthreads();
        if (c < columns) {
#pragma unroll 2
            for (int k = row; k < nk; k += 256 / kCols) {
                const float4 wa = *reinterpret_cast<const float4*>(&wts[k][0]);
                const float4 wb = *reinterpret_cast<const float4*>(&wts[k][4]);
                const float w[kW] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
                const int s = start[k] - n0;
                float f[kW];
#pragma unroll
                for (int q = 0; q < kW; ++q) {
                    f[q] = 0.0f;
                    if (q < nt) {
                        if (staged)
                            f[q] = nodes[s + q][lane];
                        else if (!zero)
                            f[q] = col[(n0 + s + q) * stride];
                    }
                }
                // pairs from the tails inwards: the small terms first
                float v = 0.0f;
#pragma unroll
                for (int q = 0; q < kW / 2; ++q) v = fmaf(w[q], f[q], fmaf(w[kW - 1 - q], f[kW - 1 - q], v));
                o[(k0 + k) * ostride] = v;
            }
        }
    }
}

// Cells in the plan's order: add[i] = sum over the 8^DIM nodes around cell i.
// A block takes kCellsBlock consecutive sorted cells, a compact group: the
// nodes that they read go to shared memory, and every lane sums one cell with
// 16-byte loads (12 of the x nodes from a multiple of 4, the weights shifted
// to them).  The block first puts its cells in the order of their nodes, so
// that the lanes of a warp read mostly the same addresses: 192 loads per cell
// in 3-D take 4.3 shared-memory wavefronts each in the plan's order (2M cells:
// 210 us).  Groups that spread over more nodes than fit read them from memory.
constexpr int kCellsBlock = 512, kBoxFloats = 10240, kCellBins = 1024;
template <int DIM>
__global__ void __launch_bounds__(256, 3) band_cells_kernel(const BandDesc* b, const float* nodes,
                                                            const float* __restrict__ xs, const float* __restrict__ ys,
                                                            const float* __restrict__ zs, int64_t n,
                                                            float* __restrict__ out) {
    __shared__ __align__(16) float box[kBoxFloats];
    __shared__ int bins[kCellBins];       // cells per bin, then of the bins before it
    __shared__ short order[kCellsBlock];  // cells of the block by bin
    __shared__ int first[3], last[3], warps[8];
    pdl_wait();
    const int64_t c0 = static_cast<int64_t>(blockIdx.x) * kCellsBlock;
    const int t = threadIdx.x, lane = t & 31;
    const int nc = static_cast<int>(min(static_cast<int64_t>(kCellsBlock), n - c0));
    if (b->n_light == 0) {
        for (int i = t; i < nc; i += 256) out[c0 + i] = 0.0f;
        return;
    }
    if (t < 3) {
        first[t] = INT_MAX;
        last[t] = 0;
    }
    for (int k = t; k < kCellBins; k += 256) bins[k] = 0;
    BandAxis ax[DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c) ax[c] = b->ax[c];
    const float* src[3] = {xs + c0, ys + c0, zs + c0};
    __syncthreads();
    constexpr int kPer = kCellsBlock / 256;
    int s[kPer][DIM];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int i = min(q * 256 + t, nc - 1);
#pragma unroll
        for (int c = 0; c < DIM; ++c) {
            float v;
            s[q][c] = band::locate(ax[c], __ldg(src[c] + i), v);
        }
    }
#pragma unroll
    for (int c = 0; c < DIM; ++c) {
        int lo = s[0][c], hi = s[0][c];
#pragma unroll
        for (int q = 1; q < kPer; ++q) {
            lo = min(lo, s[q][c]);
            hi = max(hi, s[q][c]);
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0) {
            atomicMin(&first[c], lo);
            atomicMax(&last[c], hi + kW);
        }
    }
    __syncthreads();
    const int mx = ax[0].m;
    const int64_t plane = static_cast<int64_t>(mx) * ax[1].m;
    int f0[3] = {0, 0, 0}, nb[3] = {1, 1, 1};
#pragma unroll
    for (int c = 0; c < DIM; ++c) {
        f0[c] = first[c];
        nb[c] = last[c] - first[c];
    }
    // rows of the box: an odd multiple of 4, so that the 16-byte loads of
    // neighbouring rows fall in different banks
    const int bx = nb[0] + 4;  // the last loads reach 4 past the nodes
    const int px = ((bx + 3) / 4 | 1) * 4;
    const int rows = nb[1] * nb[2];
    const bool staged = static_cast<int64_t>(px) * rows <= kBoxFloats;
    if (staged) {
        for (int r = t >> 5; r < rows; r += 8) {
            const int z = DIM > 2 ? r / nb[1] : 0, y = r - z * nb[1];
            const float* p = nodes + (f0[2] + z) * plane + static_cast<int64_t>(f0[1] + y) * mx + f0[0];
            for (int x = lane; x < px; x += 32) box[r * px + x] = x < nb[0] ? p[x] : 0.0f;
        }
    }
    // ---- order of the cells: counting sort by their first node (bins wrap
    // where the group has more of them; the order within a bin does not matter)
    int bin[kPer], rank[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        unsigned key = DIM > 2 ? static_cast<unsigned>(s[q][DIM - 1] - f0[2]) * static_cast<unsigned>(nb[1] - kW + 1) : 0u;
        key = (key + static_cast<unsigned>(s[q][1] - f0[1])) * static_cast<unsigned>(nb[0] - kW + 1) +
              static_cast<unsigned>(s[q][0] - f0[0]);
        bin[q] = static_cast<int>(key & (kCellBins - 1));
        rank[q] = q * 256 + t < nc ? atomicAdd(&bins[bin[q]], 1) : 0;
    }
    __syncthreads();
    {
        int v[kCellBins / 256], sum = 0;
#pragma unroll
        for (int k = 0; k < kCellBins / 256; ++k) {
            v[k] = sum;
            sum += bins[t * (kCellBins / 256) + k];
        }
        int run = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, run, off);
            if (lane >= off) run += o;
        }
        if (lane == 31) warps[t >> 5] = run;
        __syncthreads();
        int before = run - sum;
        for (int w = 0; w < (t >> 5); ++w) before += warps[w];
#pragma unroll
        for (int k = 0; k < kCellBins / 256; ++k) bins[t * (kCellBins / 256) + k] = before + v[k];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kPer; ++q)
        if (q * 256 + t < nc) order[bins[bin[q]] + rank[q]] = static_cast<short>(q * 256 + t);
    __syncthreads();
#pragma unroll 1
    for (int q = 0; q < kPer; ++q) {
        if (q * 256 + t >= nc) break;
        const int i = order[q * 256 + t];
        int at[DIM];
        float w[kW], wy[kW], wz[kW], v;
        at[0] = band::locate(ax[0], __ldg(src[0] + i), v);
        band::weights(v, w);
        at[1] = band::locate(ax[1], __ldg(src[1] + i), v);
        band::weights(v, wy);
        if (DIM > 2) {
            at[DIM - 1] = band::locate(ax[DIM - 1], __ldg(src[2] + i), v);
            band::weights(v, wz);
        }
        float acc = 0.0f;
        if (staged) {
            const int dx = at[0] - f0[0], sh = dx & 3;
            float w12[12];
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                float u = 0.0f;
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    if (k - h >= 0 && k - h < kW) u = sh == h ? w[k - h] : u;
                w12[k] = u;
            }
            const float* p = box + (dx - sh) + (at[1] - f0[1]) * px + (DIM > 2 ? (at[DIM - 1] - f0[2]) * nb[1] * px : 0);
#pragma unroll 1
            for (int kz = 0; kz < (DIM > 2 ? kW : 1); ++kz) {
                float a = 0.0f;
#pragma unroll
                for (int ky = 0; ky < kW; ++ky) {
                    const float4* r4 = reinterpret_cast<const float4*>(p + ky * px);
                    const float4 r0 = r4[0], r1 = r4[1], r2 = r4[2];
                    // the tails first
                    float u = w12[0] * r0.x;
                    u = fmaf(w12[11], r2.w, u);
                    u = fmaf(w12[1], r0.y, u);
                    u = fmaf(w12[10], r2.z, u);
                    u = fmaf(w12[2], r0.z, u);
                    u = fmaf(w12[9], r2.y, u);
                    u = fmaf(w12[3], r0.w, u);
                    u = fmaf(w12[8], r2.x, u);
                    u = fmaf(w12[4], r1.x, u);
                    u = fmaf(w12[7], r1.w, u);
                    u = fmaf(w12[5], r1.y, u);
                    u = fmaf(w12[6], r1.z, u);
                    a = fmaf(wy[ky], u, a);
                }
                if (DIM > 2) {
                    float u = wz[0];
#pragma unroll
                    for (int k = 1; k < kW; ++k) u = kz == k ? wz[k] : u;
                    acc = fmaf(u, a, acc);
                } else {
                    acc = a;
                }
                p += nb[1] * px;
            }
        } else {
            const float* p = nodes + (DIM > 2 ? at[DIM - 1] * plane : 0) + static_cast<int64_t>(at[1]) * mx + at[0];
#pragma unroll 1
            for (int kz = 0; kz < (DIM > 2 ? kW : 1); ++kz) {
                float a = 0.0f;
#pragma unroll
                for (int ky = 0; ky < kW; ++ky) {
                    float u = 0.0f;
#pragma unroll
                    for (int k = 0; k < kW; ++k) u = fmaf(w[k], p[static_cast<int64_t>(ky) * mx + k], u);
                    a = fmaf(wy[ky], u, a);
                }
                if (DIM > 2) {
                    float u = wz[0];
#pragma unroll
                    for (int k = 1; k < kW; ++k) u = kz == k ? wz[k] : u;
                    acc = fmaf(u, a, acc);
                } else {
                    acc = a;
                }
                p += plane;
            }
        }
        out[c0 + i] = acc;
    }
}

// Cells of a grid: y and x interpolation of the light modes from the (x, y)
// nodes at the cell's z (2-D: the nodes), plus the direct modes' partial sums
// (added in split order), mu, the maps and the loss partials.
// A block takes tx x cells of kFinRows y cells of one layer: the rows' values
// at the x nodes its cells read go to shared memory (a few values per cell,
// since nodes are wider apart than cells), then every cell takes eight of
// them.  Cells of an axis in no order may need more nodes than fit: the block
// then takes window after window of them (4096 x 4096 cells of a rough field, x
// in random order: 1320 us a call with the 64 values of a cell summed from
// memory, 408 so).  Memory-bound on the outputs where the maps are many, else on
// latency: all loads of a phase are independent.
constexpr int kFinRows = 8, kFinNodes = 320, kFinStep = kFinNodes - (kW - 1);
__global__ void __launch_bounds__(256, 4) band_finalize_kernel(const BandDesc* b, const float* mid, const float* part,
                                                               GridGeom gg, int tx, int units, MapDev map,
                                                               unsigned long long* tiles) {
    __shared__ float rows[kFinRows][kFinNodes];
    __shared__ __align__(16) float wy[kFinRows][kW];
    __shared__ int sy[kFinRows];
    __shared__ int first, last;
    __shared__ double red[8];
    pdl_wait();
    if (!b->finalize) return;
    const int t = threadIdx.x;
    const int n_light = b->n_light, n_split = b->n_splits;
    const int nx = gg.nx, ny = gg.ny;
    const int xb = (nx + tx - 1) / tx, yb = (ny + kFinRows - 1) / kFinRows;
    const bool mm = (map.bits & kMapMismatch) != 0;
    if (b->nh == 0 && tiles != nullptr && blockIdx.x == 0 && t == 0)
        atomicAdd(tiles, static_cast<unsigned long long>(b->cells.n_tiles));
    for (int u = static_cast<int>(blockIdx.x); u < units; u += static_cast<int>(gridDim.x)) {
    __syncthreads();  // the previous unit's tables are no longer read
    if (t == 0) {
        first = INT_MAX;
        last = 0;
    }
    const int k0 = (u / xb) % yb * kFinRows, l = u / xb / yb;
    const int i = u % xb * tx + (t & (tx - 1));
    const int r0 = t / tx, rstep = 256 / tx;
    float w[kW];
    int s = 0, nt = 0, mx = 0, nty = 0;
    const float* base = mid;
    if (n_light > 0) {
        const BandAxis ax = b->ax[0], ay = b->ax[1];
        mx = ax.m;
        nt = band::taps(ax);
        nty = band::taps(ay);
        base += static_cast<int64_t>(l) * ax.m * ay.m;
        if (t < kFinRows) {
            float v[kW];
            const int k = min(k0 + t, ny - 1);
            sy[t] = band::cell_weights(ay, __ldg(gg.Y + k), k, v);
#pragma unroll
            for (int q = 0; q < kW; ++q) wy[t][q] = q < nty ? v[q] : 0.0f;
        }
        const int ic = min(i, nx - 1);
        s = band::cell_weights(ax, __ldg(gg.X + ic), ic, w);
    }
    __syncthreads();
    if (n_light > 0) {
        const int lo = __reduce_min_sync(0xffffffffu, s), hi = __reduce_max_sync(0xffffffffu, s);
        if ((t & 31) == 0) {
            atomicMin(&first, lo);
            atomicMax(&last, hi + nt);
        }
    }
    __syncthreads();
    double loss = 0.0;
    const int64_t n = static_cast<int64_t>(nx) * ny * gg.nz;
    // windows of nodes: a cell belongs to the one that holds its first node
    const int n_end = n_light > 0 ? last - nt + 1 : 1;
    for (int n0 = n_light > 0 ? first : 0; n0 < n_end; n0 += kFinStep) {
        if (n_light > 0) {
            const int nn = min(kFinNodes, last - n0);
            __syncthreads();  // the previous window is no longer read
            for (int e = t; e < kFinRows * nn; e += 256) {
                const int r = e / nn, c = e - r * nn;
                const float* p = base + static_cast<int64_t>(sy[r]) * mx + n0 + c;
                float f[kW];
#pragma unroll
                for (int q = 0; q < kW; ++q) f[q] = q < nty ? p[static_cast<int64_t>(q) * mx] : 0.0f;
                float v = 0.0f;
#pragma unroll
                for (int q = 0; q < kW / 2; ++q) v = fmaf(wy[r][q], f[q], fmaf(wy[r][kW - 1 - q], f[kW - 1 - q], v));
                rows[r][c] = v;
            }
            __syncthreads();
        }
        if (i >= nx || static_cast<unsigned>(s - n0) >= static_cast<unsigned>(kFinStep)) continue;
#pragma unroll 2
        for (int r = r0; r < min(kFinRows, ny - k0); r += rstep) {
            const int64_t o = (static_cast<int64_t>(l) * ny + k0 + r) * nx + i;
            const float target = mm ? map.T[o] : 0.0f;
            float v = 0.0f;
            if (n_light > 0) {
                const float* p = &rows[r][s - n0];
#pragma unroll
                for (int q = 0; q < kW / 2; ++q) {
                    if (kW - 1 - q < nt) v = fmaf(w[kW - 1 - q], p[kW - 1 - q], v);
                    if (q < nt) v = fmaf(w[q], p[q], v);
                }
            }
            float e = 0.0f;
#pragma unroll 4
            for (int k = 0; k < n_split; ++k) two_sum_acc(v, e, part[k * n + o]);
            const float y = (v + e) + map.mu;
            map_store(map, o, y);
            if (mm) loss += mismatch_value(map, o, y, target);
        }
    }
    if (mm) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
        if ((t & 31) == 0) red[t >> 5] = loss;
        __syncthreads();
        if (t == 0) {
            double sum = 0.0;
            for (int k = 0; k < 8; ++k) sum += red[k];
            map.lpart[u] = sum;
        }
    }
    }
}

}  // namespace

int launch_band_select(const BandSelect& p, BandDesc* out, void* stream) {
    return launch_chained(band_select_kernel, 1, kSelThreads, 0, static_cast<cudaStream_t>(stream), p, out);
}

namespace {
// x cells per finalize block: a power of two from 32 to 256.
int finalize_tx(int32_t nx) {
    int tx = 32;
    while (tx < 256 && tx < nx) tx *= 2;
    return tx;
}
}  // namespace

int64_t band_finalize_blocks(const GridGeom& gg) {
    const int tx = finalize_tx(gg.nx);
    return int64_t((gg.nx + tx - 1) / tx) * ((gg.ny + kFinRows - 1) / kFinRows) * gg.nz;
}

int launch_band_lines(const BandDesc* b, float* part, const GridGeom& gg, float* mid, float* rows, int sms,
                      void* stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = launch_chained(band_sum_kernel, sms * 8, 256, 0, st, b, part);
    if (e == cudaSuccess && mid != nullptr && gg.nz > 1)
        e = launch_chained(band_line_kernel<false>, sms * 4, 256, 0, st, b, part, gg.Z, gg.nz, gg.nz, mid);
    if (e == cudaSuccess && rows != nullptr)
        e = launch_chained(band_line_kernel<true>, sms * 4, 256, 0, st, b, mid, gg.Y, gg.ny, gg.nz, rows);
    return e;
}

int launch_band_cells(const BandDesc* b, const float* nodes, int32_t dim, const float* xs, const float* ys,
                      const float* zs, int64_t n, float* out, void* stream) {
    return launch_chained(dim > 2 ? band_cells_kernel<3> : band_cells_kernel<2>,
                          static_cast<unsigned>((n + kCellsBlock - 1) / kCellsBlock), 256, 0,
                          static_cast<cudaStream_t>(stream), b, nodes, xs, ys, zs, n, out);
}

int launch_band_finalize(const BandDesc* b, const float* mid, const float* part, const GridGeom& gg,
                         const MapDev& map, unsigned long long* tiles, int sms, void* stream) {
    // a few rounds of resident blocks; a launch with nothing to do ends at once
    const int units = static_cast<int>(band_finalize_blocks(gg));
    return launch_chained(band_finalize_kernel, std::min(units, sms * 16), 256, 0, static_cast<cudaStream_t>(stream), b,
                          mid, part, gg, finalize_tx(gg.nx), units, map, tiles);
}

}  // namespace grf
