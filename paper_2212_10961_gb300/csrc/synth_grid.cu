// Spectral synthesis on Cartesian grids with the fifth-generation tensor
// cores (Icardi et al., arXiv 2212.10961, Sec. 4.1, Eq. DiscreteFT).
//
// When the cells are the tensor product of three axes -- cell (i, k, l) at
// (X_i, Y_k, Z_l) -- every term of the sum factorises,
//     A_j cos(2 pi (a_j . x + psi_j)) = Re[ Xp_ij W_jc ],
//     Xp_ij = e^{2 pi i a_jx X_i},  W_jc = A_j e^{2 pi i (psi_j + a_jy Y_k + a_jz Z_l)},
// so on a block of 128 x-cells (rows i) by 128 (y, z) cells (columns c) the
// field is a real matrix product over K = 2N:
//     Y[i, c] - mu = sum_j ( Re Xp_ij Re W_jc - Im Xp_ij Im W_jc ).
// The x phasors (operand A) are the same for every block of one x range:
// they are tabulated once per call, already in the tensor core's shared-
// memory layout, and copied in chunk by chunk.  Operand B:
//   * 3-D grids: a tile's columns are a patch of 2^p y-cells by 128 / 2^p
//     z-cells; per chunk the loader copies the patch's y phasors and
//     (amplitude, psi, z) phasors (tables stored chunk by chunk) next to A,
//     and the epilogue warps form B = WZ * Yp in shared memory;
//   * 2-D grids (and 3-D grids of one z layer): B = W * Yp is tabulated like
//     A and copied in as well.
// All phases are exactly reduced (hi/lo frequencies, FMA-split products)
// before an accurate sincospi.
//
// Precision.  Each operand value v (|v| <= 1 after scaling the amplitudes
// by a power of two S) is split into FP16 numbers hi + lo with
// |v - hi - lo| <= 2^-24; a term costs three tensor-core products
// hi.hi + hi.lo + lo.hi (the dropped lo.lo is below 2^-24).  The hi.hi
// products go to an FP32 accumulator in TMEM that takes `fc` chunks of 32
// modes and is then folded into a running FP32 sum (a few tens of folds per
// cell), so the accumulator's own rounding acts on short partial sums only;
// the two correction products, 2^-11 smaller, go to a second accumulator
// that spans the whole tile.
//
// Kernel structure (one CTA per SM, persistent over work items: tiles, or
// for grids of at most 64 tiles (tile, mode split) pairs of whole fold
// intervals whose partial fields a finalize kernel adds in split order):
//   warps 0-15: form B for each chunk (3-D; a thread forms 4 modes of two
//               columns that share a y cell), fold the accumulator, write the
//               maps (warp w reads TMEM lanes 32 (w mod 4) .., columns 32 (w / 4) ..);
//   warp 16   : one thread issues the MMAs (tcgen05.mma kind::f16, M = N = 128);
//   warp 17   : one thread issues the bulk copies; the warp owns TMEM.
// A ring of `sa` stages (A hi/lo and the chunk's tables, or A and B) and,
// in 3-D, a ring of 3 formed B stages.  TMEM (512 columns): the hi.hi
// accumulator double-buffered (2 x 128), the correction accumulator (128) and
// the running sums (128).  Every mbarrier wait is bounded and reports through
// the status word.
//
// Large calls sum only their modes of high frequency at the cells this way;
// the same kernel sums the others at the nodes of a coarse lattice, from which
// they are interpolated (band.cuh, band.cu): 256^3 cells x 4096 modes of a
// rough field 969 -> 265 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "band.cuh"
#include "device_common.cuh"
#include "grid_common.cuh"
#include "grid_tiling.cuh"
#include "launch.cuh"
#include "tcgen05.cuh"

namespace grf {

// Tiles computed by the grid path since the last grf_take_grid_tiles.
static __device__ unsigned long long g_grid_tiles;

namespace {

using gridc::gwait;
using gridc::psi_z_turns;
using gridc::tile_off;
using namespace gridt;

// Amplitude scale: the smallest power of two S >= max |A_j| (1 when all
// amplitudes vanish), so that |W| <= 1.
__device__ __forceinline__ float grid_scale(const TableHeader* h) {
    const float m = h->amp_max;
    if (!(m > 0.0f)) return 1.0f;
    int e;
    frexpf(m, &e);
    return ldexpf(1.0f, e);
}

// B of one chunk for the columns n0 and n1 (one y cell, two z cells):
// W_jc = WZ[l, j] * Yp[k, j] for the 4 modes of group kk8, from the staged
// table rows ty (y) and tw0, tw1 ((amplitude, psi, z) of the two z cells),
// written as (re, im) FP16 pairs into rows n0 and n1 of the hi and lo tiles,
// K segment kk8.
__device__ __forceinline__ void form_b(unsigned char* bhi, const float4* ty, const float4* tw0, const float4* tw1,
                                       int n0, int n1, int kk8) {
    const float4 ya = ty[0], yb = ty[1];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float4* tw = h == 0 ? tw0 : tw1;
        const uint32_t boff = tile_off(h == 0 ? n0 : n1, kk8);
        const float4 wa = tw[0], wb = tw[1];
        const float r0 = fmaf(wa.x, ya.x, -wa.y * ya.y), i0 = fmaf(wa.x, ya.y, wa.y * ya.x);
        const float r1 = fmaf(wa.z, ya.z, -wa.w * ya.w), i1 = fmaf(wa.z, ya.w, wa.w * ya.z);
        const float r2 = fmaf(wb.x, yb.x, -wb.y * yb.y), i2 = fmaf(wb.x, yb.y, wb.y * yb.x);
        const float r3 = fmaf(wb.z, yb.z, -wb.w * yb.w), i3 = fmaf(wb.z, yb.w, wb.w * yb.z);
        uint4 H, L;
        tc::split_f16x2(r0, i0, H.x, L.x);
        tc::split_f16x2(r1, i1, H.y, L.y);
        tc::split_f16x2(r2, i2, H.z, L.z);
        tc::split_f16x2(r3, i3, H.w, L.w);
        *reinterpret_cast<uint4*>(bhi + boff) = H;
        *reinterpret_cast<uint4*>(bhi + kGOpBytes + boff) = L;
    }
}

struct TileIdx {
    int mt, kt, k0, l0, pkv, plv;  // x tile, y tile, first y and z cell, valid y and z cells of the patch
};
__device__ __forceinline__ TileIdx tile_idx(const GridTiling& T, int64_t tile) {
    TileIdx t;
    t.mt = static_cast<int>(tile % T.n_mt);
    const int64_t rest = tile / T.n_mt;
    t.kt = static_cast<int>(rest % T.n_kt);
    t.k0 = t.kt << T.pk_log2;
    t.l0 = static_cast<int>(rest / T.n_kt) * (kGN >> T.pk_log2);
    t.pkv = min(1 << T.pk_log2, T.ny - t.k0);
    t.plv = min(kGN >> T.pk_log2, T.nz - t.l0);
    return t;
}

// B of a light chunk: 16 nodes (segments 2 q4, 2 q4 + 1) of column n's row
// of x nodes, from node `first` of the row, times `inv`.
__device__ __forceinline__ void form_light(unsigned char* bhi, const float* row, int first, int lp, float inv, int n,
                                           int q4) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float4 v[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int node = first + 16 * q4 + 8 * h + 4 * e;
            v[e] = node < lp ? *reinterpret_cast<const float4*>(row + node) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        uint4 H, L;
        tc::split_f16x2(v[0].x * inv, v[0].y * inv, H.x, L.x);
        tc::split_f16x2(v[0].z * inv, v[0].w * inv, H.y, L.y);
        tc::split_f16x2(v[1].x * inv, v[1].y * inv, H.z, L.z);
        tc::split_f16x2(v[1].z * inv, v[1].w * inv, H.w, L.w);
        const uint32_t boff = tile_off(n, 2 * q4 + h);
        *reinterpret_cast<uint4*>(bhi + boff) = H;
        *reinterpret_cast<uint4*>(bhi + kGOpBytes + boff) = L;
    }
}

// kLight: the band path's direct modes at the cells of a 3-D grid; a tile's
// first interval is the light modes' chunks.
template <bool kSplit, bool kLight>
__device__ __forceinline__ void grid_mma_body(const GridDesc& d, const GridTiling& T, unsigned char* gsm_raw,
                                              int32_t* status) {
    // stages on a 1024-byte boundary of the shared window (swizzle atoms)
    unsigned char* gsm = gsm_raw + ((1024u - (smem_u32(gsm_raw) & 1023u)) & 1023u);
    uint64_t* bars = reinterpret_cast<uint64_t*>(gsm + T.off_bar);
    uint64_t* afull = bars;                // [sa] stage's copies landed (transaction bytes)
    uint64_t* afree = bars + kGMaxSA;      // [sa] stage's MMAs completed
    uint64_t* bfull = bars + 2 * kGMaxSA;  // [kGSB] B formed (one arrival per epilogue warp)
    uint64_t* bfree = bfull + kGSB;        // [kGSB] B's MMAs completed
    uint64_t* accfull = bfree + kGSB;      // [2] interval's MMAs completed
    uint64_t* accfree = accfull + 2;       // [2] accumulator read by every epilogue warp
    uint64_t* corrfree = accfree + 2;      // correction accumulator read (tile end)
    uint64_t* done = corrfree + 1;         // all MMAs of this CTA completed
    uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
    volatile int32_t* abort = reinterpret_cast<volatile int32_t*>(done + 2);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const bool form = T.form != 0;
    const bool mm = (d.map.bits & kMapMismatch) != 0;
    const int SA = T.sa;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kGMaxSA; ++s) {
            mbar_init(afull + s, 1);
            mbar_init(afree + s, 1);
        }
        for (int b = 0; b < kGSB; ++b) {
            mbar_init(bfull + b, kGEpiWarps);
            mbar_init(bfree + b, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accfull + b, 1);
            mbar_init(accfree + b, kGEpiWarps);
        }
        mbar_init(corrfree, kGEpiWarps);
        mbar_init(done, 1);
        *abort = 0;
        fence_mbar_init();
    }
    if (warp == kGEpiWarps + 1) tc::alloc(tslot, kGTmemCols);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *tslot;
    pdl_wait();
    const int nl = kLight ? T.nl : 0;
    const int li = nl > 0 ? 1 : 0;    // the light chunks are an interval of their own
    const int NI = (T.nc + T.fc - 1) / T.fc + li;  // fold intervals per tile
    const int n_split = kSplit ? T.n_split : 1;
    const int pkm = (1 << T.pk_log2) - 1;

    if (warp < kGEpiWarps) {
        // ---- B formation (3-D), folds, maps ---------------------------------------
        const int q = warp & 3;           // TMEM lane quarter (rows 32 q .. 32 q + 31)
        const int h = warp >> 2;          // column block (kGColsPerWarp h ..)
        const int t = threadIdx.x;        // 0 .. 255
        const int fp = t & (kGFormPairs - 1);  // column pair this thread forms
        const int fg = t / kGFormPairs;        // 4-mode group of the chunk it forms
        const int fk = fp & pkm;               // y cell of the pair in the patch
        const int fz = (fp >> T.pk_log2) * 2;  // first z cell of the pair in the patch
        const int n0 = fk + (fz << T.pk_log2), n1 = n0 + (1 << T.pk_log2);
        const uint32_t lane_off = static_cast<uint32_t>(32 * q) << 16;
        const float S = T.scale > 0.0f ? T.scale : grid_scale(d.thdr);
        uint32_t g = 0, gi = 0;
        for (int64_t item = blockIdx.x; item < (kSplit ? T.n_items : T.n_tiles); item += gridDim.x) {
            const int64_t tile = kSplit ? item / n_split : item;
            const int split = kSplit ? static_cast<int>(item - tile * n_split) : 0;
            // the item's fold intervals iv0 .. iv1 - 1 (all of the tile's without a split)
            const int iv0 = kSplit ? NI * split / n_split : 0;
            const int NIl = kSplit ? NI * (split + 1) / n_split - iv0 : NI;
            const TileIdx ti = tile_idx(T, tile);
            // staged table rows this thread reads: y row and (amplitude, psi, z) row
            const int ry = min(fk, ti.pkv - 1);
            const int rz0 = min(fz, ti.plv - 1), rz1 = min(fz + 1, ti.plv - 1);
            const int toff_y = kGPair + ry * kGRowBytes + 32 * fg;
            const int toff_w0 = kGPair + ((1 << T.pk_log2) + rz0) * kGRowBytes + 32 * fg;
            const int toff_w1 = kGPair + ((1 << T.pk_log2) + rz1) * kGRowBytes + 32 * fg;

            // fold of interval gidx: the hi.hi accumulator into the running sum
            // (plain FP32: a few tens of folds per cell); the last fold of a
            // tile adds the correction accumulator and writes the cells
            double lsum = 0.0;  // kMapMismatch: this lane's sum of (K - T)^2 over the tile
            auto fold = [&](uint32_t gidx, bool first, bool last) -> bool {
                const uint32_t b = gidx & 1u;
                // warp-uniform outcome: the TMEM moves below are warp-wide
                if (!__all_sync(0xffffffffu, gwait(accfull + b, (gidx >> 1) & 1u, abort, status))) return false;
                tc::fence_after();
                if (!last) {
#pragma unroll 1
                    for (int blk = 0; blk < kGColsPerWarp / 16; ++blk) {  // 16 columns per TMEM round trip
                        const uint32_t col = static_cast<uint32_t>(kGColsPerWarp * h + 16 * blk);
                        uint32_t p[16], sm[16];
                        tc::ld16(tbase + lane_off + b * kGN + col, p);
                        if (!first) tc::ld16(tbase + lane_off + kGSumCol + col, sm);
                        tc::wait_ld();
                        if (blk == kGColsPerWarp / 16 - 1) {
                            tc::fence_before();
                            __syncwarp();
                            if (lane == 0) tc::mbar_arrive(accfree + b);
                        }
#pragma unroll
                        for (int cc = 0; cc < 16; ++cc)
                            sm[cc] = first ? p[cc] : __float_as_uint(__uint_as_float(sm[cc]) + __uint_as_float(p[cc]));
                        tc::st16(tbase + lane_off + kGSumCol + col, sm);
                    }
                    tc::wait_st();
                } else {
                    const int i = ti.mt * kGM + 32 * q + lane;
                    // cell of the row: x cell xi of z block zb (one block at the cells)
                    const int zb = kSplit ? i / T.xn : 0;
                    const int xi = i - zb * T.xn;
                    // a plan has fewer than 2^31 cells (and a lattice fewer nodes)
                    const uint32_t xn = static_cast<uint32_t>(T.xn), xny = xn * static_cast<uint32_t>(T.ny);
                    const uint32_t o0 = static_cast<uint32_t>(xi) + xn * static_cast<uint32_t>(ti.k0) +
                                        xny * static_cast<uint32_t>(ti.l0 + zb * T.lz);
                    // valid columns: y cells below kn, z cells below ln of the patch
                    const int kn = i < T.nx ? T.ny - ti.k0 : 0;
                    const int ln = min(T.nz, T.zn - zb * T.lz) - ti.l0;
                    float* part =
                        kSplit ? d.part + static_cast<int64_t>(split) * T.xn * T.ny * T.zn : nullptr;
#pragma unroll 1
                    for (int blk = 0; blk < kGColsPerWarp / 8; ++blk) {  // 8 columns at a time, then the maps
                        const uint32_t col = static_cast<uint32_t>(kGColsPerWarp * h + 8 * blk);
                        uint32_t p[8], sm[8], cr[8];
                        tc::ld8(tbase + lane_off + b * kGN + col, p);
                        tc::ld8(tbase + lane_off + kGCorrCol + col, cr);
                        if (!first) tc::ld8(tbase + lane_off + kGSumCol + col, sm);
                        tc::wait_ld();
                        if (blk == kGColsPerWarp / 8 - 1) {
                            tc::fence_before();
                            __syncwarp();
                            if (lane == 0) {
                                tc::mbar_arrive(accfree + b);
                                tc::mbar_arrive(corrfree);
                            }
                        }
#pragma unroll
                        for (int cc = 0; cc < 8; ++cc) {
                            float v = __uint_as_float(p[cc]);
                            if (!first) v = __uint_as_float(sm[cc]) + v;
                            v += __uint_as_float(cr[cc]);
                            const int c = static_cast<int>(col) + cc;
                            const int kc = c & pkm, lc = c >> T.pk_log2;
                            if (kc < kn && lc < ln) {
                                const uint32_t o = o0 + xn * static_cast<uint32_t>(kc) + xny * static_cast<uint32_t>(lc);
                                if (kSplit) {
                                    part[o] = v * S;
                                } else {
                                    const float y = v * S + d.map.mu;
                                    map_store(d.map, o, y);
                                    if (mm) lsum += mismatch_store(d.map, o, y);
                                }
                            }
                        }
                    }
                }
                return true;
            };

            bool ok = true;
            if (form) {
                // chunks of the item; light chunks are numbered below 0
                const int c_end = kSplit ? min((iv0 + NIl) * T.fc, T.nc) : T.nc;
                const int lcol = t >> 2;  // column whose row of x nodes this thread forms
                const int lk = min(ti.k0 + (lcol & pkm), T.ny - 1), ll = min(ti.l0 + (lcol >> T.pk_log2), T.nz - 1);
                for (int c = kSplit ? iv0 * T.fc : -nl; c < c_end; ++c, ++g) {
                    const int sb = static_cast<int>(g % kGSB);
                    const int sa = static_cast<int>(g % SA);
                    if (g >= kGSB &&
                        !__all_sync(0xffffffffu, gwait(bfree + sb, ((g / kGSB) - 1u) & 1u, abort, status))) {
                        ok = false;
                        break;
                    }
                    if (!__all_sync(0xffffffffu, gwait(afull + sa, (g / SA) & 1u, abort, status))) {
                        ok = false;
                        break;
                    }
                    const unsigned char* st = gsm + sa * T.a_stage;
                    if (kLight && c < 0)
                        form_light(gsm + T.off_b + sb * kGPair,
                                   d.light + (static_cast<int64_t>(ll) * T.ny + lk) * T.lp,
                                   d.lstart[ti.mt] + (c + nl) * kGK, T.lp, T.l_inv, lcol, t & 3);
                    else
                        form_b(gsm + T.off_b + sb * kGPair, reinterpret_cast<const float4*>(st + toff_y),
                               reinterpret_cast<const float4*>(st + toff_w0),
                               reinterpret_cast<const float4*>(st + toff_w1), n0, n1, fg);
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(bfull + sb);
                    if (c >= -1 && ((c + 1) % T.fc == 0 || c + 1 == c_end)) {
                        const int iv = (c + T.fc) / T.fc - 1 + li - (kSplit ? iv0 : 0);  // the item's interval whose chunks are all formed
                        if (iv >= 1) {
                            if (!fold(gi, iv == 1, false)) {
                                ok = false;
                                break;
                            }
                            ++gi;
                        }
                    }
                }
                if (!ok || !fold(gi, NIl == 1, true)) break;
                ++gi;
            } else {
                for (int iv = 0; iv < NIl; ++iv, ++gi) {
                    if (!fold(gi, iv == 0, iv == NIl - 1)) {
                        ok = false;
                        break;
                    }
                }
                if (!ok) break;
            }
            if (mm && !kSplit) {
                // fixed butterfly order, one partial per (tile, warp): the loss
                // does not depend on which CTA took the tile
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
                if (lane == 0) d.map.lpart[tile * kGEpiWarps + warp] = lsum;
            }
        }
    } else if (warp == kGEpiWarps) {
        // ---- MMA issue ------------------------------------------------------------
        if (lane == 0) {
            const uint32_t idesc = tc::idesc_f16_f32(kGM, kGN);
            constexpr uint32_t dhi = tc::smem_desc_sw128_hi(kGSbo);
            constexpr uint32_t tstep = kGOpBytes >> 4;  // one operand tile in descriptor units
            const uint32_t alo0 = tc::smem_desc_sw128_lo(smem_u32(gsm));
            const uint32_t blo0 = tc::smem_desc_sw128_lo(smem_u32(gsm + T.off_b));
            uint32_t g = 0, gi = 0, tile_count = 0;
            uint32_t sa = 0, pa = 0, sb = 0, pb = 0;  // ring stages and their phase parities
            bool ok = true;
            const uint32_t dc = tbase + kGCorrCol;
            for (int64_t item = blockIdx.x; item < (kSplit ? T.n_items : T.n_tiles) && ok; item += gridDim.x, ++tile_count) {
                const int split = kSplit ? static_cast<int>(item % n_split) : 0;
                const int NIl = kSplit ? NI * (split + 1) / n_split - NI * split / n_split : NI;
                // the previous item's correction accumulator has been read
                if (tile_count >= 1 && !gwait(corrfree, (tile_count - 1u) & 1u, abort, status)) {
                    ok = false;
                    break;
                }
                for (int iv = 0; iv < NIl && ok; ++iv, ++gi) {
                    const uint32_t b = gi & 1u;
                    if (gi >= 2 && !gwait(accfree + b, ((gi >> 1) - 1u) & 1u, abort, status)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after();
                    const uint32_t dt = tbase + b * kGN;
                    const int cn = kLight && li && iv == 0
                                       ? nl
                                       : min(T.fc, T.nc - (iv - li + (kSplit ? NI * split / n_split : 0)) * T.fc);
                    for (int cc = 0; cc < cn; ++cc, ++g) {
                        if (!gwait(afull + sa, pa, abort, status) || (form && !gwait(bfull + sb, pb, abort, status))) {
                            ok = false;
                            break;
                        }
                        tc::fence_after();
                        const uint32_t alo = alo0 + sa * (static_cast<uint32_t>(T.a_stage) >> 4);
                        const uint32_t blo = form ? blo0 + sb * (kGPair >> 4) : alo + (kGPair >> 4);
#pragma unroll
                        for (int ks = 0; ks < kGK / 16; ++ks) {
                            const uint32_t ko = static_cast<uint32_t>(ks) * (kGKStep >> 4);  // 16 K elements
                            const uint64_t ah = tc::desc_of(alo + ko, dhi);
                            const uint64_t al = tc::desc_of(alo + tstep + ko, dhi);
                            const uint64_t bh = tc::desc_of(blo + ko, dhi);
                            const uint64_t bl = tc::desc_of(blo + tstep + ko, dhi);
                            tc::mma_f16(dt, ah, bh, idesc, (cc | ks) != 0 ? 1u : 0u);
                            tc::mma_f16(dc, ah, bl, idesc, (iv | cc | ks) != 0 ? 1u : 0u);
                            tc::mma_f16(dc, al, bh, idesc, 1u);
                        }
                        tc::commit(afree + sa);
                        if (form) tc::commit(bfree + sb);
                        if (++sa == static_cast<uint32_t>(SA)) {
                            sa = 0;
                            pa ^= 1u;
                        }
                        if (++sb == kGSB) {
                            sb = 0;
                            pb ^= 1u;
                        }
                    }
                    if (ok) tc::commit(accfull + b);
                }
                if (ok && !d.quiet) atomicAdd(&g_grid_tiles, 1ull);
            }
            // every MMA this CTA issued has completed before TMEM is released
            tc::commit(done);
            mbar_wait_bounded(done, 0);
        }
        __syncwarp();
    } else {
        // ---- bulk copies: A chunks and, per chunk, the tables or B ---------------------
        if (lane == 0) {
            uint32_t g = 0;
            bool ok = true;
            for (int64_t item = blockIdx.x; item < (kSplit ? T.n_items : T.n_tiles) && ok; item += gridDim.x) {
                const int64_t tile = kSplit ? item / n_split : item;
                const int split = kSplit ? static_cast<int>(item - tile * n_split) : 0;
                const TileIdx ti = tile_idx(T, tile);
                const unsigned char* asrc = d.atab + static_cast<int64_t>(ti.mt) * T.nc * kGPair;
                const int c_end = kSplit ? min(NI * (split + 1) / n_split * T.fc, T.nc) : T.nc;
                for (int c = kSplit ? NI * split / n_split * T.fc : -nl; c < c_end; ++c, ++g) {
                    const int sa = static_cast<int>(g % SA);
                    if (g >= static_cast<uint32_t>(SA) &&
                        !gwait(afree + sa, ((g / SA) - 1u) & 1u, abort, status)) {
                        ok = false;
                        break;
                    }
                    unsigned char* dst = gsm + sa * T.a_stage;
                    const unsigned char* ac = asrc + static_cast<int64_t>(c) * kGPair;
                    if (kLight && c < 0) {
                        ac = d.latab + (static_cast<int64_t>(ti.mt) * nl + (c + nl)) * kGPair;
                        mbar_arrive_expect_tx(afull + sa, kGPair);
                        bulk_g2s(dst, ac, kGOpBytes, afull + sa);
                        bulk_g2s(dst + kGOpBytes, ac + kGOpBytes, kGOpBytes, afull + sa);
                    } else if (form) {
                        const uint32_t by = static_cast<uint32_t>(ti.pkv) * kGRowBytes;
                        const uint32_t bw = static_cast<uint32_t>(ti.plv) * kGRowBytes;
                        mbar_arrive_expect_tx(afull + sa, kGPair + by + bw);
                        bulk_g2s(dst, ac, kGOpBytes, afull + sa);
                        bulk_g2s(dst + kGOpBytes, ac + kGOpBytes, kGOpBytes, afull + sa);
                        bulk_g2s(dst + kGPair, d.ytab + (static_cast<int64_t>(c) * T.ny + ti.k0) * (kGRowBytes / 8), by,
                                 afull + sa);
                        bulk_g2s(dst + kGPair + (1 << T.pk_log2) * kGRowBytes,
                                 d.wztab + (static_cast<int64_t>(c) * T.nz + ti.l0) * (kGRowBytes / 8), bw,
                                 afull + sa);
                    } else {
                        const unsigned char* bc = d.btab + (static_cast<int64_t>(ti.kt) * T.nc + c) * kGPair;
                        mbar_arrive_expect_tx(afull + sa, 2 * kGPair);
                        bulk_g2s(dst, ac, kGOpBytes, afull + sa);
                        bulk_g2s(dst + kGOpBytes, ac + kGOpBytes, kGOpBytes, afull + sa);
                        bulk_g2s(dst + kGPair, bc, kGOpBytes, afull + sa);
                        bulk_g2s(dst + kGPair + kGOpBytes, bc + kGOpBytes, kGOpBytes, afull + sa);
                    }
                }
            }
            // copies still in flight land before the CTA's shared memory goes away
            for (uint32_t q = g > static_cast<uint32_t>(SA) ? g - SA : 0u; q < g; ++q)
                mbar_wait_bounded(afull + q % SA, (q / SA) & 1u);
        }
        __syncwarp();
    }
    tc::fence_before();
    __syncthreads();
    if (warp == kGEpiWarps + 1) {
        tc::fence_after();
        tc::dealloc(tbase, kGTmemCols);
    }
}

template <bool kSplit>
__global__ void __launch_bounds__(kGThreads, 1) grid_mma_kernel(GridDesc d, int32_t* status) {
    extern __shared__ __align__(1024) unsigned char gsm_dyn[];
    grid_mma_body<kSplit, false>(d, d.t, gsm_dyn, status);
}

// The same with sizes that the device chose: the light modes on the node
// lattice of the band path or the direct modes at the cells, as partial sums
// (kSplit) or with the light modes' chunks and the maps.
template <bool kSplit>
__global__ void __launch_bounds__(kGThreads, 1) grid_band_kernel(GridDesc d, const GridTiling* src, int32_t* status) {
    extern __shared__ __align__(1024) unsigned char gsm_dyn[];
    __shared__ GridTiling T;
    pdl_wait();
    if (threadIdx.x < sizeof(GridTiling) / 4)
        reinterpret_cast<uint32_t*>(&T)[threadIdx.x] = reinterpret_cast<const uint32_t*>(src)[threadIdx.x];
    __syncthreads();
    if (blockIdx.x >= T.n_items) return;  // nothing to sum, or fewer items than CTAs
    grid_mma_body<kSplit, !kSplit>(d, T, gsm_dyn, status);
}

// Tables of one call (workspace).  Work items, flattened:
//   A : (mt, chunk, row, quad of 4 modes) -> one 16-byte row segment of the
//       hi and of the lo tile ((re, -im) pairs of e^{2 pi i a_x X_i}; rows
//       beyond nx are zero);
//   3-D (form):  Y : (chunk, k, m) -> e^{2 pi i a_jy Y_k},
//                W : (chunk, l, m) -> (A_j / S) e^{2 pi i (psi_j + a_jz Z_l)}, j = 32 chunk + m;
//   2-D (load):  B : (kt, chunk, column, quad) -> (A_j / S) e^{2 pi i (psi_j + a_jy Y_k + a_jz Z_0)}
//                as (re, im) hi and lo tiles (columns beyond ny are zero).
// Node lattices of the band path also multiply A_j by the window's gains.
// Table slot of mode j of the sum; < 0: none (the chunk's padding, amplitude 0).
__device__ __forceinline__ int prep_slot(const GridPrep& p, int j) { return p.idx != nullptr ? p.idx[j] : j; }
__device__ __forceinline__ float prep_amp(const GridPrep& p, int j, const float4 c0, const float4 c1, float s_inv) {
    float amp = __ldg(&p.hot[j].w) * s_inv;
    if (p.gain_h[0] > 0.0f) amp *= band::gain(fabsf(c0.x) * p.gain_h[0]);
    if (p.gain_h[1] > 0.0f) amp *= band::gain(fabsf(c0.z) * p.gain_h[1]);
    if (p.gain_h[2] > 0.0f) amp *= band::gain(fabsf(c1.x) * p.gain_h[2]);
    return amp;
}

// I: unsigned type that holds the item count (64-bit divisions are slow).
template <class I>
__device__ __forceinline__ void grid_prep_items(const GridPrep& p, I nA, I nY, I nW) {
    const float s_inv = 1.0f / (p.scale > 0.0f ? p.scale : grid_scale(p.thdr));  // exact: a power of two
    const bool has_z = p.dim > 2;
    const I stride = static_cast<I>(gridDim.x) * blockDim.x;
    for (I idx = static_cast<I>(blockIdx.x) * blockDim.x + threadIdx.x; idx < nA + nY + nW; idx += stride) {
        if (idx < nA || (!p.form && idx < nA + nY)) {
            // an operand tile row segment: A (x phasors) or, in 2-D, B
            const bool is_a = idx < nA;
            const I u = is_a ? idx : idx - nA;
            const int quad = static_cast<int>(u & 7);
            const int r = static_cast<int>((u >> 3) & 127);
            const I rest = u >> 10;  // (mt or kt) nc + chunk
            const int tt = static_cast<int>(rest / static_cast<I>(p.nc));
            const int c = static_cast<int>(rest - static_cast<I>(tt) * static_cast<I>(p.nc));
            const int i = tt * kGM + r;  // row or y cell
            float v[8];
            if (is_a) {
                const bool in = i < p.nx;
                const int zb = i / p.xn;  // z block of the row
                const float x = in ? band::axis_at(p.ax[0], i - zb * p.xn) : 0.0f;
                const float zs = static_cast<float>(zb) * p.zstep;
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int j = in ? prep_slot(p, c * kGModes + quad * 4 + m) : -1;
                    float cs = 0.0f, sn = 0.0f;
                    if (j >= 0) {
                        const float4 c0 = __ldg(p.cold + 2 * j);
                        float t = turns_axis(c0.x, c0.y, x);
                        if (zb > 0) {
                            const float4 c1 = __ldg(p.cold + 2 * j + 1);
                            t = frac_turn(t + turns_axis(c1.x, c1.y, zs));
                        }
                        sincospif(2.0f * t, &sn, &cs);
                    }
                    v[2 * m] = cs;
                    v[2 * m + 1] = -sn;
                }
            } else {
                const bool in = i < p.ny;
                const float y = in ? band::axis_at(p.ax[1], i) : 0.0f;
                const float z = has_z ? band::axis_at(p.ax[2], 0) : 0.0f;
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int j = in ? prep_slot(p, c * kGModes + quad * 4 + m) : -1;
                    float cs = 0.0f, sn = 0.0f;
                    if (j >= 0) {
                        const float4 c0 = __ldg(p.cold + 2 * j);
                        const float4 c1 = __ldg(p.cold + 2 * j + 1);
                        const float tz = psi_z_turns(c1, z, has_z);
                        sincospif(2.0f * frac_turn(turns_axis(c0.z, c0.w, y) + tz), &sn, &cs);
                        const float amp = prep_amp(p, j, c0, c1, s_inv);
                        cs *= amp;
                        sn *= amp;
                    }
                    v[2 * m] = cs;
                    v[2 * m + 1] = sn;
                }
            }
            uint4 H, L;
            tc::split_f16x2(v[0], v[1], H.x, L.x);
            tc::split_f16x2(v[2], v[3], H.y, L.y);
            tc::split_f16x2(v[4], v[5], H.z, L.z);
            tc::split_f16x2(v[6], v[7], H.w, L.w);
            unsigned char* o = (is_a ? p.atab : p.btab) + static_cast<int64_t>(rest) * kGPair + tile_off(r, quad);
            *reinterpret_cast<uint4*>(o) = H;
            *reinterpret_cast<uint4*>(o + kGOpBytes) = L;
        } else {
            const bool is_y = idx < nA + nY;
            const I u = is_y ? idx - nA : idx - nA - nY;  // (chunk, k or l, m)
            const int m = static_cast<int>(u % kGModes);
            const I row = u / kGModes;
            const I n = static_cast<I>(is_y ? p.ny : p.nz);
            const int c = static_cast<int>(row / n);
            const int k = static_cast<int>(row - static_cast<I>(c) * n);
            const int j = prep_slot(p, c * kGModes + m);
            float cs = 0.0f, sn = 0.0f;
            if (j < 0) {
                (is_y ? p.ytab : p.wztab)[static_cast<int64_t>(row) * (kGRowBytes / 8) + m] = make_float2(0.0f, 0.0f);
                continue;
            }
            const float4 c0 = __ldg(p.cold + 2 * j);
            if (is_y) {
                sincospif(2.0f * turns_axis(c0.z, c0.w, band::axis_at(p.ax[1], k)), &sn, &cs);
                p.ytab[static_cast<int64_t>(row) * (kGRowBytes / 8) + m] = make_float2(cs, sn);
            } else {
                const float4 c1 = __ldg(p.cold + 2 * j + 1);
                const float amp = prep_amp(p, j, c0, c1, s_inv);
                sincospif(2.0f * psi_z_turns(c1, has_z ? band::axis_at(p.ax[2], k) : 0.0f, has_z), &sn, &cs);
                p.wztab[static_cast<int64_t>(row) * (kGRowBytes / 8) + m] = make_float2(amp * cs, amp * sn);
            }
        }
    }
}

__device__ __forceinline__ void grid_prep(const GridPrep& p) {
    const int64_t n_pad = static_cast<int64_t>(p.nc) * kGModes;
    const int64_t nA = static_cast<int64_t>(p.n_mt) * p.nc * kGM * 8;
    const int64_t nY = p.form ? static_cast<int64_t>(p.ny) * n_pad : static_cast<int64_t>(p.n_kt) * p.nc * kGN * 8;
    const int64_t nW = p.form ? static_cast<int64_t>(p.nz) * n_pad : 0;
    if (nA + nY + nW < (int64_t(1) << 31))
        grid_prep_items(p, static_cast<uint32_t>(nA), static_cast<uint32_t>(nY), static_cast<uint32_t>(nW));
    else
        grid_prep_items(p, static_cast<uint64_t>(nA), static_cast<uint64_t>(nY), static_cast<uint64_t>(nW));
}

__global__ void __launch_bounds__(256) grid_prep_kernel(GridPrep p) {
    pdl_wait();
    grid_prep(p);
}

// A tiles of the light chunks: row = x cell of the tile, K = x nodes from the
// tile's first one, the cell's weights times lw.
__device__ __forceinline__ void light_prep(const BandDesc* b, const float* X, const int32_t* lstart,
                                           unsigned char* latab) {
    const BandAxis ax = b->ax[0];
    const int nl = b->cells.nl;
    const float lw = b->lw;
    const uint32_t n = static_cast<uint32_t>(b->cells.n_mt) * nl * kGM * 8;
    for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
        const int seg = static_cast<int>(u & 7), r = static_cast<int>((u >> 3) & 127);
        const int rest = static_cast<int>(u >> 10);
        const int mt = rest / nl, lc = rest - mt * nl;
        const int i = mt * kGM + r;
        float v[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (i < b->cells.nx) {
            float w[band::kW];
            const int s = band::cell_weights(ax, __ldg(X + i), i, w) - (lstart[mt] + lc * kGK + 8 * seg);
            const int nt = band::taps(ax);
#pragma unroll
            for (int k = 0; k < band::kW; ++k)
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (k < nt && s + k == e) v[e] = w[k] * lw;
        }
        uint4 H, L;
        tc::split_f16x2(v[0], v[1], H.x, L.x);
        tc::split_f16x2(v[2], v[3], H.y, L.y);
        tc::split_f16x2(v[4], v[5], H.z, L.z);
        tc::split_f16x2(v[6], v[7], H.w, L.w);
        unsigned char* o = latab + static_cast<int64_t>(rest) * kGPair + tile_off(r, seg);
        *reinterpret_cast<uint4*>(o) = H;
        *reinterpret_cast<uint4*>(o + kGOpBytes) = L;
    }
}

struct SubTable {
    float4* hot;
    float4* cold;
    int32_t* kpref;
    const int32_t* table_kpref;
};

// Tables of a band-path call: those of the direct modes at the cells, those
// of the light modes at the nodes, whose sizes are the device's choice, and
// the light chunks' x weights.  `cells`, `nodes`: the host's part (table,
// table pointers, cell axes).
__device__ __forceinline__ void prep_sizes(GridPrep& p, const GridTiling& d) {
    p.nx = d.nx;
    p.ny = d.ny;
    p.nz = d.nz;
    p.nc = d.nc;
    p.n_mt = d.n_mt;
    p.n_kt = d.n_kt;
    p.form = d.form;
    p.scale = d.scale;
    p.xn = d.xn;
}
// Table of the direct modes for the kernels that take cells of any plan: the
// records of the listed slots (in table order, so still by decreasing |a|_1),
// zeros up to a whole chunk, and the prefix lengths of the extent buckets.
__device__ __forceinline__ void sub_table(const BandDesc* b, const GridPrep& p, const SubTable& o) {
    const int n = (b->nh + kChunk - 1) / kChunk * kChunk;
    const int step = gridDim.x * blockDim.x;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += step) {
        const int s = p.idx[j];
        const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        o.hot[j] = s >= 0 ? __ldg(p.hot + s) : zero;
        o.cold[2 * j] = s >= 0 ? __ldg(p.cold + 2 * s) : zero;
        o.cold[2 * j + 1] = s >= 0 ? __ldg(p.cold + 2 * s + 1) : zero;
    }
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < kBuckets; k += step) {
        const int before = __ldg(o.table_kpref + k);  // slots below this one; how many are listed
        int lo = 0, hi = b->nh;
        while (lo < hi) {
            const int mid = (lo + hi) / 2;
            if (p.idx[mid] < before)
                lo = mid + 1;
            else
                hi = mid;
        }
        o.kpref[k] = lo;
    }
}

__global__ void __launch_bounds__(256) band_prep_kernel(const BandDesc* b, GridPrep cells, GridPrep nodes,
                                                        const int32_t* lstart, unsigned char* latab, SubTable sub) {
    pdl_wait();
    if (sub.hot != nullptr) sub_table(b, cells, sub);
    if (b->nh > 0 && cells.atab != nullptr) {
        prep_sizes(cells, b->cells);
        grid_prep(cells);
    }
    if (b->n_light == 0) return;
    prep_sizes(nodes, b->nodes);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const BandAxis a = b->ax[c];
        if (!a.ident) nodes.ax[c] = AxisSrc{nullptr, a.h, a.n0};
        nodes.gain_h[c] = a.ident ? 0.0f : a.h;
    }
    nodes.zstep = static_cast<float>(b->nodes.lz) * b->ax[2].h;
    grid_prep(nodes);
    if (b->cells.nl > 0) light_prep(b, cells.ax[0].p, lstart, latab);
}

// Mode-split grids: per cell the partial fields of the splits, added in split
// order (a fixed order), plus mu, then the maps; with the mismatch bit every
// block also writes its sum of (K - T)^2 to lpart.
__global__ void __launch_bounds__(256) grid_split_finalize(const float* part, int n_split, int64_t n,
                                                           MapDev map) {
    pdl_wait();
    const int64_t o = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const bool mm = (map.bits & kMapMismatch) != 0;
    double l = 0.0;
    if (o < n) {
        float s = 0.0f, e = 0.0f;
        float v[kGMaxSplit];  // all splits' loads in flight
#pragma unroll
        for (int k = 0; k < kGMaxSplit; ++k) v[k] = k < n_split ? part[static_cast<int64_t>(k) * n + o] : 0.0f;
#pragma unroll
        for (int k = 0; k < kGMaxSplit; ++k) two_sum_acc(s, e, v[k]);
        const float y = (s + e) + map.mu;
        map_store(map, o, y);
        if (mm) l = mismatch_store(map, o, y);
    }
    if (mm) {
        __shared__ double red[8];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = l;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < 8; ++w) t += red[w];
            map.lpart[blockIdx.x] = t;
        }
    }
}

// D[128][128] = sum_K A[128][K] B[128][K] (FP16 inputs, K-contiguous rows,
// K = 64 k_chunks, FP32 result row-major) through the same layout,
// descriptors and TMEM path as the grid kernel.  One CTA of 128 threads.
__global__ void __launch_bounds__(128, 1) mma_probe_kernel(const uint16_t* A, const uint16_t* B, int32_t k_chunks,
                                                             float* D, int32_t* status) {
    __shared__ __align__(1024) unsigned char sm_raw[2 * kGOpBytes + 1024];
    // operand tiles on a 1024-byte boundary of the shared window (swizzle atoms)
    unsigned char* sm = sm_raw + ((1024u - (smem_u32(sm_raw) & 1023u)) & 1023u);
    __shared__ uint64_t bar;
    __shared__ uint32_t slot;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    if (warp == 0) tc::alloc(&slot, 128);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = slot;
    const int K = kGK * k_chunks;
    bool ok = true;
    for (int ch = 0; ch < k_chunks; ++ch) {
        // canonical layout of the 128 x 64 chunk of A and of B
        for (int e = threadIdx.x; e < kGM * kGK; e += blockDim.x) {
            const int r = e / kGK, kk = e % kGK;
            const uint32_t off = tile_off(r, kk >> 3) + static_cast<uint32_t>(kk & 7) * 2u;
            *reinterpret_cast<uint16_t*>(sm + off) = A[static_cast<int64_t>(r) * K + ch * kGK + kk];
            *reinterpret_cast<uint16_t*>(sm + kGOpBytes + off) = B[static_cast<int64_t>(r) * K + ch * kGK + kk];
        }
        fence_proxy_async_smem();
        __syncthreads();
        if (threadIdx.x == 0) {
            tc::fence_after();
            const uint32_t sa = smem_u32(sm);
            for (int ks = 0; ks < kGK / 16; ++ks) {
                const uint32_t ko = static_cast<uint32_t>(ks) * kGKStep;
                tc::mma_f16(tbase, tc::smem_desc_sw128(sa + ko, kGSbo), tc::smem_desc_sw128(sa + kGOpBytes + ko, kGSbo),
                            tc::idesc_f16_f32(kGM, kGN), (ch | ks) != 0 ? 1u : 0u);
            }
            tc::commit(&bar);
        }
        if (!mbar_wait_bounded(&bar, static_cast<uint32_t>(ch) & 1u)) {
            if (threadIdx.x == 0) atomicOr(status, 2);
            ok = false;
        }
        tc::fence_after();
        __syncthreads();  // the chunk's shared data is no longer read
        if (!ok) break;
    }
    if (ok) {
        for (int cb = 0; cb < kGN; cb += 32) {
            uint32_t r[32];
            tc::ld32(tbase + (static_cast<uint32_t>(32 * warp) << 16) + cb, r);
            tc::wait_ld();
            const int row = 32 * warp + lane;
            for (int c = 0; c < 32; ++c) D[row * kGN + cb + c] = __uint_as_float(r[c]);
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after();
        tc::dealloc(tbase, 128);
    }
}

int g_num_sms = 0;

}  // namespace

// Most nodes of a lattice for n cells of any plan.
int64_t cells_band_cap(int64_t n) { return std::max<int64_t>(n, 65536); }

namespace {

int32_t chunks_of(int64_t n_pad) { return static_cast<int32_t>(n_pad / kGModes); }
int64_t table_bytes(const GridPlan& g) { return g.a_bytes + g.y_bytes + g.w_bytes + g.b_bytes; }

// One list of table slots.
int64_t idx_bytes(const GridPlan& g) { return align256((int64_t(g.nc) * kGModes + 128) * 4); }

// Workspace of a band-path call after the grid path's own: the descriptor,
// the modes' lists, the x tiles' first nodes, the nodes' tables (those of a
// grid of as many y and z cells, with cap_mt row tiles), the light chunks, the nodes' partial sums, the (x, y)
// nodes at the z cells and the rows of x nodes at the (y, z) cells.
struct BandLayout {
    int64_t off_idx, off_lstart, off_tab, off_latab, off_part, off_mid, off_rows, total;
    int64_t cap_nodes, cap_part, cap_mid;
    int32_t cap_mt, cap_nl;
};
// All of it stays, with the grid path's own part, within ws_most.  Two parts
// give way: the nodes' x operand, down to a quarter of the cells' row tiles,
// and the light chunks' operand tiles, which have a row per cell and a column
// per x node that its tile of 128 cells reads.  That is at most all of them,
// quadratic in the x axis (65 536 x 16 x 16 cells: 17 GB), but 140 on an evenly
// spaced axis in order: at least 3 chunks of 64; a call whose tiles read more
// than there is room for sums all modes directly.
constexpr int64_t kMinLight = 3;
BandLayout band_layout(const GridGeom& gg, const GridPlan& g) {
    const int64_t n = int64_t(gg.nx) * gg.ny * gg.nz;
    BandLayout L{};
    L.cap_nodes = n / 4;
    L.cap_part = n;
    L.cap_mid = n / 2;
    L.off_idx = align256(sizeof(BandDesc));
    L.off_lstart = L.off_idx + 2 * idx_bytes(g);
    L.off_tab = L.off_lstart + align256(int64_t(g.n_mt) * 4);
    const int64_t yz = table_bytes(g) - g.a_bytes;
    const int64_t part = align256(L.cap_part * 4);
    const int64_t mid = g.form ? align256(L.cap_mid * 4) : g.max_split > 1 ? 0 : align256(n * 4);
    const int64_t rows = align256((int64_t(gg.nx) + 3) * gg.ny * gg.nz * 4);
    const int64_t tile = int64_t(g.nc) * kGPair, chunk = int64_t(g.n_mt) * kGPair;
    const int64_t chunks = g.form ? (gg.nx + 3 + kGK - 1) / kGK : 0;  // the most an x tile can read
    const int64_t left = ws_most(n) - (table_bytes(g) + g.part_bytes) - (L.off_tab + yz + part + mid + rows);
    // row tiles of the nodes: several z blocks of few x nodes, within 64 MB of tables
    const int64_t mt = std::max<int64_t>(g.n_mt, std::min<int64_t>(8, (int64_t(64) << 20) / tile));
    L.cap_mt = static_cast<int32_t>(std::min(mt, (left - std::min(chunks, kMinLight) * chunk) / tile));
    if (L.cap_mt < (g.n_mt + 3) / 4) return L;  // total 0: not offered
    L.cap_nl = static_cast<int32_t>(std::min(chunks, (left - L.cap_mt * tile) / chunk));
    L.off_latab = L.off_tab + yz + L.cap_mt * tile;
    L.off_part = L.off_latab + L.cap_nl * chunk;
    L.off_mid = L.off_part + part;
    L.off_rows = L.off_mid + mid;
    L.total = L.off_rows + rows;
    return L;
}

// What the selection may choose, from what the layout holds: the rows of the
// x operand; the y and z tables have a row per cell.
void set_limits(BandSelect& s, const BandLayout& L) {
    s.cap_nodes = L.cap_nodes;
    s.cap_part = L.cap_part;
    s.cap_mid = L.cap_mid;
    s.cap_mt = L.cap_mt;
    s.cap_nl = L.cap_nl;
    s.cap_ax[0] = L.cap_mt * kGM;
    s.cap_ax[1] = s.cap_ax[2] = INT32_MAX;
}

// Sizes at which a call on a grid may take the band path: the selection's
// modes, at least half a finalize block of x cells and 4 rows per block (its
// loss partials), and a direct sum of at least 50 us, below which the lattice's
// kernels cost more than they save (512^2 x 4096: 48 us directly, 56 with it).
constexpr double kBandMinUs = 50.0;
bool band_sizes(int32_t nx, int32_t ny, int32_t nz, int64_t n_pad) {
    return n_pad <= band::kMaxModes && nx >= 32 && ny >= 8 &&
           grid_us_per_mode(nx, ny, nz) * double(n_pad) >= kBandMinUs;
}

// SM count and shared-memory limits of the tensor-core kernels, once.
int grid_init() {
    if (g_num_sms != 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    auto allow = [&](const void* kern, int bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    allow(reinterpret_cast<const void*>(grid_mma_kernel<false>), kGSmemMax);
    allow(reinterpret_cast<const void*>(grid_mma_kernel<true>), kGSmemMax);
    allow(reinterpret_cast<const void*>(grid_band_kernel<true>), kGBandSmem);
    allow(reinterpret_cast<const void*>(grid_band_kernel<false>), kGBandSmem);
    if (e == cudaSuccess) g_num_sms = sms;
    return e;
}

// Table pointers of one synthesis at `w`.
void set_tables(GridPrep& p, GridDesc& d, const GridPlan& g, unsigned char* w) {
    p.atab = w;
    if (g.form) {
        p.ytab = reinterpret_cast<float2*>(w + g.a_bytes);
        p.wztab = reinterpret_cast<float2*>(w + g.a_bytes + g.y_bytes);
    } else {
        p.btab = w + g.a_bytes;
    }
    d.atab = p.atab;
    d.btab = p.btab;
    d.ytab = p.ytab;
    d.wztab = p.wztab;
}

int launch_band(const GridPrep& p, const GridDesc& d, const GridGeom& gg, const GridPlan& gp, int64_t n_modes,
                unsigned char* w, int32_t fc, int32_t* status, cudaStream_t st) {
    const BandLayout L = band_layout(gg, gp);
    BandDesc* b = reinterpret_cast<BandDesc*>(w);
    float* part = reinterpret_cast<float*>(w + L.off_part);
    float* mid = reinterpret_cast<float*>(w + L.off_mid);
    float* rows = reinterpret_cast<float*>(w + L.off_rows);
    unsigned char* latab = w + L.off_latab;
    // 3-D grids of many tiles add the light modes as chunks of the direct
    // sum's product; the others leave partial sums to the finalize kernel
    const bool split = gp.max_split > 1 || !gp.form;
    GridPrep pc = p, pn = p;
    BandSelect s{};
    s.hot = p.hot;
    s.cold = p.cold;
    s.n_modes = static_cast<int32_t>(n_modes);
    s.dim = p.dim;
    s.idx_h = reinterpret_cast<int32_t*>(w + L.off_idx);
    s.idx_l = reinterpret_cast<int32_t*>(w + L.off_idx + idx_bytes(gp));
    s.seg = gg.seg;
    s.status = status;
    s.X = gg.X;
    s.n[0] = gg.nx;
    s.n[1] = gg.ny;
    s.n[2] = gg.nz;
    s.us_mode = static_cast<float>(grid_us_per_mode(gg.nx, gg.ny, gg.nz));
    s.us_node = static_cast<float>(kBandNodeUs);
    s.us_fixed = static_cast<float>(kBandFixedUs);
    s.us_heavy = 12.0f;
    set_limits(s, L);
    s.fold = fc;
    s.n_mt = gp.n_mt;
    s.lstart = split ? nullptr : reinterpret_cast<int32_t*>(w + L.off_lstart);
    s.max_split = gp.max_split;
    s.split_cells = split ? 1 : 0;
    s.chunk = kGModes;
    s.loss_nb_tiles = d.t.n_tiles * kGEpiWarps;
    s.loss_nb_finalize = band_finalize_blocks(gg);
    s.thdr = p.thdr;
    pc.idx = s.idx_h;
    pn.idx = s.idx_l;
    s.cells = d.t;
    GridDesc dn = d, dc = d;
    GridPlan gn = gp;
    gn.a_bytes = align256(int64_t(L.cap_mt) * gp.nc * kGPair);
    set_tables(pn, dn, gn, w + L.off_tab);
    dn.part = part;
    dn.quiet = 1;
    // 2-D grids of many tiles: one slice of partial sums, in `mid` (2-D has no other use for it)
    if (split && dc.part == nullptr) dc.part = mid;
    dc.latab = latab;
    dc.lstart = s.lstart;
    dc.light = rows;
    unsigned long long* tiles = nullptr;
    cudaError_t e = cudaGetSymbolAddress(reinterpret_cast<void**>(&tiles), g_grid_tiles);
    if (e != cudaSuccess) return e;
    int rc = launch_band_select(s, b, st);
    if (rc != cudaSuccess) return rc;
    e = launch_chained(band_prep_kernel, g_num_sms * 5, 256, 0, st, b, pc, pn, s.lstart, latab, SubTable{});
    if (e == cudaSuccess)
        e = launch_chained(grid_band_kernel<true>, g_num_sms, kGThreads, kGBandSmem, st, dn, &b->nodes, status);
    if (e != cudaSuccess) return e;
    rc = launch_band_lines(b, part, gg, mid, split ? nullptr : rows, g_num_sms, st);
    if (rc != cudaSuccess) return rc;
    const unsigned grid = static_cast<unsigned>(std::min<int64_t>(d.t.n_tiles * gp.max_split, g_num_sms));
    e = launch_chained(split ? grid_band_kernel<true> : grid_band_kernel<false>, grid, kGThreads, kGBandSmem, st, dc,
                       &b->cells, status);
    if (e != cudaSuccess) return e;
    rc = launch_band_finalize(b, gp.form ? mid : part, dc.part, gg, d.map, tiles, g_num_sms, st);
    if (rc != cudaSuccess) return rc;
    if (d.map.bits & kMapMismatch)
        return launch_loss_sum(d.map.lpart, 0, &b->loss_nb, d.map.inv_n_mean, d.map.loss, st);
    return cudaGetLastError();
}

// Workspace of a band-path call at the cells of any plan: the descriptor, the
// modes' lists, the nodes' tables, the direct modes' table, the nodes' partial
// sums and the light modes' sums at the cells.
struct CellsLayout {
    int64_t off_idx, idx, off_tab, a_bytes, y_bytes, w_bytes, b_bytes, off_hot, off_cold, off_kpref, off_part, off_add,
        total;
    int64_t cap_nodes, cap_part;
    int32_t cap_mt, cap_yz;
};
CellsLayout cells_layout(int64_t n, int64_t n_pad, int32_t dim) {
    CellsLayout L{};
    const int64_t nc = n_pad / kGModes;
    // a node costs about a fifth of a cell; axes of up to four times a cube's
    // (2-D: a square's)
    L.cap_nodes = cells_band_cap(n);
    L.cap_part = std::max<int64_t>(L.cap_nodes, int64_t(1) << 22);
    // within the bound on the workspace: 8 bytes per node and mode and operand,
    // tiles of 128 nodes
    const double side = std::pow(double(L.cap_nodes), 1.0 / dim);
    const int64_t fixed = n_pad * 60 + L.cap_part * 4 + n * 4 + 65536;
    const int64_t per_node = dim > 2 ? n_pad * 8 + 2 * nc * kGRowBytes : n_pad * 16;
    L.cap_yz = static_cast<int32_t>(std::min({4096.0, 4.0 * side, double((ws_most(n) - fixed) / per_node - kGM - 16)})) + 16;
    if (L.cap_yz < 64) return L;  // total 0: not offered
    L.cap_mt = static_cast<int32_t>((L.cap_yz + kGM - 1) / kGM);
    int64_t off = 0;
    auto take = [&](int64_t bytes) {
        const int64_t o = off;
        off += align256(bytes);
        return o;
    };
    take(sizeof(BandDesc));
    L.idx = align256((n_pad + 128) * 4);
    L.off_idx = take(2 * L.idx);
    L.a_bytes = align256(int64_t(L.cap_mt) * nc * kGPair);
    L.y_bytes = dim > 2 ? align256(nc * L.cap_yz * kGRowBytes) : 0;
    L.w_bytes = L.y_bytes;
    L.b_bytes = dim > 2 ? 0 : align256((L.cap_yz + kGN - 1) / kGN * nc * kGPair);
    L.off_tab = take(L.a_bytes + L.y_bytes + L.w_bytes + L.b_bytes);
    L.off_hot = take((n_pad + kChunk) * 16);
    L.off_cold = take((n_pad + kChunk) * 32);
    L.off_kpref = take(kBuckets * 4);
    L.off_part = take(L.cap_part * 4);
    L.off_add = take(n * 4);
    L.total = off;
    return L;
}

void set_limits(BandSelect& s, const CellsLayout& L) {
    s.cap_nodes = L.cap_nodes;
    s.cap_part = L.cap_part;
    s.cap_mt = L.cap_mt;
    s.cap_ax[0] = L.cap_mt * kGM;
    s.cap_ax[1] = s.cap_ax[2] = L.cap_yz;
}

}  // namespace

LatticeRoom cells_room(int64_t n, int64_t n_modes, int32_t dim) {
    LatticeRoom r{};
    const int64_t n_pad = pad_modes(n_modes), nc = n_pad / kGModes;
    r.bytes = static_cast<int64_t>(cells_band_ws_bytes(n, n_modes, dim));
    if (r.bytes == 0) return r;
    const CellsLayout L = cells_layout(n, n_pad, dim);
    BandSelect s{};
    set_limits(s, L);
    for (int c = 0; c < 3; ++c) r.limit[c] = c < dim ? s.cap_ax[c] : 1;
    r.held[0] = L.a_bytes / (nc * kGPair) * kGM;
    r.held[1] = dim > 2 ? L.y_bytes / (nc * kGRowBytes) : L.b_bytes / (nc * kGPair) * kGN;
    r.held[2] = dim > 2 ? L.w_bytes / (nc * kGRowBytes) : 1;
    r.nodes = s.cap_nodes;
    r.nodes_held = (L.off_add - L.off_part) / 4;
    return r;
}

LatticeRoom grid_room(int32_t nx, int32_t ny, int32_t nz, int64_t n_pad) {
    LatticeRoom r{};
    r.bytes = static_cast<int64_t>(grid_band_ws_bytes(nx, ny, nz, n_pad));
    if (r.bytes == 0) return r;
    const GridPlan g = grid_plan(nx, ny, nz, chunks_of(n_pad));
    const BandLayout L = band_layout(GridGeom{nx, ny, nz, nullptr, nullptr, nullptr, nullptr}, g);
    BandSelect s{};
    set_limits(s, L);
    const int64_t n[3] = {nx, ny, nz};
    for (int c = 0; c < 3; ++c) r.limit[c] = std::min<int64_t>(s.cap_ax[c], n[c]);
    r.held[0] = int64_t(L.cap_mt) * kGM;
    r.held[1] = g.form ? g.y_bytes / (g.nc * kGRowBytes) : g.b_bytes / (int64_t(g.nc) * kGPair) * kGN;
    r.held[2] = g.form ? g.w_bytes / (g.nc * kGRowBytes) : 1;
    r.nodes = s.cap_nodes;
    r.nodes_held = (L.off_mid - L.off_part) / 4;
    r.base = static_cast<int64_t>(grid_ws_bytes(nx, ny, nz, n_pad));
    return r;
}

size_t grid_ws_bytes(int32_t nx, int32_t ny, int32_t nz, int64_t n_pad) {
    const GridPlan g = grid_plan(nx, ny, nz, chunks_of(n_pad));
    return static_cast<size_t>(table_bytes(g) + g.part_bytes);
}

// Whole tiles, at the rate of the tensor-core kernel on large grids (65
// Tcell.mode/s in rounds of one tile per SM of 152) or of its mode-split form.
double grid_us_per_mode(int32_t nx, int32_t ny, int32_t nz) {
    const GridPlan g = grid_plan(nx, ny, nz, 4);
    const double tile = double(kGM) * kGN;
    return g.max_split > 1 ? double(g.n_tiles) * tile / 42.0e6 : std::ceil(double(g.n_tiles) / 152.0) * 152.0 * tile / 65.0e6;
}

bool grid_splits(int32_t nx, int32_t ny, int32_t nz) { return grid_plan(nx, ny, nz, 4).max_split > 1; }

// CUDA-core kernels: 4.2 Tcell.mode/s at the cells of any plan (one hardware
// cosine each), half of it at 30 000 cells, whose tiles leave SMs idle.  The lattice's interpolation: 50 ps per cell in 3-D, 10 in 2-D.
double cells_us_per_mode(int64_t n_cells) { return 0.006 + double(n_cells) / 4.2e6; }
double cells_band_us(int64_t n_cells, int32_t dim) { return 20.0 + double(n_cells) * (dim > 2 ? 5e-5 : 1e-5); }

// The same lower limit as on grids: 250 x 130 cells x 1000 modes (45 us
// directly) cannot pay for six more launches, 126 x 63 x 31 x 2048 (130 us) gains 50.
size_t cells_band_ws_bytes(int64_t n_cells, int64_t n_modes, int32_t dim) {
    const int64_t n_pad = pad_modes(n_modes);
    if (dim < 2 || n_pad > band::kMaxModes || cells_us_per_mode(n_cells) * double(n_pad) < kBandMinUs) return 0;
    return static_cast<size_t>(cells_layout(n_cells, n_pad, dim).total);
}

int launch_cells_band(const void* table, int64_t n_modes, FwdDesc& fd, const SegInfo* seg, void* ws,
                      int32_t max_split, int64_t loss_tiles, int64_t loss_finalize, int32_t* status, void* stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (const int e = grid_init()) return e;
    const TableLayout TL = table_layout(n_modes);
    const unsigned char* tb = static_cast<const unsigned char*>(table);
    unsigned char* w = static_cast<unsigned char*>(ws);
    const CellsLayout L = cells_layout(fd.n_cells, TL.n_pad, fd.dim);
    BandDesc* b = reinterpret_cast<BandDesc*>(w);
    float* part = reinterpret_cast<float*>(w + L.off_part);
    float* add = reinterpret_cast<float*>(w + L.off_add);
    GridPrep pc{};
    pc.thdr = reinterpret_cast<const TableHeader*>(tb);
    pc.hot = fd.hot;
    pc.cold = fd.cold;
    pc.idx = reinterpret_cast<int32_t*>(w + L.off_idx);
    pc.dim = fd.dim;
    GridPrep pn = pc;
    pn.idx = reinterpret_cast<int32_t*>(w + L.off_idx + L.idx);
    GridPlan gn{};
    gn.form = fd.dim > 2;
    gn.a_bytes = L.a_bytes;
    gn.y_bytes = L.y_bytes;
    GridDesc dn{};
    set_tables(pn, dn, gn, w + L.off_tab);
    dn.thdr = pc.thdr;
    dn.part = part;
    dn.quiet = 1;
    BandSelect s{};
    s.hot = fd.hot;
    s.cold = fd.cold;
    s.thdr = pc.thdr;
    s.n_modes = static_cast<int32_t>(n_modes);
    s.dim = fd.dim;
    s.idx_h = const_cast<int32_t*>(pc.idx);
    s.idx_l = const_cast<int32_t*>(pn.idx);
    s.seg = seg;
    s.status = status;
    s.us_mode = static_cast<float>(cells_us_per_mode(fd.n_cells));
    s.us_node = static_cast<float>(kBandNodeUs);
    s.us_fixed = static_cast<float>(cells_band_us(fd.n_cells, fd.dim));
    s.us_heavy = 5.0f;
    set_limits(s, L);
    s.fold = 1;  // as exact as the direct sum (3.0e-7 of sigma); 2 would save 9 of 370 us and give 3.0e-7 to 3.1e-7
    s.chunk = kChunk;
    s.max_split = max_split;
    s.loss_nb_tiles = loss_tiles;
    s.loss_nb_finalize = loss_finalize;
    SubTable sub;
    sub.hot = reinterpret_cast<float4*>(w + L.off_hot);
    sub.cold = reinterpret_cast<float4*>(w + L.off_cold);
    sub.kpref = reinterpret_cast<int32_t*>(w + L.off_kpref);
    sub.table_kpref = fd.kpref;
    int rc = launch_band_select(s, b, st);
    if (rc != cudaSuccess) return rc;
    cudaError_t e = launch_chained(band_prep_kernel, g_num_sms * 5, 256, 0, st, b, pc, pn, nullptr, nullptr, sub);
    if (e == cudaSuccess)
        e = launch_chained(grid_band_kernel<true>, g_num_sms, kGThreads, kGBandSmem, st, dn, &b->nodes, status);
    if (e != cudaSuccess) return e;
    rc = launch_band_lines(b, part, GridGeom{}, nullptr, nullptr, g_num_sms, st);
    if (rc != cudaSuccess) return rc;
    rc = launch_band_cells(b, part, fd.dim, fd.xs, fd.ys, fd.zs, fd.n_cells, add, st);
    if (rc != cudaSuccess) return rc;
    fd.hot = sub.hot;
    fd.cold = sub.cold;
    fd.kpref = sub.kpref;
    fd.band = b;
    fd.add = add;
    return cudaSuccess;
}

size_t grid_band_ws_bytes(int32_t nx, int32_t ny, int32_t nz, int64_t n_pad) {
    if (!band_sizes(nx, ny, nz, n_pad)) return 0;
    const GridGeom gg{nx, ny, nz, nullptr, nullptr, nullptr, nullptr};
    return static_cast<size_t>(band_layout(gg, grid_plan(nx, ny, nz, chunks_of(n_pad))).total);
}

int launch_synth_grid(const void* table, int64_t n_modes, int32_t dim, const GridGeom& gg, const MapDev& map,
                      void* ws, bool band, int32_t fc, int32_t* status, void* stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const unsigned char* tb = static_cast<const unsigned char*>(table);
    const TableLayout TL = table_layout(n_modes);
    if (const int e = grid_init()) return e;
    const GridPlan gp = grid_plan(gg.nx, gg.ny, gg.nz, chunks_of(TL.n_pad));
    unsigned char* w = static_cast<unsigned char*>(ws);
    GridPrep p{};
    p.thdr = reinterpret_cast<const TableHeader*>(tb);
    p.hot = reinterpret_cast<const float4*>(tb + TL.off_hot);
    p.cold = reinterpret_cast<const float4*>(tb + TL.off_cold);
    p.ax[0].p = gg.X;
    p.ax[1].p = gg.Y;
    p.ax[2].p = gg.Z;
    p.nx = gg.nx;
    p.ny = gg.ny;
    p.nz = gg.nz;
    p.nc = gp.nc;
    p.n_mt = gp.n_mt;
    p.n_kt = gp.n_kt;
    p.dim = dim;
    p.form = gp.form ? 1 : 0;
    p.xn = gg.nx;
    GridDesc d{};
    set_tables(p, d, gp, w);
    d.thdr = p.thdr;
    set_tiling(d.t, gp, gg.nx, gg.ny, gg.nz, fc);
    d.part = gp.max_split > 1 ? reinterpret_cast<float*>(w + table_bytes(gp)) : nullptr;
    d.map = map;
    if (band) return launch_band(p, d, gg, gp, n_modes, w + table_bytes(gp) + gp.part_bytes, fc, status, st);

    const int64_t items = int64_t(gp.n_mt) * gp.nc * kGM * 8 +
                          (gp.form ? (int64_t(gg.ny) + gg.nz) * TL.n_pad : int64_t(gp.n_kt) * gp.nc * kGN * 8);
    const int pb = 256;
    const int64_t pg = std::min<int64_t>((items + pb - 1) / pb, int64_t(g_num_sms) * 16);
    cudaError_t ce = launch_chained(grid_prep_kernel, static_cast<unsigned>(pg), pb, 0, st, p);
    const unsigned grid = static_cast<unsigned>(std::min<int64_t>(d.t.n_items, g_num_sms));
    if (ce == cudaSuccess)
        ce = launch_chained(d.t.n_split > 1 ? grid_mma_kernel<true> : grid_mma_kernel<false>, grid, kGThreads, gp.smem,
                            st, d, status);
    const int64_t n = int64_t(gg.nx) * gg.ny * gg.nz;
    const int64_t fin_blocks = (n + 255) / 256;
    if (ce == cudaSuccess && d.t.n_split > 1)
        ce = launch_chained(grid_split_finalize, static_cast<unsigned>(fin_blocks), 256, 0, st, d.part, d.t.n_split, n,
                            map);
    if (ce != cudaSuccess) return ce;
    if (map.bits & kMapMismatch) {
        const int e = launch_loss_sum(map.lpart, d.t.n_split > 1 ? fin_blocks : d.t.n_tiles * kGEpiWarps, nullptr,
                                      map.inv_n_mean, map.loss, st);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

int64_t grid_loss_partials(int32_t nx, int32_t ny, int32_t nz) {
    // at most: one per (tile, warp) without a split, one per finalize block with one
    const GridPlan g = grid_plan(nx, ny, nz, 4);
    return std::max<int64_t>(g.n_tiles * kGEpiWarps, (int64_t(nx) * ny * nz + 255) / 256);
}

int64_t grid_tiles(int32_t nx, int32_t ny, int32_t nz) { return grid_plan(nx, ny, nz, 4).n_tiles; }

int take_grid_tiles(unsigned long long* tiles) {
    unsigned long long v = 0ull;
    const unsigned long long zero = 0ull;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_grid_tiles, sizeof(v));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_grid_tiles, &zero, sizeof(zero));
    if (e != cudaSuccess) return e;
    *tiles = v;
    return cudaSuccess;
}

int launch_mma_probe(const uint16_t* A, const uint16_t* B, int32_t k_chunks, float* D, int32_t* status,
                     void* stream) {
    mma_probe_kernel<<<1, 128, 0, static_cast<cudaStream_t>(stream)>>>(A, B, k_chunks, D, status);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace grf
