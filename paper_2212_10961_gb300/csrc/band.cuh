// Band-limited part of a spectral sum: modes of low frequency are summed on a
// coarse lattice of nodes and carried to the cells by interpolation.
//
// A mode whose phase advances by at most xi = 1/4 turn per node along every
// axis is, up to the aliasing error below, the interpolant of its own node
// values (Shannon's theorem with a compactly supported kernel; the gridding
// step of a non-uniform Fourier transform, Dutt and Rokhlin 1993, with the
// Kaiser-Bessel window of Jackson et al. 1991):
//     e^{2 pi i a x} = (1 / phihat(a h)) sum_n e^{2 pi i a n h} phi(x / h - n),
// phi of width W = 8 nodes per axis, separable over the axes.  So the modes of
// low frequency, with their amplitudes multiplied by the gains 1 / phihat, are
// summed at the nodes only, and every
// cell takes W^dim node values; the others are summed at the cells as before.
// The adjoint applies the same weights transposed.
//
// Error.  With beta = 0.99 pi W (1 - xi) the aliased copies of a mode along
// one axis are, relative to its amplitude, at most 1.6e-7 in RMS over the
// positions and 2.5e-7 at the worst one anywhere in the band, 3e-8 and 4e-8 at
// half of it (gen_band_weights.py).  The axes' errors add: at a corner of the
// band in 3-D 2.8e-7 in RMS, 7.5e-7 at worst.  Few modes lie there and their
// errors are unrelated, so that fields stay below the FP32 rounding of the
// direct sums (2.0e-7 to 3.5e-7 of sigma in RMS against 2.7e-7 to 4.1e-7).  Node coordinates
// n h are exact FP32 numbers (h has 8 significant bits, |n| < 2^16), so node
// phases are reduced exactly like cell phases, and x - n h is exact.
//
// Everything about the lattice (modes, spacings, sizes) is chosen on the device
// from the table and the cells' bounds by band_select_kernel, for each call:
// the table may be filled on the device's own time line, and nothing is
// remembered from one call to the next.
#pragma once

#include <cstdint>

#include "device_common.cuh"

namespace grf {
namespace band {

constexpr int kW = 8;                        // nodes per axis a cell reads
constexpr float kXi = 0.25f;                 // largest phase advance per node, turns
constexpr float kBeta = 18.661060363f;       // 0.99 pi W (1 - xi)
constexpr float kPiW = 25.132741229f;        // pi W
constexpr int kMaxModes = 65536;             // modes the selection handles (one block)
constexpr int kMaxNode = 65536;              // bound on |node index| (exact node coordinates)

// 1 / phihat(xi) relative to phihat(0), with sinh(z) / z taken as e^z / 2 z
// (z >= 17.5 in the band: the dropped e^-2z is below 1e-15).  With
// r = beta - z = q^2 / (beta + z), which carries no cancellation, it is
// e^r z / beta = e^r (1 - r / beta).
__device__ __forceinline__ float gain(float xi) {
    const float q = kPiW * xi;
    const float r = q * q / (kBeta + sqrtf(fmaf(-q, q, kBeta * kBeta)));
    return expf(r) * fmaf(-r, 1.0f / kBeta, 1.0f);
}

// ln(gain), and its derivative, in FP64.
__device__ __forceinline__ double log_gain(double xi) {
    const double q2 = 631.6546816697189 * xi * xi, beta = 18.661060362323371;  // (pi W)^2
    const double r = q2 / (beta + sqrt(beta * beta - q2));
    return r + log1p(-r / beta);
}
__device__ __forceinline__ double log_gain_slope(double xi) {
    const double pw = 25.132741228718345, beta = 18.661060362323371;
    const double z2 = beta * beta - pw * pw * xi * xi;
    const double z = sqrt(z2);
    return pw * pw * xi * (1.0 / z - 1.0 / z2);
}

// Weights of a cell at its eight nodes; v = (position between the nodes 3 and
// 4) - 1/2.  Even and odd parts of the polynomials of gen_band_weights.py,
// which give two nodes each.  FP32 error below 4e-8 of weights up to 0.436.
__device__ __forceinline__ void weights(float v, float (&w)[kW]) {
    const float c[4][10] = {
        {4.143404294e-05f, -3.294264607e-04f, 1.118412009e-03f, -2.120229416e-03f, 2.443167614e-03f,
         -1.705044066e-03f, 6.120222970e-04f, 1.789693124e-05f, -1.146915747e-04f, 3.663639291e-05f},
        {8.204627782e-03f, -2.957456186e-02f, 4.373614118e-02f, -3.193425387e-02f, 8.714604191e-03f,
         3.407949582e-03f, -3.191829193e-03f, 4.865803639e-04f, 3.132479906e-04f, -1.213801661e-04f},
        {1.155014858e-01f, -2.115766257e-01f, 1.120724156e-01f, 2.270347625e-02f, -4.075086862e-02f,
         6.638115738e-03f, 5.826086272e-03f, -2.039680956e-03f, -4.275149549e-04f, 2.610436641e-04f},
        {3.762524724e-01f, -2.150915563e-01f, -1.569276154e-01f, 1.064051464e-01f, 2.959774993e-02f,
         -2.506989613e-02f, -3.253627336e-03f, 3.746612463e-03f, 2.113322262e-04f, -3.795136290e-04f}};
    const float s = v * v;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float e = c[k][8], o = c[k][9];
#pragma unroll
        for (int q = 6; q >= 0; q -= 2) {
            e = fmaf(e, s, c[k][q]);
            o = fmaf(o, s, c[k][q + 1]);
        }
        w[k] = fmaf(v, o, e);
        w[kW - 1 - k] = fmaf(-v, o, e);
    }
}

__device__ __forceinline__ float axis_at(const AxisSrc& a, int64_t i) {
    return a.p != nullptr ? __ldg(a.p + i) : static_cast<float>(a.n0 + static_cast<int32_t>(i)) * a.h;
}

// First of the cell's eight nodes (index into the lattice, within it whatever
// x is) and the cell's offset for weights().
__device__ __forceinline__ int locate(const BandAxis& a, float x, float& v) {
    const float f = floorf(x * a.inv_h);
    v = fmaf(-f, a.h, x) * a.inv_h - 0.5f;
    return max(0, min(static_cast<int>(f) - (kW / 2 - 1) - a.n0, a.m - kW));
}

// Nodes that enter along an axis (fewer than kW on an axis that is not
// interpolated and has fewer cells), and the first node and weights of cell i
// at coordinate x.
__device__ __forceinline__ int taps(const BandAxis& a) { return a.m < kW ? a.m : kW; }
__device__ __forceinline__ int cell_weights(const BandAxis& a, float x, int i, float (&w)[kW]) {
    if (a.ident) {
        const int s = max(0, min(i, a.m - kW));
#pragma unroll
        for (int k = 0; k < kW; ++k) w[k] = k == i - s ? 1.0f : 0.0f;
        return s;
    }
    float v;
    const int s = locate(a, x, v);
    weights(v, w);
    return s;
}

}  // namespace band
}  // namespace grf
