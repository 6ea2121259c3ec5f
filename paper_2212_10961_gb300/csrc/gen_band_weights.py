"""Coefficients of the interpolation weights of the band-limited path.

The Kaiser-Bessel window of width W = 8 nodes (Kaiser and Schafer, "On the use
of the I0-sinh window for spectrum analysis", 1980),
    phi(t) = I0(beta sqrt(1 - (2 t / W)^2)) / I0(beta),  |t| <= W / 2,
with beta = 0.99 pi W (1 - xi), xi = 1/4 the largest frequency in turns per node (the factor puts the zero of the
nearest alias inside the band edge: the RMS aliasing error falls from 6.8e-7 to 1.6e-7),
divided by its integral phihat(0) = W sinh(beta) / (beta I0(beta)).  A cell at
u = v + 1/2 in [0, 1) between the nodes 3 and 4 of its eight takes the weight
phi(v + 7/2 - k) at node k; with p_k(v) that function for k = 0 .. 3 the other
four are p_{7-k}(v) = p_k(-v).  Each p_k is the least-squares polynomial of
degree 9 on Chebyshev nodes of [-1/2, 1/2], computed in FP64 and rounded to
FP32.  The script prints the coefficients, the error of their FP32 Horner
evaluation, and the aliasing error over the frequencies |xi| <= 1/4, RMS and largest over the positions.

Run: python gen_band_weights.py   (numpy and scipy)
"""
import numpy as np
from scipy.special import i0

W, XI, DEGREE = 8, 0.25, 9
BETA = 0.99 * np.pi * W * (1.0 - XI)


def transform(xi):
    """I0(beta) phihat(xi), the window's Fourier transform up to its normalisation (FP64, complex square root)."""
    z = np.sqrt(BETA ** 2 - (np.pi * W * np.asarray(xi, dtype=np.complex128)) ** 2 + 0j)
    z = np.where(np.abs(z) < 1e-6, 1e-6, z)
    return (W * np.sinh(z) / z).real


def phi(t):
    u = np.maximum(1.0 - (2.0 * t / W) ** 2, 0.0)
    return np.where(np.abs(t) <= W / 2, i0(BETA * np.sqrt(u)), 0.0) / transform(0.0)


def main():
    n = 4096
    v = 0.5 * np.cos(np.pi * (np.arange(n) + 0.5) / n)
    dense = np.linspace(-0.5, 0.5, 200_001)
    coefs = []
    for k in range(W // 2):
        c = np.polynomial.chebyshev.Chebyshev.fit(v, phi(v + 3.5 - k), DEGREE, domain=[-0.5, 0.5])
        coefs.append(c.convert(kind=np.polynomial.Polynomial).coef.astype(np.float32))
    # the mean over v of the sum of the weights is 1; rounding the coefficients
    # moved it by 3e-8, which would scale every interpolated value: node 1's
    # constant, of small magnitude, takes the difference
    x, wq = np.polynomial.legendre.leggauss(40)
    x, wq = 0.5 * x, 0.5 * wq
    total = 2.0 * sum(np.sum(wq * np.polyval(c[::-1].astype(np.float64), x)) for c in coefs)
    coefs[1][0] = np.float32(np.float64(coefs[1][0]) + 0.5 * (1.0 - total))
    for k, c in enumerate(coefs):
        acc = np.full(dense.shape, c[-1], dtype=np.float32)
        for q in c[-2::-1]:
            acc = (acc * dense.astype(np.float32) + q).astype(np.float32)
        err = np.max(np.abs(acc - phi(dense.astype(np.float32).astype(np.float64) + 3.5 - k)))
        print("{%s},  // node %d: %.1e" % (", ".join("%.9ef" % q for q in c), k, err))
    xi = np.linspace(0.0, XI, 1001)
    # relative error of a mode e^{2 pi i xi t} at position t: its aliases'
    # sum_{m != 0} r_m e^{2 pi i m t}, r_m = phihat(xi + m) / phihat(xi)
    ratios = {m: transform(xi + m) / transform(xi) for m in range(-200, 201) if m}
    rms = np.sqrt(sum(r ** 2 for r in ratios.values()))
    t = np.linspace(0.0, 1.0, 2001)
    most = np.array([np.max(np.abs(sum(r[i] * np.exp(2j * np.pi * m * t) for m, r in ratios.items())))
                     for i in range(0, 1001, 20)])
    print("beta = %.9f, gain at xi: %.4f, aliasing error over the positions: RMS at most %.2e (%.2e at xi / 2), largest "
          "%.2e (%.2e)" % (BETA, transform(0.0) / transform(XI), np.max(rms), rms[500], np.max(most), most[25]))
    # in 3-D at a corner of the band the axes' errors add: three times the
    # largest, sqrt(3) times the RMS
    print("3-D corner: RMS %.2e, largest %.2e" % (np.sqrt(3.0) * np.max(rms), 3.0 * np.max(most)))


if __name__ == "__main__":
    main()
