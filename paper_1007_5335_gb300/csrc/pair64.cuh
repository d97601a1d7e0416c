// The binary64 double-layer pair term from a table of Taylor polynomials.
//
// (1/alpha) K1(r/alpha) (d.n)/r = f(r^2) (d.n) / alpha^2 with f(rho) = K1(z)/z, z = sqrt(rho)/alpha
// (Section 3.2).  Evaluated from K1 itself a pair costs ~150 binary64 instructions (series or
// Clenshaw recurrence, exp, log, sqrt, divisions), and the binary64 pipe of this part issues one
// warp instruction in 16 cycles per SM: the pair sums are bound by that pipe.  As a function of
// rho the kernel is smooth between its singular point rho = 0 and the cut, so f is tabulated:
// every octave of rho is cut into equal bins (their number from the leading mantissa bits), each
// bin holds the 7 Taylor coefficients about its centre,
//   d^j/drho^j f = (-1/(2 alpha^2))^j K_{1+j}(z) / z^{1+j}
// (the derivative rule of z^{-n} K_n(z)).  A pair then takes 15 binary64 instructions: offsets
// 2, rho 2, t 1, Horner 6, dot product 2, accumulate 1, and no square root or division.
//   bins     128 an octave from rho = 2^-14 alpha^2 for 20 octaves (t/rho <= 1/256: the eighth
//            term is below 256^-7 = 1.4e-17 of f), 512 an octave for the six above, where f falls
//            like e^{-z} (z = 45: (z/2048)^7/7! = 4e-16); octaves start at a power of two, so
//            the two ranges reach past 2025 alpha^2 = (45 alpha)^2 whatever alpha is.
//   lookup   the bin is the top bits of rho's binary64 pattern, its centre the same bits with
//            half a bin added (integer pipe); 64 bytes per bin, four 16-byte loads from L1.
// Pairs nearer than the table (r < alpha/128) take K1 directly.
// Measured, starfish heat step in binary64 (5.6e7 near pairs, 4.2e7 upsampled, 1.5e7 trapezoid):
// 19.84 ms a step with K1 per pair, 5.03 ms with the table; u differs by 6e-17 (relative L2).
#pragma once

#include "bessel.cuh"

constexpr int PT_OCT = 20, PT_BITS = 7, PT_OCT_FAR = 6, PT_BITS_FAR = 9;
constexpr int PT_BINS = (PT_OCT << PT_BITS) + (PT_OCT_FAR << PT_BITS_FAR);   // 5632 bins, 352 KB

struct mh_pair_tab {
    const double2* c = nullptr;   // [PT_BINS][4]: coefficients 0..6, one entry of padding
    int hi0 = 0, hi1 = 0;         // high words of the first bin of the two ranges
    double inv_alpha = 0.0;
    double cut = 0.0;             // (45 alpha)^2: farther pairs are 0 (e^{-45} of the unit-distance value)
};

inline mh_pair_tab mh_pair_tab_make(const double2* c, double alpha) {
    mh_pair_tab T;
    T.c = c;
    const int e0 = std::ilogb(alpha * alpha) - 14;   // first octave: [2^e0, 2^(e0+1))
    T.hi0 = (e0 + 1023) << 20;
    T.hi1 = (e0 + PT_OCT + 1023) << 20;
    T.inv_alpha = 1.0 / alpha;
    T.cut = 2025.0 * alpha * alpha;
    return T;
}

// K1(z)/z for rho below the table (r < alpha/128; rho = 0 gives 0: the offset is 0 there).
static __device__ __noinline__ double mh_pair_near(double rho, double inv_alpha) {
    if (!(rho > 0.0)) return 0.0;
    const double z = sqrt(rho) * inv_alpha;
    return mh_k1(z) / z;
}

// f(rho) = K1(z)/z, z = sqrt(rho)/alpha; 0 beyond the cut.
__device__ __forceinline__ double mh_pair_f(double rho, const mh_pair_tab& T) {
    if (!(rho <= T.cut)) return rho > T.cut ? 0.0 : rho;   // beyond the cut; not a number stays one
    const int hi = __double2hiint(rho);
    if (hi < T.hi0) return mh_pair_near(rho, T.inv_alpha);
    const bool far = hi >= T.hi1;
    const int sh = far ? 20 - PT_BITS_FAR : 20 - PT_BITS;
    const int bin = ((hi - (far ? T.hi1 : T.hi0)) >> sh) + (far ? PT_OCT << PT_BITS : 0);
    const double t = rho - __hiloint2double((hi >> sh << sh) | (1 << (sh - 1)), 0);
    const double2* c = T.c + 4 * bin;
    const double2 a = __ldg(c), b = __ldg(c + 1), d = __ldg(c + 2), e = __ldg(c + 3);
    double v = fma(e.x, t, d.y);
    v = fma(v, t, d.x);
    v = fma(v, t, b.y);
    v = fma(v, t, b.x);
    v = fma(v, t, a.y);
    return fma(v, t, a.x);
}

// Table entries for one alpha: a thread per bin, K_n by the (stable) forward recurrence.
static __global__ void k_pair_table(mh_pair_tab T, double alpha, double2* __restrict__ out) {
    const int bin = blockIdx.x * blockDim.x + threadIdx.x;
    if (bin >= PT_BINS) return;
    const bool far = bin >= (PT_OCT << PT_BITS);
    const int sh = far ? 20 - PT_BITS_FAR : 20 - PT_BITS;
    const int i = far ? bin - (PT_OCT << PT_BITS) : bin;
    const double rho = __hiloint2double((far ? T.hi1 : T.hi0) + (i << sh) + (1 << (sh - 1)), 0);
    const double z = sqrt(rho) / alpha, d = -0.5 / (alpha * alpha);
    double km = mh_k0(z), k = mh_k1(z), scale = 1.0 / z, c[8];
    c[7] = 0.0;
    for (int j = 0; j < 7; ++j) {   // c_j = (-1/(2 alpha^2))^j / j! K_{1+j}(z) / z^{1+j}
        c[j] = scale * k;
        const double kn = km + (2.0 * (j + 1) / z) * k;
        km = k;
        k = kn;
        scale *= d / (z * (j + 1));
    }
    for (int q = 0; q < 4; ++q) out[4 * bin + q] = make_double2(c[2 * q], c[2 * q + 1]);
}
