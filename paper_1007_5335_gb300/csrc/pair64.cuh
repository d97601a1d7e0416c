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
// (the derivative rule of z^{-n} K_n(z)).
//   bins     128 an octave from rho = 2^-14 alpha^2 for 20 octaves (to z = 5.7 .. 8; |t/rho| <= 1/256 with t the
//            distance from the centre), 512 an octave for the six above, where f falls like e^{-z}
//            (1/1024); octaves start at a power of two, so the two ranges reach past 2025 alpha^2 =
//            (45 alpha)^2 whatever alpha is.
//   eighth   the first term left out, relative to f: at most 1.4e-17 for z <= 0.5, 4.2e-16 at z = 5.7, 1e-15 at
//            the cut, at the edges of a bin at the start of its octave; a 128th of that half way to the centre.
//   lookup   the bin is the top bits of rho's binary64 pattern; the bits below them, shifted up, are
//            the place in the bin, tau in [-1/2, 1/2) in units of its width (integer pipe, and one
//            subtraction).
//   terms    tau^0..3 in binary64; tau^4..6 together are at most 2.4e-10 of f for z <= 0.1, 4e-9 at z = 5.7 and
//            1.3e-8 at the cut (bin edges again), so their factor of tau^4 is formed in binary32 (1.4e-17,
//            2.4e-16, 8e-16 of f) and widened by its bits.
//   entries  the value at a centre carries the rounding of z = sqrt(rho)/alpha, z eps of e^{-z}, unless it is
//            corrected to first order (k_pair_table).
// Error of f against 30 digits, 30,000 distances over the whole range at alpha^2 = 1e-3, 2^-10 and 0.03 (rms /
// largest): table 1.2e-16 / 4.6e-16 for z < 1, 2.2e-16 / 8.4e-16 for 1 < z < 2, 1.5e-16 / 6.5e-16 above; K1 and
// its factors per pair 1.1 to 1.5e-16 / 5.6e-16, 2.6e-16 / 9.1e-16, and 2.9e-16 / 1.1e-15 (z < 5) rising to
// 2.3e-15 / 7.1e-15 (z > 20); seven binary64 coefficients the table's to three digits.
// 48 bytes per bin (four doubles, three floats, padding), three 16-byte loads from L1.
// A pair then takes 12 binary64 instructions: offsets 2, rho 2, tau 1, Horner 4, dot product 2,
// accumulate 1, and no comparison, conversion, square root or division.
// Pairs nearer than the table (r < alpha/128) take K1 directly.
// Measured, starfish heat step in binary64 (5.6e7 near pairs, 4.2e7 upsampled, 1.5e7 trapezoid):
// 19.84 ms a step with K1 per pair, 5.03 ms with seven binary64 coefficients (15 instructions; near
// field 14.8 -> 1.66 ms), 0.37 ms a step less with three of them in binary32.
#pragma once

#include <cstdint>
#include <cstring>

#include "bessel.cuh"

constexpr int PT_OCT = 20, PT_BITS = 7, PT_OCT_FAR = 6, PT_BITS_FAR = 9;
constexpr int PT_BINS = (PT_OCT << PT_BITS) + (PT_OCT_FAR << PT_BITS_FAR);   // 5632 bins, 264 KB
constexpr int PT_WORDS = 3;   // double2 per bin

struct mh_pair_tab {
    const double2* c = nullptr;   // [PT_BINS][PT_WORDS]
    int hi0 = 0, hi1 = 0;         // high words of the first bin of the two ranges
    int hi_cut = 0;               // high word of (45 alpha)^2: farther pairs are 0 (e^{-45} of the unit-distance value)
    double inv_alpha = 0.0;
};

// Outside 1e-150 < alpha < 1e150 or so the octaves leave the range of binary64 exponents: the table stays
// unused (hi0 above every number), every pair within the cut takes K1 directly.
inline mh_pair_tab mh_pair_tab_make(const double2* c, double alpha) {
    mh_pair_tab T;
    T.c = c;
    const double a2 = alpha * alpha, cut = std::fmin(2025.0 * a2, 1.7976931348623157e308);
    const bool ok = a2 >= 2.2250738585072014e-308 && a2 <= 1.7976931348623157e308;
    const int e0 = (ok ? std::ilogb(a2) : 0) - 14 + 1023;   // biased exponent of the first octave
    if (ok && e0 >= 1 && e0 + PT_OCT + PT_OCT_FAR <= 2046) {
        T.hi0 = e0 << 20;
        T.hi1 = (e0 + PT_OCT) << 20;
    } else {
        T.hi0 = T.hi1 = 0x7fffffff;
    }
    uint64_t bits;
    std::memcpy(&bits, &cut, 8);
    T.hi_cut = (int)(bits >> 32);
    T.inv_alpha = 1.0 / alpha;
    return T;
}

// Bin of a number with the high word hi, hi0 <= hi <= hi_cut.
__host__ __device__ __forceinline__ int mh_pair_bin(int hi, const mh_pair_tab& T) {
    const bool far = hi >= T.hi1;
    const int bits = far ? PT_BITS_FAR : PT_BITS;
    return ((hi - (far ? T.hi1 : T.hi0)) >> (20 - bits)) + (far ? PT_OCT << PT_BITS : 0);
}

// K1(z)/z for rho below the table (r < alpha/128; rho = 0 gives 0: the offset is 0 there).
static __device__ __noinline__ double mh_pair_near(double rho, double inv_alpha) {
    if (!(rho > 0.0)) return 0.0;
    const double z = sqrt(rho) * inv_alpha;
    return mh_k1(z) / z;
}

// f(rho) = K1(z)/z, z = sqrt(rho)/alpha; 0 beyond the cut; not a number stays one.
__device__ __forceinline__ double mh_pair_f(double rho, const mh_pair_tab& T) {
    const int hi = __double2hiint(rho), lo = __double2loint(rho);
    if (hi > T.hi_cut) return rho != rho ? rho : 0.0;
    if (hi < T.hi0) return mh_pair_near(rho, T.inv_alpha);
    const bool far = hi >= T.hi1;
    const int bits = far ? PT_BITS_FAR : PT_BITS;
    const int bin = mh_pair_bin(hi, T);
    const double2* c = T.c + PT_WORDS * bin;
    const double2 a = __ldg(c), b = __ldg(c + 1);
    const float4 q = __ldg(reinterpret_cast<const float4*>(c + 2));
    // the mantissa below the bin bits as a number in [1, 2)
    const int mh = (__funnelshift_l(lo, hi, bits) & 0xfffff) | 0x3ff00000;
    const double tau = __hiloint2double(mh, lo << bits) - 1.5;
    const float tf = __int_as_float((mh & 0xfffff) << 3 | 0x3f800000) - 1.5f;
    // (double)w by its bits (w = 0 or far below the smallest normal number comes out as some 1e-38)
    const unsigned w = __float_as_uint(fmaf(fmaf(q.z, tf, q.y), tf, q.x));
    const double h = __hiloint2double((int)((w & 0x80000000u) | (((w >> 3) & 0x0fffffffu) + (896u << 20))), (int)(w << 29));
    return fma(fma(fma(fma(h, tau, b.y), tau, b.x), tau, a.y), tau, a.x);
}

// Table entries for one alpha: a thread per bin, K_n by the (stable) forward recurrence.
static __global__ void k_pair_table(mh_pair_tab T, double alpha, double2* __restrict__ out) {
    const int bin = blockIdx.x * blockDim.x + threadIdx.x;
    if (bin >= PT_BINS || T.hi0 == 0x7fffffff) return;
    const bool far = bin >= (PT_OCT << PT_BITS);
    const int sh = far ? 20 - PT_BITS_FAR : 20 - PT_BITS;
    const int i = far ? bin - (PT_OCT << PT_BITS) : bin;
    const int first = (far ? T.hi1 : T.hi0) + (i << sh);
    const double lo = __hiloint2double(first, 0), width = 2.0 * (__hiloint2double(first + (1 << (sh - 1)), 0) - lo);
    const double rho = lo + 0.5 * width;
    const double z = sqrt(rho) / alpha, d = -0.5 * width / (alpha * alpha);
    // dz = sqrt(rho)/alpha - z: K1 falls like e^{-z}, so the rounding of z alone is z eps of an entry
    const double p = z * alpha, pe = fma(z, alpha, -p), q = p * p, qe = fma(p, p, -q);
    const double dz = (((rho - q) - qe) - 2.0 * p * pe) / (2.0 * p * alpha);
    double km = mh_k0(z), k = mh_k1(z), scale = 1.0 / z, c[7];
    for (int j = 0; j < 7; ++j) {   // c_j = (-width/(2 alpha^2))^j / j! K_{1+j}(z) / z^{1+j}
        const double kn = km + (2.0 * (j + 1) / z) * k;
        c[j] = j == 0 ? (k - dz * kn) / z : scale * k;   // (K1/z)' = -K2/z
        km = k;
        k = kn;
        scale *= d / (z * (j + 1));
    }
    out[PT_WORDS * bin] = make_double2(c[0], c[1]);
    out[PT_WORDS * bin + 1] = make_double2(c[2], c[3]);
    *reinterpret_cast<float4*>(out + PT_WORDS * bin + 2) = make_float4((float)c[4], (float)c[5], (float)c[6], 0.f);
}
