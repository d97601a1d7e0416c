// Binary64 contractions by reflection orbits.
//
// The binary64 pipe bounds the binary64 form of the multipole passes (dense products at 83 % of
// its rate), so what is left is to do fewer of them.  Every operator between two boxes depends on the
// offset of their centres and commutes with the reflections of the plane: with g a reflection in x,
// in y, or both,
//   T_{g d} = rho(g) T_d rho(g),
// where rho(g) permutes node values (node ix -> q - 1 - ix) and changes signs of expansion
// coefficients (a_n, b_n: y -> -y flips b_n; x -> -x takes a_n to (-1)^n a_n and b_n to -(-1)^n b_n).
// In a basis of components that are even or odd under both reflections ("class" c = odd in x + 2 odd
// in y) rho(g) is diagonal with the characters (-1)^(c.g), and the sources of one destination
// whose offsets are mirror images (up to four) share one product:
//   sum_g rho(g) T rho(g) x_g = sum_j T_ij X_{c(i)^c(j), j},   X_{c, j} = sum_g (-1)^(c.g) x_{g, j}.
// An offset on an axis (dx = 0 or dy = 0), or none, is its own image under a subgroup ("stab"):
// then T_ij vanishes unless c(i)^c(j) is even under it, which halves or quarters the product.
// Binary64 multiply-adds per box of a full list (p = 20, q = 8): M2L 27 x 1681 -> 18,300 (sums
// included), near tables of 9 equal neighbours 9 x 4096 -> 9,980, P2M and L2P 2624 -> 656.
// Expansions are the (a, b) components in class order; node values are transformed to even / odd
// sums and differences once per pass and back once at the end.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

// Components of a space in class order.
struct OrbSpace {
    int n = 0;
    int first[5] = {0, 0, 0, 0, 0};   // first component of each class
    std::vector<int32_t> perm;        // expansions: component in class order -> coefficient
    std::vector<int> a, b;            // node values: node column / row of the even or odd pair (a <= q - 1 - a)
    std::vector<int> cls;
};

inline OrbSpace orb_expansions(int p) {
    OrbSpace S;
    S.n = 2 * p + 1;
    for (int c = 0; c < 4; ++c) {
        S.first[c] = (int)S.perm.size();
        for (int n = 0; n <= p; ++n) {
            const int odd = n & 1;
            if (odd == c) S.perm.push_back(n == 0 ? 0 : 2 * n - 1);            // a_n: class odd
            if (n > 0 && (3 - odd) == c) S.perm.push_back(2 * n);              // b_n: class 3 (even), 2 (odd)
        }
        S.cls.resize(S.perm.size(), c);
    }
    S.first[4] = S.n;
    return S;
}

inline OrbSpace orb_nodes(int q) {
    OrbSpace S;
    S.n = q * q;
    const int even = (q + 1) / 2, odd = q / 2;
    for (int c = 0; c < 4; ++c) {
        S.first[c] = (int)S.a.size();
        for (int b = 0; b < ((c & 2) ? odd : even); ++b)
            for (int a = 0; a < ((c & 1) ? odd : even); ++a) {
                S.a.push_back(a);
                S.b.push_back(b);
            }
        S.cls.resize(S.a.size(), c);
    }
    S.first[4] = S.n;
    return S;
}

// Matrix of an operator (R x C row-major, nodes / coefficients in their plain order) in class order:
// rows H T (H: even sums and odd differences of node values), columns T H^-1.
inline std::vector<double> orb_operator(const double* T, int R, int C, const OrbSpace& rows, const OrbSpace& cols, int q) {
    std::vector<double> A((size_t)R * C), B((size_t)R * C);
    for (int r = 0; r < R; ++r)
        for (int c = 0; c < C; ++c) {
            const double* t = T + (size_t)r * C;
            if (!cols.perm.empty()) {
                A[(size_t)r * C + c] = t[cols.perm[c]];
                continue;
            }
            const int a = cols.a[c], b = cols.b[c], a2 = q - 1 - a, b2 = q - 1 - b;
            const double sx = (cols.cls[c] & 1) ? -1.0 : 1.0, sy = (cols.cls[c] & 2) ? -1.0 : 1.0;
            // u = H^-1: (even + odd) / 2 at the first node of a pair, (even - odd) / 2 at the second
            double v = t[b * q + a];
            if (a2 != a) v += sx * t[b * q + a2];
            double w = 0.0;
            if (b2 != b) {
                w = t[b2 * q + a];
                if (a2 != a) w += sx * t[b2 * q + a2];
            }
            v += sy * w;
            A[(size_t)r * C + c] = v * (a2 != a ? 0.5 : 1.0) * (b2 != b ? 0.5 : 1.0);
        }
    for (int r = 0; r < R; ++r)
        for (int c = 0; c < C; ++c) {
            if (!rows.perm.empty()) {
                B[(size_t)r * C + c] = A[(size_t)rows.perm[r] * C + c];
                continue;
            }
            const int a = rows.a[r], b = rows.b[r], a2 = q - 1 - a, b2 = q - 1 - b;
            const double sx = (rows.cls[r] & 1) ? -1.0 : 1.0, sy = (rows.cls[r] & 2) ? -1.0 : 1.0;
            auto at = [&](int bb, int aa) { return A[((size_t)bb * q + aa) * C + c]; };
            double v = at(b, a);
            if (a2 != a) v += sx * at(b, a2);
            if (b2 != b) {
                double w = at(b2, a);
                if (a2 != a) w += sx * at(b2, a2);
                v += sy * w;
            }
            B[(size_t)r * C + c] = v;
        }
    return B;
}

struct OrbDims {
    int nodes[5], exp[5];   // first component of each class, node values and expansions
};

// One operator in class order and the reflections that leave its offset alone (1: x, 2: y).
struct OrbOp {
    int64_t off;
    int32_t C, stab;
    int32_t nodes;     // columns are node values (class order already), else expansion coefficients
    int32_t pad;
};

// Task: up to four mirror-image sources of one destination (-1: none).
struct OrbSrc {
    int64_t at[4];
};

constexpr int ORB_TT = 8;        // tasks per thread, at most
constexpr int ORB_THREADS = 256;

// Words of an operator row or a source vector in shared memory: odd, so that the rows of a warp fall
// in distinct banks.
__host__ __device__ inline int orb_ld(int C) { return C | 1; }

inline size_t orb_smem(int R, int C, int groups, int characters) {
    return ((size_t)R + (size_t)characters * groups * ORB_TT) * orb_ld(C) * sizeof(double);
}

// Thread groups of a block (one row a thread, ORB_TT tasks a group): as many as two blocks on an SM
// allow, or one block where not even one group does.  0: the operator does not fit.
inline int orb_groups(int R, int C, int characters) {
    for (const size_t limit : {(size_t)112 * 1024, (size_t)200 * 1024})
        for (int g = std::min(8, ORB_THREADS / R); g >= 1; --g)
            if (orb_smem(R, C, g, characters) <= limit) return g;
    return 0;
}

// Products of TT tasks in one thread: row i (class ci) against the columns of class ci ^ c in the
// character sums c.
template <int TT>
__device__ __forceinline__ void orb_rows(const double* a, const double* z, int zs, int ld, int ci, const int* cf,
                                         int stab, double* acc) {
#pragma unroll
    for (int u = 0; u < TT; ++u) acc[u] = 0.0;
    for (int c = 0, slot = 0; c < 4; ++c) {
        if (c & stab) continue;
        const int k = ci ^ c, j0 = cf[k], j1 = cf[k + 1];
        const double* zc = z + slot * zs;
#pragma unroll 2
        for (int j = j0; j < j1; ++j) {
            const double av = a[j];
#pragma unroll
            for (int u = 0; u < TT; ++u) acc[u] = fma(av, zc[u * ld + j], acc[u]);
        }
        ++slot;
    }
}

// One block: one operator (R x C, class order) and up to ORB_TT tasks for each of its groups of R threads,
// shared evenly (a short chunk leaves no group idle).  The sources' character sums are formed as they are
// staged.  Products, expansions back in their plain order, go to temp[task][R], or with task_dst
// to dst[task_dst] (added when accumulate is set).  A task costs R C / |stab| multiply-adds of the
// binary64 pipe (a warp instruction holds its quarter of the SM for 64 clocks) and up to 8 C additions, 9 shared
// loads to 8 multiply-adds: the pipe is the bound.  A full chunk of the M2L (48 tasks, P = 41) takes
// its SM 25 us, so a phase with few tasks is cut finer (build_orbits).
// Against one product per source (4 rows x 4 tasks a thread): binary64 volume potential on 255 k nodes 553 ->
// 357 us (M2L 306 -> 196, output 94 -> 30), starfish step 4053 -> 3563 us (near tables 458 -> 120), step with curves of 64 nodes 468 -> 352 us, matrix-free solve at
// 12,288 nodes 3432 -> 3130 us.
__global__ void __launch_bounds__(ORB_THREADS) k_orbit(
    const double* __restrict__ ops, const OrbOp* __restrict__ op_of, const int32_t* __restrict__ chunk_op,
    const int32_t* __restrict__ chunk_t0, const OrbSrc* __restrict__ task_src, const int32_t* __restrict__ perm,
    OrbDims dims, int R, int row_nodes, int groups, const double* src, double* __restrict__ temp,
    const int64_t* __restrict__ task_dst, int accumulate, double* dst) {
    mh_dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int first[2][5];
    if (threadIdx.x == 0)
        for (int k = 0; k < 5; ++k) {
            first[0][k] = dims.exp[k];
            first[1][k] = dims.nodes[k];
        }
    const OrbOp op = op_of[chunk_op[blockIdx.x]];
    const int t0 = chunk_t0[blockIdx.x], nt = chunk_t0[blockIdx.x + 1] - t0;
    const int C = op.C, ld = orb_ld(C);
    const int tt = (nt + groups - 1) / groups;               // tasks per group = products a thread, 1 .. ORB_TT
    double* sA = reinterpret_cast<double*>(smem_raw);
    double* sZ = sA + R * ld;                                // [character][groups * tt][ld]
    const int zs = groups * tt * ld;
    stage_rows<double, double>(sA, ops + op.off, R * C, C, ld);
    {
        const int stride = blockDim.x, ne = nt * C;
        const int dc = stride % C, dt = stride / C;
        int c = (int)threadIdx.x % C, t = (int)threadIdx.x / C;
        for (int e = threadIdx.x; e < ne; e += stride) {
            const OrbSrc s = task_src[t0 + t];
            const int j = op.nodes ? c : perm[c];
            const double x0 = s.at[0] >= 0 ? src[s.at[0] + j] : 0.0, x1 = s.at[1] >= 0 ? src[s.at[1] + j] : 0.0;
            const double x2 = s.at[2] >= 0 ? src[s.at[2] + j] : 0.0, x3 = s.at[3] >= 0 ? src[s.at[3] + j] : 0.0;
            double* z = sZ + t * ld + c;
            if (op.stab == 3) {
                z[0] = x0;
            } else if (op.stab == 2) {        // sources at the offset and its x image
                z[0] = x0 + x1;
                z[zs] = x0 - x1;
            } else if (op.stab == 1) {        // sources at the offset and its y image
                z[0] = x0 + x2;
                z[zs] = x0 - x2;
            } else {
                const double a = x0 + x1, b = x0 - x1, r = x2 + x3, w = x2 - x3;
                z[0] = a + r;
                z[zs] = b + w;
                z[2 * zs] = a - r;
                z[3 * zs] = b - w;
            }
            c += dc;
            t += dt;
            if (c >= C) {
                c -= C;
                ++t;
            }
        }
    }
    __syncthreads();
    const int i = (int)threadIdx.x % R, g = (int)threadIdx.x / R;
    if (g >= groups || g * tt >= nt) return;
    const int* rf = first[row_nodes ? 1 : 0];
    const int* cf = first[op.nodes ? 1 : 0];
    const int ci = (i >= rf[1]) + (i >= rf[2]) + (i >= rf[3]);
    const double* a = sA + i * ld;
    const double* z = sZ + g * tt * ld;
    double acc[ORB_TT];
    switch (tt) {
        case 1: orb_rows<1>(a, z, zs, ld, ci, cf, op.stab, acc); break;
        case 2: orb_rows<2>(a, z, zs, ld, ci, cf, op.stab, acc); break;
        case 3: orb_rows<3>(a, z, zs, ld, ci, cf, op.stab, acc); break;
        case 4: orb_rows<4>(a, z, zs, ld, ci, cf, op.stab, acc); break;
        case 5: orb_rows<5>(a, z, zs, ld, ci, cf, op.stab, acc); break;
        case 6: orb_rows<6>(a, z, zs, ld, ci, cf, op.stab, acc); break;
        case 7: orb_rows<7>(a, z, zs, ld, ci, cf, op.stab, acc); break;
        default: orb_rows<8>(a, z, zs, ld, ci, cf, op.stab, acc);
    }
    const int r = row_nodes ? i : perm[i];
#pragma unroll
    for (int u = 0; u < ORB_TT; ++u) {
        const int t = g * tt + u;
        if (u >= tt || t >= nt) break;
        if (task_dst) {
            double* y = dst + task_dst[t0 + t] + r;
            *y = accumulate ? *y + acc[u] : acc[u];
        } else {
            temp[(int64_t)(t0 + t) * R + r] = acc[u];
        }
    }
}

// Node values (leaf-major, node iy q + ix) to even / odd components in class order, and back (added
// when accumulate is set).  Component k: pair columns (a, q - 1 - a), rows (b, q - 1 - b), class c in
// tab[k] = a | b << 8 | c << 16.
__global__ void k_orb_forward(const double* u, const int32_t* __restrict__ tab, int q, int64_t n, double* __restrict__ out) {
    mh_dep_wait();
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int qq = q * q, k = (int)(e % qq);
    const double* v = u + (e - k);
    const int w = tab[k], a = w & 255, b = (w >> 8) & 255, a2 = q - 1 - a, b2 = q - 1 - b;
    const bool ox = (w >> 16) & 1, oy = (w >> 17) & 1;
    double s = v[b * q + a], t = 0.0;
    if (a2 != a) s = ox ? s - v[b * q + a2] : s + v[b * q + a2];
    if (b2 != b) {
        t = v[b2 * q + a];
        if (a2 != a) t = ox ? t - v[b2 * q + a2] : t + v[b2 * q + a2];
        s = oy ? s - t : s + t;
    }
    out[e] = s;
}

// Inverse: node (ix, iy) from the four components of its pairs; at[c][b * q + a] = component.
__global__ void k_orb_back(const double* w, const int32_t* __restrict__ at, int q, int64_t n, int accumulate, double* u) {
    mh_dep_wait();
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int qq = q * q, k = (int)(e % qq), ix = k % q, iy = k / q;
    const double* v = w + (e - k);
    const int a = min(ix, q - 1 - ix), b = min(iy, q - 1 - iy);
    const bool px = a != q - 1 - a, py = b != q - 1 - b, fx = ix != a, fy = iy != b;   // paired; second of the pair
    double s[2] = {0.0, 0.0};
    for (int oy = 0; oy < 2; ++oy) {
        if (oy && !py) break;
        double r = v[at[(2 * oy) * qq + b * q + a]];
        if (px) {
            const double o = v[at[(2 * oy + 1) * qq + b * q + a]];
            r = 0.5 * (fx ? r - o : r + o);
        }
        s[oy] = r;
    }
    const double r = py ? 0.5 * (fy ? s[0] - s[1] : s[0] + s[1]) : s[0];
    u[e] = accumulate ? u[e] + r : r;
}
