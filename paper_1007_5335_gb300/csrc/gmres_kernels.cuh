// GMRES kernels around the operator products (Section 3.2): the start of a sweep from a residual,
// one Arnoldi step, and the end of a sweep.  All vectors binary64, every reduction in a fixed
// order (lanes, then warps, then the blocks of the cluster), so a solve is deterministic.
//
// An Arnoldi step moves little (k + 1 basis vectors of 8 N_Gamma bytes, from L2) but has three
// grid-wide reductions (Gram-Schmidt twice, the norm).  As separate launches it was four kernels
// of 4 to 8 us each, bound by launch and drain.  Here one thread-block cluster runs the whole
// step: each block keeps its slice of w in shared memory, partial sums are pushed into every
// block's shared memory (distributed shared memory) and a hardware cluster barrier separates the
// phases.  The binary64 pipe sets the shape of the code: a warp instruction occupies its quarter
// of the SM for 64 cycles, whatever the number of active lanes.  So 16 blocks (the largest
// cluster) share the vectors, sums over blocks are shuffle trees over lanes instead of chains,
// scalars (norms, reciprocals, the rotation) are formed by one warp and handed over through
// shared memory (a square root and a division by all 16 warps took 4 us), and the rotation of the
// column runs in a warp of its own beside the vector work.  The norm takes no reduction of its
// own: ||w - V h2||^2 = ||w||^2 - ||h2||^2 for the orthonormal V, with ||w||^2 summed beside the
// second pass's dots; h2 is at the rounding level of w, and a step where it is not (w almost in the
// span, a breakdown) forms the norm from the vector behind one more barrier.
// Measured, N_Gamma = 6144, mixed solve of 13 steps: 1083 us with the four kernels (and separate
// kernels for residual, norm, scaling and update around a sweep), 808 us with these; a step 7 us in
// the kernel at 6 basis vectors (clock counters), 23 us for the four.
#pragma once

#include <cooperative_groups.h>

#include "mh_internal.cuh"

namespace gmres_k {

namespace cg = cooperative_groups;

constexpr int GM_T = 512;   // threads per block

// Warp sum, broadcast from lane 0.
__device__ __forceinline__ double wsum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return __shfl_sync(0xffffffffu, v, 0);
}

// Sum of the values of lanes 0..m-1 of every group of m lanes (m a power of two), in every lane.
__device__ __forceinline__ double tree_sum(double v, int m) {
    for (int o = m >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Rows of a block's slice: a multiple of 32.
__host__ __device__ inline int64_t gm_rows(int64_t n, int blocks) { return ((n + blocks - 1) / blocks + 31) / 32 * 32; }

// What the interactive solver sees of a solve in progress: pinned host memory that the kernels
// write (fields first, then the counter they are published by) and the host polls.  Both counters start
// at 0 in every solve, so they stay as small as max_iter however long the boundary lives.
struct progress {
    double rn, bn, res;     // ||r||, ||b|| of the last sweep start; residual estimate of the last step
    int begins;             // sweep starts of this solve so far ...
    int started, done;      // ... and what the last one decided
    int steps;              // 2 x Arnoldi steps of this solve so far (all sweeps) + 1 if the last one ended its process
};

// Start of a sweep: r = b - ax (ax given) or r = r0 (r0 given, may alias r), its norm rn and, in
// a first sweep, ||b||; then V_0 = r / rn (and its binary32 copy), g = (rn, 0, ...).
// Accept (converged) when allowed and rn <= tol ||b||, else start an Arnoldi process with the inner target max(tol ||b||, 1e-5 rn) in mixed precision (half the
// tolerance: the binary64 residual after the sweep then lands below it instead of just above,
// which would cost another sweep), tol ||b|| in binary64.  final_check: the last residual of the
// schedule, recorded only.  recheck: a supplied residual within the tolerance starts nothing (the
// interactive solver then computes the residual).  ||b|| = 0 gives x = 0.  With loop_set, the condition of the sweep's
// Arnoldi loop (a graph WHILE node, 0 by default at every launch) is set to "start".
struct begin_args {
    const double *b, *ax, *r0;
    double *r, *V0, *g, *x;
    float* v32;
    int64_t n;
    int gsz;
    gmres_dev* gs;
    double tol;
    int mixed, may_accept, final_check, recheck, first, loop_set;
    cudaGraphConditionalHandle loop;
    progress* prog;
    int seq;   // (prog) the start's number
};

__global__ void __launch_bounds__(GM_T) k_sweep_begin(begin_args a) {
    __shared__ double red[2][GM_T / 32], all[2][16], nrm[3];
    cg::cluster_group cl = cg::this_cluster();
    mh_dep_wait();
    if (!a.first && a.gs->done) return;   // the same for every block: written after the last barrier only
    cl.barrier_arrive();              // every block of the cluster runs before the first remote store
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double bn_kept = a.first ? 0.0 : a.gs->bnorm;
    const int64_t R = gm_rows(a.n, C), e0 = R * rank, e1 = min(a.n, e0 + R);
    double s = 0.0, sb = 0.0;
    for (int64_t e = e0 + threadIdx.x; e < e1; e += GM_T) {
        const double bv = a.b[e];
        const double v = a.ax ? bv - a.ax[e] : a.r0[e];
        a.r[e] = v;
        s = fma(v, v, s);
        if (a.first) sb = fma(bv, bv, sb);
    }
    s = wsum(s);
    if (a.first) sb = wsum(sb);
    if (lane == 0) {
        red[0][warp] = s;
        red[1][warp] = sb;
    }
    __syncthreads();
    cl.barrier_wait();
    if (warp < 2) {
        const double t = tree_sum(lane < GM_T / 32 ? red[warp][lane] : 0.0, GM_T / 32);
        if (lane < C) *cl.map_shared_rank(&all[warp][rank], lane) = t;
    }
    cl.sync();
    if (warp < 2) {   // warp 0: ||r|| and its reciprocal, warp 1: ||b||
        const double q = tree_sum(lane < C ? all[warp][lane] : 0.0, C);
        const double v = sqrt(q);
        if (lane == 0) nrm[warp] = v;
        if (warp == 0 && lane == 0) nrm[2] = v > 0.0 ? 1.0 / v : 0.0;
    }
    __syncthreads();
    const double rn = nrm[0], bn = a.first ? nrm[1] : bn_kept, inv = nrm[2];
    const bool lead = rank == 0 && threadIdx.x == 0;
    bool start = rn > 0.0, conv = false;
    if (lead && a.first) {
        a.gs->done = a.gs->converged = a.gs->sweeps = a.gs->k = a.gs->total = 0;
    }
    if (bn == 0.0) {
        for (int64_t e = e0 + threadIdx.x; e < e1; e += GM_T) a.x[e] = a.r[e] = 0.0;   // b = 0: x = 0, residual 0
        start = false;
        if (lead) {
            a.gs->bnorm = 0.0;
            a.gs->done = a.gs->skip = a.gs->converged = 1;
            a.gs->rel = 0.0;
        }
    } else {
        const bool accept = a.may_accept || a.final_check;
        conv = accept && rn <= a.tol * bn;
        start = start && !conv && !a.final_check && !(a.recheck && rn <= a.tol * bn);
        if (lead) {
            if (a.first) {
                a.gs->bnorm = bn;
                a.gs->init_rel = rn / bn;
            }
            if (accept) a.gs->rel = rn / bn;
            if (conv) {
                a.gs->done = a.gs->skip = a.gs->converged = 1;
            } else if (start) {
                a.gs->skip = 0;
                a.gs->k = 0;
                a.gs->sweeps += 1;
                a.gs->target = a.mixed ? fmax(0.5 * a.tol * bn, 1e-5 * rn) : a.tol * bn;
            } else {
                a.gs->skip = 1;
            }
            if (a.loop_set) cudaGraphSetConditional(a.loop, start ? 1u : 0u);
        }
    }
    if (lead && a.prog) {
        a.prog->rn = rn;
        a.prog->bn = bn;
        a.prog->started = start;
        a.prog->done = conv || bn == 0.0;
        __threadfence_system();
        *(volatile int*)&a.prog->begins = a.seq;
    }
    if (!start) return;
    for (int64_t e = e0 + threadIdx.x; e < e1; e += GM_T) {
        const double v = a.r[e] * inv;
        a.V0[e] = v;
        if (a.v32) a.v32[e] = (float)v;
    }
    if (rank == 0)
        for (int i = threadIdx.x; i < a.gsz; i += GM_T) a.g[i] = i == 0 ? rn : 0.0;
}

// One Arnoldi step after w = A v_k: classical Gram-Schmidt twice against V_0..V_k, v_{k+1} =
// w / ||w|| (and its binary32 copy), column k of H rotated by the previous Givens rotations,
// rotation k, g updated.  k and the end of the sweep's process live on the device (gs->k,
// gs->skip; the step is skipped once it has ended), and with loop_set the condition of the graph loop is set to
// "not ended".  kcap >= k + 1 is the stride of the partial sums.
struct step_args {
    const double* V;
    double* w;        // overwritten when the slices stay in global memory
    int64_t n;
    int kcap, ldh;
    int shared_w;     // the slices of w fit in shared memory
    double *H, *cs, *sn, *g, *Vn;   // Vn = V (next column at (k + 1) n)
    float* v32;
    gmres_dev* gs;
    int m_max, loop_set;
    cudaGraphConditionalHandle loop;
    progress* prog;
};

constexpr size_t GM_SMEM_MAX = 200 * 1024;

__host__ __device__ inline size_t step_fixed(int blocks, int kcap) {
    return 2 * (size_t)blocks * (kcap + 1) + 7 * (size_t)(kcap + 1);
}

// Shared memory of a step: two sets of partial sums and the column (always), the slice of w when it
// still fits (beyond, with a slice of >= ~100 KB, the step works on w in global memory).
inline size_t step_smem(int64_t n, int blocks, int kcap, int* shared_w) {
    const size_t fixed = step_fixed(blocks, kcap) * sizeof(double);
    const size_t slice = (size_t)gm_rows(n, blocks) * sizeof(double);
    *shared_w = fixed + slice <= GM_SMEM_MAX;
    return fixed + (*shared_w ? slice : 0);
}

// Partial dots of ws (the block's slice of w) with V_0..V_{k1-1} and, for m = k1 + 1, with itself,
// pushed to part[rank] of every block.
__device__ __forceinline__ void push_dots(cg::cluster_group& cl, const double* V, int64_t n, int64_t e0, int cnt,
                                          const double* ws, int k1, int m, int cap, double* part) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    for (int i = warp; i < m; i += GM_T / 32) {
        const double* v = i < k1 ? V + (int64_t)i * n + e0 : ws;
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
        int e = lane;
        for (; e + 96 < cnt; e += 128) {
            const double v0 = v[e], v1 = v[e + 32], v2 = v[e + 64], v3 = v[e + 96];
            a0 = fma(v0, ws[e], a0);
            a1 = fma(v1, ws[e + 32], a1);
            a2 = fma(v2, ws[e + 64], a2);
            a3 = fma(v3, ws[e + 96], a3);
        }
        for (; e < cnt; e += 32) a0 = fma(v[e], ws[e], a0);
        const double t = wsum((a0 + a1) + (a2 + a3));
        if (lane < C) *cl.map_shared_rank(part + rank * cap + i, lane) = t;
    }
}

// h[i] = sum over the blocks c of part[c cap + i], i < k1: C lanes per coefficient.
__device__ __forceinline__ void sum_dots(const double* part, int C, int cap, int k1, double* h) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, per = 32 / C;
    for (int i0 = warp * per; i0 < k1; i0 += GM_T / 32 * per) {
        const int i = i0 + lane / C;
        const double v = tree_sum(i < k1 ? part[(lane % C) * cap + i] : 0.0, C);
        if (i < k1 && lane % C == 0) h[i] = v;
    }
}

// ws -= sum_i h_i V_i on the slice (threads t of nt).
__device__ __forceinline__ void subtract(const double* V, int64_t n, int64_t e0, int cnt, double* ws,
                                         const double* h, int k1, int t, int nt) {
    for (int e = t; e < cnt; e += nt) {
        const double* v = V + e0 + e;
        double a0 = ws[e], a1 = 0.0, a2 = 0.0, a3 = 0.0;
        int i = 0;
        for (; i + 4 <= k1; i += 4) {
            const double v0 = v[(int64_t)i * n], v1 = v[(int64_t)(i + 1) * n], v2 = v[(int64_t)(i + 2) * n],
                         v3 = v[(int64_t)(i + 3) * n];
            a0 = fma(-h[i], v0, a0);
            a1 = fma(-h[i + 1], v1, a1);
            a2 = fma(-h[i + 2], v2, a2);
            a3 = fma(-h[i + 3], v3, a3);
        }
        for (; i < k1; ++i) a0 = fma(-h[i], v[(int64_t)i * n], a0);
        ws[e] = k1 < 4 ? a0 : a0 + (a1 + (a2 + a3));
    }
}

__global__ void __launch_bounds__(GM_T) k_arnoldi(step_args a) {
    mh_dep_wait();
    if (a.gs->skip) return;   // the same for every block: written after the last barrier only
    extern __shared__ double sm[];
    __shared__ double npart[16], inv_s;
    cg::cluster_group cl = cg::this_cluster();
    cl.barrier_arrive();   // every block of the cluster runs before the first remote store
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = a.gs->k, k1 = k + 1, cap = a.kcap + 1;
    const int64_t R = gm_rows(a.n, C), e0 = R * rank;
    const int cnt = (int)max((int64_t)0, min(a.n - e0, R));
    double* ws = a.shared_w ? sm + step_fixed(C, a.kcap) : a.w + e0;   // the block's slice of w
    double* pA = sm;                     // [C][cap] partial dots of the first pass
    double* pB = pA + (size_t)C * cap;   // ... of the second (another block may still read pA)
    double* h1 = pB + (size_t)C * cap;
    double* h2 = h1 + cap;               // h2[k1] = ||w||^2 after the first pass
    double* cu = h2 + cap;               // c_i u_{i+1}, s_i u_{i+1} (u = h1 + h2), c_i, s_i, t_i
    double* su = cu + cap;
    double* c_s = su + cap;
    double* s_s = c_s + cap;
    double* ti = s_s + cap;
    if (a.shared_w)
        for (int e = threadIdx.x; e < cnt; e += GM_T) ws[e] = a.w[e0 + e];
    __syncthreads();
    cl.barrier_wait();
    push_dots(cl, a.V, a.n, e0, cnt, ws, k1, k1, cap, pA);
    cl.sync();
    sum_dots(pA, C, cap, k1, h1);
    __syncthreads();
    subtract(a.V, a.n, e0, cnt, ws, h1, k1, threadIdx.x, GM_T);
    __syncthreads();
    push_dots(cl, a.V, a.n, e0, cnt, ws, k1, k1 + 1, cap, pB);
    if (rank == 0)
        for (int i = threadIdx.x; i < k; i += GM_T) {
            c_s[i] = a.cs[i];
            s_s[i] = a.sn[i];
        }
    cl.sync();
    sum_dots(pB, C, cap, k1 + 1, h2);
    __syncthreads();
    // then the last warp forms ||w - V h2||^2 and, in block 0, the rotated column
    const int busy = GM_T - 32;
    double q = 0.0;
    subtract(a.V, a.n, e0, cnt, ws, h2, k1, threadIdx.x, GM_T);
    if (threadIdx.x >= busy) {
        double d = 0.0;
        for (int i = lane; i < k1; i += 32) d = fma(h2[i], h2[i], d);
        d = wsum(d);
        q = h2[k1] - d;
        const bool bad = !(q > 0.5 * h2[k1]);   // cancellation: the norm from the vector itself (below)
        if (lane == 0) inv_s = bad ? -1.0 : rsqrt(q);
    }
    __syncthreads();
    if (inv_s < 0.0) {   // the same in every block of the cluster
        if (warp == GM_T / 32 - 1) {
            double d = 0.0;
            for (int e = lane; e < cnt; e += 32) d = fma(ws[e], ws[e], d);
            d = wsum(d);
            if (lane < C) *cl.map_shared_rank(npart + rank, lane) = d;
        }
        cl.sync();
        if (warp == GM_T / 32 - 1) {
            q = tree_sum(lane < C ? npart[lane] : 0.0, C);
            q = __shfl_sync(0xffffffffu, q, 0);
            if (lane == 0) inv_s = q > 0.0 ? rsqrt(q) : 0.0;
        }
        __syncthreads();
    }
    double* vn = a.Vn + (int64_t)k1 * a.n + e0;
    if (threadIdx.x < busy) {
        const double inv = inv_s;
        for (int e = threadIdx.x; e < cnt; e += busy) {
            const double v = ws[e] * inv;
            vn[e] = v;
            if (a.v32) a.v32[e0 + e] = (float)v;
        }
        return;
    }
    if (rank != 0) return;
    // Block 0's last warp: the column u = h1 + h2 under the previous rotations (the chain over i
    // holds one operation per rotation, the rest is done for all i at once), rotation k, g.
    for (int i = lane; i < k; i += 32) {
        const double u = h1[i + 1] + h2[i + 1];
        cu[i] = c_s[i] * u;
        su[i] = s_s[i] * u;
    }
    __syncwarp();
    double t = h1[0] + h2[0];
    for (int i = 0; i < k; ++i) {
        if (lane == 0) ti[i] = t;
        t = fma(-s_s[i], t, cu[i]);
    }
    __syncwarp();
    double* hc = a.H + (int64_t)k * a.ldh;
    for (int i = lane; i < k; i += 32) hc[i] = fma(c_s[i], ti[i], su[i]);
    // den = sqrt(t^2 + ||w||^2), c = t / den, s = ||w|| / den: lane 0 and lane 1 take the two roots at once
    const double dd = fma(t, t, q);
    const double x = lane == 0 ? dd : q, rx = x > 0.0 ? rsqrt(x) : 0.0;
    const double rd = __shfl_sync(0xffffffffu, rx, 0), rq = __shfl_sync(0xffffffffu, rx, 1);
    if (lane == 0) {
        const double den = dd * rd, c = dd > 0.0 ? t * rd : 1.0, sv = (q * rq) * rd;
        const double gk = a.g[k], g1 = -sv * gk;
        a.cs[k] = c;
        a.sn[k] = sv;
        a.g[k + 1] = g1;
        a.g[k] = c * gk;
        hc[k] = den;
        hc[k1] = 0.0;
        // an estimate that is not finite ends the process too
        const bool end = !(fabs(g1) > a.gs->target) || k + 1 >= a.m_max || den == 0.0;
        const int total = a.gs->total + 1;
        a.gs->k = k + 1;
        a.gs->total = total;
        if (end) a.gs->skip = 1;
        if (a.loop_set) cudaGraphSetConditional(a.loop, end ? 0u : 1u);
        if (a.prog) {
            a.prog->res = fabs(g1);
            __threadfence_system();
            *(volatile int*)&a.prog->steps = 2 * total + (end ? 1 : 0);
        }
    }
}

// End of a sweep: R y = g (k x k upper triangular, column-major) and x += sum_i y_i V_i; with xh,
// the float-float split x = xh + xl of the residual product that follows.  Every block solves
// the small system itself, which costs less than a launch between the two: one warp, a column
// at a time, the diagonal's reciprocals formed at once and, up to 32 columns, y in registers and
// R in shared memory.
constexpr int GE_REG = 32;

__global__ void __launch_bounds__(256) k_sweep_end(const double* V, const double* H, int ldh,
                                                   const double* g, const gmres_dev* gs, int64_t n,
                                                   double* x, float* __restrict__ xh, float* __restrict__ xl) {
    mh_dep_wait();
    if (gs->done) return;
    const int k = gs->k;
    extern __shared__ double y[];   // [k]
    __shared__ double sR[GE_REG][GE_REG + 1];
    const int lane = threadIdx.x & 31;
    if (k <= GE_REG) {
        for (int e = threadIdx.x; e < GE_REG * k; e += 256) {
            const int c = e / GE_REG, r = e % GE_REG;
            if (r <= c) sR[c][r] = H[(int64_t)c * ldh + r];
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            double v = lane < k ? g[lane] : 0.0;
            const double d = lane < k ? sR[lane][lane] : 0.0;
            const double di = d != 0.0 ? 1.0 / d : 0.0;   // exact breakdown: the column adds nothing
            for (int i = k - 1; i >= 0; --i) {
                const double yi = __shfl_sync(0xffffffffu, v * di, i);
                if (lane == i) y[i] = yi;
                if (lane < i) v = fma(-sR[i][lane], yi, v);
            }
        }
    } else if (threadIdx.x < 32) {
        for (int i = lane; i < k; i += 32) y[i] = g[i];
        __syncwarp();
        for (int i = k - 1; i >= 0; --i) {
            const double* hc = H + (int64_t)i * ldh;
            const double d = hc[i];
            const double yi = d != 0.0 ? y[i] / d : 0.0;
            __syncwarp();
            for (int j = lane; j < i; j += 32) y[j] = fma(-hc[j], yi, y[j]);
            if (lane == 0) y[i] = yi;
            __syncwarp();
        }
    }
    __syncthreads();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        double a0 = 0.0, a1 = 0.0;
        int i = 0;
        for (; i + 2 <= k; i += 2) {
            a0 = fma(y[i], V[(int64_t)i * n + e], a0);
            a1 = fma(y[i + 1], V[(int64_t)(i + 1) * n + e], a1);
        }
        if (i < k) a0 = fma(y[i], V[(int64_t)i * n + e], a0);
        const double v = x[e] + (a0 + a1);
        x[e] = v;
        if (xh) {
            const float h = (float)v;
            xh[e] = h;
            xl[e] = (float)(v - (double)h);
        }
    }
}

}  // namespace gmres_k
