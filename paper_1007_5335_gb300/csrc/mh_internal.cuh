// Internal declarations shared by the libmh translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <cstdarg>
#include <cstdio>
#include <map>
#include <memory>
#include <string>
#include <vector>

#include "../../include/mh.h"

#define MH_PI 3.14159265358979323846

// Named timing region: CUDA events recorded on the context stream around each launch.
struct prof_region {
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> pending;
    double total_ms = 0.0;
    int64_t launches = 0;
    double flops = 0.0, bytes = 0.0;   // algorithmic work of the timed launches
};

struct dlp_eval;

struct mh_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    std::string err;
    int64_t launches = 0;
    bool profiling = false;
    bool capturing = false;   // inside a batch step: no cooperative launches
    bool tensor_cores = true; // binary32 contractions on the tensor cores (mh_set_tensor_cores)
    int64_t loop_nodes = 0;   // graph WHILE nodes recorded (their body kernels: loop_kernels each)
    std::map<std::string, prof_region> prof;
    std::unique_ptr<dlp_eval> eval;   // what mh_double_layer_apply at targets writes (below)
    ~mh_ctx();
};

// RAII scope: records a start/stop event pair on ctx->stream under `name` when
// profiling is enabled (mh_profile_enable), nothing otherwise.
struct prof_scope {
    mh_ctx* ctx;
    std::string name;
    double flops, bytes;
    cudaEvent_t a = nullptr, b = nullptr;
    prof_scope(mh_ctx* c, const char* n, double flops_ = 0.0, double bytes_ = 0.0);
    ~prof_scope();
};

// Records a message on ctx and returns the status.
mh_status mh_fail(mh_ctx* ctx, mh_status st, const char* fmt, ...);

#define MH_CUDA(ctx, call)                                                                      \
    do {                                                                                        \
        cudaError_t e_ = (call);                                                                \
        if (e_ != cudaSuccess)                                                                  \
            return mh_fail((ctx), e_ == cudaErrorMemoryAllocation ? MH_ERR_OOM : MH_ERR_CUDA,  \
                           "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__,    \
                           __LINE__);                                                           \
    } while (0)

#define MH_LAUNCHED(ctx)                                                                        \
    do {                                                                                        \
        (ctx)->launches++;                                                                      \
        cudaError_t e_ = cudaGetLastError();                                                    \
        if (e_ != cudaSuccess)                                                                  \
            return mh_fail((ctx), MH_ERR_CUDA, "kernel launch failed: %s (%s:%d)",              \
                           cudaGetErrorString(e_), __FILE__, __LINE__);                         \
    } while (0)

#define MH_TRY(expr)                                                                            \
    do {                                                                                        \
        mh_status s_ = (expr);                                                                  \
        if (s_ != MH_OK) return s_;                                                             \
    } while (0)

// Number of device allocations and frees made by the library (every one goes through dbuf),
// read by mh_device_alloc_calls.
extern std::atomic<int64_t> g_mh_alloc_calls;

// Device buffer with RAII free.
template <class T>
struct dbuf {
    T* p = nullptr;
    size_t n = 0;
    dbuf() = default;
    dbuf(const dbuf&) = delete;
    dbuf& operator=(const dbuf&) = delete;
    ~dbuf() { release(); }
    void release() {
        if (p) {
            g_mh_alloc_calls.fetch_add(1, std::memory_order_relaxed);
            cudaFree(p);
        }
        p = nullptr;
        n = 0;
    }
    cudaError_t alloc(size_t count) {
        release();
        if (count == 0) return cudaSuccess;
        g_mh_alloc_calls.fetch_add(1, std::memory_order_relaxed);
        const cudaError_t e = cudaMalloc((void**)&p, count * sizeof(T));
        if (e == cudaSuccess)
            n = count;   // a failed allocation leaves no room: the next reserve tries again
        else
            p = nullptr;
        return e;
    }
    cudaError_t reserve(size_t count) { return count <= n ? cudaSuccess : alloc(count); }
};

template <class... B>
inline size_t mh_bytes(const B&... b) {
    return (size_t(0) + ... + (b.n * sizeof(*b.p)));
}

#define MH_RESERVE(ctx, buf, count) MH_CUDA(ctx, (buf).reserve(count))
#define MH_ALLOC(ctx, buf, count) MH_CUDA(ctx, (buf).alloc(count))

// ---- dependent launches ----
// A kernel launched right behind another one on a stream costs about 2.2 us of drain and launch
// latency (0.9 us inside a graph); with programmatic dependent launch it is on the SMs and waiting
// when its predecessor ends (0.6 us; 16 blocks of 512 threads, chains of 500 launches).  The
// rules here: a kernel launched by mh_launch_dep calls mh_dep_wait() in every thread and before any
// return, with nothing before it but loads of set-up data (operators, weights of the geometry), so it touches
// what the stream writes only when everything before it has completed, and completes only after its
// predecessors; mh_launch_dep is used behind a kernel of
// the same stream (a launch behind an event wait, a copy or a graph's conditional node is an ordinary
// one).  The first kernel of an entry point is an ordinary launch as well: the caller's last kernel need
// not keep these rules (one that starts its dependents early and does not wait may end before its own
// predecessors).  Kernels that are launched either way call mh_dep_wait() too (no effect in an ordinary
// launch).  The wait comes before the trigger: at most one kernel waits behind the running one.
// What a kernel of the stream may have written is read by plain loads: no const __restrict__, no __ldg.  The
// read-only path asks for data that is constant over the kernel's whole life, and a dependent kernel is
// already resident while its predecessor writes; set-up data alone is read that way.
__device__ __forceinline__ void mh_dep_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... K, class... A>
inline cudaError_t mh_launch(cudaStream_t st, bool dep, void (*kernel)(K...), dim3 grid, dim3 block, size_t smem, A... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = dep ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<K>(args)...);
}

template <class... K, class... A>
inline cudaError_t mh_launch_dep(cudaStream_t st, void (*kernel)(K...), dim3 grid, dim3 block, size_t smem, A... args) {
    return mh_launch(st, true, kernel, grid, block, smem, args...);
}

// ---- L2 residency hints ----
// The binary32 operator is read once per Arnoldi step; at 6144 nodes it is 151 MB against 129 MB of
// L2, so in plain order every step streams all of it from HBM.  The first MH_L2_KEEP bytes are read
// with an evict-last hint and stay for the next step, the rest with evict-first.  k_gemv32s in a
// chain, 6144 nodes: 24.2 us without, 20.4 with 40 MB kept, 19.0 (64), 17.5 (80), 17.0 (88), 18.2
// (96), 23.5 (112): 72 MB leaves the rest of the step its share.  The share is one boundary's: in a batch
// of large problems the kept parts exceed the L2 together and give nothing.  Mixed batch steps from a zero
// density, with 72 / 24 / 0 MB kept: one problem of 7168 nodes 1290 / 1320 / 1360 us, two (7168, 8192)
// 2190 / 2040 / 2100, four (7168 to 9216) 4070 / 4015 / 4000.
constexpr int64_t MH_L2_KEEP = 72 << 20;

__device__ __forceinline__ uint64_t mh_l2_policy(bool keep) {
    uint64_t last, first;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(last));
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(first));
    return keep ? last : first;
}
__device__ __forceinline__ float4 mh_ld_hint(const float4* p, uint64_t policy) {
    float4 v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p), "l"(policy));
    return v;
}

// A second stream with fork / join events, for work that does not depend on what the context
// stream runs meanwhile: the multipole passes (latency chains, on a stream of the device's
// highest priority, so that their blocks start before queued near-field blocks) beside the
// near fields; the sums at the normal-line auxiliary points beside the double layer's
// multipole pass.  Created at set-up, outside any stream capture.
struct SideStream {
    cudaStream_t s = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    SideStream() = default;
    SideStream(const SideStream&) = delete;
    SideStream& operator=(const SideStream&) = delete;
    ~SideStream() {
        if (join) cudaEventDestroy(join);
        if (fork) cudaEventDestroy(fork);
        if (s) cudaStreamDestroy(s);
    }
    mh_status create(mh_ctx* ctx, bool high_priority = true) {
        int least = 0, greatest = 0;
        MH_CUDA(ctx, cudaDeviceGetStreamPriorityRange(&least, &greatest));
        MH_CUDA(ctx, cudaStreamCreateWithPriority(&s, cudaStreamNonBlocking, high_priority ? greatest : least));
        MH_CUDA(ctx, cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
        MH_CUDA(ctx, cudaEventCreateWithFlags(&join, cudaEventDisableTiming));
        return MH_OK;
    }
    // the side stream waits for everything issued so far on `main`
    mh_status begin(mh_ctx* ctx, cudaStream_t main) {
        MH_CUDA(ctx, cudaEventRecord(fork, main));
        MH_CUDA(ctx, cudaStreamWaitEvent(s, fork, 0));
        return MH_OK;
    }
    mh_status end(mh_ctx* ctx) {
        MH_CUDA(ctx, cudaEventRecord(join, s));
        return MH_OK;
    }
};

// Tensor-core batched contraction (contract_tc.cu): one launch over chunks of up to 128 tasks of
// one operator each; products to temp[task][R] or, with task_dst, straight to the destinations.
struct tc_launch {
    const uint16_t* img = nullptr;       // operator images (three bfloat16 parts) in the tensor-core layout
    const int64_t* img_off = nullptr;    // per operator: offset of its image (bfloat16 elements)
    const int32_t* kpad = nullptr;       // per operator: columns rounded up to 16
    const int32_t* op_C = nullptr;       // per operator: columns
    const int32_t* chunk_op = nullptr;
    const int32_t* chunk_t0 = nullptr;   // n_chunks + 1 entries
    int64_t n_chunks = 0;
    const uint16_t* spl = nullptr;       // pre-split sources: three bfloat16 planes
    int64_t plane = 0;                   // elements per plane
    const int64_t* tc_src = nullptr;     // per task: offset of its source row in a plane
    int R = 0, npad = 0, kmax = 0;
    float* temp = nullptr;
    const int64_t* task_dst = nullptr;
    int accumulate = 0;
    void* dst = nullptr;
    bool dst_double = false;
    int* err = nullptr;                  // set when a bounded wait gave up
    bool dep = false;                    // launched directly behind a kernel (mh_launch_dep)
};
int tc_pad_rows(int R);
int tc_pad_cols(int C);
void tc_operator_image(const double* op, int R, int C, int npad, int kpad, uint16_t* out);
mh_status tc_prepare(mh_ctx* ctx);
mh_status tc_contract_launch(mh_ctx* ctx, const tc_launch& a);
// Split count binary32 vectors of length len at src into the three bfloat16 planes at dst
// (rows padded with zeros to S entries).
mh_status tc_split_launch(mh_ctx* ctx, const float* src, int len, int64_t count, int S, uint16_t* planes, int64_t plane,
                          int64_t dst);
// The same from binary64 vectors at src, which are also written to dst32 in binary32.
mh_status tc_split_values(mh_ctx* ctx, const double* src, int len, int64_t count, int S, float* dst32, uint16_t* planes,
                          int64_t plane, int64_t dst, bool dep);

// Device-resident state of the sync-free GMRES (gmres_run_graph): every kernel of its fixed
// schedule reads the flags at entry and returns at once when its work is not needed.
constexpr int GMRES_LOOP_KERNELS = 2;   // kernels in the body of a graph Arnoldi loop

struct gmres_dev {
    double bnorm, rn, target, rel, init_rel;
    int done;        // converged on a binary64 residual computed in this solve
    int skip;        // done, or the Arnoldi process of the current sweep has ended
    int k;           // Arnoldi iterations of the current sweep
    int total;       // all Arnoldi iterations
    int sweeps;      // sweeps started (refinement passes in mixed precision)
    int converged;
};

// GMRES workspace (kept by the boundary so that repeated solves allocate nothing).
struct gmres_ws {
    dbuf<double> V, H, cs, sn, g, w, r;
    dbuf<gmres_dev> gs;                  // state of an interactive solve
    void* prog = nullptr;                // what the host sees of it (pinned, gmres_k::progress)
    int cluster = 0;                     // thread blocks in the cluster of an Arnoldi step (16 or 8)
    dbuf<float> v32;                     // binary32 copy of the newest Krylov vector
    cudaStream_t body_stream = nullptr;  // captures the body of a graph loop (batch graphs)
    int m = 0;
    int64_t n = 0;
    int64_t gen = 0;                     // bumped whenever the buffers are reallocated (recorded graphs hold them)
    gmres_ws() = default;
    gmres_ws(const gmres_ws&) = delete;
    gmres_ws& operator=(const gmres_ws&) = delete;
    ~gmres_ws() {
        if (body_stream) cudaStreamDestroy(body_stream);
        if (prog) cudaFreeHost(prog);
    }
};

// Assembled boundary operator for one alpha (eq. discrete_sys), row-major N x N.
struct bie_operator {
    double alpha = -1.0;
    int64_t gen = 0;     // bumped whenever a form below is allocated or released (recorded graphs hold them)
    dbuf<double> A64;
    dbuf<float> A32;
    dbuf<float> A32lo;   // A64 - A32 rounded to binary32: A32 + A32lo carries A64 to ~2^-48
    // (A64 - A32) 2^24 rounded to binary16 (bit patterns), used instead of A32lo when N is a
    // multiple of 8: A32 + 2^-24 A16lo carries A64 to 2^-35 |A| + 2^-49
    dbuf<uint16_t> A16lo;
};

// Classified target set for off-surface evaluation.
struct dlp_targets {
    int64_t n = 0;          // user targets
    int64_t n_ext = 0;      // user targets + auxiliary points of the normal-line rule
    dbuf<double> xy;        // [n_ext][2]
    dbuf<uint32_t> fine0;   // classification results before compaction (masks, nearest curves, foot data)
    dbuf<int32_t> lcurve;
    dbuf<double> ldata;
    dbuf<uint32_t> fine;    // [n_ext] bit k: use the upsampled rule on curve k
    dbuf<int32_t> region;   // [n] -1 inside Omega, k exterior side of curve k
    // normal-line rule: per line target
    int64_t n_line = 0;
    dbuf<int32_t> line_tgt;     // target index
    dbuf<int32_t> line_curve;   // curve
    dbuf<double> line_data;     // [n_line][4]: t*, d, h_s, unused
    dbuf<double> line_l;        // [n_line][5]: interpolation weights in the distance (limit, 4 auxiliary points)
    dbuf<double> line_w;        // trigonometric interpolation weights at t*, N_k per line target
    dbuf<int64_t> line_woff;    // [n_line + 1] offsets into line_w
    // fine pairs (ext target, curve)
    int64_t n_pairs = 0, n_pairs_main = 0;   // pairs of user targets come first
    double fine_nodes_main = 0, fine_nodes_aux = 0;   // work counts
    dbuf<int32_t> pair_tgt;
    // upsampled rule at the auxiliary points (at every pair of a set classified with all_groups):
    // groups of FINE_TG pairs on one curve (grp_pair, -1 padded), each group's fine nodes in
    // fine_slices slices, one block per (group, slice); partial sums per (group, slice, pair) in
    // grp_part
    int64_t n_groups = 0;
    int fine_slices = 1;
    dbuf<int32_t> grp_curve, grp_pair;
    dbuf<double> grp_part;
    dbuf<unsigned> grp_cnt;
    // evaluation workspaces (allocated once by dlp_classify)
    dbuf<double> ext, asig, part;
    size_t bytes() const {
        return mh_bytes(xy, fine0, lcurve, ldata, fine, region, line_tgt, line_curve, line_data, line_l, line_w, line_woff,
                        pair_tgt, grp_curve, grp_pair, grp_part, grp_cnt, ext, asig, part);
    }
};

// A binary64 pair table (pair64.cuh) and the alpha it holds.
struct pair_tab_buf {
    dbuf<double2> c;
    double alpha = -1.0;
};

// A density on its way to the 16x grid: Fourier coefficients, those of the sub-offsets (curves that are
// not transformed by FFT), and the density times |y'| h_f there, in binary64.
struct fine_ws {
    dbuf<double> sc, wf;
    dbuf<double2> cp;
    size_t bytes() const { return mh_bytes(sc, wf, cp); }
};

// Everything that a binary64 mh_double_layer_apply at targets writes belongs to the context, so that contexts
// on several host threads may evaluate on one boundary: the boundary is only read there (its operator for
// alpha assembled before).  Kept for the next call (some twenty allocations and frees cost ~0.3 ms) up
// to DLP_KEEP bytes: the interpolation weights alone are N_k doubles for every target within h_s/4.
struct dlp_eval {
    dlp_targets tg;
    pair_tab_buf ptab;
    fine_ws fine;
    size_t bytes() const { return tg.bytes() + fine.bytes() + mh_bytes(ptab.c); }
};
constexpr size_t DLP_KEEP = 64 << 20;

struct mh_boundary {
    int n_curves = 0;
    int64_t n = 0;                       // N_Gamma
    int alpert_order = 0;                // l (window a = l), 0 = plain trapezoid
    std::vector<int32_t> n_nodes, offset; // per curve (host)
    dbuf<int32_t> d_nn, d_off;           // per curve (device)
    dbuf<int32_t> d_curve_of;            // curve index of every node
    dbuf<double> xy;                     // [n][2]
    dbuf<double> geo;                    // [n][8]: x y x' y' x'' y'' |y'| kdiag
    dbuf<float4> geo32;                  // binary32 nodes for the classification (k_cls32)
    double cls_ox = 0, cls_oy = 0;       // their origin (mean node)
    double cls_scale = 1.0;              // and scale: a power of two that takes the extent to [1, 2)
    float cls_extent = 0;                // largest side of the nodes' bounding box, scaled
    dbuf<double> coef;                   // per curve Fourier coefficients: [off*2 ...] see boundary.cu
    dbuf<double2> tw, half;              // per node (cos, sin)(2 pi r / N) and (cos, sin)(pi r / N)
    // fine (16x) grid per curve: positions, normals, speed*h_fine
    int64_t n_fine = 0;
    std::vector<int64_t> fine_off;
    dbuf<int64_t> d_fine_off;
    dbuf<double> fine_geo;               // [n_fine][5]: x y nx ny |y'| h_f
    bie_operator op;
    gmres_ws ws;
    // binary32 source data for the mixed-precision double layer: offsets from tile
    // centres (tiles of MH_TILE nodes, fine chunks of MH_TILE fine nodes per curve)
    int64_t n_tiles = 0, n_fchunks = 0;
    std::vector<int64_t> fchunk_off;     // per curve first chunk
    dbuf<int64_t> d_fchunk_off;
    dbuf<float4> src32, fine32;          // (dx, dy, nx, ny)
    dbuf<double2> tile_c;
    dbuf<float> tile_r;                  // per source tile: largest distance of a node from its centre
    dbuf<float2> tw32;                   // binary32 copy of the twiddles e^{2 pi i r / N_k}
    dbuf<float> xhi32, xlo32;            // float-float split of the input of a residual product
    dbuf<float4> fchunk_cf;              // fine chunk centres as float-float (x_hi, x_lo, y_hi, y_lo)
    dbuf<float> fchunk_r;                // fine chunk radii
    dbuf<float> w32, wf32, x32;          // per call: weights, fine weights, GEMV input
    fine_ws fine;                        // per step: the density on the 16x grid
    pair_tab_buf ptab;                   // of the auxiliary sums of a step
    // matrix-free operator: the trapezoid sum by the on-surface multipole pass of a tree that
    // holds every node, the Alpert correction by binary64 chirp transforms per curve
    bool mfree = false;
    mh_tree* mf_tree = nullptr;          // not owned (the problem's tree)
    double mf_alpha = -1.0;
    dbuf<double> mf_cp;                  // [2 l][n] Alpert node weights (kernel x rule weight x h / pi)
    dbuf<double> mf_win;                 // [2 (a - 1)][n] own-curve window weights (kernel x |y'| h / pi)
    dbuf<double2> mf_chirp, mf_bh, mf_tw;   // per curve: e^{i pi n^2/N}, transformed chirp filter, twiddles
    dbuf<int64_t> mf_moff;               // per curve: offset of its M_k-entry blocks (twiddles at moff/2)
    dbuf<int32_t> mf_M;                  // per curve: transform length M_k (power of two >= 2 N_k - 1)
    int mf_mmax = 0;
    dbuf<double2> mf_spec;               // per call: spectra c_m, m <= N_k/2
    dbuf<double> mf_S;                   // per call: [2 l][n] interpolated density at the Alpert nodes
    dbuf<double> mf_u;                   // per call: multipole-pass output
    SideStream mf_side;                  // the Alpert transforms run there beside the multipole pass
    dbuf<double> warm_dir, warm_w, warm_scal;   // warm-start direction, its image, scalars
    dbuf<float2> fcp32;                  // fine-grid coefficients by sub-offset (binary32)
};

#define MH_TILE 128

struct mh_tree {
    double box[3];
    int q = 0, min_level = 0, max_level = 0;
    int64_t n_leaves = 0, n_boxes = 0, n_nodes = 0;
    std::vector<int32_t> lvl_start;      // box id range per level (host), size max_level+2
    dbuf<int32_t> boxes;                 // [n_boxes][3] level ix iy, level then Morton order
    dbuf<int32_t> leaf_box;              // [n_leaves] box id of each leaf (node order)
    dbuf<int32_t> box_leaf;              // [n_boxes] leaf index or -1
    dbuf<int32_t> box_parent;            // [n_boxes]
    dbuf<int32_t> box_child;             // [n_boxes][4] or -1
    dbuf<int32_t> status;                // dense per-level status map (Morton indexed), box id or -1
    std::vector<int64_t> status_off;     // per level offset into status
    dbuf<double> nodes;                  // [n_nodes][2]
    dbuf<int32_t> list_off[4], list_item[4];   // U V W X in CSR over boxes
    std::vector<int64_t> list_len;       // total items per list
    void* vol = nullptr;                 // volume operator data (volume.cu)
};

struct mh_problem {
    mh_tree* tree = nullptr;
    mh_boundary* bnd = nullptr;
    double dt = 0, alpha = 0;
    int scheme = 0;
    int p = 0;
    int ext_mode = 0;
    std::vector<double> ext_const;
    dbuf<double> d_ext_const;
    dlp_targets tg;                      // volume nodes inside Omega (classification of all nodes)
    dbuf<int32_t> region;                // [n_nodes]
    dbuf<int32_t> inside_idx;            // indices of nodes inside Omega
    int64_t n_inside = 0;
    dbuf<int32_t> bnd_leaf;              // leaf of every boundary node
    dbuf<double> B, Up, rhs;             // work arrays
    SideStream aux;                      // the normal-line auxiliary sums beside the double layer's pass
    // GMRES start (mh_problem_set_warm_start)
    int warm_mode = 0;
    int warm_arith = 0;
    struct mh_net* net = nullptr;
    bool have_prev = false;              // sig_prev holds the density entering the previous step
    dbuf<double> sig_prev, r0, c_dev;
    double* c_host = nullptr;            // pinned
    // batched stepping (mh_batch_step): sync-free GMRES with its state in gstat (device)
    bool graph_mode = false;
    gmres_dev* gstat = nullptr;
    // residual recycling: the density, right-hand side and binary64 residual the last step
    // ended with; b - A sigma for an unchanged sigma is b - rc_b + rc_r (no operator product)
    bool rc_valid = false;
    dbuf<double> rc_sigma, rc_b, rc_r, r_start;
    dbuf<int> rc_same;
    ~mh_problem() {
        if (c_host) cudaFreeHost(c_host);
    }
};

// ---- net.cu ----
// Initial guess for A x = rhs (see mh_warm_start in mh.h); c_dev receives the step length.
// save (nullable) receives the incoming sigma before x0 is written.
// r_ready: r0 already holds rhs - A sigma (binary64).
mh_status warm_start_run(mh_ctx* ctx, mh_boundary* bnd, double alpha, struct mh_net* net, int mode, int arith,
                         const double* sigma, const double* sigma_prev2, const double* rhs, double* x0, double* r0,
                         mh_precision prec, double* c_dev, double* save, bool r_ready = false);
bool net_matches(const struct mh_net* net, const mh_boundary* b);
// Workspace of the SECANT / LEARNED starts (allocated once per boundary).
mh_status warm_start_prepare(mh_ctx* ctx, mh_boundary* b);

// ---- boundary.cu ----
mh_status bie_assemble(mh_ctx* ctx, mh_boundary* b, double alpha);
mh_status bie_apply(mh_ctx* ctx, mh_boundary* b, const double* x, double* y, mh_precision prec,
                    bool dep = false);
// Matrix-free operator: set-up after volume_bie_setup on tree t (releases the dense forms; every
// later operator product of b goes through it), and one product y = A x (binary64).
mh_status bie_mfree_setup(mh_ctx* ctx, mh_boundary* b, mh_tree* t, double alpha);
mh_status bie_apply_mfree(mh_ctx* ctx, mh_boundary* b, const double* x, double* y);
// y = A x in binary64, skipped when *gate != 0 (gate nullable).
// Mixed precision: accurate to binary64 for residuals (float-float); x_split: b->xhi32, xlo32 hold x;
// dep: directly behind a kernel of the library (mh_launch_dep).
mh_status bie_apply64_gated(mh_ctx* ctx, mh_boundary* b, const double* x, double* y, const int* gate,
                            mh_precision prec, bool x_split = false, bool dep = true);
// Where the last solve left the binary64 residual rhs - A x of its result.
const double* gmres_final_residual(mh_boundary* b);
// Everything a sync-free solve in precision prec needs (binary32 operator copy).
mh_status bie_prepare(mh_ctx* ctx, mh_boundary* b, mh_precision prec);
// all_groups: the upsampled rule will run at every pair (mh_double_layer_apply), not at the auxiliary ones only.
mh_status dlp_classify(mh_ctx* ctx, mh_boundary* b, const double* xy_dev, int64_t n, dlp_targets* tg,
                       bool all_groups = false);
// Sums at the auxiliary points of the normal-line rule into tg->ext (they need sigma and its fine
// weights only, so they may run beside the pass that evaluates the other targets).
mh_status dlp_aux_sums(mh_ctx* ctx, mh_boundary* b, double alpha, dlp_targets* tg, const double* sigma,
                       mh_precision prec);
// The normal-line rule at the set's line targets, after dlp_aux_sums: out[idx[t]] = base[idx[t]] + U^h,
// with A sigma = rhs - r.
mh_status dlp_line_finish(mh_ctx* ctx, mh_boundary* b, double alpha, dlp_targets* tg, const double* rhs,
                          const double* r, const double* base, const int32_t* idx, double* out);
// Density on the 16x fine grid times |y'| h_f (binary64 in ws.wf; binary32 also in b->wf32
// when prec is mixed); spectrum64: mixed weights rounded from a binary64 spectrum, not a binary32 one.
mh_status dlp_fine_weights(mh_ctx* ctx, mh_boundary* b, const double* sigma, mh_precision prec, fine_ws& ws,
                           bool spectrum64 = false);
// r0 (nullable): the binary64 residual rhs - A x of the initial guess, computed by the caller.
mh_status gmres_run(mh_ctx* ctx, mh_boundary* b, const double* rhs, double* x, double tol, int max_iter,
                    mh_precision prec, mh_gmres_info* info, const double* r0 = nullptr);
// The same solve without host synchronisation, for capture in a CUDA graph: a fixed schedule of
// sweeps x m_max Arnoldi iterations whose kernels return at once when the device flags in gs
// say their work is not needed.  gs (device) holds the result; gmres_graph_ensure sizes the
// workspace beforehand (no allocation happens in gmres_run_graph).
mh_status gmres_graph_ensure(mh_ctx* ctx, mh_boundary* b, int m_max);
mh_status gmres_run_graph(mh_ctx* ctx, mh_boundary* b, const double* rhs, double* x, double tol, mh_precision prec,
                          const double* r0, gmres_dev* gs);
void gmres_graph_schedule(mh_precision prec, int* sweeps, int* m_max);
mh_status gmres_info_from_dev(const gmres_dev& g, double tol, mh_gmres_info* info);

// ---- tree.cu ----
void mh_gauss_legendre(int n, double* x, double* w);
const double* tree_gl_nodes(const mh_tree* t);

// ---- volume.cu ----
// dep: directly behind a kernel of the library.
mh_status volume_apply(mh_ctx* ctx, mh_tree* t, double alpha, int p, const double* b, double* up,
                       mh_precision prec, bool dep);
void volume_free(mh_tree* t);
// Threads per block of the binary32 near-field double-layer kernel (128, 256 or 512).
mh_status volume_set_near_tile(mh_ctx* ctx, mh_tree* t, int threads);
int volume_near_tile(const mh_tree* t);
// double layer through the multipole method (dipoles sorted by leaf)
mh_status volume_dipole_setup(mh_ctx* ctx, mh_tree* t, double alpha, int p, const double* dxy, const double* dnrm,
                              const int32_t* dleaf, int64_t nd, bool near_blocks);
// Strengths w[perm[j]] for dipole j; *u: U^h at every volume node (valid until the next call on the tree).
mh_status volume_dipole_apply(mh_ctx* ctx, mh_tree* t, const double* w, const int32_t* perm, mh_precision prec,
                              const double** u);
// On-surface double layer through the multipole method (binary64): set-up for the boundary
// nodes (host arrays in node order: positions, unit normals, leaf of every node), then
// u_i = -(1/(2 pi alpha^2)) sum_{d != i} w_d (1/alpha) K1(r/alpha) (y_d - x_i).nu_d / r at every
// node for device strengths w (node order).
mh_status volume_bie_setup(mh_ctx* ctx, mh_tree* t, double alpha, int p, const double* xy, const double* nrm,
                           const int32_t* leaf, int64_t nd);
bool volume_bie_ready(const mh_tree* t);
mh_status volume_bie_apply(mh_ctx* ctx, mh_tree* t, const double* sigma, const double* geo, const int32_t* curve_of,
                           const int32_t* nn, double* u);
mh_status tree_locate(mh_ctx* ctx, const mh_tree* t, const double* xy_dev, int64_t n, int32_t* leaf_out);
// Leaf interpolation U of node values at n points with known leaves; with f, c (f - U) instead of U.
mh_status tree_interpolate(mh_ctx* ctx, const mh_tree* t, const double* vals, const double* xy_dev,
                           const int32_t* leaf, int64_t n, const double* f, double c, double* out);

inline int mh_grid(int64_t n, int block) {
    int64_t g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > 2147483647LL) g = 2147483647LL;
    return (int)g;
}
