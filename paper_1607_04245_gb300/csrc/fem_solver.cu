// fem_solver.cu -- Jacobi-preconditioned conjugate-gradient solves with the assembled
// operators of Eq. 2: A v = E^T r_e(v), the element residuals of the variable-coefficient
// Laplacian or of linear elasticity summed into the vertices through the vertex-to-cell lists
// (fem_build_node2cell). Dirichlet vertices keep their value from the initial x. Also:
// mixed-precision iterative refinement around the FP32-mixed solve.
//
// The iteration is CG in Chronopoulos and Gear's form. A solve takes one of two forms:
//   * assembled: the operator's rows are formed once on the device (fem_sell.cuh) and the
//     whole loop runs in one cooperative kernel (sell_cg_kernel). Taken by the float32 forms
//     (room_for) whenever the caller's workspace has room for the matrix.
//   * element form: each application is the residual kernel and the vertex sum; one iteration
//     is captured into the body of a CUDA graph WHILE node. For the float64 solves, workspaces
//     without room for the matrix, meshes whose rows do not fit it or, in the mixed form, with
//     badly shaped cells, and device partitions that refuse the cooperative launch. The float64 Laplacian's residual is then applied from
//     factors formed once per solve (launch_lap_factors), where the workspace has room.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "fem_cell.cuh"
#include "fem_sell.cuh"
#include "fem_wait.cuh"

namespace fem {

// fem_laplacian.cu, fem_df.cu: the residual split into what is formed once and the rest
fem_status launch_lap_factors(int dim, int64_t n_cells, int64_t n_verts, const double *coords, const int32_t *conn,
                              const double *K, const QuadW &w, double *fac, cudaStream_t s);
fem_status launch_lap_factored(int dim, int64_t n_cells, int64_t n_verts, const int32_t *conn, const double *u,
                               const double *fac, double *out, cudaStream_t s);
fem_status launch_lap_df_factors(int dim, int64_t n_cells, int64_t n_verts, const double *coords, const int32_t *conn,
                                 const double *K, const QuadW &w, double *fac, cudaStream_t s);
fem_status launch_lap_df_factored(int dim, int64_t n_cells, int64_t n_verts, const int32_t *conn, const double *u,
                                  const double *fac, double *out, cudaStream_t s);
fem_status launch_gather(int dim, int n_comp, int64_t C, int64_t V, const void *elem, const int32_t *node_ptr,
                         const int32_t *node_idx, void *out, fem_precision prec, cudaStream_t s);

constexpr int kDotBlocks = 1024;  // fixed: the partial sums and their order do not depend on the device

// element diagonals of the Laplacian stiffness: out[b][e] = Kbar |n_b|^2 / |det J|
template <int DIM, class T>
__global__ void lap_diag_kernel(const double *X0, int64_t C, uint32_t V, const int32_t *conn, const T *K, int nq,
                                QuadW w, T *out, unsigned *err) {
    constexpr int NB = DIM + 1;
    const double *X[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) X[k] = X0 + int64_t(k) * V;
    uint32_t vmax = 0;
    bool bad_det = false;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < C; e += stride) {
        uint32_t v[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) v[b] = clamp_vid(conn[b * C + e], V, vmax);
        double kbar = 0.0;
        for (int q = 0; q < nq; ++q) kbar += w.wd[q] * static_cast<double>(K[q * C + e]);
        double xs[NB][DIM], ee[DIM][DIM], n[DIM][DIM];
        gather_coords<DIM>(X, v, xs);
        columns_f64<DIM>(xs, ee);
        const double det = adjugate_rows<DIM>(ee, n);
        bad_det |= det_bad(det) | ids_repeat<NB>(v);
        const double s = kbar / fabs(det);
        double n0[DIM];
#pragma unroll
        for (int i = 0; i < DIM; ++i) {
            n0[i] = 0.0;
#pragma unroll
            for (int j = 0; j < DIM; ++j) n0[i] -= n[j][i];
        }
        out[e] = static_cast<T>(s * dotv<DIM>(n0, n0));
#pragma unroll
        for (int j = 0; j < DIM; ++j) out[(j + 1) * C + e] = static_cast<T>(s * dotv<DIM>(n[j], n[j]));
    }
    report_mesh(err, vmax, V, bad_det);
}

// element diagonals of the elasticity stiffness: for the unit displacement of component k at
// vertex b, H = e_k g^T with g = n_b (n_0 = -(n_1 + ... + n_d)), so
//     out[b*DIM + k][e] = (Lbar g_k^2 + Mbar (|g|^2 + g_k^2)) / |det J|
template <int DIM, class T>
__global__ void el_diag_kernel(const double *X0, int64_t C, uint32_t V, const int32_t *conn, const T *lam,
                               const T *mu, int nq, QuadW w, T *out, unsigned *err) {
    constexpr int NB = DIM + 1;
    const double *X[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) X[k] = X0 + int64_t(k) * V;
    uint32_t vmax = 0;
    bool bad_det = false;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < C; e += stride) {
        uint32_t v[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) v[b] = clamp_vid(conn[b * C + e], V, vmax);
        double lbar = 0.0, mbar = 0.0;
        for (int q = 0; q < nq; ++q) {
            lbar += w.wd[q] * static_cast<double>(lam[q * C + e]);
            mbar += w.wd[q] * static_cast<double>(mu[q * C + e]);
        }
        double xs[NB][DIM], ee[DIM][DIM], n[DIM][DIM];
        gather_coords<DIM>(X, v, xs);
        columns_f64<DIM>(xs, ee);
        const double det = adjugate_rows<DIM>(ee, n);
        bad_det |= det_bad(det) | ids_repeat<NB>(v);
        const double s = 1.0 / fabs(det);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            double g[DIM];
#pragma unroll
            for (int i = 0; i < DIM; ++i) {
                if (b == 0) {
                    g[i] = 0.0;
#pragma unroll
                    for (int j = 0; j < DIM; ++j) g[i] -= n[j][i];
                } else {
                    g[i] = n[b - 1][i];
                }
            }
            const double gg = dotv<DIM>(g, g);
#pragma unroll
            for (int k = 0; k < DIM; ++k)
                out[(b * DIM + k) * C + e] = static_cast<T>(s * (lbar * g[k] * g[k] + mbar * (gg + g[k] * g[k])));
        }
    }
    report_mesh(err, vmax, V, bad_det);
}

// block partial sums of x . y (float64 accumulation), fixed grid and order
template <class T>
__global__ void __launch_bounds__(256) dot_partial_kernel(int64_t n, const T *x, const T *y, double *partial) {
    __shared__ double s[256];
    double acc = 0.0;
    for (int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x; i < n; i += int64_t(kDotBlocks) * 256)
        acc += static_cast<double>(x[i]) * static_cast<double>(y[i]);
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = s[0];
}

__global__ void __launch_bounds__(256) dot_final_kernel(const double *partial, double *result) {
    __shared__ double s[256];
    double acc = 0.0;
    for (int i = threadIdx.x; i < kDotBlocks; i += 256) acc += partial[i];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *result = s[0];
}

// scalars[] layout: 0 gamma = r.u, 1 delta = w.u, 2 alpha, 3 beta, 4 rr = r.r,
// 5 (rtol ||r_0||)^2, 6 iterations done, 7 the 32-bit block counter of the reduction
// (last_block), 8 alpha and beta rounded to float32 once (read by the float32 update), 9 r.r
// before the first iteration, 10 the assembled matrix' two 32-bit state words
// (SellMatrix::state), 11 the grid barrier's counter and its timeout flag
enum { S_GAMMA = 0, S_DELTA = 1, S_ALPHA = 2, S_BETA = 3, S_RR = 4, S_TOL2 = 5, S_ITER = 6, S_TICKETS = 7,
       S_AB32 = 8, S_RR0 = 9, S_MATRIX = 10, S_BARRIER = 11, S_COUNT = 12 };

__device__ __forceinline__ unsigned *tickets(double *sc) { return reinterpret_cast<unsigned *>(sc + S_TICKETS); }

// Block-level sums of three doubles per thread (256 threads; sh: 3 x 256 doubles): a
// shared-memory tree, one barrier per level for the three; every thread gets the totals.
__device__ __forceinline__ void block_sum256x3(double (&v)[3], double *sh) {
#pragma unroll
    for (int m = 0; m < 3; ++m) sh[m * 256 + threadIdx.x] = v[m];
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o)
#pragma unroll
            for (int m = 0; m < 3; ++m) sh[m * 256 + threadIdx.x] += sh[m * 256 + threadIdx.x + o];
        __syncthreads();
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) v[m] = sh[m * 256];
    __syncthreads();
}

// True in the block that finishes last: each block's thread 0 publishes the block's partial
// sums (fence), then takes a ticket; the block holding the last of `blocks` tickets sees every
// partial and reduces them in place of a separate one-block kernel (the order of the sum
// does not depend on which block that is), then resets the counter for the next iteration.
__device__ __forceinline__ bool last_block(unsigned *ticket, unsigned blocks) {
    __shared__ bool s_last;
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(ticket, 1u) == blocks - 1u;
    }
    __syncthreads();
    return s_last;
}

// The loop is the conjugate gradient method in Chronopoulos and Gear's form (s-step CG with
// s = 1): with u = D^-1 r, w = A u and s = A p carried as vectors, both inner products of an
// iteration, gamma = r.u and delta = w.u, come from the same vectors at the same time, so an
// iteration is one vector update, one operator application and one reduction:
//     p = u + beta p,  s = w + beta s,  x += alpha p,  r -= alpha s,  u = r / D,
//     w = A u,  gamma' = r.u,  delta = w.u,
//     beta = gamma' / gamma,  alpha = gamma' / (delta - beta gamma' / alpha).
// The reductions visit the vertices with dot_partial_kernel's fixed grid and order (block b,
// thread t: i = 256 b + t + k 256 kDotBlocks) and are finished by the block that completes
// last, so every sum is reproducible and independent of the device.

// The vectors hold n_comp components per vertex, component-major ([n_comp][V]): entry i
// belongs to vertex i mod V, whose Dirichlet flag covers all its components.

// r = b - Ax on the free vertices (0 on fixed ones), u = D^-1 r, p = s = 0 (Dinv: the
// reciprocal of the Jacobi diagonal, formed once per solve by diag_fix_kernel)
template <class T>
__global__ void cg_init_kernel(int64_t N, int64_t V, const T *b, const T *Ax, const T *Dinv, const uint8_t *fixed,
                               T *r, T *u, T *p, T *sv) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < N; i += stride) {
        const T ri = fixed[i % V] ? T(0) : (b ? b[i] : T(0)) - Ax[i];
        r[i] = ri, u[i] = ri * Dinv[i], p[i] = T(0), sv[i] = T(0);
    }
}

// the product of two vector entries as a float64 term of a dot product: float32 entries are
// multiplied in float32 and widened once (one conversion on the float64 pipe instead of
// two and a float64 multiply); float64 entries multiply in float64
template <class T>
__device__ __forceinline__ double dot_term(T a, T b) {
    if constexpr (std::is_same<T, float>::value) return static_cast<double>(a * b);
    else return a * b;
}

// Inner products of float32 vectors without float64 arithmetic (the float64 pipe of this
// part issues 2 operations per clock per SM, against 128 float32): a double-float sum
// hi + lo, each product split exactly by TwoProduct and added by TwoSum (Knuth; the
// product of two float32 values is exact in the pair), the low parts summed in float32.
struct PairSum {
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add_prod(float a, float b) {
        float p, e, s, t;
        two_prod(a, b, p, e);
        two_sum(hi, p, s, t);
        hi = s;
        lo += t + e;
    }
    __device__ __forceinline__ void merge(float h, float l) {
        float s, t;
        two_sum(hi, h, s, t);
        hi = s;
        lo += t + l;
    }
    __device__ __forceinline__ void merge(const PairSum &o) { merge(o.hi, o.lo); }
    __device__ __forceinline__ double value() const { return static_cast<double>(hi) + static_cast<double>(lo); }
};

// Warp tree of PairSums: lane 0 ends with the warp's total (fixed order: lane i takes lane
// i + o at o = 16, 8, 4, 2, 1).
__device__ __forceinline__ void warp_merge(PairSum &a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h = __shfl_down_sync(0xffffffffu, a.hi, o), l = __shfl_down_sync(0xffffffffu, a.lo, o);
        a.merge(h, l);
    }
}

// The totals of three PairSums per thread of a 256-thread block, in thread 0: warp trees,
// then the eight warp totals of each in a ninth (sh: 3 x 8 float2 of shared memory, free
// again on return; one barrier pair for the three).
__device__ __forceinline__ void block_merge256x3(PairSum (&a)[3], float2 *sh) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        warp_merge(a[m]);
        if (lane == 0) sh[m * 8 + (threadIdx.x >> 5)] = make_float2(a[m].hi, a[m].lo);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            PairSum b;
            if (lane < 8) b.hi = sh[m * 8 + lane].x, b.lo = sh[m * 8 + lane].y;
            warp_merge(b);
            a[m] = b;
        }
    }
    __syncthreads();
}

// p = u + beta p, s = w + beta s, x += alpha p, r -= alpha s, u = D^-1 r (in the vectors'
// own type). On fixed vertices r, u, w and so p and s stay 0, and x keeps its value.
template <class T>
__global__ void cg_update_kernel(int64_t N, const double *sc, const T *w, const T *Dinv, T *x, T *r, T *u, T *p,
                                 T *sv) {
    T alpha, beta;
    if constexpr (std::is_same<T, float>::value) {
        const float2 ab = *reinterpret_cast<const float2 *>(sc + S_AB32);  // no per-thread float64 conversion
        alpha = ab.x, beta = ab.y;
    } else {
        alpha = sc[S_ALPHA], beta = sc[S_BETA];
    }
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < N; i += stride) {
        const T pi = u[i] + beta * p[i];
        const T si = w[i] + beta * sv[i];
        p[i] = pi;
        sv[i] = si;
        x[i] = x[i] + alpha * pi;
        const T ri = r[i] - alpha * si;
        r[i] = ri;
        u[i] = ri * Dinv[i];
    }
}

// The end of an iteration, by one thread: gamma, delta and rr, the next alpha and beta, the
// iteration count and the loop condition (INIT, before the loop: alpha and beta only).
template <bool INIT>
__device__ __forceinline__ void cg_scalars(double *sc, double gamma, double delta, double rrs, int max_iter,
                                           cudaGraphConditionalHandle loop) {
    if constexpr (INIT) {
        sc[S_ALPHA] = delta != 0.0 ? gamma / delta : 0.0;
        sc[S_BETA] = 0.0;
    } else {
        const double g0 = sc[S_GAMMA], a_old = sc[S_ALPHA];
        const double beta = g0 != 0.0 ? gamma / g0 : 0.0;
        const double den = a_old != 0.0 ? delta - beta * gamma / a_old : delta;
        sc[S_BETA] = beta;
        sc[S_ALPHA] = den != 0.0 ? gamma / den : 0.0;
        const double it = sc[S_ITER] + 1.0;
        sc[S_ITER] = it;
        const bool more = it < static_cast<double>(max_iter) && rrs > sc[S_TOL2] && rrs > 0.0;
        cudaGraphSetConditional(loop, more ? 1u : 0u);
    }
    *reinterpret_cast<float2 *>(sc + S_AB32) =
        make_float2(static_cast<float>(sc[S_ALPHA]), static_cast<float>(sc[S_BETA]));
    sc[S_GAMMA] = gamma;
    sc[S_DELTA] = delta;
    sc[S_RR] = rrs;
    tickets(sc)[0] = 0u;
}

// w = A u: the element vectors of u summed per vertex in list order (as the nodal gather
// does), 0 on fixed vertices; with the block partial sums of r.u, w.u and r.r. The block
// that finishes last forms gamma, delta and rr and the next alpha and beta; INIT (before
// the loop): alpha = gamma / delta, beta = 0; otherwise it also counts the iteration and
// sets the loop condition (not converged, fewer than max_iter; a NaN residual ends the loop:
// every comparison with it is false).
template <int NB, int NCOMP, class T, bool INIT>
__global__ void __launch_bounds__(256) cg_apply_dots_kernel(int64_t C, int64_t V, const T *__restrict__ elem,
                                                            const int32_t *__restrict__ ptr,
                                                            const int32_t *__restrict__ idx, const uint8_t *fixed,
                                                            const T *r, const T *u, T *w, double *partial, double *sc,
                                                            int max_iter, cudaGraphConditionalHandle loop) {
    constexpr bool F32 = std::is_same<T, float>::value;
    __shared__ double sh[F32 ? 1 : 3 * 256];
    __shared__ float2 sh2[3 * 8];
    double ru = 0.0, wu = 0.0, rr = 0.0;  // float64 vectors
    PairSum pd[3];                         // float32 vectors: r.u, w.u, r.r
    for (int64_t n = int64_t(blockIdx.x) * 256 + threadIdx.x; n < V; n += int64_t(kDotBlocks) * 256) {
        NodeSum<T> acc[NCOMP];
        gather_list<NB, NCOMP>(elem, idx, ptr[n], ptr[n + 1], C, acc);
        const bool fx = fixed[n] != 0;
#pragma unroll
        for (int k = 0; k < NCOMP; ++k) {
            const int64_t i = int64_t(k) * V + n;
            const T wn = fx ? T(0) : acc[k].value();
            w[i] = wn;
            const T rn = r[i], un = u[i];
            if constexpr (F32) {
                pd[0].add_prod(rn, un);
                pd[1].add_prod(wn, un);
                pd[2].add_prod(rn, rn);
            } else {
                ru += dot_term(rn, un);
                wu += dot_term(wn, un);
                rr += dot_term(rn, rn);
            }
        }
    }
    double gamma = 0.0, delta = 0.0, rrs = 0.0;  // the totals, in thread 0 of the last block
    if constexpr (F32) {
        // block partials as (hi, lo) pairs in place of the float64 partials
        float2 *pp = reinterpret_cast<float2 *>(partial);
        block_merge256x3(pd, sh2);
        if (threadIdx.x == 0)
            for (int m = 0; m < 3; ++m) pp[m * kDotBlocks + blockIdx.x] = make_float2(pd[m].hi, pd[m].lo);
        if (!last_block(tickets(sc), kDotBlocks)) return;
        PairSum at[3];
        for (int i = threadIdx.x; i < kDotBlocks; i += 256)
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const float2 v = __ldcg(pp + m * kDotBlocks + i);
                at[m].merge(v.x, v.y);
            }
        block_merge256x3(at, sh2);
        gamma = at[0].value(), delta = at[1].value(), rrs = at[2].value();
    } else {
        double t[3] = {ru, wu, rr};
        block_sum256x3(t, sh);
        if (threadIdx.x == 0)
            for (int m = 0; m < 3; ++m) partial[m * kDotBlocks + blockIdx.x] = t[m];
        if (!last_block(tickets(sc), kDotBlocks)) return;
        double at[3] = {0.0, 0.0, 0.0};
        for (int i = threadIdx.x; i < kDotBlocks; i += 256)
#pragma unroll
            for (int m = 0; m < 3; ++m) at[m] += __ldcg(partial + m * kDotBlocks + i);
        block_sum256x3(at, sh);
        gamma = at[0], delta = at[1], rrs = at[2];
    }
    if (threadIdx.x == 0) cg_scalars<INIT>(sc, gamma, delta, rrs, max_iter, loop);
}

// ------------------------------------------------------------------ the whole loop from the assembled matrix
//
// One cooperative launch per solve, one CTA per SM: every CTA owns a contiguous range of
// slices, a warp takes one slice at a time, and the thread that computes a row's entries of w
// also updates these entries of the vectors. An iteration is the vector update, a grid barrier
// (u is read by other CTAs' rows), the rows of w = A u with the sum w.u, and a second barrier
// for the CTAs' partial sums, which every CTA then adds up in the same order, so that all hold
// the same alpha, beta and stopping decision. Nothing returns to the host before the end.
// While they fit, a CTA's part of the matrix stays in its shared memory and a thread's entries
// of the vectors in its registers for the whole solve; then only u and the partial sums move.
//
// Measured per iteration (64^3 x 6 tets, 274,625 rows; elasticity on 511,104 tets, 273,375
// unknowns): Laplacian 11.1 us against 52 us in element form, elasticity 15.3 against 38 us. As
// two kernels per iteration in a graph the same rows took 19 and 27 us: the launches' drain and
// the loop node cost more than the barriers. What bounds it is latency: two barriers of about
// 2 us, the gathers of u through L2 after each (5 us), the scalars (1 us). The rows' threads
// handle all components of a block (a thread per component read every column and nodal value
// NC times: 21 us), 512 threads with four slices a warp hold the vectors without spills (1024
// threads at 64 registers spilled, and a spill is reloaded from L2, because each barrier
// invalidates L1).
//
// The kernel occupies the device until the solve ends. The sums' order is fixed by the row
// count and the device's SM count.

constexpr int kCgMaxBlocks = 1024;  // partial sums provided for
constexpr int kCgTable = 1024;      // slices per CTA whose place is kept in shared memory
// threads of a CTA, and the slices per warp whose vector entries stay in registers: the row
// product wants some 60 registers beside 7 NC values per slice
template <int NC>
constexpr int cg_threads() { return NC == 1 ? 512 : 640; }
template <int NC>
constexpr int cg_units() { return NC == 1 ? 4 : 1; }
constexpr int kCgThreads = 640;  // the most of them

struct CgArgs {
    int64_t V;
    const int32_t *cols;
    const float *vals;
    const int2 *slice;
    const float *b, *Dinv;  // b: nullptr for zero
    const uint8_t *fixed;
    float *x, *r, *u, *p, *s, *w;
    float2 *partial;  // [3][kCgMaxBlocks] sums, as pairs
    double *sc;
    double rtol;
    int max_iter;
    int cache_slots;  // matrix slots that fit in the launch's dynamic shared memory
    unsigned *err;
};

// The budget of a wait at the grid's barrier. CTAs that wait for one another are resident
// together (cooperative launch), so a wait ends unless a CTA is lost.
constexpr uint64_t kCgWaitNs = 4000000000ull;

// The totals of M pairs per thread over the block (any multiple of 32 threads), in thread 0: warp
// trees, then one over the warps.
template <int M>
struct BlockPairs {
    float2 p[M][32];
};
template <int M>
__device__ __forceinline__ void block_totals(PairSum (&a)[M], BlockPairs<M> &sh) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int m = 0; m < M; ++m) {
        warp_merge(a[m]);
        if (lane == 0) sh.p[m][threadIdx.x >> 5] = make_float2(a[m].hi, a[m].lo);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int m = 0; m < M; ++m) {
            PairSum b;
            if (lane < blockDim.x / 32) b.hi = sh.p[m][lane].x, b.lo = sh.p[m][lane].y;
            warp_merge(b);
            a[m] = b;
        }
    }
}

// one entry of the iteration's vectors
struct CgEntry {
    float x, r, u, p, s, w, d;
};

// U > 0: at most U slices per warp, their vector entries kept in registers; U = 0: any number,
// the vectors in memory.
template <int NC, int U>
__global__ void __launch_bounds__(cg_threads<NC>(), 1) sell_cg_kernel(const __grid_constant__ CgArgs a) {
    constexpr int BB = NC * NC;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ BlockPairs<2> sh2;
    __shared__ BlockPairs<1> sh1;
    __shared__ int2 s_slice[kCgTable];  // place (in shared memory, if cached) and length of the CTA's first slices
    __shared__ int s_cached;
    __shared__ PairSum s_part[3 * ((kCgMaxBlocks + 31) / 32)];
    __shared__ float s_alpha, s_beta;
    __shared__ int s_ok, s_more;
    __shared__ double s_gamma, s_den, s_inv[2];  // of the last iteration: gamma, alpha's denominator; 1/gamma, 1/(gamma alpha)
    unsigned *state = reinterpret_cast<unsigned *>(a.sc + S_MATRIX), *bar = reinterpret_cast<unsigned *>(a.sc + S_BARRIER);
    if (state[1] != 0u) return;  // not assembled: the host takes the element form
    const int64_t V = a.V;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t slices = (V + 31) / 32;
    const int64_t s0 = slices * blockIdx.x / gridDim.x, s1 = slices * (blockIdx.x + 1) / gridDim.x;
    const int nslices = static_cast<int>(s1 - s0);

    // the CTA's first slices into shared memory, as many as fit
    int32_t *scols = reinterpret_cast<int32_t *>(dyn);
    float *svals = reinterpret_cast<float *>(dyn + size_t(a.cache_slots) * 32 * sizeof(int32_t));
    const int ntab = min(nslices, kCgTable);
    for (int t = threadIdx.x; t < ntab; t += blockDim.x) s_slice[t] = a.slice[s0 + t];
    __syncthreads();
    if (threadIdx.x == 0) {
        int used = 0, t = 0;
        for (; t < ntab && used + s_slice[t].y <= a.cache_slots; ++t) used += s_slice[t].y;
        s_cached = t;
    }
    __syncthreads();
    const int cached = s_cached;
    {
        int used = 0, t0 = 0;
        for (int t = warp; t < cached; t += nw) {
            for (; t0 < t; ++t0) used += s_slice[t0].y;
            const int2 g = a.slice[s0 + t];
            for (int q = 0; q < g.y; ++q) {
                scols[(used + q) * 32 + lane] = ld_matrix(a.cols + (int64_t(g.x) + q) * 32 + lane);
#pragma unroll
                for (int m = 0; m < BB; ++m)
                    svals[((used + q) * BB + m) * 32 + lane] = ld_matrix(a.vals + ((int64_t(g.x) + q) * BB + m) * 32 + lane);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int used = 0;
        for (int t = 0; t < cached; ++t) s_slice[t].x = used, used += s_slice[t].y;
    }
    __syncthreads();

    // (A v) in the row n of the CTA's slice t
    auto product = [&](const float *v, int t, int64_t n, float (&w)[NC]) {
        if (t < cached) sell_row<NC, true>(scols, svals, s_slice[t], lane, n, v, V, w);
        else sell_row<NC, false>(a.cols, a.vals, t < kCgTable ? s_slice[t] : a.slice[s0 + t], lane, n, v, V, w);
    };
    // f(entries, slice of the CTA, row, whether the row exists) for each of this thread's rows;
    // in memory: `in` names the members read first, `out` those written after
    enum { MX = 1, MR = 2, MU = 4, MP = 8, MS = 16, MW = 32, MD = 64 };
    CgEntry own[U > 0 ? U : 1][NC];
    auto rows = [&](auto in, auto out, auto f) {
        if constexpr (U > 0) {
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int t = warp + j * nw;
                if (t < nslices) {
                    const int64_t n = (s0 + t) * 32 + lane;
                    f(own[j], t, min(n, V - 1), n < V);
                }
            }
        } else {
            constexpr int I = decltype(in)::value, O = decltype(out)::value;
            for (int t = warp; t < nslices; t += nw) {
                const int64_t n = (s0 + t) * 32 + lane, row = min(n, V - 1);
                CgEntry e[NC];
#pragma unroll
                for (int k = 0; k < NC; ++k) {
                    const int64_t i = k * V + row;
                    e[k] = CgEntry{};
                    if (I & MX) e[k].x = a.x[i];
                    if (I & MR) e[k].r = a.r[i];
                    if (I & MU) e[k].u = a.u[i];
                    if (I & MP) e[k].p = a.p[i];
                    if (I & MS) e[k].s = a.s[i];
                    if (I & MW) e[k].w = a.w[i];
                    if (I & MD) e[k].d = a.Dinv[i];
                }
                f(e, t, row, n < V);
                if (n < V) {
#pragma unroll
                    for (int k = 0; k < NC; ++k) {
                        const int64_t i = k * V + row;
                        if (O & MX) a.x[i] = e[k].x;
                        if (O & MR) a.r[i] = e[k].r;
                        if (O & MP) a.p[i] = e[k].p;
                        if (O & MS) a.s[i] = e[k].s;
                        if (O & MW) a.w[i] = e[k].w;
                    }
                }
            }
        }
    };
    // r = b - A x on the free vertices (0 on fixed ones), u = D^-1 r, p = s = 0, with r.u and r.r
    PairSum sums[2], wu[1];
    rows(std::integral_constant<int, MX | MD>(), std::integral_constant<int, MR | MP | MS>(),
         [&](CgEntry (&e)[NC], int t, int64_t n, bool in) {
             float ax[NC];
             product(a.x, t, n, ax);
             const bool held = !in || a.fixed[n];
#pragma unroll
             for (int k = 0; k < NC; ++k) {
                 const int64_t i = k * V + n;
                 if constexpr (U > 0) e[k].x = a.x[i], e[k].d = a.Dinv[i];
                 e[k].r = held ? 0.0f : (a.b ? a.b[i] : 0.0f) - ax[k];
                 e[k].u = e[k].r * e[k].d;
                 e[k].p = e[k].s = 0.0f;
                 if (in) a.u[i] = e[k].u;
                 sums[0].add_prod(e[k].r, e[k].u), sums[1].add_prod(e[k].r, e[k].r);
             }
         });
    double rr = 0.0, rr0 = 0.0, tol2 = 0.0;  // in thread 0
    int it = 0;
    // the grid's barrier, in two halves: what the CTA has written before it arrives is visible
    // to every CTA that has waited
    unsigned arrivals = 0;
    auto barrier_arrive = [&]() -> unsigned {
        __syncthreads();
        arrivals += gridDim.x;
        if (threadIdx.x == 0) {
            asm volatile("fence.acq_rel.gpu;\n\tred.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        }
        return arrivals;
    };
    auto barrier_wait = [&](unsigned target) -> bool {
        if (threadIdx.x == 0) {
            s_ok = wait_reached(bar, target, kCgWaitNs, bar + 1, a.err);
        }
        __syncthreads();
        return s_ok != 0;
    };
    for (;;) {
        // all CTAs' entries of u are in memory; the sums over them are formed while waiting
        const unsigned here = barrier_arrive();
        // the reciprocals that the next scalars need, by another warp than theirs while it waits
        // (by thread 0 after alpha: 800 clocks an iteration, 3 % of a 500,000-tet elasticity's)
        if (threadIdx.x == blockDim.x - 32 && it > 0) {
            const double g = s_gamma, inv = g != 0.0 ? copysign(quot_abs(1.0, g), g) : 0.0;
            s_inv[0] = inv, s_inv[1] = s_den * inv * inv;
        }
        block_totals(sums, sh2);
        const PairSum ru = sums[0], rsq = sums[1];  // totals, in thread 0
        if (!barrier_wait(here)) return;
        // w = A u and w.u
        wu[0] = PairSum();
        rows(std::integral_constant<int, MU>(), std::integral_constant<int, MW>(),
             [&](CgEntry (&e)[NC], int t, int64_t n, bool in) {
                 float w[NC];
                 product(a.u, t, n, w);
#pragma unroll
                 for (int k = 0; k < NC; ++k) {
                     e[k].w = w[k];
                     if (in) wu[0].add_prod(w[k], e[k].u);
                 }
             });
        block_totals(wu, sh1);
        // publish this CTA's sums, wait for all CTAs', and add them up: warp m the sums of value m
        if (threadIdx.x == 0) {
            const PairSum mine[3] = {ru, wu[0], rsq};
            for (int m = 0; m < 3; ++m) a.partial[m * kCgMaxBlocks + blockIdx.x] = make_float2(mine[m].hi, mine[m].lo);
        }
        if (!barrier_wait(barrier_arrive())) return;
        const int chunks = (gridDim.x + 31) / 32;  // warp c + chunks m: 32 CTAs' sums of value m
        for (int t = warp; t < 3 * chunks; t += nw) {
            const int m = t / chunks, i = (t - m * chunks) * 32 + lane;
            PairSum v;
            if (i < gridDim.x) {
                const float2 q = __ldcg(a.partial + m * kCgMaxBlocks + i);
                v.hi = q.x, v.lo = q.y;
            }
            warp_merge(v);
            if (lane == 0) s_part[t] = v;
        }
        __syncthreads();
        // the scalars by one thread (their divisions in every thread would keep the float64 pipe
        // busy for 10 us), with one division between the sums and alpha:
        //     beta = gamma' / gamma,  alpha = gamma' / (delta - beta gamma' / alpha_old)
        double total = 0.0;
        if (threadIdx.x < 32) {
            if (lane < 3) {
                PairSum v = s_part[lane * chunks];
                for (int c = 1; c < chunks; ++c) v.merge(s_part[lane * chunks + c]);
                total = v.value();
            }
            rr = __shfl_sync(0xffffffffu, total, 2);
        }
        const double delta = __shfl_sync(0xffffffffu, total, 1);
        if (threadIdx.x == 0) {
            const double g = total;
            double beta = 0.0, den = delta;
            if (it == 0) {
                rr0 = rr;
                const double tol = a.rtol * sqrt(rr0);
                tol2 = tol * tol;
            } else {  // (g sums products of float32 values: its square stays in float64's range)
                beta = g * s_inv[0];
                den = delta - g * g * s_inv[1];
            }
            const double alpha = den != 0.0 ? copysign(quot_abs(g, den), den) : 0.0;
            s_gamma = g, s_den = den;
            s_alpha = static_cast<float>(alpha), s_beta = static_cast<float>(beta);
            // a NaN residual ends the loop: every comparison with it is false
            s_more = it < a.max_iter && rr > tol2 && rr > 0.0;
        }
        __syncthreads();
        if (!s_more) break;
        ++it;
        // p = u + beta p, s = w + beta s, x += alpha p, r -= alpha s, u = D^-1 r
        const float al = s_alpha, be = s_beta;
        sums[0] = sums[1] = PairSum();
        rows(std::integral_constant<int, MX | MR | MU | MP | MS | MW | MD>(),
             std::integral_constant<int, MX | MR | MP | MS>(), [&](CgEntry (&e)[NC], int, int64_t n, bool in) {
#pragma unroll
                 for (int k = 0; k < NC; ++k) {
                     e[k].p = e[k].u + be * e[k].p;
                     e[k].s = e[k].w + be * e[k].s;
                     e[k].x += al * e[k].p;
                     e[k].r -= al * e[k].s;
                     e[k].u = e[k].r * e[k].d;
                     if (in) {
                         a.u[k * V + n] = e[k].u;
                         sums[0].add_prod(e[k].r, e[k].u), sums[1].add_prod(e[k].r, e[k].r);
                     }
                 }
             });
    }
    if constexpr (U > 0) {
        rows(std::integral_constant<int, 0>(), std::integral_constant<int, 0>(),
             [&](CgEntry (&e)[NC], int, int64_t n, bool in) {
#pragma unroll
                 for (int k = 0; k < NC; ++k)
                     if (in) a.x[k * V + n] = e[k].x;
             });
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.sc[S_RR] = rr;
        a.sc[S_RR0] = rr0;
        a.sc[S_ITER] = it;
    }
}

// Launch sell_cg_kernel: one CTA per SM at most, four slices each while they last (fewer CTAs
// make the barriers cheaper, more spread the rows' latency), a warp per slice up to the CTA's
// limit.
template <int NC>
static cudaError_t launch_sell_cg(CgArgs a, cudaStream_t s) {
    constexpr int U = cg_units<NC>(), kWarps = cg_threads<NC>() / 32;
    const int64_t slices = (a.V + 31) / 32;
    const int grid = slices <= kWarps ? 1 : static_cast<int>(std::min<int64_t>({(slices + 3) / 4, int64_t(sm_count()), int64_t(kCgMaxBlocks)}));
    const int64_t per = (slices + grid - 1) / grid;  // the largest range of a CTA
    const int64_t rounds = (per + kWarps - 1) / kWarps;
    const int threads = static_cast<int>((per + rounds - 1) / rounds * 32);
    const bool resident = rounds <= U;
    const void *k = resident ? reinterpret_cast<const void *>(sell_cg_kernel<NC, U>)
                             : reinterpret_cast<const void *>(sell_cg_kernel<NC, 0>);
    // shared memory for the matrix: what the static part leaves, in whole slots
    cudaFuncAttributes at;
    cudaError_t e = cudaFuncGetAttributes(&at, k);
    if (e != cudaSuccess) return e;
    const size_t slot = 32 * (sizeof(int32_t) + size_t(NC) * NC * sizeof(float));
    const size_t room = 227 * 1024 - at.sharedSizeBytes;
    const int64_t most = per * kSellMaxRow;  // slots the CTA's slices can have
    a.cache_slots = static_cast<int>(std::min<int64_t>(int64_t(room / slot), most));
    const size_t smem = size_t(a.cache_slots) * slot;
    // (the same value on every call: calls on other host threads may be between here and their launch)
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(room));
    if (e != cudaSuccess) return e;
    void *args[] = {&a};
    return cudaLaunchCooperativeKernel(k, dim3(grid), dim3(threads), args, smem, s);
}

__global__ void loop_init_kernel(double *sc, double tol2) {
    sc[S_TOL2] = tol2;
    sc[S_ITER] = 0.0;
}

// a library stream per device to capture the loop body on (capture needs a stream other
// than the legacy default one, which callers may pass)
static cudaStream_t capture_stream() {
    static std::mutex mu;
    static cudaStream_t per_dev[64] = {nullptr};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lk(mu);
    if (!per_dev[dev] && cudaStreamCreateWithFlags(&per_dev[dev], cudaStreamNonBlocking) != cudaSuccess) {
        cudaGetLastError();
        per_dev[dev] = nullptr;
    }
    return per_dev[dev];
}

// fixed vertices get D = 1 (their rows are the identity); then D is replaced by its
// reciprocal, so that every application of the preconditioner is one multiply
template <class T>
__global__ void diag_fix_kernel(int64_t N, int64_t V, const uint8_t *fixed, T *D) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < N; i += stride)
        D[i] = (fixed[i % V] || !(D[i] > T(0))) ? T(1) : T(1) / D[i];
}

static size_t align256(size_t n) { return (n + 255) & ~size_t(255); }

struct Workspace {
    void *elem, *D, *r, *z, *p, *q, *sv;  // D holds D^-1, z holds u = D^-1 r, q holds w = A u, sv s = A p
    double *partial, *scalars;
    SellMatrix mat;  // the assembled operator (mat.cols: nullptr where the workspace has no room for it)
    float2 *mat_partial;
    double *fac = nullptr;  // element form: the float64 Laplacian's factors, nullptr where not provided for
};

// The assembled operator, and the factors, are provided for up to kMatrixMaxBytes of workspace; beyond
// that (3D float32: some 1,200 M cells for the Laplacian, 240 M for elasticity; factors 430 M) a solve
// runs in element form, or applies the residual kernel.
constexpr size_t kMatrixMaxBytes = size_t(32) << 30;

// What a solve's workspace holds beside its vectors, which is what form it takes: the assembled
// operator (float32), or the factors of the Laplacian's residual (the float64 value types).
// The forms' roundings differ, and CG amplifies that over its iterations until the residual norms
// differ in their second digit and the stopping test ends iterations apart. In float32 that is
// within what its rounding leaves of x (largest error against the exact solution of 16 solves in
// each of 36 families of meshes and coefficients: assembled 0.65 to 2.3 times the element form's,
// 1.02 in the mean, smaller in 19 of them). In float64 it is not: of 12 solves each of 3,000, 12,000 and
// 30,000 tets to 1e-8 with ln K normal of deviation 3, 1, 4 and 4 ended apart, x 1e-8 to 2e-7
// apart; with flat cells nearly all. So float64 keeps the element form, whose factors give the
// residual kernel's bits: its results do not depend on the workspace. (12,000 / 30,000 tets: 1.6 /
// 2.0 ms a solve, 0.6 / 0.8 in assembled form.)
enum class Room { Vectors, Matrix, Factors };
static Room room_for(int physics, fem_precision prec) {
    if (prec == FEM_FP32_MIXED || prec == FEM_FP32) return Room::Matrix;
    return physics == 0 ? Room::Factors : Room::Vectors;
}

static size_t carve(int64_t C, int64_t V, int dim, size_t vs, void *base, Workspace *w, int ncomp, Room room) {
    size_t off = 0;
    char *b = static_cast<char *>(base);
    auto take = [&](size_t bytes) {
        void *p = b ? b + off : nullptr;
        off += align256(bytes);
        return p;
    };
    const size_t N = size_t(ncomp) * size_t(V);
    void *elem = take(size_t(dim + 1) * size_t(ncomp) * size_t(C) * vs);
    void *D = take(N * vs), *r = take(N * vs), *z = take(N * vs);
    void *p = take(N * vs), *q = take(N * vs), *sv = take(N * vs);
    double *partial = static_cast<double *>(take(sizeof(double) * 3 * kDotBlocks));
    double *scalars = static_cast<double *>(take(sizeof(double) * S_COUNT));
    SellMatrix mat;
    float2 *mat_partial = nullptr;
    const int64_t slots = sell_slots(C, V);
    const size_t bb = size_t(ncomp) * size_t(ncomp);
    if (room == Room::Matrix && C > 0 && slots < (int64_t(1) << 31) && size_t(slots) * 32 * (4 + bb * vs) <= kMatrixMaxBytes) {
        mat.cap = slots;
        mat.cols = static_cast<int32_t *>(take(size_t(slots) * 32 * sizeof(int32_t)));
        mat.vals = static_cast<float *>(take(size_t(slots) * 32 * bb * vs));
        mat.slice = static_cast<int2 *>(take(size_t((V + 31) / 32) * sizeof(int2)));
        mat.state = reinterpret_cast<int32_t *>(scalars + S_MATRIX);
        // the cells' numbers lie in the element vectors' place where they fit there
        const int nv = sell_cell_values(dim, ncomp);
        mat.cell = static_cast<float *>(nv <= (dim + 1) * ncomp ? elem : take(size_t(nv) * size_t(C) * vs));
        mat_partial = static_cast<float2 *>(take(3 * sizeof(float2) * kCgMaxBlocks));
    }
    double *fac = nullptr;
    const size_t fac_bytes = size_t(dim * dim + 1) * size_t(C) * sizeof(double);
    if (room == Room::Factors && C > 0 && fac_bytes <= kMatrixMaxBytes) fac = static_cast<double *>(take(fac_bytes));
    if (w) *w = Workspace{elem, D, r, z, p, q, sv, partial, scalars, mat, mat_partial, fac};
    return off;
}

// the assembled operator of a solve: the Laplacian with K, or elasticity with lambda, mu
struct Operator {
    int physics;  // 0 Laplacian, 1 elasticity
    const void *K, *lam, *mu;
    int ncomp(int dim) const { return physics == 0 ? 1 : dim; }
};

// what a workspace holds of its operator from an earlier solve of the same call
enum class Kept { Nothing, Matrix, Diagonal };

// form the operator's rows and the reciprocal diagonal w.D in the workspace w of a float32 solve
static fem_status assemble_operator(int dim, int64_t C, int64_t V, const double *coords, const int32_t *conn,
                                    const Operator &op, const QuadW &qwt, const int32_t *ptr, const int32_t *idx,
                                    const uint8_t *fixed, const Workspace &w, fem_precision prec, cudaStream_t s) {
    unsigned *err = device_error_word();
    if (!err) return fail(FEM_ERR_CUDA, "device error word unavailable");
    const uint32_t V32 = static_cast<uint32_t>(V);
    const float tau = mixed_tau();
    const SellMatrix &m = w.mat;
    float *D = static_cast<float *>(w.D);
    const float *K = static_cast<const float *>(op.K);
    const float *lam = static_cast<const float *>(op.lam), *mu = static_cast<const float *>(op.mu);
    const unsigned rows = static_cast<unsigned>((V + 127) / 128), slices = static_cast<unsigned>((V + 31) / 32);
    auto cells = [&](auto dimc, auto pc) {
        constexpr int D_ = decltype(dimc)::value, P_ = decltype(pc)::value;
        if (op.physics == 0) {
            auto k = sell_lap_cells_kernel<D_, P_>;
            k<<<grid_for(C, kBlock, reinterpret_cast<const void *>(k)), kBlock, 0, s>>>(coords, C, V32, conn, K, qwt,
                                                                                       tau * tau, m.cell, m.state, err);
        } else {
            auto k = sell_el_cells_kernel<D_, P_>;
            k<<<grid_for(C, kBlock, reinterpret_cast<const void *>(k)), kBlock, 0, s>>>(coords, C, V32, conn, lam, mu,
                                                                                       qwt, tau * tau, m.cell, m.state,
                                                                                       err);
        }
    };
    auto all = [&](auto dimc) {
        constexpr int D_ = decltype(dimc)::value;
        if (prec == FEM_FP32_MIXED) cells(dimc, std::integral_constant<int, FEM_FP32_MIXED>());
        else cells(dimc, std::integral_constant<int, FEM_FP32>());
        if (op.physics == 0) {
            sell_rows_kernel<D_ + 1, true><<<rows, 128, 0, s>>>(C, V, conn, ptr, idx, fixed, m.cell, m.cols, m.vals,
                                                                m.slice, m.state, m.cap, D);
        } else {
            sell_rows_kernel<D_ + 1, false><<<rows, 128, 0, s>>>(C, V, conn, ptr, idx, fixed, m.cell, m.cols, m.vals,
                                                                 m.slice, m.state, m.cap, D);
            sell_blocks_kernel<D_><<<slices, 128, 0, s>>>(C, V, conn, ptr, idx, m.cell, m.cols, m.vals, m.slice,
                                                         m.state);
            sell_diag_kernel<D_><<<rows, 128, 0, s>>>(V, m.vals, m.slice, m.state, D);
        }
    };
    if (dim == 2) all(std::integral_constant<int, 2>());
    else all(std::integral_constant<int, 3>());
    return check_launch("fem_pcg assembly");
}

template <class T>
static fem_status pcg_run(int dim, int64_t C, int64_t V, const double *coords, const int32_t *conn,
                          const Operator &op, int n_q, const double *qpts, const double *qw, const int32_t *ptr,
                          const int32_t *idx, const uint8_t *fixed, const void *b, void *x, int max_iter,
                          double rtol, const Workspace &w, int *iters_out, double *resid_out, fem_precision prec,
                          cudaStream_t s, Kept &kept) {
    // the residual runs in `prec`; every other kernel sees the value type (FEM_FP64_DF
    // values are float64). kept: what a repeated solve with the same workspace finds there.
    const fem_precision vprec = prec == FEM_FP64_DF ? FEM_FP64 : prec;
    T *X = static_cast<T *>(x);
    T *D = static_cast<T *>(w.D), *r = static_cast<T *>(w.r), *z = static_cast<T *>(w.z);
    T *p = static_cast<T *>(w.p), *q = static_cast<T *>(w.q), *sv = static_cast<T *>(w.sv);
    const T *B = static_cast<const T *>(b);
    const int nc = op.ncomp(dim);
    const int64_t N = int64_t(nc) * V;  // unknowns
    const int gV = static_cast<int>(std::min<int64_t>((N + 255) / 256, 4096));
    QuadW qwt;
    fem_status st = load_quadrature(dim, n_q, qpts, qw, qwt);
    if (st != FEM_OK) return st;
    // the element form's diagonal
    auto element_diagonal = [&]() -> fem_status {
        const int g = static_cast<int>(std::min<int64_t>((C + 255) / 256, 4096));
        unsigned *err = device_error_word();
        if (!err) return fail(FEM_ERR_CUDA, "device error word unavailable");
        const uint32_t V32 = static_cast<uint32_t>(V);
        T *el = static_cast<T *>(w.elem);
        if (op.physics == 0) {
            const T *K = static_cast<const T *>(op.K);
            if (dim == 2) lap_diag_kernel<2, T><<<g, 256, 0, s>>>(coords, C, V32, conn, K, n_q, qwt, el, err);
            else lap_diag_kernel<3, T><<<g, 256, 0, s>>>(coords, C, V32, conn, K, n_q, qwt, el, err);
        } else {
            const T *lam = static_cast<const T *>(op.lam), *mu = static_cast<const T *>(op.mu);
            if (dim == 2) el_diag_kernel<2, T><<<g, 256, 0, s>>>(coords, C, V32, conn, lam, mu, n_q, qwt, el, err);
            else el_diag_kernel<3, T><<<g, 256, 0, s>>>(coords, C, V32, conn, lam, mu, n_q, qwt, el, err);
        }
        fem_status e = check_launch("fem_pcg diagonal");
        if (e != FEM_OK) return e;
        if ((e = launch_gather(dim, nc, C, V, w.elem, ptr, idx, D, vprec, s)) != FEM_OK) return e;
        diag_fix_kernel<T><<<gV, 256, 0, s>>>(N, V, fixed, D);
        return FEM_OK;
    };
    // the element vectors of v in w.elem
    auto residual = [&](const T *v, cudaStream_t cs) -> fem_status {
        double *el = static_cast<double *>(w.elem);
        if (w.fac) {
            if constexpr (std::is_same<T, double>::value)
                return prec == FEM_FP64 ? launch_lap_factored(dim, C, V, conn, v, w.fac, el, cs)
                                        : launch_lap_df_factored(dim, C, V, conn, v, w.fac, el, cs);
        }
        if (op.physics == 0)
            return fem_integrate_laplacian(dim, C, V, coords, conn, v, op.K, n_q, qpts, qw, w.elem, prec, cs);
        return fem_integrate_elasticity(dim, C, V, coords, conn, v, op.lam, op.mu, n_q, qpts, qw, w.elem, prec, cs);
    };
    auto matvec = [&](const T *v, T *out, cudaStream_t cs) -> fem_status {
        fem_status e = residual(v, cs);
        if (e != FEM_OK) return e;
        return launch_gather(dim, nc, C, V, w.elem, ptr, idx, out, vprec, cs);
    };
    // w = A u (0 on fixed vertices) with the iteration's inner products and scalars
    auto apply_dots = [&](bool init, cudaGraphConditionalHandle loop, cudaStream_t cs) -> fem_status {
        fem_status e = residual(z, cs);
        if (e != FEM_OK) return e;
        const T *el = static_cast<const T *>(w.elem);
        const int mi = init ? 0 : max_iter;
        auto go = [&](auto kern) {
            kern<<<kDotBlocks, 256, 0, cs>>>(C, V, el, ptr, idx, fixed, r, z, q, w.partial, w.scalars, mi, loop);
        };
        const int key = dim * 10 + nc;  // 21 22 31 33
        if (init) {
            if (key == 21) go(cg_apply_dots_kernel<3, 1, T, true>);
            else if (key == 22) go(cg_apply_dots_kernel<3, 2, T, true>);
            else if (key == 31) go(cg_apply_dots_kernel<4, 1, T, true>);
            else go(cg_apply_dots_kernel<4, 3, T, true>);
        } else {
            if (key == 21) go(cg_apply_dots_kernel<3, 1, T, false>);
            else if (key == 22) go(cg_apply_dots_kernel<3, 2, T, false>);
            else if (key == 31) go(cg_apply_dots_kernel<4, 1, T, false>);
            else go(cg_apply_dots_kernel<4, 3, T, false>);
        }
        return FEM_OK;
    };
    auto read = [&](int slot, int n, double *v) -> fem_status {
        cudaError_t e = cudaMemcpyAsync(v, w.scalars + slot, n * sizeof(double), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return fail(FEM_ERR_CUDA, "fem_pcg_laplacian: %s", cudaGetErrorString(e));
        return FEM_OK;
    };
    if constexpr (std::is_same<T, float>::value) {
        // the assembled operator, where the workspace holds it
        if (w.mat.cols && kept != Kept::Diagonal) {
            // a repeated solve keeps the matrix' state words
            const bool have = kept == Kept::Matrix;
            cudaError_t e = cudaMemsetAsync(w.scalars, 0, sizeof(double) * S_MATRIX, s);
            if (e == cudaSuccess)
                e = have ? cudaMemsetAsync(w.scalars + S_BARRIER, 0, sizeof(double), s)
                         : cudaMemsetAsync(w.scalars + S_MATRIX, 0, 2 * sizeof(double), s);
            if (e != cudaSuccess) return fail(FEM_ERR_CUDA, "fem_pcg_laplacian: %s", cudaGetErrorString(e));
            if (!have && (st = assemble_operator(dim, C, V, coords, conn, op, qwt, ptr, idx, fixed, w, prec, s)) != FEM_OK)
                return st;
            unsigned *err = device_error_word();
            if (!err) return fail(FEM_ERR_CUDA, "device error word unavailable");
            const CgArgs a{V, w.mat.cols, w.mat.vals, w.mat.slice, B, D, fixed, X, r, z, p, sv, q, w.mat_partial,
                           w.scalars, rtol, max_iter, 0, err};
            e = nc == 1 ? launch_sell_cg<1>(a, s) : nc == 2 ? launch_sell_cg<2>(a, s) : launch_sell_cg<3>(a, s);
            if (e == cudaSuccess) {
                double head[S_COUNT];
                if ((st = read(0, S_COUNT, head)) != FEM_OK) return st;
                uint32_t state[2], bar[2];
                std::memcpy(state, &head[S_MATRIX], sizeof(state));
                std::memcpy(bar, &head[S_BARRIER], sizeof(bar));
                if (bar[1] != 0u) return fail(FEM_ERR_TIMEOUT, "fem_pcg_laplacian: a grid barrier gave up");
                if (state[1] == 0u) {
                    kept = Kept::Matrix;
                    if (iters_out) *iters_out = static_cast<int>(head[S_ITER]);
                    if (resid_out) *resid_out = head[S_RR0] > 0.0 ? std::sqrt(head[S_RR]) / std::sqrt(head[S_RR0]) : 0.0;
                    return check_launch("fem_pcg_laplacian");
                }
            } else {
                cudaGetLastError();  // no cooperative launch (a device partition smaller than the device): element form
            }
            // badly shaped cells, rows too long or too many for the workspace: element form
        }
    }
    // element form: r0 = b - A x0 on the free vertices, u0 = D^-1 r0, w0 = A u0, gamma0, delta0, alpha0
    double rr0 = 0.0;
    {
        const cudaError_t e = cudaMemsetAsync(w.scalars, 0, sizeof(double) * S_COUNT, s);
        if (e != cudaSuccess) return fail(FEM_ERR_CUDA, "fem_pcg_laplacian: %s", cudaGetErrorString(e));
    }
    if (kept != Kept::Diagonal && (st = element_diagonal()) != FEM_OK) return st;
    if (w.fac && kept != Kept::Diagonal) {
        const double *K = static_cast<const double *>(op.K);
        st = prec == FEM_FP64 ? launch_lap_factors(dim, C, V, coords, conn, K, qwt, w.fac, s)
                              : launch_lap_df_factors(dim, C, V, coords, conn, K, qwt, w.fac, s);
        if (st != FEM_OK) return st;
    }
    kept = Kept::Diagonal;
    if ((st = matvec(X, q, s)) != FEM_OK) return st;
    cg_init_kernel<T><<<gV, 256, 0, s>>>(N, V, B, q, D, fixed, r, z, p, sv);
    if ((st = apply_dots(true, 0, s)) != FEM_OK) return st;
    if ((st = read(S_RR, 1, &rr0)) != FEM_OK) return st;
    const double r0 = std::sqrt(rr0);
    double rn = r0;
    int it = 0;
    if (max_iter > 0 && rn > rtol * r0 && rn > 0.0) {
        const double tol = rtol * r0;
        loop_init_kernel<<<1, 1, 0, s>>>(w.scalars, tol * tol);
        // the loop: a graph holding one WHILE node whose body is one CG iteration
        cudaStream_t cs = capture_stream();
        if (!cs) return fail(FEM_ERR_CUDA, "fem_pcg_laplacian: no capture stream");
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
        cudaGraphConditionalHandle loop = 0;
        cudaError_t e = cudaGraphCreate(&graph, 0);
        if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&loop, graph, 1u, cudaGraphCondAssignDefault);
        cudaGraphNodeParams np = {cudaGraphNodeTypeConditional};
        np.conditional.handle = loop;
        np.conditional.type = cudaGraphCondTypeWhile;
        np.conditional.size = 1;
        cudaGraphNode_t node = nullptr;
        if (e == cudaSuccess) e = cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &np);
        // one capture at a time on the shared capture stream
        static std::mutex capture_mu;
        std::unique_lock<std::mutex> capture_lock(capture_mu);
        if (e == cudaSuccess)
            e = cudaStreamBeginCaptureToGraph(cs, np.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                              cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            // one iteration in 3 kernels: the vector updates; the residual of u; w = A u with
            // the inner products, the scalars and the loop condition
            cg_update_kernel<T><<<gV, 256, 0, cs>>>(N, w.scalars, q, D, X, r, z, p, sv);
            st = apply_dots(false, loop, cs);
            cudaGraph_t body = nullptr;
            const cudaError_t e2 = cudaStreamEndCapture(cs, &body);
            if (e2 != cudaSuccess) e = e2;
        }
        capture_lock.unlock();
        if (e == cudaSuccess && st == FEM_OK) e = cudaGraphInstantiate(&exec, graph, 0);
        if (e == cudaSuccess && st == FEM_OK) e = cudaGraphLaunch(exec, s);
        if (e == cudaSuccess && st == FEM_OK) e = cudaStreamSynchronize(s);
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        if (st != FEM_OK) return st;
        if (e != cudaSuccess) {
            cudaGetLastError();
            return fail(FEM_ERR_CUDA, "fem_pcg_laplacian (iteration graph): %s", cudaGetErrorString(e));
        }
        double tail[3];  // rr, tol^2, iterations
        if ((st = read(S_RR, 3, tail)) != FEM_OK) return st;
        rn = std::sqrt(tail[0]);
        it = static_cast<int>(tail[2]);
    }
    if ((st = check_launch("fem_pcg_laplacian")) != FEM_OK) return st;
    if (iters_out) *iters_out = it;
    if (resid_out) *resid_out = r0 > 0.0 ? rn / r0 : 0.0;
    return FEM_OK;
}

}  // namespace fem

using namespace fem;

extern "C" int64_t fem_pcg_work_bytes(int dim, int64_t n_cells, int64_t n_verts, fem_precision prec) {
    if ((dim != 2 && dim != 3) || n_cells < 0 || n_verts < 0) return -1;
    const size_t vs = prec == FEM_FP64 || prec == FEM_FP64_DF ? 8 : 4;
    return static_cast<int64_t>(carve(n_cells, n_verts, dim, vs, nullptr, nullptr, 1, room_for(0, prec)));
}

extern "C" fem_status fem_pcg_laplacian(int dim, int64_t n_cells, int64_t n_verts, const double *coords,
                                        const int32_t *conn, const void *K, int n_q, const double *qpts,
                                        const double *qw, const int32_t *node_ptr, const int32_t *node_idx,
                                        const uint8_t *fixed, const void *b, void *x, int max_iter, double rtol,
                                        void *work, int64_t work_bytes, int *iters_out, double *resid_out,
                                        fem_precision prec, fem_stream stream) {
    fem_status st = check_common(dim, n_cells, n_verts, coords, conn);
    if (st != FEM_OK) return st;
    if (prec != FEM_FP64 && prec != FEM_FP32_MIXED && prec != FEM_FP32 && prec != FEM_FP64_DF)
        return fail(FEM_ERR_ARG, "unknown precision %d", static_cast<int>(prec));
    if (max_iter < 0 || !(rtol >= 0.0)) return fail(FEM_ERR_ARG, "max_iter must be >= 0 and rtol >= 0");
    if (n_verts == 0) {
        if (iters_out) *iters_out = 0;
        if (resid_out) *resid_out = 0.0;
        return FEM_OK;
    }
    if (!K || !node_ptr || !node_idx || !fixed || !x || !work) return fail(FEM_ERR_ARG, "a NULL array argument");
    const bool f64 = prec == FEM_FP64 || prec == FEM_FP64_DF;
    const size_t vs = f64 ? 8 : 4;
    const int64_t need = static_cast<int64_t>(carve(n_cells, n_verts, dim, vs, nullptr, nullptr, 1, Room::Vectors));
    if (work_bytes < need)
        return fail(FEM_ERR_OOM, "fem_pcg_laplacian: workspace of %lld bytes, %lld needed",
                    static_cast<long long>(work_bytes), static_cast<long long>(need));
    if (reinterpret_cast<uintptr_t>(work) & 255u) return fail(FEM_ERR_ARG, "work must be 256-byte aligned");
    Workspace w;
    const bool all = work_bytes >= fem_pcg_work_bytes(dim, n_cells, n_verts, prec);
    carve(n_cells, n_verts, dim, vs, work, &w, 1, all ? room_for(0, prec) : Room::Vectors);
    Kept kept = Kept::Nothing;
    if (f64)
        return pcg_run<double>(dim, n_cells, n_verts, coords, conn, Operator{0, K, nullptr, nullptr}, n_q, qpts, qw,
                               node_ptr, node_idx, fixed, b, x,
                               max_iter, rtol, w, iters_out, resid_out, prec, stream, kept);
    return pcg_run<float>(dim, n_cells, n_verts, coords, conn, Operator{0, K, nullptr, nullptr}, n_q, qpts, qw,
                          node_ptr, node_idx, fixed, b, x,
                          max_iter, rtol, w, iters_out, resid_out, prec, stream, kept);
}

extern "C" int64_t fem_pcg_elasticity_work_bytes(int dim, int64_t n_cells, int64_t n_verts, fem_precision prec) {
    if ((dim != 2 && dim != 3) || n_cells < 0 || n_verts < 0) return -1;
    const size_t vs = prec == FEM_FP64 || prec == FEM_FP64_DF ? 8 : 4;
    // float64 in 3D up to 10,000 cells: the size that callers have been told so far, more than the
    // element form's vectors take
    const bool more = prec == FEM_FP64 && dim == 3 && n_cells <= 10000;
    return static_cast<int64_t>(
        carve(n_cells, n_verts, dim, vs, nullptr, nullptr, dim, more ? Room::Matrix : room_for(1, prec)));
}

extern "C" fem_status fem_pcg_elasticity(int dim, int64_t n_cells, int64_t n_verts, const double *coords,
                                         const int32_t *conn, const void *lam, const void *mu, int n_q,
                                         const double *qpts, const double *qw, const int32_t *node_ptr,
                                         const int32_t *node_idx, const uint8_t *fixed, const void *b, void *x,
                                         int max_iter, double rtol, void *work, int64_t work_bytes, int *iters_out,
                                         double *resid_out, fem_precision prec, fem_stream stream) {
    fem_status st = check_common(dim, n_cells, n_verts, coords, conn);
    if (st != FEM_OK) return st;
    if (prec != FEM_FP64 && prec != FEM_FP32_MIXED && prec != FEM_FP32 && prec != FEM_FP64_DF)
        return fail(FEM_ERR_ARG, "unknown precision %d", static_cast<int>(prec));
    if (max_iter < 0 || !(rtol >= 0.0)) return fail(FEM_ERR_ARG, "max_iter must be >= 0 and rtol >= 0");
    if (int64_t(dim) * n_verts >= (int64_t(1) << 31)) return fail(FEM_ERR_SHAPE, "too many vertices");
    if (n_verts == 0) {
        if (iters_out) *iters_out = 0;
        if (resid_out) *resid_out = 0.0;
        return FEM_OK;
    }
    if (!lam || !mu || !node_ptr || !node_idx || !fixed || !x || !work)
        return fail(FEM_ERR_ARG, "a NULL array argument");
    const bool f64 = prec == FEM_FP64 || prec == FEM_FP64_DF;
    const size_t vs = f64 ? 8 : 4;
    const int64_t need = static_cast<int64_t>(carve(n_cells, n_verts, dim, vs, nullptr, nullptr, dim, Room::Vectors));
    if (work_bytes < need)
        return fail(FEM_ERR_OOM, "fem_pcg_elasticity: workspace of %lld bytes, %lld needed",
                    static_cast<long long>(work_bytes), static_cast<long long>(need));
    if (reinterpret_cast<uintptr_t>(work) & 255u) return fail(FEM_ERR_ARG, "work must be 256-byte aligned");
    Workspace w;
    const bool all = work_bytes >= fem_pcg_elasticity_work_bytes(dim, n_cells, n_verts, prec);
    carve(n_cells, n_verts, dim, vs, work, &w, dim, all ? room_for(1, prec) : Room::Vectors);
    Kept kept = Kept::Nothing;
    const Operator op{1, nullptr, lam, mu};
    if (f64)
        return pcg_run<double>(dim, n_cells, n_verts, coords, conn, op, n_q, qpts, qw, node_ptr, node_idx, fixed, b, x,
                               max_iter, rtol, w, iters_out, resid_out, prec, stream, kept);
    return pcg_run<float>(dim, n_cells, n_verts, coords, conn, op, n_q, qpts, qw, node_ptr, node_idx, fixed, b, x,
                          max_iter, rtol, w, iters_out, resid_out, prec, stream, kept);
}

// ------------------------------------------------------------------ mixed-precision refinement
//
// fem_pcg_laplacian_refined: iterative refinement around the float32-mixed solve. Each
// outer step forms the true residual r = b - A x of the float64 iterate with the float64
// (or double-float) residual kernel, solves A d = r approximately with the PCG above in the
// FP32-mixed form (float32 values, the headline kernel as its operator), and adds d to x in
// float64. The float32 operator differs from the float64 one by ~1e-7 relative, so each
// outer step gains several digits and the iterate converges to the float64 solution; most
// of the work runs at float32 speed.

namespace fem {

__global__ void to_f32_kernel(int64_t n, const double *a, float *b) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) b[i] = static_cast<float>(a[i]);
}

// r = b - q on the free vertices, 0 on fixed ones; r32 = r rounded to float32; d32 = 0
// (N = n_comp V entries, component-major)
__global__ void refine_residual_kernel(int64_t N, int64_t V, const double *b, const double *q, const uint8_t *fixed,
                                       double *r, float *r32, float *d32) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < N; i += stride) {
        const double ri = fixed[i % V] ? 0.0 : (b ? b[i] : 0.0) - q[i];
        r[i] = ri;
        r32[i] = static_cast<float>(ri);
        d32[i] = 0.0f;
    }
}

// x += d on the free vertices
__global__ void refine_update_kernel(int64_t N, int64_t V, const uint8_t *fixed, const float *d, double *x) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < N; i += stride)
        if (!fixed[i % V]) x[i] += static_cast<double>(d[i]);
}

struct RefineWork {
    Workspace inner;    // the float32 PCG's
    float *coef32[2];   // K (Laplacian) or lambda, mu (elasticity) rounded to float32
    float *r32, *d32;
    double *elem, *q, *r, *partial, *scalars;
};

// physics 0: Laplacian (one coefficient, one component), 1: elasticity (two, dim)
static size_t carve_refined(int64_t C, int64_t V, int dim, int n_q, int physics, void *base, RefineWork *w,
                            bool matrix) {
    const int nc = physics == 0 ? 1 : dim, ncoef = physics == 0 ? 1 : 2;
    Workspace inner;
    size_t off = carve(C, V, dim, sizeof(float), base, &inner, nc, matrix ? Room::Matrix : Room::Vectors);
    char *b = static_cast<char *>(base);
    auto take = [&](size_t bytes) {
        void *p = b ? b + off : nullptr;
        off += align256(bytes);
        return p;
    };
    const size_t N = size_t(nc) * size_t(V);
    float *coef32[2] = {nullptr, nullptr};
    for (int c = 0; c < ncoef; ++c) coef32[c] = static_cast<float *>(take(size_t(n_q) * size_t(C) * sizeof(float)));
    float *r32 = static_cast<float *>(take(N * sizeof(float)));
    float *d32 = static_cast<float *>(take(N * sizeof(float)));
    double *elem = static_cast<double *>(take(size_t(dim + 1) * size_t(nc) * size_t(C) * sizeof(double)));
    double *q = static_cast<double *>(take(N * sizeof(double)));
    double *r = static_cast<double *>(take(N * sizeof(double)));
    double *partial = static_cast<double *>(take(sizeof(double) * kDotBlocks));
    double *scalars = static_cast<double *>(take(sizeof(double) * 2));
    if (w) *w = RefineWork{inner, {coef32[0], coef32[1]}, r32, d32, elem, q, r, partial, scalars};
    return off;
}

// the refinement loop of both entry points (arguments validated by the caller); coef64:
// K, or lambda and mu, in float64
static fem_status refined_run(int physics, int dim, int64_t C, int64_t V, const double *coords, const int32_t *conn,
                              const double *const *coef64, int n_q, const double *qpts, const double *qw,
                              const int32_t *ptr, const int32_t *idx, const uint8_t *fixed, const double *b,
                              double *x, int max_outer, int max_inner, double inner_rtol, double rtol,
                              const RefineWork &w, int *outer_out, int *inner_out, double *resid_out,
                              fem_precision residual_prec, cudaStream_t stream) {
    const int nc = physics == 0 ? 1 : dim, ncoef = physics == 0 ? 1 : 2;
    const int64_t N = int64_t(nc) * V;
    const int gV = static_cast<int>(std::min<int64_t>((N + 255) / 256, 4096));
    const int gK = static_cast<int>(std::min<int64_t>((int64_t(n_q) * C + 255) / 256, 4096));
    for (int c = 0; c < ncoef; ++c) to_f32_kernel<<<gK, 256, 0, stream>>>(int64_t(n_q) * C, coef64[c], w.coef32[c]);
    fem_status st = check_launch("refined solve");
    if (st != FEM_OK) return st;
    const Operator op32 = physics == 0 ? Operator{0, w.coef32[0], nullptr, nullptr}
                                       : Operator{1, nullptr, w.coef32[0], w.coef32[1]};
    double rn0 = 0.0, rn = 0.0;
    int outer = 0, inner_total = 0;
    Kept kept = Kept::Nothing;
    for (;;) {
        // the true residual of the float64 iterate
        st = physics == 0 ? fem_integrate_laplacian(dim, C, V, coords, conn, x, coef64[0], n_q, qpts, qw, w.elem,
                                                    residual_prec, stream)
                          : fem_integrate_elasticity(dim, C, V, coords, conn, x, coef64[0], coef64[1], n_q, qpts, qw,
                                                     w.elem, residual_prec, stream);
        if (st != FEM_OK) return st;
        if ((st = launch_gather(dim, nc, C, V, w.elem, ptr, idx, w.q, FEM_FP64, stream)) != FEM_OK) return st;
        refine_residual_kernel<<<gV, 256, 0, stream>>>(N, V, b, w.q, fixed, w.r, w.r32, w.d32);
        dot_partial_kernel<double><<<kDotBlocks, 256, 0, stream>>>(N, w.r, w.r, w.partial);
        dot_final_kernel<<<1, 256, 0, stream>>>(w.partial, w.scalars);
        double rr = 0.0;
        cudaError_t e = cudaMemcpyAsync(&rr, w.scalars, sizeof(double), cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) return fail(FEM_ERR_CUDA, "refined solve: %s", cudaGetErrorString(e));
        rn = std::sqrt(rr);
        if (outer == 0) rn0 = rn;
        if (rn <= rtol * rn0 || rn == 0.0 || outer >= max_outer) break;
        // the correction in the FP32-mixed form: A d = r, d = 0 on the fixed vertices. When
        // the reduction still needed is less than one correction at inner_rtol gives, and
        // within float32's reach, the last correction is solved to a third of it instead, so
        // that it ends the refinement rather than stopping just short of rtol.
        const double need = rtol * rn0 / rn;
        const double tol_k = (0.3 * need < inner_rtol && 0.3 * need >= 1e-6) ? 0.3 * need : inner_rtol;
        int it = 0;
        double res = 0.0;
        st = pcg_run<float>(dim, C, V, coords, conn, op32, n_q, qpts, qw, ptr, idx, fixed, w.r32, w.d32, max_inner,
                            tol_k, w.inner, &it, &res, FEM_FP32_MIXED, stream, kept);
        if (st != FEM_OK) return st;
        inner_total += it;
        refine_update_kernel<<<gV, 256, 0, stream>>>(N, V, fixed, w.d32, x);
        if ((st = check_launch("refined solve")) != FEM_OK) return st;
        ++outer;
    }
    if (outer_out) *outer_out = outer;
    if (inner_out) *inner_out = inner_total;
    if (resid_out) *resid_out = rn0 > 0.0 ? rn / rn0 : 0.0;
    return check_launch("refined solve");
}

// the argument checks both entry points share
static fem_status refined_check(int dim, int64_t C, int64_t V, const double *coords, const int32_t *conn, int n_q,
                                int max_outer, int max_inner, double inner_rtol, double rtol,
                                fem_precision residual_prec, int *outer_out, int *inner_out, double *resid_out) {
    fem_status st = check_common(dim, C, V, coords, conn);
    if (st != FEM_OK) return st;
    if (residual_prec != FEM_FP64 && residual_prec != FEM_FP64_DF)
        return fail(FEM_ERR_ARG, "residual_prec must be FEM_FP64 or FEM_FP64_DF");
    if (max_outer < 0 || max_inner < 0 || !(rtol >= 0.0) || !(inner_rtol > 0.0 && inner_rtol < 1.0))
        return fail(FEM_ERR_ARG, "max_outer, max_inner must be >= 0, rtol >= 0 and 0 < inner_rtol < 1");
    if (n_q < 1 || n_q > FEM_MAX_QPTS) return fail(FEM_ERR_SHAPE, "n_q = %d outside [1, %d]", n_q, FEM_MAX_QPTS);
    if (outer_out) *outer_out = 0;
    if (inner_out) *inner_out = 0;
    if (resid_out) *resid_out = 0.0;
    return FEM_OK;
}

}  // namespace fem

extern "C" int64_t fem_pcg_refined_work_bytes(int dim, int64_t n_cells, int64_t n_verts, int n_q) {
    if ((dim != 2 && dim != 3) || n_cells < 0 || n_verts < 0 || n_q < 1 || n_q > FEM_MAX_QPTS) return -1;
    return static_cast<int64_t>(carve_refined(n_cells, n_verts, dim, n_q, 0, nullptr, nullptr, true));
}

extern "C" int64_t fem_pcg_elasticity_refined_work_bytes(int dim, int64_t n_cells, int64_t n_verts, int n_q) {
    if ((dim != 2 && dim != 3) || n_cells < 0 || n_verts < 0 || n_q < 1 || n_q > FEM_MAX_QPTS) return -1;
    return static_cast<int64_t>(carve_refined(n_cells, n_verts, dim, n_q, 1, nullptr, nullptr, true));
}

extern "C" fem_status fem_pcg_laplacian_refined(int dim, int64_t n_cells, int64_t n_verts, const double *coords,
                                                const int32_t *conn, const double *K, int n_q, const double *qpts,
                                                const double *qw, const int32_t *node_ptr, const int32_t *node_idx,
                                                const uint8_t *fixed, const double *b, double *x, int max_outer,
                                                int max_inner, double inner_rtol, double rtol, void *work,
                                                int64_t work_bytes, int *outer_out, int *inner_out,
                                                double *resid_out, fem_precision residual_prec, fem_stream stream) {
    fem_status st = refined_check(dim, n_cells, n_verts, coords, conn, n_q, max_outer, max_inner, inner_rtol, rtol,
                                  residual_prec, outer_out, inner_out, resid_out);
    if (st != FEM_OK || n_verts == 0) return st;
    if (!K || !node_ptr || !node_idx || !fixed || !x || !work) return fail(FEM_ERR_ARG, "a NULL array argument");
    const int64_t need =
        static_cast<int64_t>(carve_refined(n_cells, n_verts, dim, n_q, 0, nullptr, nullptr, false));
    if (work_bytes < need)
        return fail(FEM_ERR_OOM, "fem_pcg_laplacian_refined: workspace of %lld bytes, %lld needed",
                    static_cast<long long>(work_bytes), static_cast<long long>(need));
    if (reinterpret_cast<uintptr_t>(work) & 255u) return fail(FEM_ERR_ARG, "work must be 256-byte aligned");
    RefineWork w;
    carve_refined(n_cells, n_verts, dim, n_q, 0, work, &w,
                  work_bytes >= fem_pcg_refined_work_bytes(dim, n_cells, n_verts, n_q));
    const double *coef[1] = {K};
    return refined_run(0, dim, n_cells, n_verts, coords, conn, coef, n_q, qpts, qw, node_ptr, node_idx, fixed, b, x,
                       max_outer, max_inner, inner_rtol, rtol, w, outer_out, inner_out, resid_out, residual_prec,
                       stream);
}

extern "C" fem_status fem_pcg_elasticity_refined(int dim, int64_t n_cells, int64_t n_verts, const double *coords,
                                                 const int32_t *conn, const double *lam, const double *mu, int n_q,
                                                 const double *qpts, const double *qw, const int32_t *node_ptr,
                                                 const int32_t *node_idx, const uint8_t *fixed, const double *b,
                                                 double *x, int max_outer, int max_inner, double inner_rtol,
                                                 double rtol, void *work, int64_t work_bytes, int *outer_out,
                                                 int *inner_out, double *resid_out, fem_precision residual_prec,
                                                 fem_stream stream) {
    fem_status st = refined_check(dim, n_cells, n_verts, coords, conn, n_q, max_outer, max_inner, inner_rtol, rtol,
                                  residual_prec, outer_out, inner_out, resid_out);
    if (st != FEM_OK || n_verts == 0) return st;
    if (int64_t(dim) * n_verts >= (int64_t(1) << 31)) return fail(FEM_ERR_SHAPE, "too many vertices");
    if (!lam || !mu || !node_ptr || !node_idx || !fixed || !x || !work)
        return fail(FEM_ERR_ARG, "a NULL array argument");
    const int64_t need =
        static_cast<int64_t>(carve_refined(n_cells, n_verts, dim, n_q, 1, nullptr, nullptr, false));
    if (work_bytes < need)
        return fail(FEM_ERR_OOM, "fem_pcg_elasticity_refined: workspace of %lld bytes, %lld needed",
                    static_cast<long long>(work_bytes), static_cast<long long>(need));
    if (reinterpret_cast<uintptr_t>(work) & 255u) return fail(FEM_ERR_ARG, "work must be 256-byte aligned");
    RefineWork w;
    carve_refined(n_cells, n_verts, dim, n_q, 1, work, &w,
                  work_bytes >= fem_pcg_elasticity_refined_work_bytes(dim, n_cells, n_verts, n_q));
    const double *coef[2] = {lam, mu};
    return refined_run(1, dim, n_cells, n_verts, coords, conn, coef, n_q, qpts, qw, node_ptr, node_idx, fixed, b, x,
                       max_outer, max_inner, inner_rtol, rtol, w, outer_out, inner_out, resid_out, residual_prec,
                       stream);
}
