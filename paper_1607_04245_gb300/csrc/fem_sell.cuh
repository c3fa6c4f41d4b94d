// fem_sell.cuh -- the assembled operator of the float32 PCG solves, built on the device inside
// the call and stored in sliced ELLPACK form.
//
// A solve applies one operator hundreds of times, and per application the element form costs
// the geometry of every cell again, the element vectors' trip to memory and the scattered
// vertex sum over them. Assembled, the operator of a P1 mesh has one entry per pair of
// vertices that share a cell (about 14 per vertex in 3D, 6 in 2D). Its constant fields give
// zero (sum_b grad phi_b = 0 on every cell), so the diagonal is minus the sum of the row's
// other entries and an application is
//     w_i = sum_{j != i} A_ij (u_j - u_i),
// from the off-diagonal entries alone: differences of nodal values, as the element kernels
// form them, so that a constant (elasticity: a rigid translation) gives exactly zero and no
// digits of a smooth field are lost to the cancellation of a_ii u_i against the rest.
//
// Storage: slices of 32 rows (one warp); slice s holds len slots of 32 lanes, slot k of lane l
// at (off + k) * 32 + l, so that every read of cols and vals is coalesced. Rows shorter than
// their slice's longest are padded with (own row, 0), which contributes 0 * (u_i - u_i).
// For vector fields an entry is an NC x NC block, its component (k, i) at
// ((off + slot) * NC * NC + k * NC + i) * 32 + lane. Slices take their room with one atomic
// each: where a slice lies depends on the order in which warps arrive, what it holds does not
// (a row's entries are in the order in which its sorted cell list meets them), so results
// are bitwise reproducible. Rows of Dirichlet vertices are left empty (w = 0 there).
//
// A mesh with cells that the mixed form's shape test rejects is not assembled: the residual
// kernels apply such cells in float64, and their large entries rounded to float32 would lose what
// cancels between them (8^3 x 6 tets flattened to 1e-2 and 1e-3, a smooth field, the rounding of
// the entries alone: errors of one application 1.4e-6 and 6.2e-6 of its largest value; 2.4e-8 and
// 5.2e-8 with such cells in float64).
#pragma once

#include "fem_cell.cuh"

namespace fem {

constexpr int kSellMaxRow = 64;  // longest row that is assembled; a mesh with a longer one is solved in element form

struct SellMatrix {
    int32_t *cols = nullptr;   // [cap][32]; nullptr: no room in the workspace, element form
    float *vals = nullptr;     // [cap][NC * NC][32]
    int2 *slice = nullptr;     // (off, len) per slice of 32 rows
    int32_t *state = nullptr;  // [0] slots taken, [1] nonzero: element form (1: did not fit, 2: badly shaped cells)
    float *cell = nullptr;     // per-cell numbers the rows are summed from (sell_cell_values())
    int64_t cap = 0;           // slots
};

// slots provided for: 2E directed vertex pairs of a conforming mesh are 2V + 2C plus (3D) its
// boundary faces; half as much again for padding and boundary, and a floor for tiny meshes
inline int64_t sell_slots(int64_t C, int64_t V) { return (3 * (V + C)) / 32 + 2 * ((V + 31) / 32) + 64; }

// values per cell that the rows are assembled from: the Laplacian's off-diagonal entries, one
// per pair of local vertices; elasticity: d adjugate rows and the two Lame sums, padded to a
// multiple of 16 bytes
__host__ __device__ constexpr int sell_cell_values(int dim, int nc) {
    return nc == 1 ? dim * (dim + 1) / 2 : (dim == 3 ? 12 : 6);
}

// index of the pair (a, b), a != b, of a simplex' NB vertices: (0,1) (0,2) .. (1,2) ..
template <int NB>
__device__ __forceinline__ int pair_index(int a, int b) {
    const int lo = min(a, b), hi = max(a, b);
    return lo * (2 * NB - lo - 1) / 2 + hi - lo - 1;
}

// ------------------------------------------------------------------ per-cell numbers

// Off-diagonal entries of the Laplacian's element matrices, Kbar (n_a . n_b) / |det J|, in the
// geometry of the precision form P. The mixed form's badly shaped cells are recorded in state.
template <int DIM, int P>
__global__ void __launch_bounds__(kBlock) sell_lap_cells_kernel(const double *X0, int64_t C, uint32_t V,
                                                                const int32_t *conn, const float *K, QuadW w,
                                                                float tau2, float *out, int32_t *state, unsigned *err) {
    constexpr int NB = DIM + 1, NP = sell_cell_values(DIM, 1);
    const double *X[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) X[k] = X0 + int64_t(k) * V;
    uint32_t vmax = 0;
    bool bad_det = false, bad_shape = false;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < C; e += stride) {
        uint32_t v[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) v[b] = clamp_vid(ld_stream(conn + b * C + e), V, vmax);
        qsum_t<P> ks;
        ks.first(w.wf[0], ld_stream(K + e));
        for (int q = 1; q < w.nq; ++q) ks.add(w.wf[q], ld_stream(K + q * C + e));
        double xs[NB][DIM];
        gather_coords<DIM>(X, v, xs);
        float ec[DIM][DIM], n[DIM][DIM];
        if constexpr (P == FEM_FP32_MIXED) columns_mixed<DIM>(xs, ec);
        else columns_f32<DIM>(xs, ec);
        const float det = adjugate_rows<DIM>(ec, n);
        if constexpr (P == FEM_FP32_MIXED) {
            if (!shape_ok<DIM>(ec, det, tau2)) {
                bad_shape = true;
                continue;
            }
        } else {
            bad_det |= det_bad(det) | ids_repeat<NB>(v);
        }
        const float s = quot_abs(ks.value(), det);
        float n0[DIM];
#pragma unroll
        for (int i = 0; i < DIM; ++i) {
            n0[i] = n[0][i];
#pragma unroll
            for (int j = 1; j < DIM; ++j) n0[i] = n0[i] + n[j][i];
        }
        float r[NP];
        int p = 0;
#pragma unroll
        for (int b = 0; b < DIM; ++b) r[p++] = -(s * dotv<DIM>(n0, n[b]));
#pragma unroll
        for (int a = 0; a < DIM; ++a)
#pragma unroll
            for (int b = a + 1; b < DIM; ++b) r[p++] = s * dotv<DIM>(n[a], n[b]);
        if constexpr (NP == 6) {
            float2 *dst = reinterpret_cast<float2 *>(out + e * NP);
#pragma unroll
            for (int i = 0; i < 3; ++i) dst[i] = float2{r[2 * i], r[2 * i + 1]};
        } else {
#pragma unroll
            for (int i = 0; i < NP; ++i) out[e * NP + i] = r[i];
        }
    }
    if (bad_shape) atomicOr(state + 1, 2);
    report_mesh(err, vmax, V, bad_det);
}

// Elasticity: the adjugate rows g_1 .. g_d and the factors sl, sm of the entries' blocks
//     A_ab[k][i] = sl g_a[k] g_b[i] + sm (g_a[i] g_b[k] + delta_ki g_a . g_b),
// g_0 = -(g_1 + .. + g_d), with g = n / sqrt|det J|, sl = Lbar, sm = Mbar, which stay in
// float32's range wherever the entries do (n ~ L^2 and 1 / |det J| ~ L^-3 would not).
template <int DIM, int P>
__global__ void __launch_bounds__(kBlock) sell_el_cells_kernel(const double *X0, int64_t C, uint32_t V,
                                                               const int32_t *conn, const float *lam,
                                                               const float *mu, QuadW w, float tau2,
                                                               float *out, int32_t *state, unsigned *err) {
    constexpr int NB = DIM + 1, NV = sell_cell_values(DIM, DIM);
    const double *X[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) X[k] = X0 + int64_t(k) * V;
    uint32_t vmax = 0;
    bool bad_det = false, bad_shape = false;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < C; e += stride) {
        uint32_t v[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) v[b] = clamp_vid(ld_stream(conn + b * C + e), V, vmax);
        qsum_t<P> ls, ms;
        ls.first(w.wf[0], ld_stream(lam + e));
        ms.first(w.wf[0], ld_stream(mu + e));
        for (int q = 1; q < w.nq; ++q) {
            ls.add(w.wf[q], ld_stream(lam + q * C + e));
            ms.add(w.wf[q], ld_stream(mu + q * C + e));
        }
        double xs[NB][DIM];
        gather_coords<DIM>(X, v, xs);
        float ec[DIM][DIM], n[DIM][DIM];
        if constexpr (P == FEM_FP32_MIXED) columns_mixed<DIM>(xs, ec);
        else columns_f32<DIM>(xs, ec);
        const float det = adjugate_rows<DIM>(ec, n);
        if constexpr (P == FEM_FP32_MIXED) {
            if (!shape_ok<DIM>(ec, det, tau2)) {
                bad_shape = true;
                continue;
            }
        } else {
            bad_det |= det_bad(det) | ids_repeat<NB>(v);
        }
        float r[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) r[i] = 0.0f;
        const float y = __frsqrt_rn(fabsf(det));
#pragma unroll
        for (int j = 0; j < DIM; ++j)
#pragma unroll
            for (int i = 0; i < DIM; ++i) r[j * DIM + i] = n[j][i] * y;
        r[DIM * DIM] = ls.value(), r[DIM * DIM + 1] = ms.value();
        float2 *dst = reinterpret_cast<float2 *>(out + e * NV);
#pragma unroll
        for (int i = 0; i < NV / 2; ++i) dst[i] = float2{r[2 * i], r[2 * i + 1]};
    }
    if (bad_shape) atomicOr(state + 1, 2);
    report_mesh(err, vmax, V, bad_det);
}

// ------------------------------------------------------------------ rows

// sums of a row's entries, compensated (TwoSum, as the nodal sum)
struct RowSums {
    float2 s[kSellMaxRow];
    __device__ __forceinline__ void start(int p, float x) { s[p] = make_float2(x, 0.0f); }
    __device__ __forceinline__ void add(int p, float x) {
        float t, e;
        const float2 o = s[p];
        two_sum(o.x, x, t, e);
        s[p] = make_float2(t, o.y + e);
    }
    __device__ __forceinline__ float value(int p) const { return s[p].x + s[p].y; }
};

// The rows' columns (and, LAP, their entries and the reciprocal diagonal): one thread per row
// walks the row's cells in list order, looks every other vertex up among the columns found so
// far (a per-thread array: rows have about 14 entries) and appends it if it is new; the warp's
// longest row is the slice's length.
template <int NB, bool LAP>
__global__ void __launch_bounds__(128) sell_rows_kernel(int64_t C, int64_t V, const int32_t *__restrict__ conn,
                                                        const int32_t *__restrict__ ptr,
                                                        const int32_t *__restrict__ idx, const uint8_t *fixed,
                                                        const float *__restrict__ cell, int32_t *cols, float *vals,
                                                        int2 *slice, int32_t *state, int64_t cap, float *Dinv) {
    if (state[1] & 2) return;  // badly shaped cells: not assembled
    constexpr int NP = NB * (NB - 1) / 2;
    const int64_t n = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    int32_t col[kSellMaxRow];
    RowSums sum;
    int m = 0;
    bool over = false;
    if (n < V && !fixed[n]) {
        const int32_t e1 = ptr[n + 1];
        for (int32_t j = ptr[n]; j < e1 && !over; ++j) {
            const int32_t t = __ldg(idx + j);
            const int32_t c = t / NB, a = t - c * NB;
#pragma unroll
            for (int o = 1; o < NB; ++o) {
                const int b = a + o < NB ? a + o : a + o - NB;
                const int32_t v = static_cast<int32_t>(clamp_vid(__ldg(conn + b * C + c), static_cast<uint32_t>(V)));
                if (v == n) continue;  // repeated vertex (reported by the cell pass)
                float x = 0.0f;
                if constexpr (LAP) x = __ldg(cell + int64_t(c) * NP + pair_index<NB>(a, b));
                int p = 0;
                while (p < m && col[p] != v) ++p;
                if (p < m) {
                    if constexpr (LAP) sum.add(p, x);
                } else if (m < kSellMaxRow) {
                    col[m] = v;
                    if constexpr (LAP) sum.start(m, x);
                    ++m;
                } else {
                    over = true;
                }
            }
        }
    }
    int len = m;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) len = max(len, __shfl_xor_sync(0xffffffffu, len, o));
    const bool any_over = __any_sync(0xffffffffu, over);
    int off = 0;
    if (lane == 0) {
        off = atomicAdd(state, len);
        if (any_over || int64_t(off) + len > cap) atomicOr(reinterpret_cast<unsigned *>(state) + 1, 1u);
    }
    off = __shfl_sync(0xffffffffu, off, 0);
    if (any_over || int64_t(off) + len > cap) len = 0;
    if (lane == 0 && n < V) slice[n >> 5] = make_int2(off, len);
    float d = 0.0f;
    for (int k = 0; k < len; ++k) {
        const int64_t at = (int64_t(off) + k) * 32 + lane;
        cols[at] = k < m ? col[k] : static_cast<int32_t>(min(n, V - 1));
        if constexpr (LAP) {
            const float x = k < m ? sum.value(k) : 0.0f;
            vals[at] = x;
            d -= x;
        }
    }
    if constexpr (LAP) {
        if (n < V) Dinv[n] = d > 0.0f ? 1.0f / d : 1.0f;
    }
}

// Elasticity: the blocks. A warp takes one slot of a slice, its lanes the 32 rows: each lane
// walks its row's cells in list order and sums the blocks of those that hold its column, in
// registers.
template <int DIM>
__global__ void __launch_bounds__(128) sell_blocks_kernel(int64_t C, int64_t V, const int32_t *__restrict__ conn,
                                                          const int32_t *__restrict__ ptr,
                                                          const int32_t *__restrict__ idx,
                                                          const float *__restrict__ cell, const int32_t *cols, float *vals,
                                                          const int2 *slice, const int32_t *state) {
    if (state[1] != 0) return;  // not assembled
    constexpr int NB = DIM + 1, NV = sell_cell_values(DIM, DIM), BB = DIM * DIM;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t s = blockIdx.x;  // one slice per CTA, its slots over the warps
    const int2 sl = slice[s];
    const int64_t n = s * 32 + lane;
    const int32_t j0 = n < V ? ptr[n] : 0, j1 = n < V ? ptr[n + 1] : 0;
    for (int k = warp; k < sl.y; k += nw) {
        const int64_t slot = int64_t(sl.x) + k;
        const int32_t want = cols[slot * 32 + lane];
        NodeSum<float> acc[BB];
        if (want != n) {
            for (int32_t j = j0; j < j1; ++j) {
                const int32_t t = __ldg(idx + j);
                const int32_t c = t / NB, a = t - c * NB;
                int b = -1;
#pragma unroll
                for (int o = 0; o < NB; ++o)
                    if (o != a && static_cast<int32_t>(clamp_vid(__ldg(conn + o * C + c), static_cast<uint32_t>(V))) == want) b = o;
                if (b < 0) continue;
                const float *g = cell + int64_t(c) * NV;
                float ga[DIM], gb[DIM];
#pragma unroll
                for (int i = 0; i < DIM; ++i) {
                    float all = 0.0f;
#pragma unroll
                    for (int r = 0; r < DIM; ++r) all += __ldg(g + r * DIM + i);
                    ga[i] = a == 0 ? -all : __ldg(g + (a - 1) * DIM + i);
                    gb[i] = b == 0 ? -all : __ldg(g + (b - 1) * DIM + i);
                }
                const float sL = __ldg(g + BB), sM = __ldg(g + BB + 1);
                const float dot = sM * dotv<DIM>(ga, gb);
#pragma unroll
                for (int r = 0; r < DIM; ++r)
#pragma unroll
                    for (int i = 0; i < DIM; ++i) {
                        float x = (sL * ga[r]) * gb[i] + (sM * ga[i]) * gb[r];
                        if (r == i) x += dot;
                        acc[r * DIM + i].add(x);
                    }
            }
        }
#pragma unroll
        for (int q = 0; q < BB; ++q) vals[(slot * BB + q) * 32 + lane] = acc[q].value();
    }
}

// Elasticity: the reciprocal diagonal, from the blocks' diagonal components
template <int NC>
__global__ void __launch_bounds__(128) sell_diag_kernel(int64_t V, const float *vals, const int2 *slice, const int32_t *state,
                                                        float *Dinv) {
    if (state[1] != 0) return;  // not assembled
    const int64_t n = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (n >= V) return;
    const int lane = threadIdx.x & 31;
    const int2 sl = slice[n >> 5];
    float d[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) d[k] = 0.0f;
    for (int q = 0; q < sl.y; ++q)
#pragma unroll
        for (int k = 0; k < NC; ++k) d[k] -= vals[((int64_t(sl.x) + q) * NC * NC + k * NC + k) * 32 + lane];
#pragma unroll
    for (int k = 0; k < NC; ++k) Dinv[k * V + n] = d[k] > 0.0f ? 1.0f / d[k] : 1.0f;
}

// ------------------------------------------------------------------ application

// sums of products along a row, as pairs (TwoProduct and TwoSum)
struct DotRow {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float a, float b) {
        float p, e, t, f;
        two_prod(a, b, p, e);
        two_sum(s, p, t, f);
        s = t;
        c += e + f;
    }
    __device__ __forceinline__ float value() const { return s + c; }
};

// a matrix word: read once per application, so kept out of L1 (which the nodal values share),
// but not marked evict-first: the next application wants it from L2
__device__ __forceinline__ int32_t ld_matrix(const int32_t *p) {
    int32_t v;
    asm("ld.global.nc.L1::no_allocate.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_matrix(const float *p) {
    float v;
    asm("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// w = (A u) in row n, all components, lane `lane` of slice sl: a thread reads a column and its
// nodal values once for the NC rows of the block. The columns of up to J slots first, then
// batches of B slots, their nodal values (and, unless they lie in shared memory, their entries)
// in flight together. u is read with ordinary loads: other CTAs write it between barriers.
// SHARED: cols and vals lie in shared memory.
template <int NC, bool SHARED>
__device__ __forceinline__ void sell_row(const int32_t *__restrict__ cols, const float *__restrict__ vals, int2 sl,
                                         int lane, int64_t n, const float *u, int64_t V, float (&w)[NC]) {
    constexpr int BB = NC * NC;
    constexpr int J = SHARED || NC == 1 ? 16 : 8;
    constexpr int B = SHARED ? (NC == 1 ? 16 : 8) : (NC == 1 ? 8 : 4);
    DotRow acc[NC];
    float ui[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) ui[m] = u[m * V + n];
    const int32_t *c = cols + int64_t(sl.x) * 32 + lane;
    const float *v = vals + int64_t(sl.x) * BB * 32 + lane;
    for (int q = 0; q < sl.y; q += J, c += J * 32, v += J * BB * 32) {
        int32_t j[J];
#pragma unroll
        for (int i = 0; i < J; ++i) {
            j[i] = static_cast<int32_t>(n);
            if (q + i < sl.y) j[i] = SHARED ? c[i * 32] : ld_matrix(c + i * 32);
        }
#pragma unroll
        for (int i0 = 0; i0 < J; i0 += B) {
            if (q + i0 >= sl.y) break;
            float a[SHARED ? 1 : B][SHARED ? 1 : BB], x[B][NC];
#pragma unroll
            for (int i = 0; i < B; ++i) {
#pragma unroll
                for (int m = 0; m < NC; ++m) x[i][m] = u[m * V + j[i0 + i]];
                if constexpr (!SHARED) {
#pragma unroll
                    for (int m = 0; m < BB; ++m) {
                        a[i][m] = 0.0f;
                        if (q + i0 + i < sl.y) a[i][m] = ld_matrix(v + ((i0 + i) * BB + m) * 32);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < B; ++i) {
                if (q + i0 + i >= sl.y) break;
#pragma unroll
                for (int m = 0; m < NC; ++m) x[i][m] = x[i][m] - ui[m];
#pragma unroll
                for (int k = 0; k < NC; ++k)
#pragma unroll
                    for (int m = 0; m < NC; ++m)
                        acc[k].add(SHARED ? v[((i0 + i) * BB + k * NC + m) * 32] : a[SHARED ? 0 : i][SHARED ? 0 : k * NC + m],
                                   x[i][m]);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) w[k] = acc[k].value();
}

}  // namespace fem
