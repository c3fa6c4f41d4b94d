// fem_cell.cuh -- per-cell device arithmetic shared by the integration kernels.
//
// Geometry of a P1 simplex (reference vertices 0, e_1, ..., e_d):
//   columns of the Jacobian   e_j = x_j - x_0                  (j = 1..d)
//   adjugate rows             n_j = det(J) * (row j of J^{-1})
//       2D: n_1 = (e_2y, -e_2x), n_2 = (-e_1y, e_1x)
//       3D: n_1 = e_2 x e_3, n_2 = e_3 x e_1, n_3 = e_1 x e_2
//   determinant               det J = e_1 . n_1
// so the physical basis gradients are G_j = J^{-T} grad_ref phi_j = n_j / det J for
// j >= 1 and G_0 = -(G_1 + ... + G_d). All kernels work with n_j and det J and divide
// once per cell.
#pragma once

#include <cfloat>
#include <type_traits>

#include "fem_f2.cuh"
#include "fem_internal.cuh"

namespace fem {

template <int P>
using val_t = typename std::conditional<P == FEM_FP64, double, float>::type;

// ------------------------------------------------------------------ row access (cell-indexed arrays)

template <int CPT>
__device__ __forceinline__ void load_row(const int32_t *p, int32_t (&v)[CPT]) {
    if constexpr (CPT == 4) {
        int4 t = ld_stream(reinterpret_cast<const int4 *>(p));
        v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
    } else if constexpr (CPT == 2) {
        int2 t = __ldcs(reinterpret_cast<const int2 *>(p));
        v[0] = t.x, v[1] = t.y;
    } else {
#pragma unroll
        for (int i = 0; i < CPT; ++i) v[i] = ld_stream(p + i);
    }
}

template <int CPT>
__device__ __forceinline__ void load_row(const float *p, float (&v)[CPT]) {
    if constexpr (CPT == 4) {
        float4 t = ld_stream(reinterpret_cast<const float4 *>(p));
        v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
    } else if constexpr (CPT == 2) {
        float2 t = __ldcs(reinterpret_cast<const float2 *>(p));
        v[0] = t.x, v[1] = t.y;
    } else {
#pragma unroll
        for (int i = 0; i < CPT; ++i) v[i] = ld_stream(p + i);
    }
}

template <int CPT>
__device__ __forceinline__ void load_row(const double *p, double (&v)[CPT]) {
    if constexpr (CPT == 4) {
        double2 a = ld_stream(reinterpret_cast<const double2 *>(p));
        double2 b = ld_stream(reinterpret_cast<const double2 *>(p) + 1);
        v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
    } else if constexpr (CPT == 2) {
        double2 a = ld_stream(reinterpret_cast<const double2 *>(p));
        v[0] = a.x, v[1] = a.y;
    } else {
#pragma unroll
        for (int i = 0; i < CPT; ++i) v[i] = ld_stream(p + i);
    }
}

template <int CPT>
__device__ __forceinline__ void store_row(float *p, const float (&v)[CPT]) {
    if constexpr (CPT == 4) {
        __stcs(reinterpret_cast<float4 *>(p), make_float4(v[0], v[1], v[2], v[3]));
    } else if constexpr (CPT == 2) {
        __stcs(reinterpret_cast<float2 *>(p), make_float2(v[0], v[1]));
    } else {
#pragma unroll
        for (int i = 0; i < CPT; ++i) __stcs(p + i, v[i]);
    }
}

template <int CPT>
__device__ __forceinline__ void store_row(double *p, const double (&v)[CPT]) {
    if constexpr (CPT == 4) {
        __stcs(reinterpret_cast<double2 *>(p), make_double2(v[0], v[1]));
        __stcs(reinterpret_cast<double2 *>(p) + 1, make_double2(v[2], v[3]));
    } else if constexpr (CPT == 2) {
        __stcs(reinterpret_cast<double2 *>(p), make_double2(v[0], v[1]));
    } else {
#pragma unroll
        for (int i = 0; i < CPT; ++i) __stcs(p + i, v[i]);
    }
}

// The CPT cells that thread g of a grid-stride loop owns. STRIDED = false: consecutive ones, whose
// rows are read and written as one vector (the rows must be aligned for it). STRIDED = true: cells
// 32 apart, lane l of a warp taking l, l + 32, .. of the warp's 32 CPT cells, so that every access
// is a coalesced one of single values whatever the rows' alignment and the cell count; cells past
// the last are computed as copies of it and not stored.
template <int CPT, bool STRIDED>
struct Cells {
    int64_t c0, C;
    static __host__ __device__ int64_t groups(int64_t C) {
        return STRIDED ? (C + 32 * CPT - 1) / (32 * CPT) * 32 : (C + CPT - 1) / CPT;
    }
    __device__ __forceinline__ Cells(int64_t g, int64_t n) : c0(STRIDED ? (g >> 5) * (32 * CPT) + (g & 31) : g * CPT), C(n) {}
    __device__ __forceinline__ int64_t at(int i) const { return STRIDED ? min(c0 + 32 * i, C - 1) : c0 + i; }
    __device__ __forceinline__ bool in(int i) const { return !STRIDED || c0 + 32 * i < C; }
    template <class T>
    __device__ __forceinline__ void load(const T *row, T (&v)[CPT]) const {
        if constexpr (STRIDED) {
#pragma unroll
            for (int i = 0; i < CPT; ++i) v[i] = ld_stream(row + at(i));
        } else {
            load_row<CPT>(row + c0, v);
        }
    }
    template <class T>
    __device__ __forceinline__ void store(T *row, const T (&v)[CPT]) const {
        if constexpr (STRIDED) {
#pragma unroll
            for (int i = 0; i < CPT; ++i)
                if (in(i)) __stcs(row + c0 + 32 * i, v[i]);
        } else {
            store_row<CPT>(row + c0, v);
        }
    }
};

// ------------------------------------------------------------------ generic arithmetic
// The cell algebra below is written once for double, float and f2 (two cells per value).

// (both overloads are declared here: an unqualified fma() inside namespace fem must never
// resolve a double call to the float version)
__device__ __forceinline__ double fma(double a, double b, double c) { return ::fma(a, b, c); }
__device__ __forceinline__ float fma(float a, float b, float c) { return fmaf(a, b, c); }

// a*b - c*d
__device__ __forceinline__ double diffprod(double a, double b, double c, double d) { return fma(a, b, -(c * d)); }
__device__ __forceinline__ float diffprod(float a, float b, float c, float d) { return fmaf(a, b, -(c * d)); }
__device__ __forceinline__ f2 diffprod(f2 a, f2 b, f2 c, f2 d) { return a * b - c * d; }

// num / |den| in float64. The IEEE division is about a dozen float64 instructions and the
// float64 forms are bound by the float64 pipe, so: |den| = m 2^e with m in [1, 2) (integer
// operations on the exponent field); a float32 reciprocal of m, truncated to 23 bits, as the
// seed (relative error below 2^-22); two Newton-Raphson steps y <- y + y (1 - m y) in
// float64, each squaring the relative error, so the second ends at the float64 rounding
// level; the exponent put back and one product -- five float64 instructions, a result
// within about two units in the last place of the correctly rounded quotient. |den|
// outside [2^-1000, 2^1001) (zero, subnormal, infinite, NaN or extreme) takes the IEEE
// division.
__device__ __forceinline__ double quot_abs(double num, double den) {
    const uint32_t hw = static_cast<uint32_t>(__double2hiint(den)) & 0x7fffffffu;
    const uint32_t lw = static_cast<uint32_t>(__double2loint(den));
    const int ef = static_cast<int>(hw >> 20);  // biased exponent of |den|
    if (ef < 23 || ef > 2023) return num / fabs(den);
    const double m = __hiloint2double(static_cast<int>((hw & 0x000fffffu) | 0x3ff00000u), static_cast<int>(lw));
    const float yf = __frcp_rn(__uint_as_float(0x3f800000u | ((hw & 0x000fffffu) << 3) | (lw >> 29)));
    // yf in [0.5, 1]: widen it to float64 exactly with integer operations
    const uint32_t fb = __float_as_uint(yf);
    double y = __hiloint2double(static_cast<int>(((((fb >> 23) & 0xffu) + 896u) << 20) | ((fb & 0x7fffffu) >> 3)),
                                static_cast<int>(fb << 29));
    y = fma(y, fma(-m, y, 1.0), y);
    y = fma(y, fma(-m, y, 1.0), y);
    // 1 / |den| = y 2^-(ef - 1023): y's exponent field stays inside [22, 2023]
    const uint32_t yh = static_cast<uint32_t>(__double2hiint(y)) - (static_cast<uint32_t>(ef - 1023) << 20);
    return num * __hiloint2double(static_cast<int>(yh), __double2loint(y));
}
// float32: the fast reciprocal (the mixed form's tolerance is far above its error)
__device__ __forceinline__ float quot_abs(float num, float den) { return __fdividef(num, fabsf(den)); }
__device__ __forceinline__ f2 quot_abs(f2 num, f2 den) {
    return f2_make(__fdividef(f2_x(num), fabsf(f2_x(den))), __fdividef(f2_y(num), fabsf(f2_y(den))));
}

// -x and (first term of a sum) 0 + x, which turns -0 into +0, with integer operations: either is an
// addition on the float64 pipe otherwise, two of a tet's 58 in the residual
// (1,572,864 tets, us: residual 166.5 -> 159.9, adjoint 246.3 -> 240.4, elasticity 340 -> 330, three
// fields 403 -> 377)
__device__ __forceinline__ double neg(double x) {
    return __hiloint2double(__double2hiint(x) ^ static_cast<int>(0x80000000u), __double2loint(x));
}
__device__ __forceinline__ double from_zero(double x) {
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
    return __hiloint2double(static_cast<int>(hi == 0x80000000u && lo == 0u ? 0u : hi), static_cast<int>(lo));
}
__device__ __forceinline__ float from_zero(float x) { return 0.0f + x; }
__device__ __forceinline__ f2 from_zero(f2 x) { return f2{0ull} + x; }
__device__ __forceinline__ float neg(float x) { return -x; }
__device__ __forceinline__ f2 neg(f2 x) { return f2{0ull} - x; }

template <class T> __device__ __forceinline__ T zero();
template <> __device__ __forceinline__ double zero<double>() { return 0.0; }
template <> __device__ __forceinline__ float zero<float>() { return 0.0f; }
template <> __device__ __forceinline__ f2 zero<f2>() { return f2{0ull}; }

// ------------------------------------------------------------------ geometry

template <int DIM, class T>
__device__ __forceinline__ T adjugate_rows(const T (&e)[DIM][DIM], T (&n)[DIM][DIM]) {
    if constexpr (DIM == 2) {
        n[0][0] = e[1][1], n[0][1] = -e[1][0];
        n[1][0] = -e[0][1], n[1][1] = e[0][0];
        return diffprod(e[0][0], e[1][1], e[0][1], e[1][0]);
    } else {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const T *a = e[(j + 1) % 3], *b = e[(j + 2) % 3];
            n[j][0] = diffprod(a[1], b[2], a[2], b[1]);
            n[j][1] = diffprod(a[2], b[0], a[0], b[2]);
            n[j][2] = diffprod(a[0], b[1], a[1], b[0]);
        }
        return fma(e[0][2], n[0][2], fma(e[0][1], n[0][1], e[0][0] * n[0][0]));
    }
}

template <int DIM, class T>
__device__ __forceinline__ T dotv(const T *a, const T *b) {
    T s = a[0] * b[0];
#pragma unroll
    for (int i = 1; i < DIM; ++i) s = fma(a[i], b[i], s);
    return s;
}

// Gather the float64 coordinates of a cell's vertices: x[b][k] = X[k][v[b]].
template <int DIM>
__device__ __forceinline__ void gather_coords(const double *const (&X)[DIM], const uint32_t (&v)[DIM + 1],
                                              double (&x)[DIM + 1][DIM]) {
#pragma unroll
    for (int b = 0; b <= DIM; ++b)
#pragma unroll
        for (int k = 0; k < DIM; ++k) x[b][k] = ld_gather(X[k] + v[b]);
}

// Float64 Jacobian columns e_j = x_j - x_0.
template <int DIM>
__device__ __forceinline__ void columns_f64(const double (&x)[DIM + 1][DIM], double (&e)[DIM][DIM]) {
#pragma unroll
    for (int j = 0; j < DIM; ++j)
#pragma unroll
        for (int k = 0; k < DIM; ++k) e[j][k] = x[j + 1][k] - x[0][k];
}

// The differences x[j + 1] - x[0], bitwise those of the float64 subtraction, with integer
// operations: the float64 pipe issues 2 lanes a clock and SM, the integer pipes about 100, and the
// float64 kernels wait for the former. The values are brought to fixed point at their largest
// exponent (53 significant bits, 9 to spare), subtracted exactly as 64-bit integers, normalised and
// packed again. Returns false, with d unusable, where that does not give the correctly rounded
// difference: a nonzero value more than 9 binades below the largest; -0, subnormal or non-finite
// values; a difference below the normal range or of more than 53 significant bits (vertex
// coordinates of one cell hardly ever have one).
template <int N>
__device__ __forceinline__ bool exact_differences(const double (&x)[N], double (&d)[N - 1]) {
    uint32_t hw[N], lw[N], ex[N], top = 0;
#pragma unroll
    for (int b = 0; b < N; ++b) {
        hw[b] = static_cast<uint32_t>(__double2hiint(x[b]));
        lw[b] = static_cast<uint32_t>(__double2loint(x[b]));
        ex[b] = (hw[b] >> 20) & 0x7ffu;
        top = max(top, ex[b]);
    }
    bool ok = top < 0x7feu;
    uint32_t fh[N], fl[N];
#pragma unroll
    for (int b = 0; b < N; ++b) {
        const bool zero = (hw[b] | lw[b]) == 0u;  // +0 (-0 is left to the subtraction: its sign counts)
        const int up = static_cast<int>(ex[b] - top) + 9;
        ok = ok && (zero || (up >= 0 && ex[b] != 0u));
        const uint32_t mh = (hw[b] & 0xfffffu) | 0x100000u;
        uint32_t h = __funnelshift_l(lw[b], mh, up), l = lw[b] << (up & 31);
        h = zero ? 0u : h;
        const uint32_t s = static_cast<uint32_t>(static_cast<int32_t>(hw[b]) >> 31);
        // two's complement of the magnitude where the sign is set
        const uint64_t f = ((static_cast<uint64_t>(h ^ s) << 32) | (l ^ s)) - (static_cast<uint64_t>(s) << 32 | s);
        fh[b] = static_cast<uint32_t>(f >> 32), fl[b] = static_cast<uint32_t>(f);
    }
    const uint64_t f0 = (static_cast<uint64_t>(fh[0]) << 32) | fl[0];
    uint32_t dropped = 0;
#pragma unroll
    for (int j = 1; j < N; ++j) {
        const uint64_t df = ((static_cast<uint64_t>(fh[j]) << 32) | fl[j]) - f0;
        const uint64_t s = static_cast<uint64_t>(static_cast<int64_t>(df) >> 63);
        const uint64_t mag = (df ^ s) - s;
        const uint32_t mh = static_cast<uint32_t>(mag >> 32), ml = static_cast<uint32_t>(mag);
        const bool small = mh == 0u;
        const uint32_t h = small ? ml : mh, l = small ? 0u : ml;
        const int n = __clz(static_cast<int>(h));
        const uint32_t bh = __funnelshift_l(l, h, n), bl = l << (n & 31);  // leading one at bit 63
        // the leading one of a value at exponent `top` is bit 61
        const int e = static_cast<int>(top) + 2 - n - (small ? 32 : 0);
        const bool none = h == 0u;
        ok = ok && (none || e >= 1);
        const uint32_t hi = (static_cast<uint32_t>(s) & 0x80000000u) + (static_cast<uint32_t>(e - 1) << 20) + (bh >> 11);
        const uint32_t lo = __funnelshift_r(bl, bh, 11);
        dropped |= bl;
        d[j - 1] = __hiloint2double(static_cast<int>(none ? 0u : hi), static_cast<int>(none ? 0u : lo));
    }
    return ok && (dropped & 0x7ffu) == 0u;
}

// out of line: written in place the compiler would execute it predicated in every cell, and a
// float64 instruction takes its time on the pipe even where every lane is switched off
static __device__ __noinline__ double subtract_out_of_line(double a, double b) { return a - b; }

// Cells from which the float64 kernels take their columns so: below, a scheduler has one or two warps of 32 cells, whose time is their
// own latency, which the integer operations lengthen. Us, subtractions / integer columns, 1,572,864
// tets: residual 192 / 167, adjoint 272 / 246, elasticity 366 / 340, reaction-diffusion 375 / 351,
// three fields 429 / 403; 50,000: 8.0 / 7.6, 14.1 / 13.9, 14.5 / 13.8, 15.2 / 15.2, 16.8 / 16.2;
// 25,000: 5.0 / 5.3, 10.2 / 10.4, 8.4 / 8.6, 9.3 / 9.7, 9.8 / 10.1. The kernels that use it take one
// cell per thread; double-float kernels, which the instruction issue bounds, lose a third by it.
constexpr int64_t kExactFrom = 60000;

// columns_f64, bit for bit, axis by axis by exact_differences where they give them
template <int DIM>
__device__ __forceinline__ void columns_f64_int(const double (&x)[DIM + 1][DIM], double (&e)[DIM][DIM],
                                                bool by_integer) {
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        double a[DIM + 1], d[DIM];
#pragma unroll
        for (int b = 0; b <= DIM; ++b) a[b] = x[b][k];
        if (by_integer) {
            if (!exact_differences<DIM + 1>(a, d)) {
#pragma unroll
                for (int j = 0; j < DIM; ++j) d[j] = subtract_out_of_line(a[j + 1], a[0]);
            }
        } else {
#pragma unroll
            for (int j = 0; j < DIM; ++j) d[j] = a[j + 1] - a[0];
        }
#pragma unroll
        for (int j = 0; j < DIM; ++j) e[j][k] = d[j];
    }
}

// Float32 Jacobian columns from float64 coordinates split into (hi, lo) pairs:
// e_jk = (hi_jk - hi_0k) + (lo_jk - lo_0k); exact up to float32 rounding of the result.
template <int DIM>
__device__ __forceinline__ void columns_mixed(const double (&x)[DIM + 1][DIM], float (&e)[DIM][DIM]) {
    float hi[DIM + 1][DIM], lo[DIM + 1][DIM];
#pragma unroll
    for (int b = 0; b <= DIM; ++b)
#pragma unroll
        for (int k = 0; k < DIM; ++k)
            split_f64(static_cast<uint32_t>(__double2loint(x[b][k])), static_cast<uint32_t>(__double2hiint(x[b][k])),
                      hi[b][k], lo[b][k]);
#pragma unroll
    for (int j = 0; j < DIM; ++j)
#pragma unroll
        for (int k = 0; k < DIM; ++k) e[j][k] = fmaf(lo[j + 1][k] - lo[0][k], 0x1p-23f, hi[j + 1][k] - hi[0][k]);
}

// The same for two cells at once (lane x: cell xa, lane y: cell xb).
template <int DIM>
__device__ __forceinline__ void columns_mixed2(const double (&xa)[DIM + 1][DIM], const double (&xb)[DIM + 1][DIM],
                                               f2 (&e)[DIM][DIM]) {
    f2 hi[DIM + 1][DIM], lo[DIM + 1][DIM];
#pragma unroll
    for (int b = 0; b <= DIM; ++b)
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            float ha, la, hb, lb;
            split_f64(static_cast<uint32_t>(__double2loint(xa[b][k])), static_cast<uint32_t>(__double2hiint(xa[b][k])),
                      ha, la);
            split_f64(static_cast<uint32_t>(__double2loint(xb[b][k])), static_cast<uint32_t>(__double2hiint(xb[b][k])),
                      hb, lb);
            hi[b][k] = f2_make(ha, hb);
            lo[b][k] = f2_make(la, lb);
        }
    const f2 scale = f2_splat(0x1p-23f);
#pragma unroll
    for (int j = 0; j < DIM; ++j)
#pragma unroll
        for (int k = 0; k < DIM; ++k) e[j][k] = fma(lo[j + 1][k] - lo[0][k], scale, hi[j + 1][k] - hi[0][k]);
}

// Float32 Jacobian columns from coordinates rounded to float32 (FP32 ablation).
template <int DIM>
__device__ __forceinline__ void columns_f32(const double (&x)[DIM + 1][DIM], float (&e)[DIM][DIM]) {
    float xf[DIM + 1][DIM];
#pragma unroll
    for (int b = 0; b <= DIM; ++b)
#pragma unroll
        for (int k = 0; k < DIM; ++k)
            xf[b][k] = round_f64_to_f32(static_cast<uint32_t>(__double2loint(x[b][k])),
                                        static_cast<uint32_t>(__double2hiint(x[b][k])));
#pragma unroll
    for (int j = 0; j < DIM; ++j)
#pragma unroll
        for (int k = 0; k < DIM; ++k) e[j][k] = xf[j + 1][k] - xf[0][k];
}

// The same for two cells at once.
template <int DIM>
__device__ __forceinline__ void columns_f32_2(const double (&xa)[DIM + 1][DIM], const double (&xb)[DIM + 1][DIM],
                                              f2 (&e)[DIM][DIM]) {
    f2 xf[DIM + 1][DIM];
#pragma unroll
    for (int b = 0; b <= DIM; ++b)
#pragma unroll
        for (int k = 0; k < DIM; ++k)
            xf[b][k] = f2_make(round_f64_to_f32(static_cast<uint32_t>(__double2loint(xa[b][k])),
                                                static_cast<uint32_t>(__double2hiint(xa[b][k]))),
                               round_f64_to_f32(static_cast<uint32_t>(__double2loint(xb[b][k])),
                                                static_cast<uint32_t>(__double2hiint(xb[b][k]))));
#pragma unroll
    for (int j = 0; j < DIM; ++j)
#pragma unroll
        for (int k = 0; k < DIM; ++k) e[j][k] = xf[j + 1][k] - xf[0][k];
}

// Shape test of the mixed form: det^2 >= tau^2 prod_j |e_j|^2 (Hadamard ratio >= tau),
// with det^2 inside float32's normal range; failing cells take the float64 path.
template <int DIM>
__device__ __forceinline__ bool shape_ok(const float (&e)[DIM][DIM], float det, float tau2) {
    float p = dotv<DIM>(e[0], e[0]);
#pragma unroll
    for (int j = 1; j < DIM; ++j) p *= dotv<DIM>(e[j], e[j]);
    float d2 = det * det;
    return d2 >= fmaxf(tau2 * p, FLT_MIN) && d2 <= FLT_MAX;
}

// The shape test for two cells: (ok of lane x, ok of lane y).
template <int DIM>
__device__ __forceinline__ void shape_ok2(const f2 (&e)[DIM][DIM], f2 det, float tau2, bool &oka, bool &okb) {
    f2 p = dotv<DIM>(e[0], e[0]);
#pragma unroll
    for (int j = 1; j < DIM; ++j) p = p * dotv<DIM>(e[j], e[j]);
    const f2 d2 = det * det;
    const f2 lim = p * f2_splat(tau2);
    const float da = f2_x(d2), db = f2_y(d2);
    oka = da >= fmaxf(f2_x(lim), FLT_MIN) && da <= FLT_MAX;
    okb = db >= fmaxf(f2_y(lim), FLT_MIN) && db <= FLT_MAX;
}

// ------------------------------------------------------------------ quadrature sums

// sum_q w_q c_q, plain (FMA chain) -- float64 form and float32 ablation
template <class T>
struct PlainSum {
    T s;
    __device__ __forceinline__ void first(T w, T c) { s = w * c; }
    __device__ __forceinline__ void add(T w, T c) { s = fma(w, c, s); }
    __device__ __forceinline__ T value() const { return s; }
    __device__ __forceinline__ double value_f64() const { return static_cast<double>(s); }
};

// sum_q w_q c_q compensated: Dot2 (Ogita, Rump, Oishi 2005) with TwoProduct and TwoSum;
// the result is as accurate as if computed in twice the working precision.
struct Dot2Sum {
    float s, c;
    __device__ __forceinline__ void first(float w, float x) { two_prod(w, x, s, c); }
    __device__ __forceinline__ void add(float w, float x) {
        float p, pe, se;
        two_prod(w, x, p, pe);
        two_sum(s, p, s, se);
        c += pe + se;
    }
    __device__ __forceinline__ float value() const { return s + c; }
    __device__ __forceinline__ double value_f64() const { return static_cast<double>(s) + static_cast<double>(c); }
};

// Dot2 for two cells at once. The compensation is kept negated (m = -c): TwoProduct's
// error term then comes out of one FMA, m_p = fma(-w, x, p) = p - w x exactly, with p
// the correctly rounded product (mul_rn_exact), and no negation is needed anywhere.
struct Dot2Sum2 {
    f2 s, m;
    __device__ __forceinline__ void first(float w, f2 x) {
        s = mul_rn_exact(f2_splat(w), x);
        m = fma(f2_splat(-w), x, s);
    }
    __device__ __forceinline__ void add(float w, f2 x) {
        const f2 p = mul_rn_exact(f2_splat(w), x);
        const f2 mp = fma(f2_splat(-w), x, p);
        const f2 t = s + p;
        const f2 bb = t - s;
        const f2 se = (s - (t - bb)) + (p - bb);
        s = t;
        m = m + (mp - se);
    }
    __device__ __forceinline__ f2 value() const { return s - m; }
    __device__ __forceinline__ double value_f64_x() const { return double(f2_x(s)) - double(f2_x(m)); }
    __device__ __forceinline__ double value_f64_y() const { return double(f2_y(s)) - double(f2_y(m)); }
};

// sum_q w_q c_q in plain f32x2 (FP32 ablation)
struct PlainSum2 {
    f2 s;
    __device__ __forceinline__ void first(float w, f2 x) { s = f2_splat(w) * x; }
    __device__ __forceinline__ void add(float w, f2 x) { s = fma(f2_splat(w), x, s); }
    __device__ __forceinline__ f2 value() const { return s; }
    __device__ __forceinline__ double value_f64_x() const { return double(f2_x(s)); }
    __device__ __forceinline__ double value_f64_y() const { return double(f2_y(s)); }
};

// fixed-order sum of a vertex's list entries (the nodal gather E^T): plain in float64,
// compensated (TwoSum) in float32
template <class T>
struct NodeSum {
    T s = T(0);
    __device__ __forceinline__ void add(T x) { s += x; }
    __device__ __forceinline__ T value() const { return s; }
};

template <>
struct NodeSum<float> {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x) {
        float t, e;
        two_sum(s, x, t, e);
        s = t;
        c += e;
    }
    __device__ __forceinline__ float value() const { return s + c; }
};

// Sums of the element vectors' entries idx[b .. e) (entry t = NB cell + a stands for row
// a * NCOMP + k, cell `cell`, of elem) into acc[k], one by one in list order. The loads of eight
// entries are in flight together, of a remainder those of four, two and one: each batch costs two
// dependent loads' latency, and a remainder taken entry by entry up to seven times that (triangles'
// lists have 6 entries: 1,000,000 / 50,000 cells, two float32 components, 10.7 -> 9.9 / 2.8 -> 2.6 us).
template <int NB, int NCOMP, int N, class T>
__device__ __forceinline__ void gather_batch(const T *__restrict__ elem, const int32_t *__restrict__ idx, int64_t C,
                                             NodeSum<T> (&acc)[NCOMP]) {
    int32_t t[N];
    T val[N][NCOMP];
#pragma unroll
    for (int i = 0; i < N; ++i) t[i] = __ldg(idx + i);
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int k = 0; k < NCOMP; ++k) {
            const int32_t cell = t[i] / NB, a = t[i] - cell * NB;
            val[i][k] = __ldg(elem + int64_t(a * NCOMP + k) * C + cell);
        }
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int k = 0; k < NCOMP; ++k) acc[k].add(val[i][k]);
}

template <int NB, int NCOMP, class T>
__device__ __forceinline__ void gather_list(const T *__restrict__ elem, const int32_t *__restrict__ idx, int32_t b,
                                            int32_t e, int64_t C, NodeSum<T> (&acc)[NCOMP]) {
    int32_t j = b;
    for (; j + 8 <= e; j += 8) gather_batch<NB, NCOMP, 8>(elem, idx + j, C, acc);
    if (j + 4 <= e) gather_batch<NB, NCOMP, 4>(elem, idx + j, C, acc), j += 4;
    if (j + 2 <= e) gather_batch<NB, NCOMP, 2>(elem, idx + j, C, acc), j += 2;
    if (j < e) gather_batch<NB, NCOMP, 1>(elem, idx + j, C, acc);
}

template <int P>
using qsum_t = typename std::conditional<P == FEM_FP64, PlainSum<double>,
                                         typename std::conditional<P == FEM_FP32_MIXED, Dot2Sum, PlainSum<float>>::type>::type;

}  // namespace fem
