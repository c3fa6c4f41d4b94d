// fem_mesh.cu -- vertex-to-cell lists (the transpose of the connectivity, i.e. the
// assembly operator E of Eq. 2 as lists), the deterministic nodal gather E^T applied
// to element vectors, and the mesh validation pass.
#include "fem_cell.cuh"

namespace fem {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

static int64_t scan_tiles_for(int64_t n) { return (n + kScanTile - 1) / kScanTile; }

// ------------------------------------------------------------------ scan (three passes)

// Exclusive prefix sum of x over the CTA (kScanThreads threads); the CTA total is
// stored to *total (shared memory) and is visible to every thread on return.
__device__ __forceinline__ int32_t block_exclusive_scan(int32_t x, int32_t *total) {
    constexpr int kWarps = kScanThreads / 32;
    __shared__ int32_t warp_off[kWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_off[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        int32_t t = lane < kWarps ? warp_off[lane] : 0;
        int32_t ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += y;
        }
        if (lane < kWarps) warp_off[lane] = ti - t;
        if (lane == 31) *total = ti;
    }
    __syncthreads();
    const int32_t off = warp_off[wid];
    __syncthreads();  // warp_off may be reused by the next call
    return off + incl - x;
}

// in-place inclusive scan of one tile; the tile's total goes to tile_sums[tile]
__global__ void __launch_bounds__(kScanThreads) scan_tiles_kernel(int32_t *data, int64_t n, int32_t *tile_sums) {
    pdl_wait();
    __shared__ int32_t s_total;
    const int64_t base = int64_t(blockIdx.x) * kScanTile + int64_t(threadIdx.x) * kScanItems;
    int32_t v[kScanItems];
    int32_t run = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        run += (base + i < n) ? data[base + i] : 0;
        v[i] = run;  // inclusive within the thread
    }
    const int32_t off = block_exclusive_scan(run, &s_total);
#pragma unroll
    for (int i = 0; i < kScanItems; ++i)
        if (base + i < n) data[base + i] = v[i] + off;
    if (threadIdx.x == 0) tile_sums[blockIdx.x] = s_total;
}

// exclusive scan of the tile sums in place (one CTA, chunks of a tile with a carry)
__global__ void __launch_bounds__(kScanThreads) scan_sums_kernel(int32_t *sums, int64_t n) {
    pdl_wait();
    __shared__ int32_t s_total;
    int32_t carry = 0;
    for (int64_t c = 0; c < n; c += kScanTile) {
        const int64_t base = c + int64_t(threadIdx.x) * kScanItems;
        int32_t v[kScanItems], run = 0;
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) {
            v[i] = run;  // exclusive within the thread
            run += (base + i < n) ? sums[base + i] : 0;
        }
        const int32_t off = block_exclusive_scan(run, &s_total);
#pragma unroll
        for (int i = 0; i < kScanItems; ++i)
            if (base + i < n) sums[base + i] = carry + off + v[i];
        carry += s_total;
        __syncthreads();
    }
}

// data[i] += the sums of the tiles before i's (summed: tile_sums holds these offsets already;
// otherwise the CTA, one per tile, adds them up); cursor[i + 1] = data[i], cursor[0] = 0
__global__ void __launch_bounds__(kScanThreads) add_offsets_kernel(int32_t *data, int64_t n, const int32_t *tile_sums,
                                                                   bool summed, int32_t *cursor) {
    pdl_wait();
    __shared__ int32_t s_total;
    const int64_t tile = blockIdx.x;
    int32_t off;
    if (summed) {
        off = tile_sums[tile];
    } else {
        int32_t part = 0;
        for (int64_t t = threadIdx.x; t < tile; t += kScanThreads) part += tile_sums[t];
        block_exclusive_scan(part, &s_total);
        off = s_total;
    }
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int64_t j = tile * kScanTile + int64_t(i) * kScanThreads + threadIdx.x;
        if (j < n) {
            const int32_t x = data[j] + off;
            data[j] = x;
            if (j + 1 < n) cursor[j + 1] = x;
        }
    }
    if (tile == 0 && threadIdx.x == 0) cursor[0] = 0;
}

// data[0..n) inclusive-scanned in place, cursor[0..n) the exclusive sums; workspace
// tile_sums[scan_tiles_for(n)]. Up to kSumTiles tiles the tiles' offsets are summed where they
// are used, one kernel less.
constexpr int64_t kSumTiles = 2048;
static fem_status scan_with_cursor(int32_t *data, int64_t n, int32_t *tile_sums, int32_t *cursor, cudaStream_t s) {
    const int64_t tiles = scan_tiles_for(n);
    const unsigned grid = static_cast<unsigned>(tiles);
    const bool summed = tiles > kSumTiles;
    launch_overlapped(scan_tiles_kernel, grid, kScanThreads, 0, s, data, n, tile_sums);
    if (summed) launch_overlapped(scan_sums_kernel, 1, kScanThreads, 0, s, tile_sums, tiles);
    const int32_t *sums = tile_sums;
    launch_overlapped(add_offsets_kernel, grid, kScanThreads, 0, s, data, n, sums, summed, cursor);
    return check_launch("scan");
}

// ------------------------------------------------------------------ vertex-to-cell lists
//
// zero, count, scan (two kernels), fill, sort, launched overlapped. On 524,286 tets (93,000
// vertices; ncu, cold caches, us): count 10.3, scan 9, fill 11.7 (14 with one atomic per cell and
// vertex), sort 12.5; the lists and the adjoint after them 66 -> 57 us with the eight-lane sort, 110
// with the sort by one thread per vertex in local memory (41), a scan of four kernels and plain
// launches. What bounds them is latency: of the atomics that return a place, and of the chain
// pointer -> list -> place -> list per vertex.

__global__ void __launch_bounds__(kBlock) zero_kernel(int32_t *data, int64_t n) {
    pdl_wait();
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) data[i] = 0;
}

// One atomic per run of equal vertices among a warp's 32 cells (in one row): meshes that list the
// cells of one vertex or one grid box together have such runs, and atomics on one address go one
// by one. Lanes without a cell carry an id no vertex has. Every lane gets the old value of its
// vertex' counter plus its place in the run.
__device__ __forceinline__ int32_t warp_add(int32_t *counters, uint32_t v, bool in) {
    const int lane = threadIdx.x & 31;
    const uint32_t w = in ? v : 0xffffffffu;
    const uint32_t before = __shfl_up_sync(0xffffffffu, w, 1);
    const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || before != w);
    const unsigned from = heads & (0xffffffffu >> (31 - lane));  // heads at or below this lane
    const int head = 31 - __clz(from);
    const unsigned above = heads & ~(0xffffffffu >> (31 - lane));
    const int end = above ? __ffs(above) - 1 : 32;
    int32_t old = 0;
    if (in && lane == head) old = atomicAdd(counters + v, end - lane);
    return __shfl_sync(0xffffffffu, old, head) + lane - head;
}

template <int NB>
__global__ void __launch_bounds__(kBlock) count_kernel(const int32_t *conn, int64_t C, uint32_t V, int32_t *ptr1,
                                                       unsigned *err) {
    pdl_wait();
    uint32_t vmax = 0;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    const int64_t warps_end = (C + 31) / 32 * 32;  // whole warps: warp_add is a warp's work
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < warps_end; e += stride) {
        const bool in = e < C;
        uint32_t v[NB];
#pragma unroll
        for (int a = 0; a < NB; ++a) v[a] = in ? clamp_vid(conn[a * C + e], V, vmax) : 0u;
#pragma unroll
        for (int a = 0; a < NB; ++a) warp_add(ptr1, v[a], in);
    }
    report_mesh(err, vmax, V, false);
}

template <int NB>
__global__ void __launch_bounds__(kBlock) fill_kernel(const int32_t *conn, int64_t C, uint32_t V, int32_t *cursor,
                                                      int32_t *idx) {
    pdl_wait();
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    const int64_t warps_end = (C + 31) / 32 * 32;
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < warps_end; e += stride) {
        const bool in = e < C;
        uint32_t v[NB];
        int32_t pos[NB];
#pragma unroll
        for (int a = 0; a < NB; ++a) v[a] = in ? clamp_vid(conn[a * C + e], V) : 0u;
#pragma unroll
        for (int a = 0; a < NB; ++a) pos[a] = warp_add(cursor, v[a], in);
        if (in)
#pragma unroll
            for (int a = 0; a < NB; ++a) idx[pos[a]] = static_cast<int32_t>(e * NB + a);
    }
}

// Sort every vertex' list: cell order, independent of the order in which the atomics above
// landed. G = 8 lanes per vertex (32: 20.6 us on the mesh above, 4: 13.0). In 3D (24 entries are usual)
// lists of 9 to 32 entries are sorted in registers by a network: counting smaller entries took 442
// instructions per warp and 82 % of the issue slots (lists of 1,000,000 tets 51.9 -> 44.9 us,
// 200,000: 20.1 -> 19.1; 2D, with 6 entries, would lose 0.5 %). Other lists of up to kSortShared
// entries go to shared memory, where an entry's place is the number of smaller ones (all entries of
// a list are distinct). Longer ones are sorted in place by the eight lanes with bitonic merges (lists
// of meshes of hubs, us, by insertion sort of one lane -> so: 5000 of 129 entries 861 -> 159, 2000 of
// 400 4708 -> 236, 500 of 1000 19,510 -> 353; by a thread per vertex they took 677, 3500, 19,490).
constexpr int kSortShared = 128;

// 32 values over 8 lanes, four to a lane, into ascending order (entry 4 lane + i in x[i]): bitonic
// merges of 2, 4, .. 32 whose first step compares with the mirrored entry, so that every step is
// ascending and the smaller value goes to the lower place. Nine of the fifteen steps stay in a lane.
__device__ __forceinline__ void sort32(int32_t (&x)[4], int lane, unsigned mask) {
    auto order = [&](int a, int b) {
        const int32_t lo = min(x[a], x[b]), hi = max(x[a], x[b]);
        x[a] = lo, x[b] = hi;
    };
    auto halves = [&]() { order(0, 2), order(1, 3), order(0, 1), order(2, 3); };
    auto across = [&](int with, int bit, bool mirror) {
        int32_t y[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) y[i] = __shfl_xor_sync(mask, x[mirror ? 3 - i : i], with, 8);
        const bool lower = (lane & bit) == 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = lower ? min(x[i], y[i]) : max(x[i], y[i]);
    };
    order(0, 1), order(2, 3), order(0, 3), order(1, 2), order(0, 1), order(2, 3);
    across(1, 1, true), halves();
    across(3, 2, true), across(1, 1, false), halves();
    across(7, 4, true), across(2, 2, false), across(1, 1, false), halves();
}

template <int G, bool NETWORK>
__global__ void __launch_bounds__(kBlock) sort_segments_kernel(const int32_t *ptr, int32_t *idx, int64_t V) {
    pdl_wait();
    __shared__ __align__(16) int32_t list[kBlock / G][kSortShared + 4];  // + 4: the groups' rows in different banks
    const int lane = threadIdx.x % G, group = threadIdx.x / G;
    const unsigned mask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << ((threadIdx.x & 31) / G * G);
    const int64_t stride = int64_t(gridDim.x) * (kBlock / G);
    int32_t *s = list[group];
    for (int64_t n = int64_t(blockIdx.x) * (kBlock / G) + group; n < V; n += stride) {
        const int32_t b = ptr[n], m = ptr[n + 1] - b;
        if (NETWORK && G == 8 && m > 8 && m <= 32) {
            int32_t x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = lane + i * 8 < m ? idx[b + lane + i * 8] : 0x7fffffff;
            sort32(x, lane, mask);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (lane * 4 + i < m) idx[b + lane * 4 + i] = x[i];
        } else if (m <= kSortShared) {
            // padded to a multiple of four with the largest value, which no entry exceeds
            const int pad = (m + 3) & ~3;
            for (int k = lane; k < pad; k += G) s[k] = k < m ? idx[b + k] : 0x7fffffff;
            __syncwarp(mask);
            for (int k = lane; k < m; k += G) {
                const int32_t x = s[k];
                int r = 0;
                for (int j = 0; j < m; j += 4) {
                    const int4 q = *reinterpret_cast<const int4 *>(s + j);
                    r += (q.x < x) + (q.y < x) + (q.z < x) + (q.w < x);
                }
                idx[b + r] = x;
            }
            __syncwarp(mask);
        } else {
            // in place, by the same merges as sort32's; entries past the end count as the largest,
            // and no exchange reaches them
            int32_t *p = idx + b;
            const uint32_t len = static_cast<uint32_t>(m);
            auto step = [&](uint32_t d, uint32_t mirror) {
                for (uint32_t q = lane;; q += G) {
                    const uint32_t i = 2 * (q & ~(d - 1)) + (q & (d - 1)), j = mirror ? i ^ mirror : i + d;
                    if (i >= len) break;
                    if (j < len) {
                        const int32_t x = p[i], y = p[j];
                        if (x > y) p[i] = y, p[j] = x;
                    }
                }
                __syncwarp(mask);
            };
            for (uint64_t k = 2; k / 2 < len; k *= 2) {
                step(static_cast<uint32_t>(k / 2), static_cast<uint32_t>(k - 1));
                for (uint32_t d = static_cast<uint32_t>(k / 4); d > 0; d /= 2) step(d, 0u);
            }
        }
    }
}

// ------------------------------------------------------------------ nodal gather


template <int NB, int NCOMP, class T>
__global__ void gather_kernel(int64_t C, int64_t V, const T *__restrict__ elem, const int32_t *__restrict__ ptr,
                              const int32_t *__restrict__ idx, T *__restrict__ out) {
    pdl_wait();  // overlapped launch: the previous kernel's writes are visible from here
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t n = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; n < V; n += stride) {
        // (A warp reading 32 vertices' lists together with coalesced loads and summing from shared
        // memory was slower: 60.4 against 48.8 us for the adjoint on 1,572,864 tets.)
        NodeSum<T> acc[NCOMP];
        gather_list<NB, NCOMP>(elem, idx, ptr[n], ptr[n + 1], C, acc);
#pragma unroll
        for (int k = 0; k < NCOMP; ++k) out[k * V + n] = acc[k].value();
    }
}

// Large 3D meshes (lists of 24 entries, more than 512 vertices per SM) in one-warp CTAs, which
// hold 1024 threads to an SM: with all 2048 the sectors that neighbouring vertices' lists share
// are gone from L1 before their second use (1,000,000 tets, one component 14.6 -> 11.1 us in
// float32, 21.3 -> 15.7 in float64; three 26.5 -> 22.9, 53.3 -> 36.7; 400,000 tets 7.4 -> 8.8 in
// float32, so not there). Small meshes (at most 128 vertices per SM)
// in CTAs of 128 threads (50,000 tets, three components, float64: 8.3 -> 7.2 us against 256). 2D lists (6 entries) want full occupancy: one-warp CTAs take 35
// against 19.5 us on 2,097,152 triangles. Rejected: list indices by 16-byte loads (no change in
// 3D, 22-60 % slower in 2D), 12 or 24 entries in flight, larger CTAs.
template <int NB, class T>
static void launch_gather_t(int n_comp, int64_t C, int64_t V, const void *elem, const int32_t *ptr,
                            const int32_t *idx, void *out, cudaStream_t s) {
    const T *el = static_cast<const T *>(elem);
    T *o = static_cast<T *>(out);
    const int64_t sms = sm_count();
    const unsigned cta = NB == 4 && V > 512 * sms ? kWarpCta : (V > 128 * sms ? kBlock : 128);
    const unsigned grid = static_cast<unsigned>((V + cta - 1) / cta);
    switch (n_comp) {
        case 1: {
            auto k = gather_kernel<NB, 1, T>;
            launch_overlapped(k, grid, cta, 0, s, C, V, el, ptr, idx, o);
        } break;
        case 2: {
            auto k = gather_kernel<NB, 2, T>;
            launch_overlapped(k, grid, cta, 0, s, C, V, el, ptr, idx, o);
        } break;
        default: {
            auto k = gather_kernel<NB, 3, T>;
            launch_overlapped(k, grid, cta, 0, s, C, V, el, ptr, idx, o);
        } break;
    }
}

fem_status launch_gather(int dim, int n_comp, int64_t C, int64_t V, const void *elem, const int32_t *node_ptr,
                         const int32_t *node_idx, void *out, fem_precision prec, cudaStream_t s) {
    if (V == 0) return FEM_OK;
    const bool f64 = prec == FEM_FP64 || prec == FEM_FP64_DF;  // float64 values either way
    if (dim == 2) {
        if (f64) launch_gather_t<3, double>(n_comp, C, V, elem, node_ptr, node_idx, out, s);
        else launch_gather_t<3, float>(n_comp, C, V, elem, node_ptr, node_idx, out, s);
    } else {
        if (f64) launch_gather_t<4, double>(n_comp, C, V, elem, node_ptr, node_idx, out, s);
        else launch_gather_t<4, float>(n_comp, C, V, elem, node_ptr, node_idx, out, s);
    }
    return check_launch("nodal gather");
}

// ------------------------------------------------------------------ mesh validation

template <int DIM>
__global__ void check_mesh_kernel(const double *X0, int64_t C, uint32_t V, const int32_t *conn, float tau2,
                                  unsigned long long *counts) {
    constexpr int NB = DIM + 1;
    __shared__ unsigned long long s_cnt[4];
    if (threadIdx.x < 4) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long c_bad = 0, c_degen = 0, c_fallback = 0, c_neg = 0;
    const double *X[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) X[k] = X0 + int64_t(k) * V;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; c < C; c += stride) {
        uint32_t v[NB];
        bool ids_ok = true;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            int32_t id = conn[b * C + c];
            if (id < 0 || static_cast<uint32_t>(id) >= V) ++c_bad, ids_ok = false;
            v[b] = clamp_vid(id, V);
        }
        if (!ids_ok) continue;
        double xs[NB][DIM], e[DIM][DIM], n[DIM][DIM];
        gather_coords<DIM>(X, v, xs);
        columns_f64<DIM>(xs, e);
        double det = adjugate_rows<DIM>(e, n);
        // degenerate to rounding: |det J| <= 16 eps_64 prod_j |e_j| (FMA contraction can
        // leave a rounding residue instead of an exact zero for repeated vertices)
        double pn = 1.0;
#pragma unroll
        for (int j = 0; j < DIM; ++j) pn *= sqrt(dotv<DIM>(e[j], e[j]));
        const bool degenerate = !(fabs(det) > 16.0 * DBL_EPSILON * pn) || !isfinite(det);
        if (degenerate) ++c_degen;
        else if (det < 0.0) ++c_neg;
        float ef[DIM][DIM], nf[DIM][DIM];
        columns_mixed<DIM>(xs, ef);
        float detf = adjugate_rows<DIM>(ef, nf);
        if (!shape_ok<DIM>(ef, detf, tau2)) ++c_fallback;
    }
    atomicAdd(&s_cnt[0], c_bad);
    atomicAdd(&s_cnt[1], c_degen);
    atomicAdd(&s_cnt[2], c_fallback);
    atomicAdd(&s_cnt[3], c_neg);
    __syncthreads();
    if (threadIdx.x < 4 && s_cnt[threadIdx.x]) atomicAdd(counts + threadIdx.x, s_cnt[threadIdx.x]);
}

}  // namespace fem

using namespace fem;

extern "C" int64_t fem_node2cell_work_size(int64_t n_verts) {
    if (n_verts < 0) return 0;
    return n_verts + scan_tiles_for(n_verts) + 1;
}

extern "C" fem_status fem_build_node2cell(int dim, int64_t n_cells, int64_t n_verts, const int32_t *conn,
                                          int32_t *node_ptr, int32_t *node_idx, int32_t *work, fem_stream stream) {
    if (dim != 2 && dim != 3) return fail(FEM_ERR_ARG, "dim = %d, must be 2 or 3", dim);
    if (n_cells < 0 || n_verts < 0) return fail(FEM_ERR_ARG, "negative size");
    if ((dim + 1) * n_cells >= (int64_t(1) << 31) || n_verts >= (int64_t(1) << 31))
        return fail(FEM_ERR_SHAPE, "mesh too large for int32 indexing");
    if (n_cells > 0 && (n_verts < 1 || !conn)) return fail(FEM_ERR_ARG, "cells without vertices or NULL conn");
    fem_status st;
    if (!node_ptr || (n_verts > 0 && !work) || (n_cells > 0 && !node_idx))
        return fail(FEM_ERR_ARG, "node_ptr, node_idx or work is NULL");
    cudaStream_t s = stream;
    if (n_cells == 0 || n_verts == 0) {
        if (cudaMemsetAsync(node_ptr, 0, sizeof(int32_t) * (n_verts + 1), s) != cudaSuccess)
            return check_launch("node2cell memset");
        return check_launch("node2cell");
    }
    const uint32_t V = static_cast<uint32_t>(n_verts);
    unsigned *err = device_error_word();
    if (!err) return fail(FEM_ERR_CUDA, "device error word unavailable");
    int32_t *cursor = work;
    const int32_t *ptr = node_ptr;
    {
        auto k = zero_kernel;
        launch_overlapped(k, grid_for(n_verts + 1, kBlock, reinterpret_cast<const void *>(k)), kBlock, 0, s, node_ptr, n_verts + 1);
    }
    auto lists = [&](auto nb) {
        constexpr int NBC = decltype(nb)::value;
        {
            auto k = count_kernel<NBC>;
            launch_overlapped(k, grid_for(n_cells, kBlock, reinterpret_cast<const void *>(k)), kBlock, 0, s, conn, n_cells, V, node_ptr + 1, err);
        }
        const fem_status e = scan_with_cursor(node_ptr + 1, n_verts, work + n_verts, cursor, s);
        if (e != FEM_OK) return e;
        {
            auto k = fill_kernel<NBC>;
            launch_overlapped(k, grid_for(n_cells, kBlock, reinterpret_cast<const void *>(k)), kBlock, 0, s, conn, n_cells, V, cursor, node_idx);
        }
        auto k = sort_segments_kernel<8, NBC == 4>;
        launch_overlapped(k, grid_for(n_verts * 8, kBlock, reinterpret_cast<const void *>(k)), kBlock, 0, s, ptr, node_idx, n_verts);
        return FEM_OK;
    };
    st = dim == 2 ? lists(std::integral_constant<int, 3>()) : lists(std::integral_constant<int, 4>());
    if (st != FEM_OK) return st;
    return check_launch("fem_build_node2cell");
}

extern "C" fem_status fem_gather_nodes(int dim, int n_comp, int64_t n_cells, int64_t n_verts, const void *elem,
                                       const int32_t *node_ptr, const int32_t *node_idx, void *out,
                                       fem_precision prec, fem_stream stream) {
    if (dim != 2 && dim != 3) return fail(FEM_ERR_ARG, "dim = %d", dim);
    if (n_comp < 1 || n_comp > 3) return fail(FEM_ERR_ARG, "n_comp = %d", n_comp);
    if (n_cells < 0 || n_verts < 0) return fail(FEM_ERR_ARG, "negative size");
    if (prec != FEM_FP64 && prec != FEM_FP32_MIXED && prec != FEM_FP32 && prec != FEM_FP64_DF)
        return fail(FEM_ERR_ARG, "unknown precision %d", static_cast<int>(prec));
    if (n_verts > 0 && (!node_ptr || !out)) return fail(FEM_ERR_ARG, "NULL argument");
    if (n_cells > 0 && (!elem || !node_idx)) return fail(FEM_ERR_ARG, "NULL argument");
    return launch_gather(dim, n_comp, n_cells, n_verts, elem, node_ptr, node_idx, out, prec, stream);
}

extern "C" fem_status fem_check_mesh(int dim, int64_t n_cells, int64_t n_verts, const double *coords,
                                     const int32_t *conn, int64_t *counts, fem_stream stream) {
    fem_status st = check_common(dim, n_cells, n_verts, coords, conn);
    if (st != FEM_OK) return st;
    if (!counts) return fail(FEM_ERR_ARG, "counts is NULL");
    if (cudaMemsetAsync(counts, 0, 4 * sizeof(int64_t), stream) != cudaSuccess) return check_launch("check memset");
    if (n_cells == 0) return check_launch("fem_check_mesh");
    float tau = mixed_tau();
    unsigned long long *cnt = reinterpret_cast<unsigned long long *>(counts);
    const uint32_t V = static_cast<uint32_t>(n_verts);
    if (dim == 2) {
        auto k = check_mesh_kernel<2>;
        k<<<grid_for(n_cells, kBlock, reinterpret_cast<const void *>(k)), kBlock, 0, stream>>>(coords, n_cells, V,
                                                                                              conn, tau * tau, cnt);
    } else {
        auto k = check_mesh_kernel<3>;
        k<<<grid_for(n_cells, kBlock, reinterpret_cast<const void *>(k)), kBlock, 0, stream>>>(coords, n_cells, V,
                                                                                              conn, tau * tau, cnt);
    }
    return check_launch("fem_check_mesh");
}
