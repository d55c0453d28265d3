// The fast summation for the 3D kernel G(r) = 1/(4 pi r): binning, spreading, interpolation,
// near field and output (the transform is in kernels_fft.cu).
//
// The paper names the 3D Green function as the next step with the same pipeline; each
// kernel here is the 2D one with a third coordinate:
//   spreading    g_k = sum_j q_j psi(k1 - u_j1) psi(k2 - u_j2) psi(k3 - u_j3) over the
//                (2m)^3 grid lines around each source; one warp per source, lanes 0..6m-1
//                hold the window values of the three coordinates and every lane owns
//                (2m)^3 / 32 taps.  FP32: shared tiles of the source cell with a TwoSum
//                compensation plane, flushed once per item (m = 4: k_spread3_runs, a tile per
//                block; other widths: k_spread3_tile, a tile per warp); FP64 (or tiles too large
//                for shared memory, or few sources): global atomics (k_spread3);
//   interpolation phi and grad phi from the same taps, the window and its slope;
//   near field   q (1/(4 pi r) - T_I(r)) and its gradient for 0 < r < eps_I over the 27
//                cells around, -q T_I(0) for coincident points.  FP32: warp items over the
//                targets with candidate lists (k_near3_warp) or, when sources outnumber
//                targets three to one, over the sources (k_near3_src); pairs closer than
//                eps_I / 8 take their difference from hi + lo coordinates.  FP64: thread per
//                target (k_near3_f64);
//   output       phi = s phi~, H = -s^2 grad~ phi~ (1/r is homogeneous of degree -1).
// Grid layout: g[z][y][x], x fastest, edge n_a (the active window); a point's base grid
// line per coordinate is packed into 10 bits each.
#include "near_warp.cuh"
#include "sort_shared.cuh"

namespace fs {

namespace {

template <typename real> using real2_t = typename Cplx<real>::type;

__device__ __forceinline__ int b3x(int p) { return p & 1023; }
__device__ __forceinline__ int b3y(int p) { return (p >> 10) & 1023; }
__device__ __forceinline__ int b3z(int p) { return (p >> 20) & 1023; }

__global__ void k_rmax3(const double *__restrict__ xyz, int64_t n, unsigned long long *out)
{
    double best = 0.0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const double x = xyz[3 * k], y = xyz[3 * k + 1], z = xyz[3 * k + 2];
        best = fmax(best, x * x + y * y + z * z);
    }
    for (int o = 16; o > 0; o >>= 1)
        best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax(out, (unsigned long long)__double_as_longlong(best));   // non-negative: bit order = value order
}

// Window grid line of torus coordinate s x: floor(n_os s x) + n_os/2 - window_lo, and the
// fraction n_os s x - floor(n_os s x); `outside` is set when the taps leave the active window (the
// point lies beyond the admissible radius).
__device__ __forceinline__ int grid_line3(double x, double s, int n_os, int window_lo, int m, int n_a, double &frac,
                                          bool &outside)
{
    const double v = (double)n_os * (s * x);
    const double fl = floor(v);
    frac = v - fl;
    int b = (int)fl + n_os / 2 - window_lo;
    if (b - m + 1 < 0 || b + m > n_a - 1) {
        outside = true;
        b = b - m + 1 < 0 ? m - 1 : n_a - 1 - m;
        frac = 0.0;
    }
    return b;
}

__global__ void k_point_keys3(const double *__restrict__ xyz, int64_t n, double s, int n_os, int window_lo, int n_a,
                              int m, CellGrid3 cg, int *__restrict__ key, int *__restrict__ count, int *status)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n)
        return;
    int b[3], sc[3];
    bool outside = false;
    for (int d = 0; d < 3; ++d) {
        double f;
        b[d] = grid_line3(xyz[3 * k + d], s, n_os, window_lo, m, n_a, f, outside);
        // sub-cell from the offset inside the cell, (b mod cell + frac) / cell in [0, 1)
        const int sidx = (int)(((double)(b[d] % cg.cell) + f) * cg.sub / cg.cell);
        sc[d] = sidx < cg.sub ? sidx : cg.sub - 1;
    }
    if (outside)
        atomicExch(status, 1);
    int morton = 0;
    for (int bit = 0; bit < 2; ++bit)
        morton |= (((sc[2] >> bit) & 1) << (3 * bit)) | (((sc[1] >> bit) & 1) << (3 * bit + 1)) |
                  (((sc[0] >> bit) & 1) << (3 * bit + 2));
    const int kk = cg.key(b[0] / cg.cell, b[1] / cg.cell, b[2] / cg.cell) * cg.sub3() + morton;
    key[k] = kk;
    atomicAdd(&count[kk], 1);
}

template <typename real>
__global__ void k_gather_points3(const double *__restrict__ xyz, const int *__restrict__ perm, int64_t n, double s,
                                 int n_os, int window_lo, int n_a, int m, int cell,
                                 double *__restrict__ pos, real *__restrict__ frac, int *__restrict__ base,
                                 float4 *__restrict__ hi, float4 *__restrict__ lo)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n)
        return;
    const int64_t i = perm[k];
    int b[3];
    double fr[3];
    bool outside;   // k_point_keys3 reports it
    for (int d = 0; d < 3; ++d) {
        b[d] = grid_line3(xyz[3 * i + d], s, n_os, window_lo, m, n_a, fr[d], outside);
        pos[3 * k + d] = s * xyz[3 * i + d];
        frac[3 * k + d] = (real)fr[d];
    }
    base[k] = b[0] | (b[1] << 10) | (b[2] << 20);
    if (hi) {
        // offset from the lower corner of the point's cell as hi + lo: 48 bits of at most a cell's width,
        // which end some bits above or below the coordinate's last place
        float o[3], l[3];
        for (int d = 0; d < 3; ++d) {
            const double corner = (double)((b[d] / cell) * cell + window_lo) / n_os - 0.5;
            const double off = s * xyz[3 * i + d] - corner;
            o[d] = (float)off;
            l[d] = (float)(off - (double)o[d]);
        }
        hi[k] = make_float4(o[0], o[1], o[2], 0.f);
        lo[k] = make_float4(l[0], l[1], l[2], 0.f);
    }
}

// Points of a cell into slabs, strips and pieces (CellSplit3): one block per cell, three sorts of a run.
constexpr int kOrder3Threads = 256;
__global__ void __launch_bounds__(kOrder3Threads) k_cell_order3(const int *__restrict__ start, CellGrid3 cg, int cap,
                                                                const double *__restrict__ xyz, double s, int n_os,
                                                                int window_lo, int n_a, int m, int *__restrict__ perm)
{
    __shared__ unsigned long long key[kOrderRun];
    __shared__ unsigned q[3][kOrderRun];
    __shared__ int idx[kOrderRun];
    const int S3 = cg.sub3();
    const int a = start[(int64_t)blockIdx.x * S3], count = start[(int64_t)(blockIdx.x + 1) * S3] - a;
    if (count <= cap)
        return;
    bool outside;   // k_point_keys3 reports it
    for (int r = 0; r < CellSplit::runs(count); ++r) {
        const int first = a + CellSplit::run_first(count, r), n = a + CellSplit::run_first(count, r + 1) - first;
        const CellSplit3 split(n, cap);
        int n2 = 2;
        while (n2 < n)
            n2 <<= 1;
        __syncthreads();   // the previous run's keys are read
        for (int t = threadIdx.x; t < n2; t += blockDim.x) {
            unsigned long long k = ~0ull;
            if (t < n) {
                const int i = perm[first + t];
                for (int d = 0; d < 3; ++d) {
                    double f;
                    const int b = grid_line3(xyz[3 * (int64_t)i + d], s, n_os, window_lo, m, n_a, f, outside);
                    q[d][t] = (unsigned)((((double)(b % cg.cell) + f) / cg.cell) * 4194304.0);   // 22 bits
                }
                idx[t] = i;
                k = ((unsigned long long)q[0][t] << 16) | (unsigned)t;
            }
            key[t] = k;
        }
        __syncthreads();
        // a pass per axis: sort, then number each point's slab (strip) and key it by the next axis
        for (int axis = 0; axis < 3; ++axis) {
            sort_shared(key, n2);
            if (axis == 2)
                break;
            for (int t = threadIdx.x; t < n; t += blockDim.x) {
                int slab = 0;
                while (t >= split.slab_first(slab + 1))
                    ++slab;
                int part = slab << 8;
                if (axis == 1) {
                    const int k = split.slab_piece(slab + 1) - split.slab_piece(slab), t0 = split.slab_first(slab);
                    const int len = split.slab_first(slab + 1) - t0;
                    int strip = 0;
                    while (t - t0 >= CellSplit3::strip_first(k, len, strip + 1))
                        ++strip;
                    part |= strip;
                }
                const unsigned slot = (unsigned)key[t] & 0xffffu;
                key[t] = ((unsigned long long)part << 48) | ((unsigned long long)q[axis + 1][slot] << 16) | slot;
            }
            __syncthreads();
        }
        for (int t = threadIdx.x; t < n; t += blockDim.x)
            perm[first + t] = idx[(unsigned)key[t] & 0xffffu];
    }
}

// One warp per source: lanes 0..M2-1, M2..2M2-1, 2M2..3M2-1 evaluate the x, y, z window values
// (x times q), every lane adds its taps (t = lane + 32 i: x fastest) to the grid.
template <typename real, int M2>
__global__ void __launch_bounds__(256) k_spread3(int64_t M, const int *__restrict__ base, const real *__restrict__ frac,
                                                 const real *__restrict__ q, Window<real> w, WindowPoly wp,
                                                 real *__restrict__ grid, int n_a)
{
    constexpr int m = M2 / 2;
    constexpr int TAPS = M2 * M2 * M2;
    constexpr int PER = (TAPS + 31) / 32;
    const int lane = threadIdx.x & 31;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int dim = lane / M2, jw = lane - (lane / M2) * M2;
    // software pipeline: the next source's record is in flight while this one is spread
    int64_t j = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int nb = 0;
    real nf = real(0), nq = real(0);
    if (j < M) {
        nb = base[j];
        nf = lane < 3 * M2 ? frac[3 * j + dim] : real(0);
        nq = q[j];
    }
    for (; j < M; j += warps) {
        const int packed = nb;
        const real fr = nf, qj = nq;
        if (j + warps < M) {
            nb = base[j + warps];
            nf = lane < 3 * M2 ? frac[3 * (j + warps) + dim] : real(0);
            nq = q[j + warps];
        }
        real wv = real(0);
        if (lane < 3 * M2) {
            if constexpr (sizeof(real) == 4)
                wv = poly_eval<kPolyD>(wp.c[jw], (float)fr - 0.5f);
            else
                wv = kb_value<real>(w, fr, m - 1 - jw);
            if (dim == 0)
                wv *= qj;
        }
        const int x0 = b3x(packed) - m + 1, y0 = b3y(packed) - m + 1, z0 = b3z(packed) - m + 1;
        if constexpr (M2 == 8) {
            // t = lane + 32 i: tx = lane % 8 for every i, ty takes two values (i even / odd) and
            // tz = i / 2, so 11 shuffles serve the 16 taps of a lane
            const real vx = __shfl_sync(0xffffffffu, wv, lane & 7);
            const real vxy0 = vx * __shfl_sync(0xffffffffu, wv, 8 + (lane >> 3));
            const real vxy1 = vx * __shfl_sync(0xffffffffu, wv, 12 + (lane >> 3));
            real* row = grid + ((int64_t)z0 * n_a + (y0 + (lane >> 3))) * n_a + (x0 + (lane & 7));
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const real vz = __shfl_sync(0xffffffffu, wv, 16 + (i >> 1));
                atomicAdd(row + ((int64_t)(i >> 1) * n_a + 4 * (i & 1)) * n_a, ((i & 1) ? vxy1 : vxy0) * vz);
            }
        } else {
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                const int t = lane + 32 * i;
                const int tx = t % M2, ty = (t / M2) % M2, tz = t / (M2 * M2);
                const real vx = __shfl_sync(0xffffffffu, wv, tx);
                const real vy = __shfl_sync(0xffffffffu, wv, M2 + ty);
                const real vz = __shfl_sync(0xffffffffu, wv, 2 * M2 + (tz < M2 ? tz : 0));
                if (t < TAPS)
                    atomicAdd(grid + ((int64_t)(z0 + tz) * n_a + (y0 + ty)) * n_a + (x0 + tx), vx * vy * vz);
            }
        }
    }
}

// FP32 spreading through warp-private tiles in shared memory (items of at most
// kSpread3ItemMax sources of one cell).  Each warp owns a tile covering the cell's taps, edge
// P = cell + 2m - 1 grid lines, plus a compensation plane: a warp handles one source at a time
// and every tap of a source is a distinct cell, so the read-modify-write needs no atomics, and
// the rounding error of each addition is recovered exactly (TwoSum) into the compensation
// plane.  The warps' tiles are summed and added to the grid once per item with global atomics.
// This replaces 512 global atomics per source (at m = 4) by 2 shared reads and 2 writes per tap.
constexpr int kSpread3Warps = 4;

template <int M2>
__global__ void __launch_bounds__(kSpread3Warps * 32) k_spread3_tile(const int2 *__restrict__ items,
                                                                     const int *__restrict__ base,
                                                                     const float *__restrict__ frac,
                                                                     const float *__restrict__ q, WindowPoly wp,
                                                                     int cell, float *__restrict__ grid, int n_a)
{
    constexpr int m = M2 / 2;
    constexpr int TAPS = M2 * M2 * M2;
    constexpr int PER = (TAPS + 31) / 32;
    extern __shared__ float tiles[];
    const int P = cell + M2 - 1, P3 = P * P * P;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *acc = tiles + (size_t)warp * 2 * P3;   // value plane, then compensation plane
    const int2 it = items[blockIdx.x];
    for (int i = lane; i < 2 * P3; i += 32)
        acc[i] = 0.f;
    const int pk = base[it.x];
    const int ox = (b3x(pk) / cell) * cell - (m - 1), oy = (b3y(pk) / cell) * cell - (m - 1),
              oz = (b3z(pk) / cell) * cell - (m - 1);
    const int dim = lane / M2, jw = lane - (lane / M2) * M2;
    float pc[kPolyD + 1];   // this lane's window polynomial
#pragma unroll
    for (int k = 0; k <= kPolyD; ++k)
        pc[k] = wp.c[lane < 3 * M2 ? jw : 0][k];
    __syncwarp();
    // software pipeline: the next source's record is in flight while this one is spread
    const int end = it.x + it.y;
    int j = it.x + warp;
    int nb = 0;
    float nf = 0.f, nq = 0.f;
    if (j < end) {
        nb = base[j];
        nf = lane < 3 * M2 ? frac[3 * j + dim] : 0.f;
        nq = q[j];
    }
    for (; j < end; j += kSpread3Warps) {
        const int packed = nb;
        const float fr = nf, qj = nq;
        if (j + kSpread3Warps < end) {
            nb = base[j + kSpread3Warps];
            nf = lane < 3 * M2 ? frac[3 * (j + kSpread3Warps) + dim] : 0.f;
            nq = q[j + kSpread3Warps];
        }
        float wv = 0.f;
        if (lane < 3 * M2) {
            wv = poly_eval<kPolyD>(pc, fr - 0.5f);
            if (dim == 0)
                wv *= qj;
        }
        const int lx = b3x(packed) - m + 1 - ox, ly = b3y(packed) - m + 1 - oy, lz = b3z(packed) - m + 1 - oz;
        float v[PER];
        int idx[PER];
        bool on[PER];
        if constexpr (M2 == 8) {
            const float vx = __shfl_sync(0xffffffffu, wv, lane & 7);
            const float vxy0 = vx * __shfl_sync(0xffffffffu, wv, 8 + (lane >> 3));
            const float vxy1 = vx * __shfl_sync(0xffffffffu, wv, 12 + (lane >> 3));
            const int row = (lz * P + ly + (lane >> 3)) * P + lx + (lane & 7);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                v[i] = ((i & 1) ? vxy1 : vxy0) * __shfl_sync(0xffffffffu, wv, 16 + (i >> 1));
                idx[i] = row + ((i >> 1) * P + 4 * (i & 1)) * P;
                on[i] = true;
            }
        } else {
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                const int t = lane + 32 * i;
                const int tx = t % M2, ty = (t / M2) % M2, tz = t / (M2 * M2);
                const float vx = __shfl_sync(0xffffffffu, wv, tx);
                const float vy = __shfl_sync(0xffffffffu, wv, M2 + ty);
                const float vz = __shfl_sync(0xffffffffu, wv, 2 * M2 + (tz < M2 ? tz : 0));
                v[i] = vx * vy * vz;
                idx[i] = ((lz + tz) * P + (ly + ty)) * P + (lx + tx);
                on[i] = t < TAPS;
            }
        }
        // a source's taps are distinct cells: all reads before the writes
        float old[PER], cmp[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (on[i]) {
                old[i] = acc[idx[i]];
                cmp[i] = acc[P3 + idx[i]];
            }
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (on[i]) {
                const float s = old[i] + v[i];
                const float bb = s - old[i];
                acc[idx[i]] = s;
                acc[P3 + idx[i]] = cmp[i] + ((old[i] - (s - bb)) + (v[i] - bb));
            }
        __syncwarp();
    }
    __syncthreads();
    for (int i = threadIdx.x; i < P3; i += blockDim.x) {
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < kSpread3Warps; ++w)
            v += tiles[(size_t)w * 2 * P3 + i] + tiles[(size_t)w * 2 * P3 + P3 + i];
        const int x = i % P, y = (i / P) % P, z = i / (P * P);
        const int gx = ox + x, gy = oy + y, gz = oz + z;
        if (v != 0.f && gx >= 0 && gx < n_a && gy >= 0 && gy < n_a && gz >= 0 && gz < n_a)
            atomicAdd(grid + ((int64_t)gz * n_a + gy) * n_a + gx, v);
    }
}

// FP32 spreading at 2m = 8 through one shared tile per block, sources of a cell in the order of their
// base grid lines (k_spread3_order).  Warp w of the block's four adds, for every source of the item,
// the taps on the tile planes z = w (mod 4): two of the source's eight, a plane belongs to one warp,
// and a lane holds one x and two y of both planes, four taps.  So the tile is shared without atomics
// (21.6 KB for 6-line cells, ten blocks per SM) where a tile per warp left three blocks of four.
// Consecutive sources with the same base lines (4.5 of them at 970 per 6^3-line cell) have the same
// taps and are summed in registers, value and TwoSum error, before the tile is read and written.
// The weights of 128 sources at a time are evaluated a source per thread, coefficients from the
// constant bank, into shared memory.  Rows are 16 floats, pairs of rows rotated by 8, so that the 8
// x and 4 y of a warp's access fall on 32 banks.
// It is bound by the shared-memory pipe and the issue slots (about 140 instructions a source over the
// four warps, against some 300 and 64 conflicting shared accesses).  Measured: 1.59M quadrature
// points of the 384,000-tetrahedron cube 1330 -> 421 us; 2^18 points of a ball (41 per cell) 206 us
// with global atomics, 162 us here.
constexpr int kSpread3RunThreads = 128;
constexpr int kSpread3WeightPitch = 25;   // 24 weights a source, odd
template <int kM2 = 8>
__global__ void __launch_bounds__(kSpread3RunThreads) k_spread3_runs(const int2 *__restrict__ items,
                                                                     const int *__restrict__ base,
                                                                     const float *__restrict__ frac,
                                                                     const int *__restrict__ order,
                                                                     const float *__restrict__ q, WindowPoly wp,
                                                                     int cell, float *__restrict__ grid, int n_a)
{
    constexpr int m = kM2 / 2;
    static_assert(kM2 == 8, "two planes, two rows and one column of taps a lane");
    extern __shared__ __align__(16) float sm[];
    const int P = cell + kM2 - 1, plane = P * P * 16;   // words of the value tile; the compensation tile follows
    float *acc = sm, *wt = sm + 2 * plane;
    int *bs = reinterpret_cast<int *>(wt + kSpread3RunThreads * kSpread3WeightPitch);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int2 it = items[blockIdx.x];
    for (int i = threadIdx.x; i < plane / 2; i += kSpread3RunThreads)
        reinterpret_cast<float4 *>(acc)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int pk0 = base[it.x];
    const int ox = (b3x(pk0) / cell) * cell - (m - 1), oy = (b3y(pk0) / cell) * cell - (m - 1),
              oz = (b3z(pk0) / cell) * cell - (m - 1);
    int run = -1, z0 = 0, at[4] = {0, 0, 0, 0};
    float2 s0 = f2(0.f), s1 = s0, c0 = s0, c1 = s0;   // planes z0, z0 + 4: rows y, y + 4
    auto flush = [&]() {
        const float v[4] = {s0.x, s0.y, s1.x, s1.y}, c[4] = {c0.x, c0.y, c1.x, c1.y};
        float old[4], cmp[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            old[k] = acc[at[k]];
            cmp[k] = acc[plane + at[k]];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float t = old[k] + v[k], bb = t - old[k];
            acc[at[k]] = t;
            acc[plane + at[k]] = cmp[k] + (((old[k] - (t - bb)) + (v[k] - bb)) + c[k]);
        }
        __syncwarp();   // the next run's cells may be other lanes' of this one
    };
    for (int first = 0; first < it.y; first += kSpread3RunThreads) {
        const int n = min(kSpread3RunThreads, it.y - first);
        __syncthreads();   // the last weights are read (and the tile is zeroed)
        if (threadIdx.x < n) {
            const int j = it.x + first + threadIdx.x;
            float *o = wt + threadIdx.x * kSpread3WeightPitch;
            const float qj = q[order[j]];
            bs[threadIdx.x] = base[j];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const float t = frac[3 * (int64_t)j + d] - 0.5f, s = t * t;
#pragma unroll
                for (int a = 0; a < m; ++a) {
                    float e, od;
                    poly_even_odd<kPolyD>(wp.c[a], s, e, od);
                    o[8 * d + a] = fmaf(t, od, e) * (d == 0 ? qj : 1.f);
                    o[8 * d + kM2 - 1 - a] = fmaf(-t, od, e) * (d == 0 ? qj : 1.f);
                }
            }
        }
        __syncthreads();
        for (int i = 0; i < n; ++i) {
            const int pk = bs[i];
            if (pk != run) {
                if (run >= 0)
                    flush();
                run = pk;
                const int lz = b3z(pk) - m + 1 - oz, y = b3y(pk) - m + 1 - oy + (lane >> 3),
                          x = b3x(pk) - m + 1 - ox + (lane & 7);
                z0 = (warp - lz) & 3;
                const int r = (lz + z0) * P + y;   // tile row of plane z0 and row y
                at[0] = r * 16 + ((x + 8 * ((y >> 1) & 1)) & 15);
                at[1] = at[0] + 4 * 16;
                at[2] = at[0] + 4 * P * 16;
                at[3] = at[1] + 4 * P * 16;
                s0 = s1 = c0 = c1 = f2(0.f);
            }
            const float *o = wt + i * kSpread3WeightPitch;
            const float wx = o[lane & 7];
            const float2 wxy = make_float2(wx * o[8 + (lane >> 3)], wx * o[12 + (lane >> 3)]);
            const float2 v0 = mul2(wxy, f2(o[16 + z0])), v1 = mul2(wxy, f2(o[20 + z0]));
            const float2 t0 = add2(s0, v0), t1 = add2(s1, v1);
            const float2 b0 = add2(t0, make_float2(-s0.x, -s0.y)), b1 = add2(t1, make_float2(-s1.x, -s1.y));
            const float2 e0 = add2(add2(s0, fma2(b0, f2(1.f), make_float2(-t0.x, -t0.y))),
                                   add2(v0, make_float2(-b0.x, -b0.y)));
            const float2 e1 = add2(add2(s1, fma2(b1, f2(1.f), make_float2(-t1.x, -t1.y))),
                                   add2(v1, make_float2(-b1.x, -b1.y)));
            c0 = add2(c0, e0);
            c1 = add2(c1, e1);
            s0 = t0;
            s1 = t1;
        }
    }
    if (run >= 0)
        flush();
    __syncthreads();
    for (int i = threadIdx.x; i < plane; i += kSpread3RunThreads) {
        const int x = i & 15, r = i >> 4, y = r % P, z = r / P;
        const float v = acc[i] + acc[plane + i];
        const int gx = ox + ((x - 8 * ((y >> 1) & 1)) & 15), gy = oy + y, gz = oz + z;
        if (v != 0.f && gx >= 0 && gx < n_a && gy >= 0 && gy < n_a && gz >= 0 && gz < n_a)
            atomicAdd(grid + ((int64_t)gz * n_a + gy) * n_a + gx, v);
    }
}

// Sort keys of the run order: cell key x cell^3 + base grid lines inside the cell.
__global__ void k_spread3_keys(const int *__restrict__ base, int64_t M, CellGrid3 cg, int *__restrict__ key,
                               int *__restrict__ count)
{
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= M)
        return;
    const int pk = base[j], c = cg.cell;
    const int x = b3x(pk), y = b3y(pk), z = b3z(pk);
    const int k = cg.key(x / c, y / c, z / c) * (c * c * c) + ((z % c) * c + y % c) * c + x % c;
    key[j] = k;
    atomicAdd(&count[k], 1);
}

__global__ void k_spread3_order(const int *__restrict__ order, int64_t M, const int *__restrict__ base,
                                const float *__restrict__ frac, int *__restrict__ run_base,
                                float *__restrict__ run_frac)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= M)
        return;
    const int64_t j = order[k];
    run_base[k] = base[j];
    for (int d = 0; d < 3; ++d)
        run_frac[3 * k + d] = frac[3 * j + d];
}

// phi~ and grad~ phi~ at the targets from the filtered grid (thread per target).
template <typename real, int M2>
__global__ void __launch_bounds__(256) k_interp3(int64_t N, const int *__restrict__ base, const real *__restrict__ frac,
                                                 Window<real> w, WindowPoly wp, const real *__restrict__ grid, int n_a,
                                                 real n_os, real *__restrict__ phi_s, real *__restrict__ grad_s,
                                                 bool acc)
{
    constexpr int m = M2 / 2;
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= N)
        return;
    real wt[3][M2], dt[3][M2];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const real fr = frac[3 * k + d];
#pragma unroll
        for (int a = 0; a < M2; ++a) {
            if constexpr (sizeof(real) == 4) {
                wt[d][a] = poly_eval<kPolyD>(wp.c[a], (float)fr - 0.5f);
                dt[d][a] = poly_eval<kPolyD - 1>(wp.d[a], (float)fr - 0.5f);
            } else {
                kb_value_slope<real>(w, fr, m - 1 - a, wt[d][a], dt[d][a]);
            }
        }
    }
    const int packed = base[k];
    const int x0 = b3x(packed) - m + 1, y0 = b3y(packed) - m + 1, z0 = b3z(packed) - m + 1;
    real phi = 0, gx = 0, gy = 0, gz = 0;
    for (int c = 0; c < M2; ++c) {
        real t = 0, tx = 0, ty = 0;
        for (int b = 0; b < M2; ++b) {
            const real *row = grid + ((int64_t)(z0 + c) * n_a + (y0 + b)) * n_a + x0;
            real s = 0, sx = 0;
#pragma unroll
            for (int a = 0; a < M2; ++a) {
                const real g = __ldg(row + a);
                s += wt[0][a] * g;
                sx += dt[0][a] * g;
            }
            t += wt[1][b] * s;
            tx += wt[1][b] * sx;
            ty += dt[1][b] * s;
        }
        phi += wt[2][c] * t;
        gx += wt[2][c] * tx;
        gy += wt[2][c] * ty;
        gz += dt[2][c] * t;
    }
    // acc: the near field was stored first (it ran beside spreading and the transform)
    phi_s[k] = acc ? phi_s[k] + phi : phi;
    grad_s[3 * k] = acc ? grad_s[3 * k] + n_os * gx : n_os * gx;
    grad_s[3 * k + 1] = acc ? grad_s[3 * k + 1] + n_os * gy : n_os * gy;
    grad_s[3 * k + 2] = acc ? grad_s[3 * k + 2] + n_os * gz : n_os * gz;
}

// FP32 interpolation and output at 2m = 8, for plans whose near field was stored first (k_interp3 with
// acc, then k_unpermute3, in one pass): eight lanes a target, lane a its taps of column x = a, so that
// a grid row of 8 taps is one 32-byte read where a thread per target reads 32 rows a request.  A
// lane holds its tap's value and slope polynomials in registers for all its targets; the y and z
// weights of a target's lanes go through shared memory.  Bound by the L1's sector rate (128 a
// target).  2^18 targets of a ball: 127 + 9 us -> about 75 us (the step 617 -> 566 us).
constexpr int kInterp3Threads = 256;
__global__ void __launch_bounds__(kInterp3Threads) k_interp3_out(int64_t N, const int *__restrict__ base,
                                                                 const float *__restrict__ frac, WindowPoly wp,
                                                                 const float *__restrict__ grid, int n_a, float n_os,
                                                                 const float *__restrict__ phi_s,
                                                                 const float *__restrict__ grad_s,
                                                                 const int *__restrict__ perm, double s,
                                                                 void *__restrict__ phi_out, void *__restrict__ H_out,
                                                                 int out_f64)
{
    constexpr int m = 4, M2 = 8, kPitch = 36;   // 32 weights a target; 16-byte aligned, spread over the banks
    __shared__ __align__(16) float wt[kInterp3Threads / M2][kPitch];
    const int lane = threadIdx.x & 31, a = lane & 7, slot = threadIdx.x >> 3;
    float pc[kPolyD + 1], pd[kPolyD];
#pragma unroll
    for (int k = 0; k <= kPolyD; ++k)
        pc[k] = wp.c[a][k];
#pragma unroll
    for (int k = 0; k < kPolyD; ++k)
        pd[k] = wp.d[a][k];
    const int64_t step = (int64_t)gridDim.x * (kInterp3Threads / M2);
    // (whole warps stay together: a warp's four targets are consecutive)
    for (int64_t first = (int64_t)blockIdx.x * (kInterp3Threads / M2) + (slot & ~3); first < N; first += step) {
        const int64_t k = first + (slot & 3);
        const int64_t kk = k < N ? k : N - 1;
        const int packed = base[kk];
        const float fx = frac[3 * kk] - 0.5f, fy = frac[3 * kk + 1] - 0.5f, fz = frac[3 * kk + 2] - 0.5f;
        const float wx = poly_eval<kPolyD>(pc, fx), dx = poly_eval<kPolyD - 1>(pd, fx);
        __syncwarp();
        wt[slot][a] = poly_eval<kPolyD>(pc, fy);
        wt[slot][8 + a] = poly_eval<kPolyD - 1>(pd, fy);
        wt[slot][16 + a] = poly_eval<kPolyD>(pc, fz);
        wt[slot][24 + a] = poly_eval<kPolyD - 1>(pd, fz);
        __syncwarp();
        float wy[M2], dy[M2];
#pragma unroll
        for (int i = 0; i < M2; i += 4) {
            const float4 u = *reinterpret_cast<const float4 *>(&wt[slot][i]);
            const float4 v = *reinterpret_cast<const float4 *>(&wt[slot][8 + i]);
            wy[i] = u.x;
            wy[i + 1] = u.y;
            wy[i + 2] = u.z;
            wy[i + 3] = u.w;
            dy[i] = v.x;
            dy[i + 1] = v.y;
            dy[i + 2] = v.z;
            dy[i + 3] = v.w;
        }
        const float *row = grid + ((int64_t)(b3z(packed) - m + 1) * n_a + (b3y(packed) - m + 1)) * n_a +
                           (b3x(packed) - m + 1 + a);
        float A = 0.f, B = 0.f, C = 0.f;   // sums over y, z of g w w, g d w, g w d
#pragma unroll 2
        for (int c = 0; c < M2; ++c) {
            float g[M2];
#pragma unroll
            for (int b = 0; b < M2; ++b)
                g[b] = __ldg(row + b * n_a);
            row += (int64_t)n_a * n_a;
            float t = 0.f, ty = 0.f;
#pragma unroll
            for (int b = 0; b < M2; ++b) {
                t = fmaf(wy[b], g[b], t);
                ty = fmaf(dy[b], g[b], ty);
            }
            const float wz = wt[slot][16 + c], dz = wt[slot][24 + c];
            A = fmaf(wz, t, A);
            B = fmaf(wz, ty, B);
            C = fmaf(dz, t, C);
        }
        // sums over x: lanes 0, 2, 4, 6 of a target end with phi, d/dx, d/dy, d/dz
        const float v0 = wx * A, v1 = dx * A, v2 = wx * B, v3 = wx * C;
        const bool h4 = a & 4, h2 = a & 2;
        const float p = (h4 ? v2 : v0) + __shfl_xor_sync(0xffffffffu, h4 ? v0 : v2, 4);
        const float q = (h4 ? v3 : v1) + __shfl_xor_sync(0xffffffffu, h4 ? v1 : v3, 4);
        float r = (h2 ? q : p) + __shfl_xor_sync(0xffffffffu, h2 ? p : q, 2);
        r += __shfl_xor_sync(0xffffffffu, r, 1);
        if (k >= N || (a & 1))
            continue;
        const int64_t i = perm[k];
        if (a == 0) {
            const double v = s * (double)(phi_s[k] + r);
            if (phi_out && out_f64)
                ((double *)phi_out)[i] = v;
            else if (phi_out)
                ((float *)phi_out)[i] = (float)v;
        } else if (H_out) {
            const int d = (a >> 1) - 1;
            const double v = -s * s * (double)(grad_s[3 * k + d] + n_os * r);
            if (out_f64)
                ((double *)H_out)[3 * i + d] = v;
            else
                ((float *)H_out)[3 * i + d] = (float)v;
        }
    }
}

// FP64 near-field correction at target k (thread per target) over the 27 cells around its cell.
__global__ void __launch_bounds__(256) k_near3_f64(int64_t N, const int *__restrict__ tgt_base,
                                                   const double *__restrict__ tgt_pos,
                                                   const double *__restrict__ src_pos,
                                                   const int *__restrict__ src_start, CellGrid3 cg,
                                                   const double *__restrict__ q, NearParams<double> np,
                                                   double *__restrict__ phi_s, double *__restrict__ grad_s)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= N)
        return;
    const int packed = tgt_base[k];
    const int c1 = b3x(packed) / cg.cell, c2 = b3y(packed) / cg.cell, c3 = b3z(packed) / cg.cell;
    const double xt0 = tgt_pos[3 * k], xt1 = tgt_pos[3 * k + 1], xt2 = tgt_pos[3 * k + 2];
    const double inv4pi = 1.0 / (4.0 * kPi);
    const int S3 = cg.sub3();
    double phi = 0, g0 = 0, g1 = 0, g2 = 0;
    for (int e1 = max(c1 - 1, 0); e1 <= min(c1 + 1, cg.n_c - 1); ++e1)
        for (int e2 = max(c2 - 1, 0); e2 <= min(c2 + 1, cg.n_c - 1); ++e2)
            for (int e3 = max(c3 - 1, 0); e3 <= min(c3 + 1, cg.n_c - 1); ++e3) {
                const int key = cg.key(e1, e2, e3);
                const int end = src_start[(key + 1) * S3];
                for (int j = src_start[key * S3]; j < end; ++j) {
                    const double dx = xt0 - src_pos[3 * j];
                    const double dy = xt1 - src_pos[3 * j + 1];
                    const double dz = xt2 - src_pos[3 * j + 2];
                    const double r2 = dx * dx + dy * dy + dz * dz;
                    if (!(r2 < np.eps2))
                        continue;
                    const double qj = q[j];
                    if (r2 == 0.0) {
                        phi -= qj * np.beta[0];
                        continue;
                    }
                    const double u2 = r2 * np.inv_eps2;
                    double t = np.beta[np.p - 1];
                    for (int i = np.p - 2; i >= 0; --i)
                        t = t * u2 + np.beta[i];
                    double tp = 0.0;
                    if (np.p > 1) {
                        tp = np.dbeta[np.p - 2];
                        for (int i = np.p - 3; i >= 0; --i)
                            tp = tp * u2 + np.dbeta[i];
                    }
                    const double inv_r = 1.0 / sqrt(r2);
                    const double val = inv4pi * inv_r - t;
                    const double coef = -inv4pi * inv_r * inv_r * inv_r - tp;
                    phi += qj * val;
                    g0 += qj * coef * dx;
                    g1 += qj * coef * dy;
                    g2 += qj * coef * dz;
                }
            }
    phi_s[k] += phi;
    grad_s[3 * k] += g0;
    grad_s[3 * k + 1] += g1;
    grad_s[3 * k + 2] += g2;
}

// ---- FP32 near field: warp items, candidate lists, packed pairs
//
// As the 2D traversal (near_warp.cuh): a warp takes a piece of a cell, at most 8, 16 or 32 targets, one
// per lane (the 32 / lanes groups of the warp take different candidates); reads the sources of the
// 27 cells around 32 at a time, keeps those within eps_I of the piece's box, and appends them to
// lists in shared memory, negated in the piece's frame and in units of eps_I, which all lanes
// evaluate two candidates to a packed operation.  Pairs beyond eps_I get charge 0.  Sources within
// eps_I / 8 of the box go to a second list with hi + lo coordinates.  Their differences are good to
// 2^-45 of a cell edge (a few roundings of the low words), FP32's relative accuracy and better down to
// kNear3Exact eps_I.  Pairs closer than that get charge 0 in the lists: the coincident ones (equal
// FP64 positions) are accounted from the per-target lists built with the plan, and targets that have
// others, marked when the plan is built, take those from the FP64 positions at the end
// (near3_touching).  FP64 differences of all close pairs, at a 64th of the FP32 rate, were half of the
// source-major kernel's time.
// Measured, 2^18 points of a ball (41 per cell, p = 3): 380 us with items of 64 targets (two per lane,
// the box a whole cell: 0.13 of the pair slots useful) and FP64 close pairs, 249 us here; list building
// is the larger part of it.
constexpr int kNear3Warps = 4;
constexpr int kNear3Cap = 256;        // far candidates per warp
constexpr int kNear3CloseCap = 64;    // close candidates per warp

__device__ __forceinline__ float rsqrt_approx(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// w = min(r^2, 1): pairs beyond eps_I land on 1, where near3_pair drops their charge
__device__ __forceinline__ float2 near3_w(float2 dx, float2 dy, float2 dz)
{
    const float2 r = fma2(dy, dy, mul2(dx, dx));
    return make_float2(__saturatef(fmaf(dz.x, dz.x, r.x)), __saturatef(fmaf(dz.y, dz.y, r.y)));
}

struct Near3Sums {
    float2 phi, gx, gy, gz;
};

// The packed pair arithmetic of two candidates at (w, dx, dy, dz) (units of eps_I), 0 < w <= 1.
template <int P>
__device__ __forceinline__ void near3_pair(const Near3Params &np, float2 w, float2 dx, float2 dy, float2 dz,
                                           float2 qq, Near3Sums &a)
{
    const float2 c1 = f2(np.c1);
    const float2 qe = make_float2(w.x < 1.f ? qq.x : 0.f, w.y < 1.f ? qq.y : 0.f);
    const float2 rs = make_float2(rsqrt_approx(w.x), rsqrt_approx(w.y));
    float2 t = f2(np.nbeta[P - 1]);
#pragma unroll
    for (int i = P - 2; i >= 0; --i)
        t = fma2(t, w, f2(np.nbeta[i]));
    float2 u = f2(0.f);
    if constexpr (P >= 2) {
        u = f2(np.dbeta2[P - 2]);
#pragma unroll
        for (int i = P - 3; i >= 0; --i)
            u = fma2(u, w, f2(np.dbeta2[i]));
    }
    const float2 val = fma2(c1, rs, t);                            // c1 w^-1/2 - P(w)
    const float2 gc = fma2(c1, mul2(mul2(rs, rs), rs), u);         // c1 w^-3/2 + 2 P'(w)
    a.phi = fma2(qe, val, a.phi);
    const float2 qc = mul2(qe, gc);
    a.gx = fma2(qc, dx, a.gx);
    a.gy = fma2(qc, dy, a.gy);
    a.gz = fma2(qc, dz, a.gz);
}

// A pair of candidates close to the item's box: charge 0 below kNear3Exact2 (near3_touching and the lists of
// coincident pairs account for those).
template <int P>
__device__ __forceinline__ void near3_pair_close(const Near3Params &np, float2 dx, float2 dy, float2 dz, float2 qq,
                                                 Near3Sums &a)
{
    float2 w = near3_w(dx, dy, dz);
    if (w.x < kNear3Exact2)
        qq.x = 0.f;
    if (w.y < kNear3Exact2)
        qq.y = 0.f;
    w.x = fmaxf(w.x, kNear3Exact2);
    w.y = fmaxf(w.y, kNear3Exact2);
    near3_pair<P>(np, w, dx, dy, dz, qq, a);
}

struct Near3List {
    float x[kNear3Cap], y[kNear3Cap], z[kNear3Cap], q[kNear3Cap];
    float cx[kNear3CloseCap], cy[kNear3CloseCap], cz[kNear3CloseCap], cq[kNear3CloseCap];
    float lx[kNear3CloseCap], ly[kNear3CloseCap], lz[kNear3CloseCap];
    __device__ __forceinline__ void put(int at, float px, float py, float pz, float pq)
    {
        x[at] = px;
        y[at] = py;
        z[at] = pz;
        q[at] = pq;
    }
    __device__ __forceinline__ void put_close(int at, float3 p, float3 l, float pq)
    {
        cx[at] = p.x;
        cy[at] = p.y;
        cz[at] = p.z;
        lx[at] = l.x;
        ly[at] = l.y;
        lz[at] = l.z;
        cq[at] = pq;
    }
    // pads n entries to a multiple of `unit` (at most 32); returns the padded count
    __device__ __forceinline__ int pad(int n, int unit, int lane)
    {
        const int full = (n + unit - 1) & ~(unit - 1);
        if (n + lane < full)
            put(n + lane, kPadPos, kPadPos, kPadPos, 0.f);
        return full;
    }
    __device__ __forceinline__ int pad_close(int n, int unit, int lane)
    {
        const int full = (n + unit - 1) & ~(unit - 1);
        if (n + lane < full)
            put_close(n + lane, make_float3(kPadPos, kPadPos, kPadPos), make_float3(0.f, 0.f, 0.f), 0.f);
        return full;
    }
};

__device__ __forceinline__ float4 four(const float *p, int e) { return *reinterpret_cast<const float4 *>(p + 4 * e); }
__device__ __forceinline__ float2 half_of(float4 v, int h) { return h ? make_float2(v.z, v.w) : make_float2(v.x, v.y); }

// n candidates (a multiple of 4 x groups); group g takes every groups-th four of them.
template <int P>
__device__ __forceinline__ void near3_eval(const Near3List &L, int n, int g, int groups, float3 X,
                                           const Near3Params &np, Near3Sums &a)
{
#pragma unroll 2
    for (int e = g; e < n >> 2; e += groups) {
        const float4 x = four(L.x, e), y = four(L.y, e), z = four(L.z, e), q = four(L.q, e);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 dx = add2(f2(X.x), half_of(x, h)), dy = add2(f2(X.y), half_of(y, h)),
                         dz = add2(f2(X.z), half_of(z, h));
            near3_pair<P>(np, near3_w(dx, dy, dz), dx, dy, dz, half_of(q, h), a);
        }
    }
}

template <int P>
__device__ __forceinline__ void near3_eval_close(const Near3List &L, int n, int g, int groups, float3 X, float3 XL,
                                                 const Near3Params &np, Near3Sums &a)
{
    const float2 ie = f2(np.inv_eps);
    for (int e = g; e < n >> 2; e += groups) {
        const float4 x = four(L.cx, e), y = four(L.cy, e), z = four(L.cz, e), q = four(L.cq, e);
        const float4 lx = four(L.lx, e), ly = four(L.ly, e), lz = four(L.lz, e);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 dx = mul2(add2(add2(f2(X.x), half_of(x, h)), add2(f2(XL.x), half_of(lx, h))), ie);
            const float2 dy = mul2(add2(add2(f2(X.y), half_of(y, h)), add2(f2(XL.y), half_of(ly, h))), ie);
            const float2 dz = mul2(add2(add2(f2(X.z), half_of(z, h)), add2(f2(XL.z), half_of(lz, h))), ie);
            near3_pair_close<P>(np, dx, dy, dz, half_of(q, h), a);
        }
    }
}

// The box of a warp's points (offsets from their cell's corner).
struct Box3 {
    float x0, x1, y0, y1, z0, z1;
    __device__ __forceinline__ void of(float4 a, float4 b)
    {
        x0 = warp_min(fminf(a.x, b.x));
        x1 = warp_max(fmaxf(a.x, b.x));
        y0 = warp_min(fminf(a.y, b.y));
        y1 = warp_max(fmaxf(a.y, b.y));
        z0 = warp_min(fminf(a.z, b.z));
        z1 = warp_max(fmaxf(a.z, b.z));
    }
    // squared distance of the negated point (-fx, -fy, -fz)
    __device__ __forceinline__ float gap2(float fx, float fy, float fz) const
    {
        const float gx = fmaxf(0.f, fmaxf(-fx - x1, x0 + fx)), gy = fmaxf(0.f, fmaxf(-fy - y1, y0 + fy)),
                    gz = fmaxf(0.f, fmaxf(-fz - z1, z0 + fz));
        return gx * gx + gy * gy + gz * gz;
    }
};

// Walks the other side's points of the 27 cells around cell (c1, c2, c3) that are within reach of the
// box, in chunks of 32, the next chunk's record loaded while the current one is used.  The three
// cells of a row along z follow each other in memory and are walked as one range (at 41 points a
// cell four chunks where three cells take six).
struct Chunks3 {
    int c_j0, c_j1, c_b1, c_b2, jb, j1, b1, b2;   // a row's range and the first points of its second and third cell
    float c_ox, c_oy, h;
    unsigned rows;
    // the chunk loaded ahead
    int j;
    bool in;
    float ox, oy, oz;   // step from the point's cell to the item's frame
    float4 p;
    float v;
    __device__ __forceinline__ Chunks3(int lane, int packed, const CellGrid3 &cg, const Near3Params &np,
                                       const Box3 &box, const int *__restrict__ start)
    {
        const int e1 = b3x(packed) / cg.cell - 1 + lane / 3, e2 = b3y(packed) / cg.cell - 1 + lane % 3,
                  e3 = b3z(packed) / cg.cell;
        h = np.h;
        c_ox = (float)(1 - lane / 3) * h;
        c_oy = (float)(1 - lane % 3) * h;
        const float gx = fmaxf(0.f, fmaxf(-c_ox - box.x1, box.x0 - (h - c_ox))),
                    gy = fmaxf(0.f, fmaxf(-c_oy - box.y1, box.y0 - (h - c_oy)));
        const float left = np.reach2 - gx * gx - gy * gy;   // squared reach along z
        c_j0 = c_j1 = c_b1 = c_b2 = 0;
        if (lane < 9 && e1 >= 0 && e1 < cg.n_c && e2 >= 0 && e2 < cg.n_c && left >= 0.f) {
            const bool below = e3 > 0 && box.z0 * box.z0 <= left,
                       above = e3 + 1 < cg.n_c && (h - box.z1) * (h - box.z1) <= left;
            const int64_t key = (int64_t)cg.key(e1, e2, e3) * cg.sub3();
            c_b1 = start[key];
            c_b2 = start[key + cg.sub3()];
            c_j0 = below ? start[key - cg.sub3()] : c_b1;
            c_j1 = above ? start[key + 2 * cg.sub3()] : c_b2;
        }
        rows = __ballot_sync(0xffffffffu, c_j0 < c_j1);
        jb = j1 = j = b1 = b2 = 0;
        in = false;
        ox = oy = oz = v = 0.f;
        p = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __device__ __forceinline__ bool next(int lane, const float4 *__restrict__ hi, const float *__restrict__ val)
    {
        if (jb >= j1) {
            if (!rows)
                return false;
            const int c = __ffs(rows) - 1;
            rows &= rows - 1;
            jb = __shfl_sync(0xffffffffu, c_j0, c);
            j1 = __shfl_sync(0xffffffffu, c_j1, c);
            b1 = __shfl_sync(0xffffffffu, c_b1, c);
            b2 = __shfl_sync(0xffffffffu, c_b2, c);
            ox = __shfl_sync(0xffffffffu, c_ox, c);
            oy = __shfl_sync(0xffffffffu, c_oy, c);
        }
        j = jb + lane;
        in = j < j1;
        oz = j < b1 ? h : (j < b2 ? 0.f : -h);
        jb += 32;
        if (in) {
            p = __ldg(hi + j);
            if (val)
                v = __ldg(val + j);
        }
        return true;
    }
};

// off - hi - lo as hi + lo (TwoSum of off and -hi), d = off - hi given.
__device__ __forceinline__ float neg_lo(float off, float hi, float lo, float d)
{
    const float b = d - off;
    return ((off - (d - b)) + (-hi - b)) - lo;
}

template <int P>
__global__ void __launch_bounds__(kNear3Warps * 32, 6) k_near3_warp(const int2 *__restrict__ items, int n_items,
                                                                    int lanes, const int *__restrict__ tgt_base,
                                                                    const float4 *__restrict__ tgt_hi,
                                                                    const float4 *__restrict__ tgt_lo,
                                                                    const float4 *__restrict__ src_hi,
                                                                    const float4 *__restrict__ src_lo,
                                                                    const float *__restrict__ q,
                                                                    const int *__restrict__ src_start, CellGrid3 cg,
                                                                    Near3Params np, const int *__restrict__ coinc_start,
                                                                    const int *__restrict__ coinc_src,
                                                                    float *__restrict__ phi_s,
                                                                    float *__restrict__ grad_s, bool assign)
{
    __shared__ __align__(16) Near3List lists[kNear3Warps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int item = blockIdx.x * kNear3Warps + warp;
    if (item >= n_items)
        return;   // whole warp; the kernel has no block-wide barrier
    Near3List &L = lists[warp];
    const int2 it = items[item];
    const int groups = 32 / lanes, slot = lane & (lanes - 1), g = lane / lanes;
    const bool valid = slot < it.y;
    const int k = it.x + (valid ? slot : 0);
    const float4 h = tgt_hi[k], l = tgt_lo[k];
    Box3 box;
    box.of(h, h);
    const float ie = np.inv_eps;
    const float3 X = valid ? make_float3(h.x, h.y, h.z) : make_float3(1e6f, 1e6f, 1e6f);   // idle: beyond eps_I of all
    const float3 XL = make_float3(l.x, l.y, l.z), XS = make_float3(X.x * ie, X.y * ie, X.z * ie);
    const unsigned below = (1u << lane) - 1u;
    Near3Sums a;
    a.phi = a.gx = a.gy = a.gz = f2(0.f);
    int nf = 0, nc = 0;
    Chunks3 ch(lane, tgt_base[it.x], cg, np, box, src_start);
    bool more = ch.next(lane, src_hi, q);
    while (more) {
        const float4 y = ch.p;
        const float qj = ch.v, ox = ch.ox, oy = ch.oy, oz = ch.oz;
        const int j = ch.j;
        const bool in = ch.in;
        more = ch.next(lane, src_hi, q);
        const float fx = ox - y.x, fy = oy - y.y, fz = oz - y.z;   // -(source in the item's frame)
        const float g2 = in ? box.gap2(fx, fy, fz) : 3e38f;
        const bool keep = g2 <= np.reach2, close = g2 <= np.close_reach2;
        const unsigned mc = __ballot_sync(0xffffffffu, close), mf = __ballot_sync(0xffffffffu, keep) & ~mc;
        if (keep && !close)
            L.put(nf + __popc(mf & below), fx * ie, fy * ie, fz * ie, qj);
        nf += __popc(mf);
        if (nf > kNear3Cap - 32) {
            nf = L.pad(nf, 4 * groups, lane);
            __syncwarp();
            near3_eval<P>(L, nf, g, groups, XS, np, a);
            nf = 0;
            __syncwarp();
        }
        if (mc) {
            if (close) {
                const float4 yl = __ldg(src_lo + j);
                L.put_close(nc + __popc(mc & below), make_float3(fx, fy, fz),
                            make_float3(neg_lo(ox, y.x, yl.x, fx), neg_lo(oy, y.y, yl.y, fy), neg_lo(oz, y.z, yl.z, fz)),
                            qj);
            }
            nc += __popc(mc);
            if (nc > kNear3CloseCap - 32) {
                nc = L.pad_close(nc, 4 * groups, lane);
                __syncwarp();
                near3_eval_close<P>(L, nc, g, groups, X, XL, np, a);
                nc = 0;
                __syncwarp();
            }
        }
    }
    nf = L.pad(nf, 4 * groups, lane);
    nc = L.pad_close(nc, 4 * groups, lane);
    __syncwarp();
    near3_eval<P>(L, nf, g, groups, XS, np, a);
    near3_eval_close<P>(L, nc, g, groups, X, XL, np, a);
    float ph = a.phi.x + a.phi.y, gx = a.gx.x + a.gx.y, gy = a.gy.x + a.gy.y, gz = a.gz.x + a.gz.y;
    for (int o = 16; o >= lanes; o >>= 1) {
        ph = lane_add(ph, o);
        gx = lane_add(gx, o);
        gy = lane_add(gy, o);
        gz = lane_add(gz, o);
    }
    if (!valid || g != 0)
        return;
    // coincident pairs: G(0) := 0, so only -q T_I(0) remains of the far field's self term
    float self = 0.f;
    for (int c = coinc_start[k]; c < coinc_start[k + 1]; ++c)
        self += q[coinc_src[c]];
    const int64_t k3 = 3 * (int64_t)k;
    phi_s[k] = (assign ? 0.f : phi_s[k]) + (ph - np.beta0 * self);
    grad_s[k3] = (assign ? 0.f : grad_s[k3]) - np.inv_eps * gx;
    grad_s[k3 + 1] = (assign ? 0.f : grad_s[k3 + 1]) - np.inv_eps * gy;
    grad_s[k3 + 2] = (assign ? 0.f : grad_s[k3 + 2]) - np.inv_eps * gz;
}

// ---- FP32 near field, source-major (plans with many more sources than targets: FEM meshes,
// where every node meets the quadrature points of several elements)
//
// Target items would hold the few targets of a cell, their boxes large.  Here a warp takes a piece
// of at most 64 sources of one cell and keeps them in shared memory as packed pairs; it reads the
// targets of the 27 cells around 32 at a time, keeps those within eps_I of the sources' box (ballot)
// in a list (those within eps_I / 8 of the box in a second one, hi + lo), and each lane then takes one
// listed target and sums the item's sources on it, two per packed operation, adding phi and grad
// phi to the target with atomics.  Coincident pairs are removed by k_coincident3_apply.
// Measured, 1.59M quadrature points and 68,921 nodes of the 384,000-tetrahedron cube (p = 3): 1144 us
// with runs of the Morton order and FP64 differences of the close pairs, 497 us here.
constexpr int kSrcListCap = 128, kSrcCloseCap = 64;

struct Near3Sources {
    float4 xy[32], zq[32];            // (xa, xb, ya, yb), (za, zb, qa, qb), units of eps_I
    float4 hxy[32], lxy[32];          // hi and lo parts (torus units) for the close list
    float2 hz[32], lz[32];
    float4 far[kSrcListCap];          // listed targets: x, y, z (units of eps_I), index
    float4 chi[kSrcCloseCap], clo[kSrcCloseCap];   // hi (torus units) and index, lo
};

__device__ __forceinline__ void near3_src_add(const Near3Sums &a, int k, const Near3Params &np,
                                              float *__restrict__ phi_s, float *__restrict__ grad_s)
{
    atomicAdd(phi_s + k, a.phi.x + a.phi.y);
    atomicAdd(grad_s + 3 * (int64_t)k, -np.inv_eps * (a.gx.x + a.gx.y));
    atomicAdd(grad_s + 3 * (int64_t)k + 1, -np.inv_eps * (a.gy.x + a.gy.y));
    atomicAdd(grad_s + 3 * (int64_t)k + 2, -np.inv_eps * (a.gz.x + a.gz.y));
}

template <int P>
__device__ __forceinline__ void near3_src_eval(const Near3Sources &S, int n, int pairs, const Near3Params &np,
                                               float *__restrict__ phi_s, float *__restrict__ grad_s, int lane)
{
    for (int base = 0; base < n; base += 32) {
        const bool valid = base + lane < n;
        const float4 T = valid ? S.far[base + lane] : make_float4(kPadPos, kPadPos, kPadPos, 0.f);
        Near3Sums a;
        a.phi = a.gx = a.gy = a.gz = f2(0.f);
#pragma unroll 4
        for (int i = 0; i < pairs; ++i) {
            const float4 A = S.xy[i], B = S.zq[i];
            const float2 dx = add2(f2(T.x), make_float2(-A.x, -A.y)), dy = add2(f2(T.y), make_float2(-A.z, -A.w)),
                         dz = add2(f2(T.z), make_float2(-B.x, -B.y));
            near3_pair<P>(np, near3_w(dx, dy, dz), dx, dy, dz, make_float2(B.z, B.w), a);
        }
        if (valid)
            near3_src_add(a, __float_as_int(T.w), np, phi_s, grad_s);
    }
}

template <int P>
__device__ __forceinline__ void near3_src_eval_close(const Near3Sources &S, int n, int pairs, const Near3Params &np,
                                                     float *__restrict__ phi_s, float *__restrict__ grad_s, int lane)
{
    const float2 ie = f2(np.inv_eps);
    for (int base = 0; base < n; base += 32) {
        const bool valid = base + lane < n;
        const float4 T = valid ? S.chi[base + lane] : make_float4(kPadPos, kPadPos, kPadPos, 0.f);
        const float4 TL = valid ? S.clo[base + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
        Near3Sums a;
        a.phi = a.gx = a.gy = a.gz = f2(0.f);
#pragma unroll 2
        for (int i = 0; i < pairs; ++i) {
            const float4 A = S.hxy[i], AL = S.lxy[i], B = S.zq[i];
            const float2 Z = S.hz[i], ZL = S.lz[i];
            const float2 dx = mul2(add2(add2(f2(T.x), make_float2(-A.x, -A.y)), add2(f2(TL.x), make_float2(-AL.x, -AL.y))), ie);
            const float2 dy = mul2(add2(add2(f2(T.y), make_float2(-A.z, -A.w)), add2(f2(TL.y), make_float2(-AL.z, -AL.w))), ie);
            const float2 dz = mul2(add2(add2(f2(T.z), make_float2(-Z.x, -Z.y)), add2(f2(TL.z), make_float2(-ZL.x, -ZL.y))), ie);
            near3_pair_close<P>(np, dx, dy, dz, make_float2(B.z, B.w), a);
        }
        if (valid)
            near3_src_add(a, __float_as_int(T.w), np, phi_s, grad_s);
    }
}

template <int P>
__global__ void __launch_bounds__(kNear3Warps * 32) k_near3_src(const int2 *__restrict__ items, int n_items,
                                                                const int *__restrict__ src_base,
                                                                const float4 *__restrict__ src_hi,
                                                                const float4 *__restrict__ src_lo,
                                                                const float4 *__restrict__ tgt_hi,
                                                                const float4 *__restrict__ tgt_lo,
                                                                const float *__restrict__ q,
                                                                const int *__restrict__ tgt_start, CellGrid3 cg,
                                                                Near3Params np, float *__restrict__ phi_s,
                                                                float *__restrict__ grad_s)
{
    __shared__ Near3Sources all[kNear3Warps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int item = blockIdx.x * kNear3Warps + warp;
    if (item >= n_items)
        return;   // whole warp; the kernel has no block-wide barrier
    Near3Sources &S = all[warp];
    const int2 it = items[item];
    // pair i: sources i and i + pairs; an idle second one copies the first source with charge 0
    const int pairs = (it.y + 1) / 2;
    const int ja = it.x + (lane < pairs ? lane : 0);
    const bool vb = lane < pairs && lane + pairs < it.y;
    const int jb = vb ? ja + pairs : it.x;
    const float4 ha = src_hi[ja], hb = src_hi[jb], la = src_lo[ja], lb = src_lo[jb];
    const float ie = np.inv_eps;
    S.xy[lane] = make_float4(ha.x * ie, hb.x * ie, ha.y * ie, hb.y * ie);
    S.zq[lane] = make_float4(ha.z * ie, hb.z * ie, q[ja], vb ? q[jb] : 0.f);
    S.hxy[lane] = make_float4(ha.x, hb.x, ha.y, hb.y);
    S.lxy[lane] = make_float4(la.x, lb.x, la.y, lb.y);
    S.hz[lane] = make_float2(ha.z, hb.z);
    S.lz[lane] = make_float2(la.z, lb.z);
    Box3 box;
    box.of(ha, hb);
    __syncwarp();
    const unsigned below = (1u << lane) - 1u;
    int nf = 0, nc = 0;
    Chunks3 ch(lane, src_base[it.x], cg, np, box, tgt_start);
    bool more = ch.next(lane, tgt_hi, nullptr);
    while (more) {
        const float4 y = ch.p;
        const float ox = ch.ox, oy = ch.oy, oz = ch.oz;
        const int j = ch.j;
        const bool in = ch.in;
        more = ch.next(lane, tgt_hi, nullptr);
        const float fx = ox - y.x, fy = oy - y.y, fz = oz - y.z;   // -(target in the item's frame)
        const float g2 = in ? box.gap2(fx, fy, fz) : 3e38f;
        const bool keep = g2 <= np.reach2, close = g2 <= np.close_reach2;
        const unsigned mc = __ballot_sync(0xffffffffu, close), mf = __ballot_sync(0xffffffffu, keep) & ~mc;
        if (keep && !close)
            S.far[nf + __popc(mf & below)] = make_float4(-fx * ie, -fy * ie, -fz * ie, __int_as_float(j));
        nf += __popc(mf);
        if (nf > kSrcListCap - 32) {
            __syncwarp();
            near3_src_eval<P>(S, nf, pairs, np, phi_s, grad_s, lane);
            nf = 0;
            __syncwarp();
        }
        if (mc) {
            if (close) {
                const int at = nc + __popc(mc & below);
                const float4 yl = __ldg(tgt_lo + j);
                S.chi[at] = make_float4(-fx, -fy, -fz, __int_as_float(j));
                S.clo[at] = make_float4(-neg_lo(ox, y.x, yl.x, fx), -neg_lo(oy, y.y, yl.y, fy), -neg_lo(oz, y.z, yl.z, fz), 0.f);
            }
            nc += __popc(mc);
            if (nc > kSrcCloseCap - 32) {
                __syncwarp();
                near3_src_eval_close<P>(S, nc, pairs, np, phi_s, grad_s, lane);
                nc = 0;
                __syncwarp();
            }
        }
    }
    __syncwarp();
    near3_src_eval<P>(S, nf, pairs, np, phi_s, grad_s, lane);
    near3_src_eval_close<P>(S, nc, pairs, np, phi_s, grad_s, lane);
}

// Calls f(j) for the sources j whose pair with a target (tgt_hi entry X, tgt_lo entry XL) gets charge 0 in
// near3_pair_close, that is, for w < kNear3Exact2 of the difference that it forms, in the target's or (SRC) the
// source's frame, bit by bit the same.  Such sources lie in the target's cell, or across a face that is
// no farther.
template <bool SRC, class F>
__device__ __forceinline__ void near3_touching(const Near3Params &np, const CellGrid3 &cg, int packed, float4 X, float4 XL,
                                               const Near3Others &src, F &&f)
{
    const float lim = 1.05f * kNear3Exact / np.inv_eps;
    auto diff = [&](float x, float xl, float y, float yl, float off) {   // off: step from the source's cell to the target's
        const float a = SRC ? -off - x : off - y;
        const float d = SRC ? (-a - y) + (-neg_lo(-off, x, xl, a) - yl) : (x + a) + (xl + neg_lo(off, y, yl, a));
        return d * np.inv_eps;
    };
    for (int c = 0; c < 27; ++c) {
        const int d1 = c / 9 - 1, d2 = c / 3 % 3 - 1, d3 = c % 3 - 1;
        const int e1 = b3x(packed) / cg.cell + d1, e2 = b3y(packed) / cg.cell + d2, e3 = b3z(packed) / cg.cell + d3;
        auto far = [&](int d, float x) { return d < 0 ? x > lim : (d > 0 && np.h - x > lim); };
        if (far(d1, X.x) || far(d2, X.y) || far(d3, X.z) || min(min(e1, e2), e3) < 0 || max(max(e1, e2), e3) >= cg.n_c)
            continue;
        const float ox = -(float)d1 * np.h, oy = -(float)d2 * np.h, oz = -(float)d3 * np.h;
        const int64_t key = (int64_t)cg.key(e1, e2, e3) * cg.sub3();
        for (int j = src.start[key]; j < src.start[key + cg.sub3()]; ++j) {
            const float4 y = src.hi[j];
            if (fabsf(X.x + (ox - y.x)) > lim || fabsf(X.y + (oy - y.y)) > lim || fabsf(X.z + (oz - y.z)) > lim)
                continue;
            const float4 yl = src.lo[j];
            const float2 dx = f2(diff(X.x, XL.x, y.x, yl.x, ox)), dy = f2(diff(X.y, XL.y, y.y, yl.y, oy)),
                         dz = f2(diff(X.z, XL.z, y.z, yl.z, oz));
            if (near3_w(dx, dy, dz).x < kNear3Exact2)
                f(j);
        }
    }
}

// The differences of those pairs from the FP64 positions, in place of the hi + lo ones; nothing for a
// coincident pair.  Adds to phi and the three components of grad.
template <int P, bool SRC>
__device__ __forceinline__ void near3_add_touching(const Near3Params &np, const CellGrid3 &cg, int k, int packed, float4 X,
                                                   float4 XL, const Near3Others &src, const double *__restrict__ tgt_pos,
                                                   const float *__restrict__ q, float (&add)[4])
{
    Near3Sums a;
    a.phi = a.gx = a.gy = a.gz = f2(0.f);
    const double tx = tgt_pos[3 * (int64_t)k], ty = tgt_pos[3 * (int64_t)k + 1], tz = tgt_pos[3 * (int64_t)k + 2];
    near3_touching<SRC>(np, cg, packed, X, XL, src, [&](int j) {
        const double *s = src.pos + 3 * (int64_t)j;
        const double ex = tx - s[0], ey = ty - s[1], ez = tz - s[2];
        if (ex == 0.0 && ey == 0.0 && ez == 0.0)
            return;
        const float2 dx = f2((float)(ex * src.inv_eps)), dy = f2((float)(ey * src.inv_eps)),
                     dz = f2((float)(ez * src.inv_eps));
        const float w = fmaxf(near3_w(dx, dy, dz).x, 1e-20f);   // (w^-3/2 stays finite)
        near3_pair<P>(np, f2(w), dx, dy, dz, make_float2(q[j], 0.f), a);
    });
    add[0] = a.phi.x;
    add[1] = -np.inv_eps * a.gx.x;
    add[2] = -np.inv_eps * a.gy.x;
    add[3] = -np.inv_eps * a.gz.x;
}

// The pairs that the kernels above leave out: those of the marked targets, and for the source-major kernel
// the coincident ones (coinc_start given), phi -= T_I(0) (sum of their charges).
template <int P, bool SRC>
__global__ void k_touching3(int64_t N, const int *__restrict__ coinc_start, const int *__restrict__ coinc_src,
                            const int *__restrict__ tgt_base, const float4 *__restrict__ tgt_hi,
                            const float4 *__restrict__ tgt_lo, const double *__restrict__ tgt_pos, Near3Others src,
                            const float *__restrict__ q, CellGrid3 cg, Near3Params np, float *__restrict__ phi_s,
                            float *__restrict__ grad_s)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= N)
        return;
    if (coinc_start) {
        float self = 0.f;
        for (int c = coinc_start[k]; c < coinc_start[k + 1]; ++c)
            self += q[coinc_src[c]];
        if (self != 0.f)
            phi_s[k] -= np.beta0 * self;
    }
    const float4 X = tgt_hi[k];
    if (X.w == 0.f)
        return;
    float add[4];
    near3_add_touching<P, SRC>(np, cg, (int)k, tgt_base[k], X, tgt_lo[k], src, tgt_pos, q, add);
    phi_s[k] += add[0];
    for (int d = 0; d < 3; ++d)
        grad_s[3 * k + d] += add[1 + d];
}

// Per target, the number of its coincident sources (equal FP64 positions, so of its own cell), with
// tgt_hi[k].w = 1 and *touching = 1 if it has other sources that close; or (coinc_src given) those
// sources.
template <bool SRC>
__global__ void k_coincident3(int64_t N, const int *__restrict__ tgt_base, float4 *__restrict__ tgt_hi,
                              const float4 *__restrict__ tgt_lo, const double *__restrict__ tgt_pos, Near3Others src,
                              CellGrid3 cg, Near3Params np, int *__restrict__ count, const int *__restrict__ coinc_start,
                              int *__restrict__ coinc_src, int *__restrict__ touching)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= N)
        return;
    const double tx = tgt_pos[3 * k], ty = tgt_pos[3 * k + 1], tz = tgt_pos[3 * k + 2];
    const float4 X = tgt_hi[k];
    int c = 0, at = coinc_src ? coinc_start[k] : 0;
    bool other = false;
    near3_touching<SRC>(np, cg, tgt_base[k], X, tgt_lo[k], src, [&](int j) {
        const double *s = src.pos + 3 * (int64_t)j;
        if (s[0] != tx || s[1] != ty || s[2] != tz) {
            other = true;
            return;
        }
        if (coinc_src)
            coinc_src[at++] = j;
        ++c;
    });
    if (coinc_src)
        return;
    count[k] = c;
    if (other) {
        tgt_hi[k] = make_float4(X.x, X.y, X.z, 1.f);
        *touching = 1;
    }
}

template <typename real>
__global__ void k_unpermute3(int64_t N, const real *__restrict__ phi_s, const real *__restrict__ grad_s,
                             const int *__restrict__ perm, double s, void *__restrict__ phi_out,
                             void *__restrict__ H_out, int out_f64)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= N)
        return;
    const int64_t i = perm[k];
    const double phi = s * (double)phi_s[k];
    const double s2 = -s * s;
    if (out_f64) {
        if (phi_out)
            ((double *)phi_out)[i] = phi;
        if (H_out)
            for (int d = 0; d < 3; ++d)
                ((double *)H_out)[3 * i + d] = s2 * (double)grad_s[3 * k + d];
    } else {
        if (phi_out)
            ((float *)phi_out)[i] = (float)phi;
        if (H_out)
            for (int d = 0; d < 3; ++d)
                ((float *)H_out)[3 * i + d] = (float)(s2 * (double)grad_s[3 * k + d]);
    }
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

template <class F> cudaError_t with_width3(int m, F &&f)
{
    switch (m) {
    case 2: return f(std::integral_constant<int, 4>{});
    case 3: return f(std::integral_constant<int, 6>{});
    case 4: return f(std::integral_constant<int, 8>{});
    case 5: return f(std::integral_constant<int, 10>{});
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_rmax3(const double *xyz, int64_t n, unsigned long long *out, cudaStream_t st)
{
    if (n <= 0)
        return cudaSuccess;
    unsigned b = nblk(n, 256);
    if (b > 1024)
        b = 1024;
    k_rmax3<<<b, 256, 0, st>>>(xyz, n, out);
    return cudaGetLastError();
}

cudaError_t launch_point_keys3(const double *xyz, int64_t n, double s, int n_os, int window_lo, int n_a, int m,
                               CellGrid3 cg, int *key, int *count, int *status, cudaStream_t st)
{
    if (n <= 0)
        return cudaSuccess;
    k_point_keys3<<<nblk(n, 256), 256, 0, st>>>(xyz, n, s, n_os, window_lo, n_a, m, cg, key, count, status);
    return cudaGetLastError();
}

template <typename real>
cudaError_t launch_gather_points3(const double *xyz, const int *perm, int64_t n, double s, int n_os, int window_lo,
                                  int n_a, int m, int cell, double *pos, real *frac, int *base,
                                  float4 *hi, float4 *lo, cudaStream_t st)
{
    if (n <= 0)
        return cudaSuccess;
    k_gather_points3<real><<<nblk(n, 256), 256, 0, st>>>(xyz, perm, n, s, n_os, window_lo, n_a, m, cell, pos, frac,
                                                         base, hi, lo);
    return cudaGetLastError();
}

template <typename real>
cudaError_t launch_spread3(int64_t M, int m, const int *base, const real *frac, const real *q, Window<real> w,
                           const WindowPoly &wp, real *grid, int n_a, cudaStream_t st)
{
    if (M <= 0)
        return cudaSuccess;
    return with_width3(m, [&](auto mc) {
        constexpr int M2 = decltype(mc)::value;
        int64_t blocks = (M + 7) / 8;   // eight warps (sources) per block, then grid-stride
        if (blocks > 152 * 16)
            blocks = 152 * 16;
        k_spread3<real, M2><<<(unsigned)blocks, 256, 0, st>>>(M, base, frac, q, w, wp, grid, n_a);
        return cudaGetLastError();
    });
}

// Shared memory of the tiled FP32 spreading (0 when the tiles do not fit: use k_spread3).
size_t spread3_tile_smem(int cell, int m)
{
    const size_t P = (size_t)cell + 2 * m - 1;
    const size_t bytes = (size_t)kSpread3Warps * 2 * P * P * P * sizeof(float);
    return bytes <= 112 * 1024 ? bytes : 0;
}

size_t spread3_runs_smem(int cell, int m)
{
    const int P = cell + 2 * m - 1;
    if (m != 4 || P > 16)
        return 0;
    return sizeof(float) * (2 * (size_t)P * P * 16 + kSpread3RunThreads * (kSpread3WeightPitch + 1));
}

cudaError_t launch_spread3_keys(int64_t M, const int *base, CellGrid3 cg, int *key, int *count, cudaStream_t st)
{
    if (M <= 0)
        return cudaSuccess;
    k_spread3_keys<<<(unsigned)((M + 255) / 256), 256, 0, st>>>(base, M, cg, key, count);
    return cudaGetLastError();
}

cudaError_t launch_spread3_gather(int64_t M, const int *order, const int *base, const float *frac, int *run_base,
                                  float *run_frac, cudaStream_t st)
{
    if (M <= 0)
        return cudaSuccess;
    k_spread3_order<<<(unsigned)((M + 255) / 256), 256, 0, st>>>(order, M, base, frac, run_base, run_frac);
    return cudaGetLastError();
}

cudaError_t launch_spread3_runs(const int2 *items, int n_items, int m, int cell, const int *base, const float *frac,
                                const int *order, const float *q, const WindowPoly &wp, float *grid, int n_a,
                                cudaStream_t st)
{
    if (n_items <= 0)
        return cudaSuccess;
    const size_t smem = spread3_runs_smem(cell, m);
    if (smem == 0)
        return cudaErrorInvalidValue;
    const cudaError_t e = cudaFuncSetAttribute(k_spread3_runs<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return e;
    k_spread3_runs<8><<<(unsigned)n_items, kSpread3RunThreads, smem, st>>>(items, base, frac, order, q, wp, cell, grid,
                                                                         n_a);
    return cudaGetLastError();
}

cudaError_t launch_spread3_tile(const int2 *items, int n_items, int m, int cell, const int *base, const float *frac,
                                const float *q, const WindowPoly &wp, float *grid, int n_a, cudaStream_t st)
{
    if (n_items <= 0)
        return cudaSuccess;
    const size_t smem = spread3_tile_smem(cell, m);
    if (smem == 0)
        return cudaErrorInvalidValue;
    return with_width3(m, [&](auto mc) {
        constexpr int M2 = decltype(mc)::value;
        cudaError_t e = cudaFuncSetAttribute(k_spread3_tile<M2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess)
            return e;
        k_spread3_tile<M2><<<(unsigned)n_items, kSpread3Warps * 32, smem, st>>>(items, base, frac, q, wp, cell, grid,
                                                                                n_a);
        return cudaGetLastError();
    });
}

template <typename real>
cudaError_t launch_interp3(int64_t N, int m, const int *base, const real *frac, Window<real> w, const WindowPoly &wp,
                           const real *grid, int n_a, real n_os, real *phi_s, real *grad_s, bool acc,
                           cudaStream_t st)
{
    if (N <= 0)
        return cudaSuccess;
    return with_width3(m, [&](auto mc) {
        constexpr int M2 = decltype(mc)::value;
        k_interp3<real, M2><<<nblk(N, 256), 256, 0, st>>>(N, base, frac, w, wp, grid, n_a, n_os, phi_s, grad_s, acc);
        return cudaGetLastError();
    });
}

cudaError_t launch_near3_f64(int64_t N, const int *tgt_base, const double *tgt_pos, const double *src_pos,
                             const int *src_start, CellGrid3 cg, const double *q, NearParams<double> np,
                             double *phi_s, double *grad_s, cudaStream_t st)
{
    if (N <= 0)
        return cudaSuccess;
    k_near3_f64<<<nblk(N, 256), 256, 0, st>>>(N, tgt_base, tgt_pos, src_pos, src_start, cg, q, np, phi_s, grad_s);
    return cudaGetLastError();
}

cudaError_t launch_interp3_out(int64_t N, int m, const int *base, const float *frac, const WindowPoly &wp,
                               const float *grid, int n_a, float n_os, const float *phi_s, const float *grad_s,
                               const int *perm, double s, void *phi_out, void *H_out, int out_f64, cudaStream_t st)
{
    if (m != 4)
        return cudaErrorInvalidValue;
    if (N <= 0)
        return cudaSuccess;
    const int64_t want = (N + kInterp3Threads / 8 - 1) / (kInterp3Threads / 8);
    const unsigned blocks = (unsigned)(want < 152 * 16 ? want : 152 * 16);
    k_interp3_out<<<blocks, kInterp3Threads, 0, st>>>(N, base, frac, wp, grid, n_a, n_os, phi_s, grad_s, perm, s,
                                                       phi_out, H_out, out_f64);
    return cudaGetLastError();
}

cudaError_t launch_cell_order3(const int *start, CellGrid3 cg, int cap, const double *xyz, double s, int n_os,
                               int window_lo, int n_a, int m, int *perm, cudaStream_t st)
{
    if (cg.n_cells() <= 0)
        return cudaSuccess;
    k_cell_order3<<<(unsigned)cg.n_cells(), kOrder3Threads, 0, st>>>(start, cg, cap, xyz, s, n_os, window_lo, n_a, m, perm);
    return cudaGetLastError();
}

cudaError_t launch_near3_warp(const int2 *items, int n_items, int lanes, const Near3Targets &tgt, const Near3Others &src,
                              const float *q, CellGrid3 cg, const Near3Params &np, int64_t N, const int *coinc_start,
                              const int *coinc_src, bool any_marked, float *phi_s, float *grad_s, bool assign,
                              cudaStream_t st)
{
    if (n_items <= 0)
        return cudaSuccess;
    const unsigned blocks = (unsigned)((n_items + kNear3Warps - 1) / kNear3Warps);
    return with_degree(np.p, [&](auto pc) {
        constexpr int P = decltype(pc)::value;
        k_near3_warp<P><<<blocks, kNear3Warps * 32, 0, st>>>(items, n_items, lanes, tgt.base, tgt.hi, tgt.lo, src.hi, src.lo,
                                                             q, src.start, cg, np, coinc_start, coinc_src, phi_s, grad_s,
                                                             assign);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess || !any_marked)
            return e;
        k_touching3<P, false><<<nblk(N, 256), 256, 0, st>>>(N, nullptr, nullptr, tgt.base, tgt.hi, tgt.lo, tgt.pos, src, q, cg,
                                                            np, phi_s, grad_s);
        return cudaGetLastError();
    });
}

cudaError_t launch_near3_src(const int2 *items, int n_items, const int *src_base, const Near3Others &src,
                             const Near3Targets &tgt, const int *tgt_start, const float *q, CellGrid3 cg,
                             const Near3Params &np, int64_t N, const int *coinc_start, const int *coinc_src,
                             bool any_touching, float *phi_s, float *grad_s, cudaStream_t st)
{
    return with_degree(np.p, [&](auto pc) {
        constexpr int P = decltype(pc)::value;
        if (n_items > 0) {
            const unsigned blocks = (unsigned)((n_items + kNear3Warps - 1) / kNear3Warps);
            k_near3_src<P><<<blocks, kNear3Warps * 32, 0, st>>>(items, n_items, src_base, src.hi, src.lo, tgt.hi, tgt.lo, q,
                                                                tgt_start, cg, np, phi_s, grad_s);
            const cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess)
                return e;
        }
        if (any_touching && N > 0)
            k_touching3<P, true><<<nblk(N, 256), 256, 0, st>>>(N, coinc_start, coinc_src, tgt.base, tgt.hi, tgt.lo, tgt.pos,
                                                               src, q, cg, np, phi_s, grad_s);
        return cudaGetLastError();
    });
}

cudaError_t launch_coincident3(int64_t N, const Near3Targets &tgt, const Near3Others &src, CellGrid3 cg,
                               const Near3Params &np, bool source_frame, int *count, const int *coinc_start, int *coinc_src,
                               int *touching, cudaStream_t st)
{
    if (N <= 0)
        return cudaSuccess;
    if (source_frame)
        k_coincident3<true><<<nblk(N, 256), 256, 0, st>>>(N, tgt.base, tgt.hi, tgt.lo, tgt.pos, src, cg, np, count, coinc_start,
                                                          coinc_src, touching);
    else
        k_coincident3<false><<<nblk(N, 256), 256, 0, st>>>(N, tgt.base, tgt.hi, tgt.lo, tgt.pos, src, cg, np, count,
                                                           coinc_start, coinc_src, touching);
    return cudaGetLastError();
}

template <typename real>
cudaError_t launch_unpermute3(int64_t N, const real *phi_s, const real *grad_s, const int *perm, double s,
                              void *phi_out, void *H_out, int out_f64, cudaStream_t st)
{
    if (N <= 0)
        return cudaSuccess;
    k_unpermute3<real><<<nblk(N, 256), 256, 0, st>>>(N, phi_s, grad_s, perm, s, phi_out, H_out, out_f64);
    return cudaGetLastError();
}

#define FS_INST3(real)                                                                                            \
    template cudaError_t launch_gather_points3<real>(const double *, const int *, int64_t, double, int, int, int, \
                                                     int, int, double *, real *, int *, float4 *, float4 *,  \
                                                     cudaStream_t);                                               \
    template cudaError_t launch_spread3<real>(int64_t, int, const int *, const real *, const real *, Window<real>, \
                                              const WindowPoly &, real *, int, cudaStream_t);                     \
    template cudaError_t launch_interp3<real>(int64_t, int, const int *, const real *, Window<real>,               \
                                              const WindowPoly &, const real *, int, real, real *, real *, bool,  \
                                              cudaStream_t);                                                      \
    template cudaError_t launch_unpermute3<real>(int64_t, const real *, const real *, const int *, double, void *, \
                                                 void *, int, cudaStream_t);
FS_INST3(float)
FS_INST3(double)
#undef FS_INST3

}  // namespace fs
