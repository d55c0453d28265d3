// FP64 near field of the 2D path: warp-per-point traversal, shared by the forward correction, the
// adjoint potential and the Hessian.
//
// GB300 issues two FP64 operations per SM and cycle, a 64th of the FP32 rate, so the time is the
// number of FP64 warp instructions (16 cycles each) and nothing else.  A warp takes one own point;
// its lanes test the other points of the 3 x 3 cells in FP32 (the cell-relative positions, with a
// margin for their rounding), queue those within reach in shared memory (ballot), and evaluate 32 of
// them at a time in FP64, every lane a pair: a pair within eps_I costs its own arithmetic and
// nothing of its neighbours', where a thread per point diverged (0.4 of the lanes useful) and ran
// CUDA's log and divide.  With w = r^2 / eps_I^2 and s = 1 - w a pair takes 20 + 2 p instructions:
//   log: table of 129 reciprocals c_i of the mantissa with -log c_i, and a degree-6 series in
//        r = m c_i - 1, |r| <= 2^-8 (P. T. P. Tang, Table-driven implementation of the logarithm
//        function, ACM TOMS 16, 1990); the exponent's multiple of ln 2 from a second table;
//   1/w: the 20-bit hardware approximation y and one third-order step y (1 + e + e^2), e = 1 - w y;
//   T_I: the two polynomials Ptilde and P' of the far field's own coefficients.
// Measured (32,768 points, n = 256, 10.0e6 pairs within eps_I, p = 6): 3.03 ms with a thread per
// target, 0.67 ms here; the FP64 pipe's bound for the pairs is 0.53 ms.
#pragma once

#include "near_warp.cuh"

namespace fs {

struct Near64Tables {
    double2 log[kLogTab];
    double ln2[kLogExp];
    // the whole block; ends with a barrier
    __device__ __forceinline__ void load(const double *__restrict__ t)
    {
        for (int i = threadIdx.x; i < kLogTab; i += blockDim.x)
            log[i] = make_double2(t[2 * i], t[2 * i + 1]);
        for (int i = threadIdx.x; i < kLogExp; i += blockDim.x)
            ln2[i] = t[2 * kLogTab + i];
        __syncthreads();
    }
    // log of w in (0, 1]; exactly 0 at 1.  The table of the exponent's multiples ends at 2^-127, a pair
    // 7.7e-20 eps_I apart (such pairs are found near the origin alone, where doubles are that fine): below
    // it CUDA's log, on a branch that ordinary warps do not take.
    __device__ __forceinline__ double ln(double w) const
    {
        const int hi = __double2hiint(w);
        if (hi < (1024 - kLogExp) << 20)
            return ::log(w);
        const double2 c = log[((hi & 0xfffff) + 0x1000) >> 13];
        const double r = fma(__hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(w)), c.x, -1.0);
        double t = fma(r, -1.0 / 6.0, 1.0 / 5.0);
        t = fma(r, t, -1.0 / 4.0);
        t = fma(r, t, 1.0 / 3.0);
        t = fma(r, t, -1.0 / 2.0);
        return (ln2[1023 - (hi >> 20)] + c.y) + fma(r * r, t, r);
    }
};

__device__ __forceinline__ double near64_rcp(double w)
{
    if (__double2hiint(w) < 0x00100000)
        return 1.0 / w;   // subnormal: the approximation would flush it
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(w));
    const double e = fma(-w, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// The functions of a pair at w in (0, 1], s = 1 - w, y = 1 / w (P = T_I - k(eps_I)), from the far field's
// own coefficients (near64_params):
//   4 pi f            = s (4 pi Ptilde(w)) - ln w            (f = G - T_I)
//   -2 pi eps_I^2 c   = y + 4 pi P'(w)                       (c = f'(r) / r)
//   2 pi eps_I^2 c'   = y^2 - 4 pi P''(w)                    (c' = dc / dw)
template <int P> __device__ __forceinline__ double near64_horner(const double *c, int n, double w)
{
    double t = n > 0 ? c[n - 1] : 0.0;
#pragma unroll
    for (int i = n - 2; i >= 0; --i)
        t = fma(t, w, c[i]);
    return t;
}

template <int P> __device__ __forceinline__ double near64_f(const Near64Params &np, const Near64Tables &tab, double w, double s)
{
    if constexpr (P == 1)
        return np.f[0] - tab.ln(w);
    else
        return fma(s, near64_horner<P>(np.f, P - 1, w), -tab.ln(w));
}
template <int P> __device__ __forceinline__ double near64_c(const Near64Params &np, double w, double y)
{
    return P == 1 ? y : y + near64_horner<P>(np.c, P - 1, w);
}
template <int P> __device__ __forceinline__ double near64_cp(const Near64Params &np, double w, double y)
{
    return P < 3 ? y * y : fma(y, y, -near64_horner<P>(np.cp, P - 2, w));
}

constexpr int kNear64Warps = 4;

// Sums v[0..3] over the warp; lane 8 i returns v[i]'s.  Six additions where four separate
// reductions take twenty.
__device__ __forceinline__ double near64_reduce4(const double *v, int lane)
{
    const bool hi = lane & 16, mid = lane & 8;
    const double a = (hi ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[2], 16);
    const double b = (hi ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, hi ? v[1] : v[3], 16);
    double r = (mid ? b : a) + __shfl_xor_sync(0xffffffffu, mid ? a : b, 8);
    for (int o = 4; o > 0; o >>= 1)
        r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}

// One own point k by one warp.  Op: kV (4 or 5) sums v[], init(), pair(np, tab, j, in, w, dx, dy) with
// d = own - other in torus units, in: 0 < w < 1 (else w = 1 is handed over and nothing may be added),
// coincident(np, j), store(np, k, i, sum) for sum i.
template <class Op>
__device__ __forceinline__ void near64_point(int64_t k, int lane, const Near64Sides &sd, const CellGrid &cg,
                                             const Near64Params &np, const Near64Tables &tab, Op &op, int *queue)
{
    const double2 X = sd.own_pos[k];
    const float2 xh = sd.own_hi[k];
    const int packed = sd.own_base[k], c1 = base1(packed) / cg.cell, c2 = base2(packed) / cg.cell;
    const unsigned below = (1u << lane) - 1u;
    // lane c < 9: cell c of the 3 x 3 around the point's, if it holds points and is within reach
    const float c_ox = (float)(1 - lane / 3) * np.h, c_oy = (float)(1 - lane % 3) * np.h;
    int c_j0 = 0, c_j1 = 0;
    {
        const int e1 = c1 - 1 + lane / 3, e2 = c2 - 1 + lane % 3;
        const float gx = fmaxf(0.f, fmaxf(-c_ox - xh.x, xh.x - (np.h - c_ox)));
        const float gy = fmaxf(0.f, fmaxf(-c_oy - xh.y, xh.y - (np.h - c_oy)));
        if (lane < 9 && e1 >= 0 && e1 < cg.n_c && e2 >= 0 && e2 < cg.n_c && gx * gx + gy * gy <= np.reach2) {
            const int key = cg.key(e1, e2) * kSub;
            c_j0 = sd.oth_start[key];
            c_j1 = sd.oth_start[key + kSub];
        }
    }
    unsigned cells = __ballot_sync(0xffffffffu, c_j0 < c_j1);
    op.init();
    int nq = 0;
    auto eval = [&](int first, int count) {
        __syncwarp();
        if (lane < count) {
            const int j = queue[first + lane];
            const double2 Y = sd.oth_pos[j];
            const double dx = X.x - Y.x, dy = X.y - Y.y;
            double w = fma(dy, dy, dx * dx) * np.inv_eps2;
            const int hi = __double2hiint(w);
            const bool zero = (hi | __double2loint(w)) == 0, in = hi < 0x3ff00000 && !zero;
            if (zero)
                op.coincident(np, j);
            w = in ? w : 1.0;
            op.pair(np, tab, j, in, w, dx, dy);
        }
        __syncwarp();
    };
    while (cells) {
        const int c = __ffs(cells) - 1;
        cells &= cells - 1;
        const int j1 = __shfl_sync(0xffffffffu, c_j1, c);
        const float px = xh.x + __shfl_sync(0xffffffffu, c_ox, c), py = xh.y + __shfl_sync(0xffffffffu, c_oy, c);
        for (int jb = __shfl_sync(0xffffffffu, c_j0, c); jb < j1; jb += 32) {
            const int j = jb + lane;
            bool keep = false;
            if (j < j1) {
                const float2 y = __ldg(sd.oth_hi + j);
                const float fx = px - y.x, fy = py - y.y;
                keep = fx * fx + fy * fy <= np.reach2;
            }
            const unsigned mk = __ballot_sync(0xffffffffu, keep);
            if (keep)
                queue[nq + __popc(mk & below)] = j;
            nq += __popc(mk);
            if (nq >= 32) {
                nq -= 32;
                eval(nq, 32);
            }
        }
    }
    eval(0, nq);
    const double r = near64_reduce4(op.v, lane);
    if ((lane & 7) == 0)
        op.store(np, k, lane >> 3, r);
    if constexpr (Op::kV == 5) {
        double t = op.v[4];
        for (int o = 16; o > 0; o >>= 1)
            t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0)
            op.store(np, k, 4, t);
    }
}

// Persistent: each warp takes every n-th point (points of a dense cell go to different warps).
template <class Op>
__global__ void __launch_bounds__(32 * kNear64Warps) k_near64(int64_t N, Near64Sides sd, CellGrid cg, Near64Params np, Op op)
{
    __shared__ Near64Tables tab;
    __shared__ int queue[kNear64Warps][64];
    tab.load(sd.tables);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t k = blockIdx.x * (int64_t)kNear64Warps + w; k < N; k += (int64_t)gridDim.x * kNear64Warps)
        near64_point(k, lane, sd, cg, np, tab, op, queue[w]);
}

template <class Op>
cudaError_t launch_near64_points(int64_t N, const Near64Sides &sd, CellGrid cg, const Near64Params &np, const Op &op,
                                 cudaStream_t st)
{
    if (N <= 0)
        return cudaSuccess;
    const int64_t blocks = (N + kNear64Warps - 1) / kNear64Warps;
    k_near64<Op><<<(unsigned)(blocks < 152 * 8 ? blocks : 152 * 8), 32 * kNear64Warps, 0, st>>>(N, sd, cg, np, op);
    return cudaGetLastError();
}

}  // namespace fs
