// Near-field correction (step g) and return to physical units.
//
// The far field uses the kernel smoothed inside eps_I ("the price to pay is an
// afterwards correction in the smoothing zone"): for every pair closer than
// eps_I it holds T_I(r) instead of G(r) = -(1/2 pi) log r, so
//     phi_i  += q_j (G(r) - T_I(r))                       0 < r < eps_I
//     grad_i += q_j (-(1/2 pi) / r^2 - T_I'(r)/r) d        d = x~_i - y~_j
//     phi_i  -= q_j T_I(0), coinc_i += q_j                  r = 0 (G(0) := 0)
// Cells are at least eps_I wide, so a target's partners lie in the 3 x 3 cells
// around its own.
//
// FP64 path: one warp per target (near64.cuh).
//
// FP32 path: one warp per work item, a compact piece of a cell of at most 32 targets (one per
// lane), over the sources near the item's bounding box (near_warp.cuh).
// The value and gradient use the cancellation-free forms of G - T_I and of its
// radial derivative over r, c (w - 1)^(p-1) / w with w = r^2 / eps_I^2.
//
// The output kernel adds the far and near fields and rescales:
//     phi = phi~ + (log s / 2 pi) (sum_j q_j - coinc_i),   H = -s grad~ phi,
// scattering back to the caller's target order.
#include <cmath>

#include "internal.h"
#include "output.cuh"
#include "near64.cuh"
#include "near_fwd.cuh"

namespace fs {

namespace {

// phi += q f, grad += q c d, and the coincident charge (4 pi f and -2 pi eps_I^2 c are summed).
template <int P> struct Near64Fwd {
    static constexpr int kV = 4;
    const double *__restrict__ q;
    double *__restrict__ phi_s;
    double *__restrict__ grad_s;
    double *__restrict__ coinc;
    double v[4];

    __device__ __forceinline__ void init() { v[0] = v[1] = v[2] = v[3] = 0.0; }
    __device__ __forceinline__ void coincident(const Near64Params &np, int j)
    {
        const double qj = q[j];
        v[0] -= qj * (4.0 * kPi * np.beta0);
        v[3] += qj;
    }
    __device__ __forceinline__ void pair(const Near64Params &np, const Near64Tables &tab, int j, bool in, double w, double dx,
                                         double dy)
    {
        const double qj = in ? q[j] : 0.0;
        v[0] = fma(qj, near64_f<P>(np, tab, w, 1.0 - w), v[0]);
        const double t = qj * near64_c<P>(np, w, near64_rcp(w));
        v[1] = fma(t, dx, v[1]);
        v[2] = fma(t, dy, v[2]);
    }
    __device__ __forceinline__ void store(const Near64Params &np, int64_t k, int i, double r) const
    {
        if (i == 0)
            phi_s[k] += r * (1.0 / (4.0 * kPi));
        else if (i == 3)
            coinc[k] = r;
        else
            grad_s[2 * k + i - 1] -= r * (np.inv_eps2 / (2.0 * kPi));
    }
};

// Batched FP64 near field: block -> (instance, block of its targets), blockIdx.y = right-hand side;
// the block's warps take its targets in turn.
template <int P>
__global__ void __launch_bounds__(32 * kNear64Warps) k_batch_near64(const BatchInst<double> *__restrict__ inst,
                                                                    BlockMap bm, const double *__restrict__ tables,
                                                                    int per_block)
{
    __shared__ Near64Tables tab;
    __shared__ int queue[kNear64Warps][64];
    __shared__ Near64Params np;
    tab.load(tables);
    const int i = bm.inst[blockIdx.x], r = blockIdx.y;
    const BatchInst<double> &b = inst[i];
    for (int t = threadIdx.x; t < (int)(sizeof(np) / sizeof(int)); t += blockDim.x)
        reinterpret_cast<int *>(&np)[t] = reinterpret_cast<const int *>(&b.np64)[t];
    __syncthreads();
    const Near64Sides sd{b.tgt_base, b.tgt_pos, b.tgt_hi, b.src_pos, b.src_hi, b.src_start, tables};
    const CellGrid cg = b.cg;
    const int64_t N = b.N, first = (int64_t)(blockIdx.x - bm.first[i]) * per_block;
    Near64Fwd<P> op{};
    op.q = b.q + (int64_t)r * b.M;
    op.phi_s = b.phi_s + (int64_t)r * N;
    op.grad_s = b.grad_s + 2 * (int64_t)r * N;
    op.coinc = b.coinc + (int64_t)r * N;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t k = first + w; k < first + per_block && k < N; k += kNear64Warps)
        near64_point(k, lane, sd, cg, np, tab, op, queue[w]);
}

// Plan-time statistics: pairs with r < eps_I and with r < eps_I / 8 (coincident pairs
// included), counted by the same traversal and the same FP32 differences as the field
// kernel.  Each lane adds its counts to one of kCountSlots counter pairs (summed on the host).
static_assert(kNearCountSlots == 64, "counter slots");
constexpr int kCountSlots = kNearCountSlots;
struct NearCount {
    static constexpr int kMinBlocks = 6;
    static constexpr int kUnroll = 1;
    static constexpr bool kSat = false;
    unsigned long long *__restrict__ counts;   // 2 * kCountSlots
    unsigned n_near, n_close;

    __device__ __forceinline__ void init() { n_near = n_close = 0; }
    static constexpr int kR = 1;   // candidate-list traversal: no values per other point
    __device__ __forceinline__ void fetch(int, float (&v)[1]) const { v[0] = 0.f; }
    __device__ __forceinline__ void set_q(const float2 (&)[1]) {}
    __device__ __forceinline__ void coincident(const NearParams<float> &, int)
    {
        ++n_near;
        ++n_close;
    }
    __device__ __forceinline__ void pair2(const NearParams<float> &np, float2 w, float2, float2)
    {
        n_near += (w.x < np.eps2 ? 1u : 0u) + (w.y < np.eps2 ? 1u : 0u);
        n_close += (w.x < np.close2 ? 1u : 0u) + (w.y < np.close2 ? 1u : 0u);
    }
    __device__ __forceinline__ void row_begin() {}
    __device__ __forceinline__ void row_end() {}
    __device__ __forceinline__ void fold() {}
    __device__ __forceinline__ void reduce(int o)
    {
        n_near += __shfl_xor_sync(0xffffffffu, n_near, o);
        n_close += __shfl_xor_sync(0xffffffffu, n_close, o);
    }
    __device__ __forceinline__ void store(int64_t)
    {
        const int slot = (threadIdx.x + 7 * blockIdx.x) & (kCountSlots - 1);
        atomicAdd(&counts[2 * slot], (unsigned long long)n_near);
        atomicAdd(&counts[2 * slot + 1], (unsigned long long)n_close);
    }
};

// Batched FP32 near field: one warp per item (first target, count, instance, lanes); all R
// right-hand sides in one candidate-list traversal.
template <int P, int R>
__global__ void __launch_bounds__(32 * kNearWarps, NearFwd<P, R, true>::kMinBlocks * 4 / kNearWarps) k_batch_near32(int64_t n_items,
                                                                               const int4 *__restrict__ items,
                                                                               const BatchInst<float> *__restrict__ inst,
                                                                               bool assign)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (warp >= n_items)
        return;
    const int4 it = items[warp];
    const BatchInst<float> &b = inst[it.z];
    const NearSides sd{b.tgt_base, b.tgt_hi, b.tgt_lo, b.src_hi, b.src_lo, b.src_start};
    const CellGrid cg = b.cg;
    const NearParams<float> np = b.np;
    NearFwd<P, R, true> op;
    op.q = b.q;
    op.phi_s = b.phi_s;
    op.grad_s = b.grad_s;
    op.coinc = b.coinc;
    op.q_stride = b.M;
    op.n_stride = b.N;
    op.rcoef = np.rcoef * sqrtf(np.eps2);
    op.assign = assign;
    __shared__ __align__(16) NearList<R> L[kNearWarps];
    near_traverse_list(make_int2(it.x, it.y), it.w, lane, sd, cg, np, op, L[threadIdx.x >> 5]);
}

template <typename real>
__device__ __forceinline__ void unpermute_point(int64_t k, const real *__restrict__ phi_s,
                                                const real *__restrict__ grad_s, const real *__restrict__ coinc,
                                                const int *__restrict__ perm, double shift, double q_sum, double s,
                                                void *__restrict__ phi_out, void *__restrict__ H_out, int out_is_f64)
{
    output_point<real>(k, phi_s[k], grad_s[2 * k], grad_s[2 * k + 1], coinc[k], perm, shift, q_sum, s, phi_out, H_out,
                       out_is_f64);
}

template <typename real>
__global__ void k_unpermute(int64_t N, const real *__restrict__ phi_s, const real *__restrict__ grad_s,
                            const real *__restrict__ coinc, const int *__restrict__ perm, double shift,
                            const double *__restrict__ q_sum, double s, void *__restrict__ phi_out,
                            void *__restrict__ H_out, int out_is_f64)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k < N)
        unpermute_point(k, phi_s, grad_s, coinc, perm, shift, q_sum[0], s, phi_out, H_out, out_is_f64);
}

// Batched output: block -> (instance, block of its targets), blockIdx.y = right-hand side;
// writes the caller's (nrhs, N) and (nrhs, N, 2) buffers of each instance.
template <typename real>
__global__ void k_batch_unpermute(const BatchInst<real> *__restrict__ inst, const BatchIO *__restrict__ io,
                                  BlockMap bm, int out_is_f64)
{
    const int i = bm.inst[blockIdx.x];
    const BatchInst<real> &b = inst[i];
    const int64_t k = (int64_t)(blockIdx.x - bm.first[i]) * blockDim.x + threadIdx.x;
    const int64_t N = b.N;
    if (k >= N)
        return;
    const int r = blockIdx.y;
    const size_t osz = out_is_f64 ? 8 : 4;
    void *po = io[i].phi ? (unsigned char *)io[i].phi + (size_t)r * N * osz : nullptr;
    void *ho = io[i].H ? (unsigned char *)io[i].H + (size_t)r * N * 2 * osz : nullptr;
    unpermute_point(k, b.phi_s + (int64_t)r * N, b.grad_s + 2 * (int64_t)r * N, b.coinc + (int64_t)r * N,
                    b.tgt_perm, b.shift, b.q_sum[r], b.s, po, ho, out_is_f64);
}

}  // namespace

Near64Params near64_params(const NearParams<double> &np)
{
    Near64Params o{};
    o.eps2 = np.eps2;
    o.inv_eps2 = np.inv_eps2;
    o.beta0 = np.beta[0];
    o.hess0 = np.p > 1 ? 2.0 * np.beta[1] * np.inv_eps2 : 0.0;
    o.h = (float)np.hcell;
    const float reach = sqrtf((float)np.eps2) * (1.f + 1e-4f) + 1e-5f;
    o.reach2 = reach * reach;
    o.p = np.p;
    const double four_pi = 4.0 * kPi;
    for (int k = 0; k + 1 < np.p; ++k)
        o.f[k] = -four_pi * np.nptilde[k];
    if (np.p == 1)
        o.f[0] = -four_pi * np.pbeta[0];      // p = 1: P is a constant
    for (int k = 1; k < np.p; ++k)
        o.c[k - 1] = four_pi * k * np.beta[k];
    for (int k = 2; k < np.p; ++k)
        o.cp[k - 2] = four_pi * k * (k - 1) * np.beta[k];
    return o;
}

cudaError_t launch_near64(int64_t N, const Near64Sides &sd, CellGrid cg, const double *q, const NearParams<double> &np,
                          double *phi_s, double *grad_s, double *coinc, cudaStream_t st)
{
    return with_degree(np.p, [&](auto pc) {
        Near64Fwd<decltype(pc)::value> op{};
        op.q = q;
        op.phi_s = phi_s;
        op.grad_s = grad_s;
        op.coinc = coinc;
        return launch_near64_points(N, sd, cg, near64_params(np), op, st);
    });
}

cudaError_t launch_near32(int64_t n_items, const int2 *items, int lanes, const int *tgt_base, const float2 *tgt_hi,
                          const float2 *tgt_lo, const float2 *src_hi, const float2 *src_lo, const int *src_start,
                          CellGrid cg, const float *q, NearParams<float> np, float *phi_s, float *grad_s, float *coinc,
                          bool assign, cudaStream_t st)
{
    const NearSides sd{tgt_base, tgt_hi, tgt_lo, src_hi, src_lo, src_start};
    return with_degree(np.p, [&](auto pc) {
        NearFwd<decltype(pc)::value, 1> op{};
        op.q = q;
        op.phi_s = phi_s;
        op.grad_s = grad_s;
        op.coinc = coinc;
        op.q_stride = 0;
        op.n_stride = 0;
        op.rcoef = (float)((double)np.rcoef * std::sqrt((double)np.eps2));
        op.assign = assign;
        return launch_near_list(n_items, items, lanes, sd, cg, np, op, st);
    });
}

cudaError_t launch_near_src32(int64_t n_items, const int2 *items, const int *src_base, const float2 *src_hi,
                              const float2 *src_lo, const float2 *tgt_hi, const float2 *tgt_lo, const int *tgt_start,
                              CellGrid cg, const float *q, NearParams<float> np, float *phi_s, float *grad_s,
                              float *coinc, cudaStream_t st)
{
    if (n_items <= 0)
        return cudaSuccess;
    const NearSides sd{src_base, src_hi, src_lo, tgt_hi, tgt_lo, tgt_start};
    const unsigned blocks = (unsigned)((n_items + 3) / 4);
    return with_degree(np.p, [&](auto pc) {
        constexpr int P = decltype(pc)::value;
        k_near_src32<P><<<blocks, 128, 0, st>>>(n_items, items, sd, cg, np, q, phi_s, grad_s, coinc);
        return cudaGetLastError();
    });
}

template <typename real>
cudaError_t launch_unpermute(int64_t N, const real *phi_s, const real *grad_s, const real *coinc, const int *perm,
                             double shift, const double *q_sum, double s, void *phi_out, void *H_out, int out_is_f64,
                             cudaStream_t st)
{
    if (N <= 0)
        return cudaSuccess;
    k_unpermute<real><<<(unsigned)((N + 255) / 256), 256, 0, st>>>(N, phi_s, grad_s, coinc, perm, shift, q_sum, s,
                                                                   phi_out, H_out, out_is_f64);
    return cudaGetLastError();
}

template cudaError_t launch_unpermute<float>(int64_t, const float *, const float *, const float *, const int *,
                                             double, const double *, double, void *, void *, int, cudaStream_t);
template cudaError_t launch_unpermute<double>(int64_t, const double *, const double *, const double *, const int *,
                                              double, const double *, double, void *, void *, int, cudaStream_t);

cudaError_t launch_near_count32(int64_t n_items, const int2 *items, int lanes, const int *tgt_base, const float2 *tgt_hi,
                                const float2 *tgt_lo, const float2 *src_hi, const float2 *src_lo, const int *src_start,
                                CellGrid cg, NearParams<float> np, unsigned long long *counts, cudaStream_t st)
{
    const NearSides sd{tgt_base, tgt_hi, tgt_lo, src_hi, src_lo, src_start};
    NearCount op{};
    op.counts = counts;
    return launch_near_list(n_items, items, lanes, sd, cg, np, op, st);
}

cudaError_t launch_batch_near32(int64_t n_items, const int4 *items, const BatchInst<float> *inst, int p, int nrhs,
                                bool assign, cudaStream_t st)
{
    if (n_items <= 0 || nrhs <= 0)
        return cudaSuccess;
    const unsigned blocks = (unsigned)((n_items + kNearWarps - 1) / kNearWarps);
    constexpr int T = 32 * kNearWarps;
    return with_degree(p, [&](auto pc) {
        constexpr int P = decltype(pc)::value;
        switch (nrhs) {
        case 1: k_batch_near32<P, 1><<<blocks, T, 0, st>>>(n_items, items, inst, assign); break;
        case 2: k_batch_near32<P, 2><<<blocks, T, 0, st>>>(n_items, items, inst, assign); break;
        case 3: k_batch_near32<P, 3><<<blocks, T, 0, st>>>(n_items, items, inst, assign); break;
        case 4: k_batch_near32<P, 4><<<blocks, T, 0, st>>>(n_items, items, inst, assign); break;
        default: return cudaErrorInvalidValue;
        }
        return cudaGetLastError();
    });
}

cudaError_t launch_batch_near64(const BatchInst<double> *inst, BlockMap bm, int blocks, int nrhs, int p,
                                const double *tables, cudaStream_t st)
{
    if (blocks <= 0 || nrhs <= 0)
        return cudaSuccess;
    return with_degree(p, [&](auto pc) {
        k_batch_near64<decltype(pc)::value><<<dim3((unsigned)blocks, (unsigned)nrhs), 32 * kNear64Warps, 0, st>>>(
            inst, bm, tables, 256);
        return cudaGetLastError();
    });
}

template <typename real>
cudaError_t launch_batch_unpermute(const BatchInst<real> *inst, const BatchIO *io, BlockMap bm, int blocks, int nrhs,
                                   int out_is_f64, cudaStream_t st)
{
    if (blocks <= 0 || nrhs <= 0)
        return cudaSuccess;
    k_batch_unpermute<real><<<dim3((unsigned)blocks, (unsigned)nrhs), 256, 0, st>>>(inst, io, bm, out_is_f64);
    return cudaGetLastError();
}

template cudaError_t launch_batch_unpermute<float>(const BatchInst<float> *, const BatchIO *, BlockMap, int, int, int,
                                                   cudaStream_t);
template cudaError_t launch_batch_unpermute<double>(const BatchInst<double> *, const BatchIO *, BlockMap, int, int,
                                                    int, cudaStream_t);

}  // namespace fs
