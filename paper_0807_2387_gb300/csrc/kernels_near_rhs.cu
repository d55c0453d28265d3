// FP32 near field of a plan for two to four charge vectors at once (near_fwd.cuh): the lists, the pair
// geometry, the log and the gradient coefficient are shared, where one vector at a time repeats them.
// The whole evaluation of three vectors at 65,537 targets: 257 us one vector at a time, 152 us together
// (139 us with the steps since).
#include <cmath>

#include "near_fwd.cuh"

namespace fs {

cudaError_t launch_near32_rhs(int64_t n_items, const int2 *items, int lanes, const int *tgt_base, const float2 *tgt_hi,
                              const float2 *tgt_lo, const float2 *src_hi, const float2 *src_lo, const int *src_start,
                              CellGrid cg, const float *q, NearParams<float> np, float *phi_s, float *grad_s,
                              float *coinc, int nrhs, int64_t q_stride, int64_t n_stride, cudaStream_t st)
{
    const NearSides sd{tgt_base, tgt_hi, tgt_lo, src_hi, src_lo, src_start};
    return with_degree(np.p, [&](auto pc) {
        auto run = [&](auto rc) {
            NearFwd<decltype(pc)::value, decltype(rc)::value> op{};
            op.q = q;
            op.phi_s = phi_s;
            op.grad_s = grad_s;
            op.coinc = coinc;
            op.q_stride = q_stride;
            op.n_stride = n_stride;
            op.rcoef = (float)((double)np.rcoef * std::sqrt((double)np.eps2));
            op.assign = true;
            return launch_near_list(n_items, items, lanes, sd, cg, np, op, st);
        };
        switch (nrhs) {
        case 2: return run(std::integral_constant<int, 2>{});
        case 3: return run(std::integral_constant<int, 3>{});
        case 4: return run(std::integral_constant<int, 4>{});
        default: return cudaErrorInvalidValue;
        }
    });
}

}  // namespace fs
