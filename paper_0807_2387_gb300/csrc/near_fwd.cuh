// The forward FP32 near-field correction as an operation of the candidate-list traversal.
#pragma once

#include "near_warp.cuh"

namespace fs {

// Forward correction at the targets for R right-hand sides at once (the pair geometry, the
// log and the gradient coefficient are shared): phi += q f, grad += q c d for two candidates per
// packed operation; the factor c_ln of f (near_g2) and rc eps_I of c are applied once at the
// store (d arrives in units of eps_I).  A plan's sums are split into partial sums per list evaluation,
// for any number of right-hand sides, so that a vector's rounding error does not depend on the vectors
// beside it: 12,000 sources of one sign around 6,000 targets in a cell (p = 4), RMS error against FP64
// 1.2e-7 of phi and 1.9e-7 of H, alone and together; with one running sum a vector 3.1e-7 and 9.5e-7.
// 100,003 sources and 65,537 targets, an evaluation of 2 / 3 / 4 vectors 107.5 / 129 / 158 us (running sums
// 107.7 / 127.4 / 152.3 us).  Four vectors need up to 168 registers and run at three blocks per SM: 20,000 points at p = 8
// 50.6 us against 61 us with spills at four blocks.  The batched kernel, which reads its constants from
// memory, keeps running sums where it holds several right-hand sides.
// Right-hand side r reads q + r q_stride and writes at r n_stride.
template <int P, int R, bool BATCH = false> struct NearFwd {
    static constexpr int kMinBlocks = BATCH ? 4 : (R == 1 ? 6 : (R == 4 ? 3 : 4));   // of four warps per SM
    static constexpr int kUnroll = (R == 1 && !BATCH) ? 2 : 4;
    // |w - 1|^(p-1) / w, the gradient coefficient over rc up to the sign (-1)^(p-1) (applied at the
    // store), as 2^((p-1) log2(1 - w) - log2 w) (log2 w is shared with the value; w = 1 gives 2^-inf):
    // four MUFU operations and one FMA a pair of candidates, against two and the power's
    // multiplications.  2.26 -> 2.19 ms at 2^20 points (p = 8) against alternating the two.  Several
    // right-hand sides add FMA work that hides the difference (batched replay the same either way).
    static constexpr bool kExp2 = P >= 5 && R == 1 && !BATCH;
    static constexpr bool kRows = R == 1 || !BATCH;
    static constexpr bool kSat = P >= 2;   // f(1) = 0 and (w - 1)^(p-1) = 0: clamping w masks a pair
    static constexpr float kPhi = P >= 2 ? kLnCoef : 1.f;   // unit of the phi sums
    const float *__restrict__ q;
    float *__restrict__ phi_s;
    float *__restrict__ grad_s;
    float *__restrict__ coinc;
    int64_t q_stride, n_stride;
    float rcoef;   // rc eps_I: the pair differences arrive in units of eps_I
    bool assign;   // store phi_s / grad_s instead of adding (the far field is added later)
    float2 qj[R];
    float2 phi[R], gx[R], gy[R];
    float qc[R];
    float2 rphi[kRows ? R : 1], rgx[kRows ? R : 1], rgy[kRows ? R : 1];

    __device__ __forceinline__ float2 &acc_phi(int r) { return kRows ? rphi[kRows ? r : 0] : phi[r]; }
    __device__ __forceinline__ float2 &acc_gx(int r) { return kRows ? rgx[kRows ? r : 0] : gx[r]; }
    __device__ __forceinline__ float2 &acc_gy(int r) { return kRows ? rgy[kRows ? r : 0] : gy[r]; }

    __device__ __forceinline__ void init()
    {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            phi[r] = gx[r] = gy[r] = f2(0.f);
            qc[r] = 0.f;
        }
    }
    // candidate-list traversal: the R charges of source j, and those of a pair of candidates
    static constexpr int kR = R;
    __device__ __forceinline__ void fetch(int j, float (&v)[R]) const
    {
#pragma unroll
        for (int r = 0; r < R; ++r)
            v[r] = __ldg(q + r * q_stride + j);
    }
    __device__ __forceinline__ void set_q(const float2 (&v)[R])
    {
#pragma unroll
        for (int r = 0; r < R; ++r)
            qj[r] = v[r];
    }
    __device__ __forceinline__ void coincident(const NearParams<float> &np, int t)
    {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float qs = comp(qj[r], t);
            add_comp(acc_phi(r), t, -qs * (np.beta[0] / kPhi));   // G(0) := 0 removes the far field's T_I(0)
            qc[r] += qs;
        }
    }
    __device__ __forceinline__ void pair2(const NearParams<float> &np, float2 w, float2 dx, float2 dy)
    {
        float2 val, coef;
        if constexpr (P >= 2) {
            const float2 s = fma2(w, f2(-1.f), f2(1.f)), lw = lg2_2(w);
            val = near_g2<P>(np, w, s, lw);
            if constexpr (kExp2)
                coef = ex2_2(fma2(f2((float)(P - 1)), lg2_2(s), make_float2(-lw.x, -lw.y)));   // s = 0: 2^-inf
            else
                coef = mul2(ipow2<P - 1>(s), rcp_2(w));
        } else {
            val = near_f2<P>(np, w);
            coef = rcp_2(w);
#pragma unroll
            for (int r = 0; r < R; ++r)
                qj[r] = select2(w, np.eps2, qj[r]);
        }
        if constexpr (R >= 3) {
            // three or more right-hand sides: the pair's gradient vector once, then one FMA per
            // component and right-hand side (batched replay 8.01 -> 7.77 ms at three)
            const float2 cdx = mul2(coef, dx), cdy = mul2(coef, dy);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                acc_phi(r) = fma2(qj[r], val, acc_phi(r));
                acc_gx(r) = fma2(qj[r], cdx, acc_gx(r));
                acc_gy(r) = fma2(qj[r], cdy, acc_gy(r));
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                acc_phi(r) = fma2(qj[r], val, acc_phi(r));
                const float2 tq = mul2(qj[r], coef);
                acc_gx(r) = fma2(tq, dx, acc_gx(r));
                acc_gy(r) = fma2(tq, dy, acc_gy(r));
            }
        }
    }
    __device__ __forceinline__ void row_begin()
    {
        if constexpr (kRows)
#pragma unroll
            for (int r = 0; r < R; ++r)
                rphi[r] = rgx[r] = rgy[r] = f2(0.f);
    }
    __device__ __forceinline__ void row_end()
    {
        if constexpr (kRows)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                phi[r] = add2(phi[r], rphi[r]);
                gx[r] = add2(gx[r], rgx[r]);
                gy[r] = add2(gy[r], rgy[r]);
            }
    }
    __device__ __forceinline__ void fold()
    {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            phi[r].x += phi[r].y;
            gx[r].x += gx[r].y;
            gy[r].x += gy[r].y;
        }
    }
    __device__ __forceinline__ void reduce(int o)
    {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            phi[r].x = lane_add(phi[r].x, o);
            gx[r].x = lane_add(gx[r].x, o);
            gy[r].x = lane_add(gy[r].x, o);
            qc[r] = lane_add(qc[r], o);
        }
    }
    __device__ __forceinline__ void store(int64_t k)
    {
        const float rc = (P >= 2 && (P - 1) % 2 == 1) ? -rcoef : rcoef;   // coef is |w - 1|^(p-1) / w
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t kk = k + r * n_stride;
            const float p = kPhi * phi[r].x, x = rc * gx[r].x, y = rc * gy[r].x;
            phi_s[kk] = assign ? p : phi_s[kk] + p;
            grad_s[2 * kk] = assign ? x : grad_s[2 * kk] + x;
            grad_s[2 * kk + 1] = assign ? y : grad_s[2 * kk + 1] + y;
            coinc[kk] = qc[r];
        }
    }
};

}  // namespace fs
