// Plan object of the FEM-NFFT fast summation and the host helpers shared by the plan
// entry points (femnfft.cu) and the batched solves (batch.cu).  Private to the library.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

#include "../../include/femnfft.h"
#include "internal.h"

namespace fs {

// Records msg as the calling thread's last error and returns st.
fs_status fail(fs_status st, const std::string &msg);

constexpr int kStages = 8;

// Several arrays in one allocation (a cudaMalloc takes about 30 us where arrays are some megabytes large, and
// so does a cudaFree): take() each with no base to add the sizes up, then again with the allocation as
// the base for the pointers.
struct Parts {
    unsigned char *base = nullptr;
    size_t used = 0;
    template <typename T> void take(T **out, size_t count)
    {
        *out = base ? reinterpret_cast<T *>(base + used) : nullptr;
        used += (count * sizeof(T) + 255) / 256 * 256;
    }
};

// A cell's run of near-field items: `count` items of one size from item `first` on, and the
// estimated pair work of each.
struct NearCell {
    int64_t work;
    int first, count;
};
constexpr int kSrcMajorItem = 64;   // sources per item of the source-major near field
constexpr int kSms = 152;           // streaming multiprocessors of a GB300
constexpr int kRhsGroup = 4;       // charge vectors a plan evaluates together at most
constexpr int kSpreadChunk = 512;   // sources per spreading work item
// 2D plans whose occupied spreading tiles hold fewer sources than this on average spread with
// global atomics (the plan's choice in plan_init).  Zero: on GB300 the tiles won at every
// density measured, from 1.4 to over 700 sources per occupied tile (uniform discs of 2^10 to
// 2^20 points on n = 128 and 512 grids, m = 5: 12.9 vs 19.9 us at the sparse end, 170 vs
// 545 us at the dense end), so direct spreading is used only when FS_FLAG_SPREAD_DIRECT asks.
constexpr double kDirectSpreadBelow = 0.0;

}  // namespace fs

#define FS_CUDA(call)                                                                                   \
    do {                                                                                                \
        cudaError_t e_ = (call);                                                                        \
        if (e_ != cudaSuccess)                                                                          \
            return fs::fail(FS_ECUDA, std::string(#call) + " failed: " + cudaGetErrorString(e_));       \
    } while (0)

#define FS_TRY(expr)                                                                                    \
    do {                                                                                                \
        fs_status s_ = (expr);                                                                          \
        if (s_ != FS_OK)                                                                                \
            return s_;                                                                                  \
    } while (0)

struct fs_plan {
    // parameters
    int precision = 32;
    int n = 0, n_os = 0, m = 0, p = 0;
    double sigma = 0, eps_I = 0, eps_B = 0, s = 1.0;
    int64_t M = 0, N = 0;
    int window_lo = 0, n_a = 0, pitch = 0, ld = 0;
    fs::CellGrid cg{};
    int n_keys = 0;
    unsigned flags = 0;
    cudaStream_t stream = nullptr;
    int device = 0;
    bool kahan = true;
    fs::KernelParams kp{};
    double beta[fs::kMaxP] = {0};
    fs::WindowPoly wpoly{};               // window polynomials (per tap) of FP32 plans
    fs::WindowPoly64 wpoly64{};           // and of FP64 plans
    // device memory
    std::vector<void *> allocs;
    int64_t bytes = 0;
    int *status = nullptr;
    int *status_host = nullptr;           // page-locked copy of *status (fs_solve_host)
    int *src_perm = nullptr, *tgt_perm = nullptr;
    int *src_base = nullptr, *tgt_base = nullptr;
    void *src_frac = nullptr, *tgt_frac = nullptr;
    double2 *src_pos = nullptr, *tgt_pos = nullptr;
    float2 *src_pos32 = nullptr, *tgt_pos32 = nullptr;
    double *near64_tables = nullptr;      // FP64 plans (Near64Sides)
    float2 *src_lo32 = nullptr, *tgt_lo32 = nullptr;
    int *src_start = nullptr, *tgt_start = nullptr;
    std::vector<int> src_cells, tgt_cells;   // the cells' first points (host)
    int src_cap = 0, tgt_cap = 0;            // points per piece of a cell: 8, 16, 32 (64: source-major)
    fs::SpreadItem *items = nullptr;
    int n_items = 0;
    fs::SpreadItem *tgt_items = nullptr;  // adjoint: spreading at the targets
    int n_tgt_items = 0;
    // adjoint workspace (allocated by the first fs_adjoint call)
    void *adj_c = nullptr, *adj_dn = nullptr, *adj_df = nullptr;
    void *adj_a = nullptr, *adj_ga = nullptr, *adj_cg = nullptr, *adj_hess = nullptr;
    double *adj_gsum = nullptr;
    int2 *near_items = nullptr;       // FP32 near field: (first target, count <= tgt_cap) per warp
    int64_t n_near_items = 0;
    std::vector<int2> near_items_h;   // host copies (merged into batch work lists)
    std::vector<fs::NearCell> near_cells_h;
    std::vector<fs::SpreadItem> items_h;
    int2 *adj_items = nullptr;        // FP32 adjoint: (first source, count <= min(src_cap, 32))
    int64_t n_adj_items = 0;
    int2 *src_near_items = nullptr;   // source-major near field: (first source, count <= 64)
    int64_t n_src_near_items = 0;
    bool src_major = false;           // FP32 forward near field over source items (many more sources than targets)
    void *mul = nullptr, *tw = nullptr;
    void *grid = nullptr, *spec = nullptr;   // grid: zero between evaluations (grid_dirty: not known to be)
    void *field = nullptr;            // the filtered grid (without memory for it, the grid)
    bool member = false;              // of a batch, which has its own grids: field is not allocated before the first charges
    bool grid_dirty = false, grid_recorded = false;
    void *grid_comp = nullptr;        // direct spreading (FP32): compensation plane of the grid
    bool spread_direct = false;       // spread with global atomics instead of shared-memory tiles
    // grid, field, spec and (FP32) the near field's sums hold rhs_cap charge vectors, evaluated together; the
    // sums are phi_s, grad_s from rhs_cap sums_n and coinc from 3 rhs_cap sums_n on (FP64: of one vector)
    void *phi_s = nullptr, *grad_s = nullptr, *coinc = nullptr;
    int64_t sums_n = 0;
    int rhs_cap = 1;
    void *rhs_block = nullptr;        // their allocation for rhs_cap > 1
    // charges
    void *q_sorted = nullptr;
    double *q_sum = nullptr;
    int nrhs = 0, nrhs_cap = 0;
    // FEM
    bool is_fem = false;
    int64_t Nv = 0, Nt = 0, Ne = 0;
    const double2 *nodes = nullptr;   // caller's (valid while the plan is used)
    int *tris = nullptr, *bedges = nullptr;
    double2 *fem_tri_coef = nullptr;      // per triangle: its charge = sum_k M_k . coef_k (k_fem_tri_coef)
    double2 *fem_src = nullptr;
    int *src_inv_perm = nullptr;      // source index -> sorted index (charges assembled into cell order)
    // host staging for fs_solve_host
    void *d_q_stage = nullptr, *d_phi_stage = nullptr, *d_H_stage = nullptr;
    size_t q_stage_bytes = 0, phi_stage_bytes = 0, H_stage_bytes = 0;
    // stats
    int64_t near_pairs = 0, near_pairs_fp64 = 0;
    // timing
    cudaEvent_t ev[fs::kStages + 1] = {};
    cudaEvent_t ev_q0 = nullptr, ev_q1 = nullptr;
    bool events = false;
    // FP32 plans: the near field runs on a second stream beside spreading and the transform
    // (fork after the charges, join before the interpolation adds the far field)
    bool overlap = false;
    cudaStream_t aux = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    cudaEvent_t ev_n0 = nullptr, ev_n1 = nullptr, ev_j = nullptr;   // timing of the overlapped stages

    // Memory the plan can do without (null, and no error text, if there is none).
    void *try_alloc(size_t nbytes, cudaError_t *error = nullptr)
    {
        void *p_ = nullptr;
        const cudaError_t e = cudaMalloc(&p_, nbytes);
        if (error)
            *error = e;
        if (e != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        allocs.push_back(p_);
        bytes += (int64_t)nbytes;
        return p_;
    }
    template <typename T> fs_status alloc(T **out, size_t count)
    {
        const size_t nbytes = std::max<size_t>(count, 1) * sizeof(T);
        cudaError_t e = cudaSuccess;
        *out = static_cast<T *>(try_alloc(nbytes, &e));
        if (!*out)
            return fs::fail(FS_ENOMEM, "cudaMalloc of " + std::to_string(nbytes) + " bytes failed: " +
                                       cudaGetErrorString(e));
        return FS_OK;
    }
    fs_status alloc_bytes(void **out, size_t nbytes)
    {
        unsigned char *p_ = nullptr;
        FS_TRY(alloc(&p_, nbytes));
        *out = p_;
        return FS_OK;
    }
    void release(void *ptr)
    {
        if (!ptr)
            return;
        auto it = std::find(allocs.begin(), allocs.end(), ptr);
        if (it != allocs.end()) {
            cudaFree(ptr);
            allocs.erase(it);
        }
    }
    // Whether an evaluation submits the near field before the spreading.  Where points crowd, one item
    // (a warp) takes a good part of the near field's time, and its start must not wait for the
    // spreading's blocks: 300,001 points in eight clusters, longest item 2.8e5 candidate pairs, host
    // call 555 us with the spreading first and 527 us with the near field first.  Elsewhere the order
    // makes no difference beyond 1.5 % (1,000 targets 40.7 us against 41.3 us with the near field first,
    // whose submission delays the longer chain); uniform 262,144 points have items of up to 5.7e4 pairs.
    bool near_first() const { return !near_cells_h.empty() && near_cells_h[0].work >= (1 << 16); }
    // Whether the transform's kernels start before the kernel ahead of them has ended (launch_chained):
    // where the row kernels (over all vectors; the columns are about as many) and the spreading of one
    // vector (n_items) have at most a block per SM.  There a launch's latency counts: evaluations of 1,000 and 4,096 points 35.8 -> 24.5 and 31.8 -> 24.6 us on the GPU.
    // With more blocks the waiting ones keep slots that the spreading or the near field needs: 32,768
    // points in FP64 875 -> 992 us, the disc mesh 131 -> 145, a training step of 262,144 points 974 -> 988.
    bool chained(int n_items, int nrhs) const
    {
        return n_items > 0 && n_items <= fs::kSms && (n_a + 1) / 2 * nrhs <= fs::kSms && !spread_direct;
    }
    size_t rsize() const { return precision == 64 ? 8 : 4; }
};

namespace fs {

// Modified Bessel function I_0 (power series, FP64).
double bessel_i0(double x);
// Per-tap polynomial form of the normalised Kaiser-Bessel window (FP32 kernels) for
// oversampling sigma and half-width m.
void build_window_poly(double sigma, int m, WindowPoly *wp);
// The FP64 kernels' (kept per (sigma, m) for the process: a few of at most 4 KB).
void build_window_poly64(double sigma, int m, WindowPoly64 *wp);

// Validates the parameters and builds the plan (binning, tables, items) on its stream.
fs_status plan_create_common(const double *src, int64_t M, const double *tgt, int64_t N, int n_grid,
                             double sigma_os, int m, double eps_I, const fs_opts *opts, fs_plan *pl);
// Waits for the plan's stream and frees everything it owns.
void plan_destroy(fs_plan *pl);

template <typename real> inline const WinPoly<real> &win_poly(const fs_plan *pl)
{
    if constexpr (sizeof(real) == 8)
        return pl->wpoly64;
    else
        return pl->wpoly;
}

template <typename real> inline Window<real> make_window(double sigma, int m_window)
{
    const double b = kPi * (2.0 - 1.0 / sigma);
    const double m = m_window;
    Window<real> w;
    w.m = (real)m;
    w.m2 = (real)(m * m);
    w.b = (real)b;
    w.bm = (real)(b * m);
    w.S = (real)(m * b / (1.0 - std::exp(-2.0 * b * m)));
    return w;
}

template <typename real> inline Window<real> make_window(const fs_plan *pl)
{
    return make_window<real>(pl->sigma, pl->m);
}

template <typename real> inline NearParams<real> make_near(const fs_plan *pl)
{
    NearParams<real> np{};
    np.p = pl->p;
    np.eps2 = (real)(pl->eps_I * pl->eps_I);
    np.inv_eps2 = (real)(1.0 / (pl->eps_I * pl->eps_I));
    np.close2 = (real)((pl->eps_I / 8.0) * (pl->eps_I / 8.0));
    np.hcell = (real)((double)pl->cg.cell / pl->n_os);
    for (int k = 0; k < pl->p; ++k)
        np.beta[k] = (real)pl->beta[k];
    for (int k = 1; k < pl->p; ++k)
        np.dbeta[k - 1] = (real)(2.0 * k * pl->beta[k] / (pl->eps_I * pl->eps_I));
    // T_I - k(eps_I) vanishes at r = eps_I; and since k - T_I has a zero of order p there, the
    // gradient numerator R(w) = -(1/2pi) - sum_k 2k beta_k w^k (degree p-1) is c (w-1)^(p-1).
    const double k_eps = -std::log(pl->eps_I) / (2.0 * kPi);
    for (int k = 0; k < pl->p; ++k)
        np.pbeta[k] = (real)(k == 0 ? pl->beta[0] - k_eps : pl->beta[k]);
    // synthetic division of P by (w - 1): Ptilde_{p-2} = a_{p-1}, Ptilde_k = a_{k+1} + Ptilde_{k+1}
    // (the remainder P(1) vanishes in exact arithmetic and is dropped)
    {
        double a[kMaxP] = {0}, t[kMaxP] = {0};
        for (int k = 0; k < pl->p; ++k)
            a[k] = k == 0 ? pl->beta[0] - k_eps : pl->beta[k];
        for (int k = pl->p - 2; k >= 0; --k)
            t[k] = a[k + 1] + (k + 1 <= pl->p - 2 ? t[k + 1] : 0.0);
        for (int k = 0; k + 1 < pl->p; ++k)
            np.nptilde[k] = (real)(-t[k]);
        const double c_ln = -std::log(2.0) / (4.0 * kPi);
        for (int k = 0; k + 1 < pl->p; ++k)
            np.ptln[k] = (real)(t[k] / c_ln);
    }
    // R(w) = c (w-1)^(p-1) with R(0) = -(1/2pi) gives c = (-1)^p / (2pi), independent of beta
    np.rcoef = (real)(((pl->p % 2 == 0) ? 1.0 : -1.0) / (2.0 * kPi * pl->eps_I * pl->eps_I));
    return np;
}

inline Near64Sides near64_sides(const fs_plan *pl, bool own_targets)
{
    if (own_targets)
        return {pl->tgt_base, pl->tgt_pos, pl->tgt_pos32, pl->src_pos, pl->src_pos32, pl->src_start, pl->near64_tables};
    return {pl->src_base, pl->src_pos, pl->src_pos32, pl->tgt_pos, pl->tgt_pos32, pl->tgt_start, pl->near64_tables};
}

}  // namespace fs
