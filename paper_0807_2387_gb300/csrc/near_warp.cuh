// Warp-cooperative FP32 near-field traversal, shared by the forward correction
// (phi and grad phi at the targets; one or several charge vectors), the Hessian of phi at
// the targets, the adjoint potential at the sources and the plan's pair statistics.
//
// A work item is a piece of a cell: at most 8, 16 or 32 consecutive "own" points (one per lane),
// compact because the cells are sorted into pieces (CellSplit).  The warp forms the bounding box of
// its points, reads the "other" points of the neighbour cells within eps_I of that box 32 at a
// time, keeps those within eps_I of the box (ballot) and appends them to candidate lists in shared
// memory, which all lanes then evaluate with branch-free masked arithmetic.  Positions are FP32
// offsets from the cell corner stored as hi + lo; candidates within eps_I / 8 of the box go to a
// second list that carries their position in the item's frame as hi + lo as well, so the pair
// difference keeps full FP32 relative accuracy for nearly coincident points, and exactly
// coincident pairs are detected (G(0) := 0).
//
// With w = r^2 / eps_I^2 and f = G - T_I (T_I the inner polynomial of the
// regularised kernel, p-fold contact with G at r = eps_I):
//     f(w)      = -(ln 2 / 4 pi) log2 w - P(w),      P = T_I - k(eps_I), P(1) = 0
//     c(w)      = f'(r) / r = rc (w - 1)^(p-1) / w,  rc = (-1)^p / (2 pi eps_I^2)
//     c'(w)     = dc/dw = rc (w - 1)^(p-2) ((p - 2) w + 1) / w^2
// (the (p-1)-fold root at w = 1 keeps c free of cancellation near r = eps_I), so
// grad f = c d and Hess f = c I + (2 c' / eps_I^2) d d^T for d = own - other.
//
// An own point meets two candidates at a time, their arithmetic done as packed pairs
// (Blackwell's two-wide FP32 add, multiply and fma: one instruction for both).  Pairs beyond eps_I are masked without a select where the forms allow it:
// with w clamped to 1, P(w) = (w - 1) Ptilde(w) and (w - 1)^(p-1) vanish exactly, as
// does log2(1).
#pragma once

#include <type_traits>

#include "internal.h"

namespace fs {

__device__ __forceinline__ float warp_min(float v)
{
    for (int o = 16; o > 0; o >>= 1)
        v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ float warp_max(float v)
{
    for (int o = 16; o > 0; o >>= 1)
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Single MUFU operations (approximate, flush-to-zero): log2 with ~2^-22 absolute error on
// (0, 16), and the reciprocal with ~1 ulp error; both arguments here are normal numbers.
__device__ __forceinline__ float lg2_approx(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ---- packed pairs of FP32 values (x: the first candidate, y: the second)

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 lg2_2(float2 w) { return make_float2(lg2_approx(w.x), lg2_approx(w.y)); }
__device__ __forceinline__ float2 rcp_2(float2 w) { return make_float2(rcp_approx(w.x), rcp_approx(w.y)); }
__device__ __forceinline__ float2 ex2_2(float2 w) { return make_float2(ex2_approx(w.x), ex2_approx(w.y)); }
__device__ __forceinline__ float2 select2(float2 r2, float eps2, float2 v)
{
    return make_float2(r2.x < eps2 ? v.x : 0.f, r2.y < eps2 ? v.y : 0.f);
}
__device__ __forceinline__ float comp(float2 v, int t) { return t == 0 ? v.x : v.y; }
__device__ __forceinline__ void add_comp(float2 &v, int t, float a)
{
    if (t == 0)
        v.x += a;
    else
        v.y += a;
}

template <int E> __device__ __forceinline__ float2 ipow2(float2 x)
{
    if constexpr (E == 0) {
        return f2(1.f);
    } else if constexpr (E == 1) {
        return x;
    } else {
        const float2 h = ipow2<E / 2>(x);
        if constexpr (E % 2 == 0)
            return mul2(h, h);
        else
            return mul2(mul2(h, h), x);
    }
}

// f = G - T_I at w (clamped to <= 1 by the caller for p >= 2, where f(1) = 0 exactly).
template <int P> __device__ __forceinline__ float2 near_f2(const NearParams<float> &np, float2 w)
{
    const float c_ln = -0.69314718055994531f / (4.0f * 3.14159265358979324f);   // -(ln 2) / (4 pi)
    if constexpr (P == 1) {
        return fma2(f2(c_ln), lg2_2(w), f2(-np.pbeta[0]));
    } else {
        float2 t = f2(np.nptilde[P - 2]);
#pragma unroll
        for (int i = P - 3; i >= 0; --i)
            t = fma2(t, w, f2(np.nptilde[i]));
        return fma2(f2(c_ln), lg2_2(w), mul2(add2(w, f2(-1.f)), t));   // c_ln log2 w - (w - 1) Ptilde(w)
    }
}

// f / c_ln with c_ln = -(ln 2) / (4 pi), applied by the caller at the store: since P(w) =
// (w - 1) Ptilde(w), f / c_ln = log2 w + s Ptilde(w) / c_ln with s = 1 - w: one FMA after the
// polynomial.  w <= 1 (clamped) and degree p >= 2.
constexpr float kLnCoef = -0.69314718055994531f / (4.0f * 3.14159265358979324f);
template <int P> __device__ __forceinline__ float2 near_g2(const NearParams<float> &np, float2 w, float2 s, float2 lw)
{
    float2 t = f2(np.ptln[P - 2]);
#pragma unroll
    for (int i = P - 3; i >= 0; --i)
        t = fma2(t, w, f2(np.ptln[i]));
    return fma2(s, t, lw);
}

// c / rc = (w - 1)^(p-1) / w and c' / rc = (w - 1)^(p-2) ((p - 2) w + 1) / w^2 (rc applied by the caller),
// for degrees whose pairs are not clamped (p <= 2).
template <int P> __device__ __forceinline__ void near_c_cp2(float2 w, float2 &c, float2 &cp)
{
    static_assert(P <= 2, "clamped pairs use near_b2");
    const float2 rw = rcp_2(w);
    if constexpr (P == 1) {
        c = rw;
        cp = mul2(f2(-1.f), mul2(rw, rw));
    } else {
        c = mul2(rw, add2(w, f2(-1.f)));
        cp = mul2(rw, rw);
    }
}

// The same for p >= 3 from s = 1 - w: with b = s^(p-2) / w and h = p - 2 + 1 / w,
// c / rc = (-1)^(p-1) b s and c' / rc = (-1)^p b h, the signs applied by the caller at the store.  The
// gradients' pair work is bound by the FMA pipe: weighting b instead of c and c', sharing s with
// near_g2 and the adjoint's dipoles read with their sign took 5 of 33 packed operations of an adjoint
// pair and 2 of 23 of a Hessian pair (training step of 262,144 points, p = 6: 1025 -> 991 us).
template <int P> __device__ __forceinline__ void near_b2(float2 w, float2 s, float2 &b, float2 &h)
{
    const float2 rw = rcp_2(w);
    b = mul2(ipow2<P - 2>(s), rw);
    h = add2(rw, f2((float)(P - 2)));
}

// The two point sets of a traversal: the items' own points and the other side's.
struct NearSides {
    const int *own_base;
    const float2 *own_hi, *own_lo;
    const float2 *oth_hi, *oth_lo;
    const int *oth_start;
};

// ---- candidate-list traversal
//
// The lanes read the other points of each neighbour cell within reach of the box 32 at a time
// (a cell is one contiguous range, so the chunks are full, where sub-cells would hold only a
// few points each), test each against the box (ballot) and append those within reach to the
// warp's lists in shared memory: "far" candidates (beyond eps_I / 8 of the box: no pair can
// need the refined difference) shifted into the item's cell frame, negated and in units of eps_I,
// with their Op::kR values (charges, or the adjoint's weights); "close" candidates the same way as
// hi + lo (the TwoSum of the cell step and -y_hi, with -y_lo added to the low part), for the
// refined path.  A list is one array per component (an append is one address, a read four
// candidates per 16 bytes), padded with far-away entries of value 0 to a whole number of rounds
// and evaluated when it fills and at the end: broadcast shared loads and no per-candidate test or
// vote in the far loop.  Partial sums are kept per list evaluation (op.row_begin / row_end).
//
// An item holds at most `lanes` own points, one per lane; the 32 / lanes groups of the warp take
// different candidates and their sums are added at the end (op.reduce).  Small items have small
// boxes, so more of the evaluated pairs lie within eps_I, and there are more of them to fill the
// GPU; large ones build fewer lists (near_item_lanes).
//
// What bounds it (2^20-point mixture, 32 lanes, 2.2e9 pairs within eps_I, 0.75 of the evaluated ones):
// the issue slots; a pair of candidates is 26 instructions (34 FMA-pipe cycles and 40 of the MUFU
// pipe for 64 pair slots), 1.2e9 of the 1.78e9 in all, the lists are most of the rest.  2.75 ms
// with items of 64 targets (two per lane, runs of the Morton sub-cell order) -> 2.18 ms.  Tried and
// not kept: bounding boxes of groups of 32 other points tested before the points (2.23 ms; at 45
// points per cell 49 against 43 us); the lists' entries (first point, mask) kept with the plan
// (2.09 ms, at 45 per cell 51 against 41 us, 40 bytes per target and twice the plan's time);
// alternating the gradient's exp2 and power forms (2.26 ms).
//
// An Op provides kMinBlocks, kUnroll (fours of candidates), kR, kSat (w = min(r2, 1) is all it needs: the clamp rides on the last
// FMA of r2), init(), fetch(j, v) (the kR values of other point j), set_q(v) (those of a pair of
// candidates), coincident(np, t) (candidate t of the pair coincides with the own point),
// pair2(np, w, dx, dy) (both candidates packed; dx, dy in units of eps_I, w = r^2, and np carries
// eps2 = inv_eps2 = 1; pairs with w >= 1 must contribute nothing), row_begin(), row_end(), fold()
// (the two packed halves of each sum together), reduce(o) (add the sums of the lane at xor distance
// o) and store(k).
constexpr int kListCap = 256;    // far candidates per warp
constexpr int kCloseCap = 64;    // close candidates per warp
constexpr float kPadPos = 1e9f;  // a padding entry's position: beyond eps_I of every point (idle lanes sit at 1e6 / eps_I)

__device__ __forceinline__ float2 near_w2(bool sat, float2 dx, float2 dy)
{
    const float2 m = mul2(dx, dx);
    if (sat)
        return make_float2(__saturatef(fmaf(dy.x, dy.x, m.x)), __saturatef(fmaf(dy.y, dy.y, m.y)));
    return fma2(dy, dy, m);
}

// Four values of each of the R arrays of stride `cap`, as two pairs.
template <int R>
__device__ __forceinline__ void near_list_q(const float *s_q, int cap, int e, float2 (&qa)[R], float2 (&qb)[R])
{
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float4 q = *reinterpret_cast<const float4 *>(s_q + r * cap + 4 * e);
        qa[r] = make_float2(q.x, q.y);
        qb[r] = make_float2(q.z, q.w);
    }
}

// n candidates (a multiple of 4 x groups); group g of `groups` takes every groups-th four of them.
template <class Op>
__device__ __forceinline__ void near_eval_far(const float *s_x, const float *s_y, const float *s_q, int n, int g,
                                              int groups, float2 X, float2 Y, const NearParams<float> &np, Op &op)
{
    op.row_begin();
    const int quads = n >> 2;
#pragma unroll(Op::kUnroll)
    for (int e = g; e < quads; e += groups) {
        const float4 x = *reinterpret_cast<const float4 *>(s_x + 4 * e), y = *reinterpret_cast<const float4 *>(s_y + 4 * e);
        float2 qa[Op::kR], qb[Op::kR];
        near_list_q<Op::kR>(s_q, kListCap, e, qa, qb);
        {
            const float2 dx = add2(X, make_float2(x.x, x.y)), dy = add2(Y, make_float2(y.x, y.y));
            op.set_q(qa);
            op.pair2(np, near_w2(Op::kSat, dx, dy), dx, dy);
        }
        {
            const float2 dx = add2(X, make_float2(x.z, x.w)), dy = add2(Y, make_float2(y.z, y.w));
            op.set_q(qb);
            op.pair2(np, near_w2(Op::kSat, dx, dy), dx, dy);
        }
    }
    op.row_end();
}

// Close candidates carry their negated position in the item's frame as hi + lo
// (n = -(offset of the cell step) - y, TwoSum-exact at list time), so the difference
// d = (x_hi + n_hi) + (x_lo + n_lo) keeps full FP32 relative accuracy however small it is:
// when x_hi and -n_hi are close the first sum is exact (Sterbenz), and when they are not,
// d is of their size and one rounding is harmless.  Exactly coincident points give d = 0
// (G(0) := 0); they are handled on a warp-uniform branch.  The exact difference is then scaled
// by ie = 1 / eps_I, the unit of every difference handed to the Op.
template <class Op>
__device__ __forceinline__ void near_eval_close(const float *s_x, const float *s_y, const float *s_lx,
                                                const float *s_ly, const float *s_q, int n, int g, int groups,
                                                float2 X, float2 Y, float2 XL, float2 YL, float ie,
                                                const NearParams<float> &np, Op &op)
{
    op.row_begin();
    for (int e = g; e < n >> 2; e += groups) {
        const float4 x = *reinterpret_cast<const float4 *>(s_x + 4 * e), y = *reinterpret_cast<const float4 *>(s_y + 4 * e);
        const float4 lx = *reinterpret_cast<const float4 *>(s_lx + 4 * e), ly = *reinterpret_cast<const float4 *>(s_ly + 4 * e);
        float2 q2[2][Op::kR];
        near_list_q<Op::kR>(s_q, kCloseCap, e, q2[0], q2[1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 hx = h ? make_float2(x.z, x.w) : make_float2(x.x, x.y);
            const float2 hy = h ? make_float2(y.z, y.w) : make_float2(y.x, y.y);
            const float2 ox = h ? make_float2(lx.z, lx.w) : make_float2(lx.x, lx.y);
            const float2 oy = h ? make_float2(ly.z, ly.w) : make_float2(ly.x, ly.y);
            op.set_q(q2[h]);
            const float2 ex = add2(add2(X, hx), add2(XL, ox));
            const float2 ey = add2(add2(Y, hy), add2(YL, oy));
            const float2 dx = mul2(ex, f2(ie)), dy = mul2(ey, f2(ie));   // in units of eps_I
            float2 w = near_w2(Op::kSat, dx, dy);
            const bool z0 = ex.x == 0.f && ey.x == 0.f, z1 = ex.y == 0.f && ey.y == 0.f;
            if (__any_sync(0xffffffffu, z0 || z1)) {
                if (z0) {
                    op.coincident(np, 0);
                    w.x = 1.f;                        // masked out
                }
                if (z1) {
                    op.coincident(np, 1);
                    w.y = 1.f;
                }
            }
            op.pair2(np, w, dx, dy);
        }
    }
    op.row_end();
}

// A warp's lists: x, y and the R values of kListCap far candidates; x, y, their low parts and the R
// values of kCloseCap close ones.
template <int R> struct NearList {
    float x[kListCap], y[kListCap], q[kListCap * R];
    float cx[kCloseCap], cy[kCloseCap], lx[kCloseCap], ly[kCloseCap], cq[kCloseCap * R];
    __device__ __forceinline__ void put(int at, float px, float py, const float (&v)[R])
    {
        x[at] = px;
        y[at] = py;
#pragma unroll
        for (int r = 0; r < R; ++r)
            q[r * kListCap + at] = v[r];
    }
    __device__ __forceinline__ void put_close(int at, float px, float py, float plx, float ply, const float (&v)[R])
    {
        cx[at] = px;
        cy[at] = py;
        lx[at] = plx;
        ly[at] = ply;
#pragma unroll
        for (int r = 0; r < R; ++r)
            cq[r * kCloseCap + at] = v[r];
    }
    // pads n entries to a multiple of `unit` (at most 32); returns the padded count
    __device__ __forceinline__ int pad(int n, int unit, int lane)
    {
        const float none[R] = {};
        const int full = (n + unit - 1) & ~(unit - 1);
        if (n + lane < full)
            put(n + lane, kPadPos, kPadPos, none);
        return full;
    }
    __device__ __forceinline__ int pad_close(int n, int unit, int lane)
    {
        const float none[R] = {};
        const int full = (n + unit - 1) & ~(unit - 1);
        if (n + lane < full)
            put_close(n + lane, kPadPos, kPadPos, 0.f, 0.f, none);
        return full;
    }
};

template <class Op>
__device__ __forceinline__ void near_traverse_list(int2 item, int lanes, int lane, const NearSides &sd,
                                                   const CellGrid &cg, const NearParams<float> &np, Op &op,
                                                   NearList<Op::kR> &L)
{
    constexpr int R = Op::kR;
    const float h = np.hcell, eps = sqrtf(np.eps2);
    const int groups = 32 / lanes, slot = lane & (lanes - 1), g = lane / lanes;
    const bool valid = slot < item.y;
    const int64_t k = item.x + (valid ? slot : 0);
    const int packed = sd.own_base[k];
    const int c1 = base1(packed) / cg.cell, c2 = base2(packed) / cg.cell;   // the item's cell
    float2 xh = sd.own_hi[k];
    const float2 xl = sd.own_lo[k];
    // bounding box in the item's frame, offsets from its cell's corner (idle lanes hold the first point)
    const float tx0 = warp_min(xh.x), tx1 = warp_max(xh.x);
    const float ty0 = warp_min(xh.y), ty1 = warp_max(xh.y);
    if (!valid)
        xh = make_float2(1e6f, 1e6f);             // idle lanes: every pair lands beyond eps_I
    const float2 X = f2(xh.x), Y = f2(xh.y), XL = f2(xl.x), YL = f2(xl.y);
    // the Op sees differences in units of eps_I, so w = r^2 needs no scaling per pair: the far
    // list holds sources in those units and the item's points are scaled once here
    const float ie = sqrtf(np.inv_eps2);
    const float2 XS = mul2(X, f2(ie)), YS = mul2(Y, f2(ie));
    NearParams<float> nps = np;
    nps.eps2 = 1.f;
    nps.inv_eps2 = 1.f;
    nps.close2 = 1.f / 64.f;
    const float margin = 1e-4f * eps + 1e-5f;
    const float reach = eps + margin;
    const float reach2 = reach * reach;
    const float close_reach = sqrtf(np.close2) + margin;
    const float close_reach2 = close_reach * close_reach;
    const unsigned below = (1u << lane) - 1u;
    int nf = 0, nc = 0;
    op.init();
    // the 3 x 3 cells around the item's (cells are at least eps_I wide), one per lane: those with
    // points and within reach of the box
    int c_j0 = 0, c_j1 = 0;
    float c_ox = 0.f, c_oy = 0.f;                 // step from the cell's frame to the item's
    if (lane < 9) {
        const int ex = c1 - 1 + lane / 3, ey = c2 - 1 + lane % 3;
        c_ox = (float)(c1 - ex) * h;
        c_oy = (float)(c2 - ey) * h;
        const float gapx = fmaxf(0.f, fmaxf(-c_ox - tx1, tx0 - (h - c_ox)));
        const float gapy = fmaxf(0.f, fmaxf(-c_oy - ty1, ty0 - (h - c_oy)));
        if (ex >= 0 && ex < cg.n_c && ey >= 0 && ey < cg.n_c && gapx * gapx + gapy * gapy <= reach2) {
            const int kbase = cg.key(ex, ey) * kSub;
            c_j0 = sd.oth_start[kbase];
            c_j1 = sd.oth_start[kbase + kSub];
        }
    }
    unsigned cells = __ballot_sync(0xffffffffu, c_j0 < c_j1);
    // their points in chunks of 32, each chunk's loads issued while the one before is listed
    int jb = 0, j1 = 0;
    float offx = 0.f, offy = 0.f;
    auto next_cell = [&]() {
        const int c = cells ? __ffs(cells) - 1 : 31;   // lane 31: an empty range
        cells &= cells - 1;
        jb = __shfl_sync(0xffffffffu, c_j0, c);
        j1 = __shfl_sync(0xffffffffu, c_j1, c);
        offx = __shfl_sync(0xffffffffu, c_ox, c);
        offy = __shfl_sync(0xffffffffu, c_oy, c);
    };
    float2 ny = make_float2(0.f, 0.f);
    float nq[R];
#pragma unroll
    for (int r = 0; r < R; ++r)
        nq[r] = 0.f;
    auto load = [&]() {
        if (jb + lane < j1) {
            ny = __ldg(sd.oth_hi + jb + lane);
            op.fetch(jb + lane, nq);
        }
    };
    next_cell();
    load();
    while (jb < j1) {
        const float2 yh = ny;
        const int j = jb + lane;
        const bool in = j < j1;
        const float ox = offx, oy = offy;
        float qv[R];
#pragma unroll
        for (int r = 0; r < R; ++r)
            qv[r] = nq[r];
        jb += 32;
        if (jb >= j1)
            next_cell();
        load();
        const float fx = ox - yh.x, fy = oy - yh.y;   // -(source in the item's frame)
        const float gx = fmaxf(0.f, fmaxf(-fx - tx1, tx0 + fx));
        const float gy = fmaxf(0.f, fmaxf(-fy - ty1, ty0 + fy));
        const float g2 = gx * gx + gy * gy;
        const bool keep = in && g2 <= reach2, close = in && g2 <= close_reach2;
        const unsigned mc = __ballot_sync(0xffffffffu, close), mf = __ballot_sync(0xffffffffu, keep) & ~mc;
        if (keep && !close)   // -(source in the item's frame), in units of eps_I
            L.put(nf + __popc(mf & below), fx * ie, fy * ie, qv);
        nf += __popc(mf);
        if (nf > kListCap - 32) {
            nf = L.pad(nf, 4 * groups, lane);
            __syncwarp();
            near_eval_far(L.x, L.y, L.q, nf, g, groups, XS, YS, nps, op);
            nf = 0;
            __syncwarp();
        }
        if (mc) {
            if (close) {
                const float2 yl = __ldg(sd.oth_lo + j);
                // -(source in the item's frame) = off - y_hi - y_lo as hi + lo (TwoSum of off and -y_hi)
                const float bx = fx - ox, by = fy - oy;
                const float lx = ((ox - (fx - bx)) + (-yh.x - bx)) - yl.x;
                const float ly = ((oy - (fy - by)) + (-yh.y - by)) - yl.y;
                L.put_close(nc + __popc(mc & below), fx, fy, lx, ly, qv);
            }
            nc += __popc(mc);
            if (nc > kCloseCap - 32) {
                nc = L.pad_close(nc, 4 * groups, lane);
                __syncwarp();
                near_eval_close(L.cx, L.cy, L.lx, L.ly, L.cq, nc, g, groups, X, Y, XL, YL, ie, nps, op);
                nc = 0;
                __syncwarp();
            }
        }
    }
    nf = L.pad(nf, 4 * groups, lane);
    nc = L.pad_close(nc, 4 * groups, lane);
    __syncwarp();
    near_eval_far(L.x, L.y, L.q, nf, g, groups, XS, YS, nps, op);
    near_eval_close(L.cx, L.cy, L.lx, L.ly, L.cq, nc, g, groups, X, Y, XL, YL, ie, nps, op);
    op.fold();
    for (int o = 16; o >= lanes; o >>= 1)
        op.reduce(o);
    if (valid && g == 0)
        op.store(k);
}

__device__ __forceinline__ float lane_add(float v, int o) { return v + __shfl_xor_sync(0xffffffffu, v, o); }

// Warps per block of the candidate-list kernels (a warp per item).  An Op's kMinBlocks counts
// blocks of four warps.
constexpr int kNearWarps = 4;
template <class Op>
__global__ void __launch_bounds__(32 * kNearWarps, Op::kMinBlocks * 4 / kNearWarps) k_near_list(int64_t n_items, const int2 *__restrict__ items,
                                                                   int lanes, NearSides sd, CellGrid cg,
                                                                   NearParams<float> np, Op op)
{
    __shared__ __align__(16) NearList<Op::kR> L[kNearWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (warp >= n_items)
        return;                                   // whole warp past the end; no block-wide barrier follows
    near_traverse_list(items[warp], lanes, lane, sd, cg, np, op, L[w]);
}

template <class Op> cudaError_t launch_near_list(int64_t n_items, const int2 *items, int lanes, const NearSides &sd,
                                                 CellGrid cg, const NearParams<float> &np, const Op &op,
                                                 cudaStream_t st)
{
    if (n_items <= 0)
        return cudaSuccess;
    const unsigned blocks = (unsigned)((n_items + kNearWarps - 1) / kNearWarps);
    k_near_list<Op><<<blocks, 32 * kNearWarps, 0, st>>>(n_items, items, lanes, sd, cg, np, op);
    return cudaGetLastError();
}

// ---- source-major forward near field (FP32), for plans with many more sources than targets
//
// FEM plans put several quadrature points around every node, so a cell holds few targets and
// a target item's box would be large.  Here a warp takes a piece of at most 64 sources of one
// cell and keeps them in shared memory as packed pairs; it reads the targets of the 3 x 3 cells
// around 32 at a time, lists those within reach of the sources' box (those within eps_I / 8 of it in a
// second list, hi + lo), and each lane then takes one listed target and sums the item's sources
// on it, two per packed operation; phi, grad phi and the coincident charge are added to the target
// with atomics.  The pair arithmetic is NearFwd's.
// Measured, disc mesh of 50,311 nodes and 301,086 quadrature points (p = 6): 101 us with runs of the
// Morton order and a branch per close pair, 72 us here (items of 32 sources 76 us).
constexpr int kSrcMajorCap = 128, kSrcMajorClose = 64;   // listed targets per warp

struct NearSources {
    float4 xy[32];                    // (xa, xb, ya, yb) of the pairs, units of eps_I
    float4 hi[32], lo[32];            // the same as hi and lo parts (torus units)
    float2 q[32];
    float4 far[kSrcMajorCap];         // listed targets: x, y (units of eps_I), index
    float4 close[kSrcMajorClose];     // x, y as hi parts, then lo parts (torus units)
    int close_k[kSrcMajorClose];
};

// The sums of a lane's target: phi in units of c_ln (P >= 2), the gradient of rcoef.
struct NearSrcSums {
    float2 phi, gx, gy;
};

template <int P>
__device__ __forceinline__ void near_src_pair(const NearParams<float> &np, float2 w, float2 dx, float2 dy, float2 q2,
                                              NearSrcSums &a)
{
    float2 val, coef;
    if constexpr (P >= 2) {
        const float2 s = fma2(w, f2(-1.f), f2(1.f)), lw = lg2_2(w);
        val = near_g2<P>(np, w, s, lw);
        if constexpr (P >= 5)
            coef = ex2_2(fma2(f2((float)(P - 1)), lg2_2(s), make_float2(-lw.x, -lw.y)));
        else
            coef = mul2(ipow2<P - 1>(s), rcp_2(w));
    } else {
        val = near_f2<P>(np, w);
        coef = rcp_2(w);
        q2 = select2(w, 1.f, q2);
    }
    a.phi = fma2(q2, val, a.phi);
    const float2 tq = mul2(q2, coef);
    a.gx = fma2(tq, dx, a.gx);
    a.gy = fma2(tq, dy, a.gy);
}

template <int P>
__device__ __forceinline__ void near_src_add(const NearSrcSums &a, int k, float cq, float rcoef,
                                             float *__restrict__ phi_s, float *__restrict__ grad_s,
                                             float *__restrict__ coinc)
{
    const float rc = (P >= 2 && (P - 1) % 2 == 1) ? -rcoef : rcoef;   // coef is |w - 1|^(p-1) / w
    atomicAdd(phi_s + k, (P >= 2 ? kLnCoef : 1.f) * (a.phi.x + a.phi.y));
    atomicAdd(grad_s + 2 * (int64_t)k, rc * (a.gx.x + a.gx.y));
    atomicAdd(grad_s + 2 * (int64_t)k + 1, rc * (a.gy.x + a.gy.y));
    if (cq != 0.f)
        atomicAdd(coinc + k, cq);
}

template <int P>
__device__ __forceinline__ void near_src_far(const NearSources &S, int n, int pairs, int lane,
                                             const NearParams<float> &np, float rcoef, float *__restrict__ phi_s,
                                             float *__restrict__ grad_s, float *__restrict__ coinc)
{
    for (int base = 0; base < n; base += 32) {
        const bool valid = base + lane < n;
        const float4 T = valid ? S.far[base + lane] : make_float4(kPadPos, kPadPos, 0.f, 0.f);
        NearSrcSums a;
        a.phi = a.gx = a.gy = f2(0.f);
#pragma unroll 8
        for (int i = 0; i < pairs; ++i) {
            const float4 s = S.xy[i];
            const float2 dx = add2(f2(T.x), make_float2(-s.x, -s.y)), dy = add2(f2(T.y), make_float2(-s.z, -s.w));
            near_src_pair<P>(np, near_w2(P >= 2, dx, dy), dx, dy, S.q[i], a);
        }
        if (valid)
            near_src_add<P>(a, __float_as_int(T.z), 0.f, rcoef, phi_s, grad_s, coinc);
    }
}

template <int P>
__device__ __forceinline__ void near_src_close(const NearSources &S, int n, int pairs, int lane, float ie,
                                               const NearParams<float> &np, float rcoef, float *__restrict__ phi_s,
                                               float *__restrict__ grad_s, float *__restrict__ coinc)
{
    for (int base = 0; base < n; base += 32) {
        const bool valid = base + lane < n;
        const float4 T = valid ? S.close[base + lane] : make_float4(kPadPos, kPadPos, 0.f, 0.f);
        NearSrcSums a;
        a.phi = a.gx = a.gy = f2(0.f);
        float cq = 0.f;
        for (int i = 0; i < pairs; ++i) {
            const float4 h = S.hi[i], l = S.lo[i];
            const float2 q2 = S.q[i];
            const float2 ex = add2(add2(f2(T.x), make_float2(-h.x, -h.y)), add2(f2(T.z), make_float2(-l.x, -l.y)));
            const float2 ey = add2(add2(f2(T.y), make_float2(-h.z, -h.w)), add2(f2(T.w), make_float2(-l.z, -l.w)));
            const float2 dx = mul2(ex, f2(ie)), dy = mul2(ey, f2(ie));
            float2 w = near_w2(P >= 2, dx, dy);
            const bool z0 = ex.x == 0.f && ey.x == 0.f, z1 = ex.y == 0.f && ey.y == 0.f;
            if (z0 || z1) {
                // coincident: G(0) := 0; an idle second source has charge 0
                const float qs = (z0 ? q2.x : 0.f) + (z1 ? q2.y : 0.f);
                a.phi.x -= qs * (np.beta[0] / (P >= 2 ? kLnCoef : 1.f));
                cq += qs;
                w.x = z0 ? 1.f : w.x;
                w.y = z1 ? 1.f : w.y;
            }
            near_src_pair<P>(np, w, dx, dy, q2, a);
        }
        if (valid)
            near_src_add<P>(a, S.close_k[base + lane], cq, rcoef, phi_s, grad_s, coinc);
    }
}

template <int P>
__global__ void __launch_bounds__(128) k_near_src32(int64_t n_items, const int2 *__restrict__ items, NearSides sd,
                                                    CellGrid cg, NearParams<float> np, const float *__restrict__ q,
                                                    float *__restrict__ phi_s, float *__restrict__ grad_s,
                                                    float *__restrict__ coinc)
{
    __shared__ NearSources all[4];
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (warp >= n_items)
        return;                                   // whole warp past the end; no block-wide barrier follows
    NearSources &S = all[threadIdx.x >> 5];
    const int2 item = items[warp];
    // pair i: the item's sources i and i + pairs (own side); an idle second one copies the first
    // source with charge 0
    const int pairs = (item.y + 1) / 2;
    const int64_t ja = item.x + (lane < pairs ? lane : 0);
    const bool vb = lane < pairs && lane + pairs < item.y;
    const int64_t jb = vb ? ja + pairs : item.x;
    const float2 ha = sd.own_hi[ja], hb = sd.own_hi[jb], la = sd.own_lo[ja], lb = sd.own_lo[jb];
    const float ie = sqrtf(np.inv_eps2);
    S.hi[lane] = make_float4(ha.x, hb.x, ha.y, hb.y);
    S.lo[lane] = make_float4(la.x, lb.x, la.y, lb.y);
    S.xy[lane] = make_float4(ha.x * ie, hb.x * ie, ha.y * ie, hb.y * ie);
    S.q[lane] = make_float2(__ldg(q + ja), vb ? __ldg(q + jb) : 0.f);
    const int packed = sd.own_base[item.x];
    const int c1 = base1(packed) / cg.cell, c2 = base2(packed) / cg.cell;
    const float h = np.hcell, eps = sqrtf(np.eps2);
    // the sources' box in the item's frame (offsets from the item cell's corner)
    const float lx = warp_min(fminf(ha.x, hb.x)), hx = warp_max(fmaxf(ha.x, hb.x));
    const float ly = warp_min(fminf(ha.y, hb.y)), hy = warp_max(fmaxf(ha.y, hb.y));
    const float margin = 1e-4f * eps + 1e-5f;
    const float reach = eps + margin, reach2 = reach * reach;
    const float close_reach = sqrtf(np.close2) + margin, close_reach2 = close_reach * close_reach;
    const unsigned below = (1u << lane) - 1u;
    const float rcoef = np.rcoef * eps;           // the differences are in units of eps_I
    __syncwarp();
    int nf = 0, nc = 0;
    for (int e1 = max(c1 - 1, 0); e1 <= min(c1 + 1, cg.n_c - 1); ++e1) {
        const float ox = (float)(e1 - c1) * h;        // cell step into the item's frame
        const float gxc = fmaxf(0.f, fmaxf(ox - hx, lx - (ox + h)));
        for (int e2 = max(c2 - 1, 0); e2 <= min(c2 + 1, cg.n_c - 1); ++e2) {
            const float oy = (float)(e2 - c2) * h;
            const float gyc = fmaxf(0.f, fmaxf(oy - hy, ly - (oy + h)));
            if (gxc * gxc + gyc * gyc > reach2)
                continue;                             // the whole cell is beyond reach (warp-uniform)
            const int kbase = cg.key(e1, e2) * kSub;
            const int j0 = sd.oth_start[kbase], j1 = sd.oth_start[kbase + kSub];
            for (int jb0 = j0; jb0 < j1; jb0 += 32) {
                const int j = jb0 + lane;
                float2 th = make_float2(0.f, 0.f);
                if (j < j1)
                    th = __ldg(sd.oth_hi + j);
                const float tx = ox + th.x, ty = oy + th.y;
                const float dxb = fmaxf(0.f, fmaxf(tx - hx, lx - tx));
                const float dyb = fmaxf(0.f, fmaxf(ty - hy, ly - ty));
                const float g2 = j < j1 ? dxb * dxb + dyb * dyb : 3e38f;
                const bool keep = g2 <= reach2, close = g2 <= close_reach2;
                const unsigned mc = __ballot_sync(0xffffffffu, close), mf = __ballot_sync(0xffffffffu, keep) & ~mc;
                if (keep && !close)
                    S.far[nf + __popc(mf & below)] = make_float4(tx * ie, ty * ie, __int_as_float(j), 0.f);
                nf += __popc(mf);
                if (nf > kSrcMajorCap - 32) {
                    __syncwarp();
                    near_src_far<P>(S, nf, pairs, lane, np, rcoef, phi_s, grad_s, coinc);
                    nf = 0;
                    __syncwarp();
                }
                if (mc) {
                    if (close) {
                        const int at = nc + __popc(mc & below);
                        const float2 tl = __ldg(sd.oth_lo + j);
                        // step + hi + lo as hi + lo (TwoSum of the step and hi)
                        const float bx = tx - ox, by = ty - oy;
                        S.close[at] = make_float4(tx, ty, ((ox - (tx - bx)) + (th.x - bx)) + tl.x,
                                                  ((oy - (ty - by)) + (th.y - by)) + tl.y);
                        S.close_k[at] = j;
                    }
                    nc += __popc(mc);
                    if (nc > kSrcMajorClose - 32) {
                        __syncwarp();
                        near_src_close<P>(S, nc, pairs, lane, ie, np, rcoef, phi_s, grad_s, coinc);
                        nc = 0;
                        __syncwarp();
                    }
                }
            }
        }
    }
    __syncwarp();
    near_src_far<P>(S, nf, pairs, lane, np, rcoef, phi_s, grad_s, coinc);
    near_src_close<P>(S, nc, pairs, lane, ie, np, rcoef, phi_s, grad_s, coinc);
}

// Calls f(std::integral_constant<int, P>) for the expansion degree p in 1..16.
template <class F> cudaError_t with_degree(int p, F &&f)
{
    switch (p) {
#define FS_P_CASE(P)                                                                                             \
    case P:                                                                                                      \
        return f(std::integral_constant<int, P>{});
        FS_P_CASE(1)
        FS_P_CASE(2)
        FS_P_CASE(3)
        FS_P_CASE(4)
        FS_P_CASE(5)
        FS_P_CASE(6)
        FS_P_CASE(7)
        FS_P_CASE(8)
        FS_P_CASE(9)
        FS_P_CASE(10)
        FS_P_CASE(11)
        FS_P_CASE(12)
        FS_P_CASE(13)
        FS_P_CASE(14)
        FS_P_CASE(15)
        FS_P_CASE(16)
#undef FS_P_CASE
    default:
        return cudaErrorInvalidValue;
    }
}

}  // namespace fs
