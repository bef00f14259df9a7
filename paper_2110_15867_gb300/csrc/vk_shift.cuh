// vk_shift.cuh -- the FP32 march of position sweeps that shift whole cells (sweep_shift32.cu,
// sweep_strided.cu).
#pragma once

#include "vk_common.cuh"

namespace vk {

// The FP32 march of these sweeps, with the flux written in the cells themselves (34
// operations a face) where every other kernel takes differences (31): over a drift of
// whole-cell shifts the two forms' roundings, both right to 7e-8 of the 2-norm, were driven
// apart in single cells by the limiter (3e-5 of the rms after six sweeps), more than these
// sweeps' results may change.  What that costs was measured one line per thread: 4 % (32 x 24 x 32
// x 16 x 16 x 32 cells: 1.665 against 1.597 ms, three sweeps); in pairs, now 1.020 ms, it is not known.
// X = float: one line; float2: two lines as f32x2 pairs, the same operations one by one.
template <typename X> struct CellCoef { // weights of fbar, Courant fraction, f_UL's factor
    X w[5], s, alpha;
};
__device__ __forceinline__ CellCoef<float> to_cell(const LineCoefT<float> &k)
{
    return CellCoef<float>{{k.w[0], k.w[1], k.w[2], k.w[3], k.w[4]}, k.s, k.alpha};
}
__device__ __forceinline__ CellCoef<float2> to_cell2(const LineCoefT<float> &a, const LineCoefT<float> &b)
{
    CellCoef<float2> k;
#pragma unroll
    for (int m = 0; m < 5; ++m) k.w[m] = make_float2(a.w[m], b.w[m]);
    k.s = make_float2(a.s, b.s);
    k.alpha = make_float2(a.alpha, b.alpha);
    return k;
}
template <typename X> __device__ __forceinline__ X cell_curv(X a, X b, X c) { return vadd(vfma(splat<X>(-2.0), b, a), c); }
template <typename X> __device__ __forceinline__ X minmod_curv(X d0, X d1)
{
    const X a = vsub(vmul(splat<X>(4.0), d0), d1), b = vsub(vmul(splat<X>(4.0), d1), d0); // (4 x is exact)
    return mn2(mx2(mn2(mn3(a, b, d0), d1), splat<X>(0.0)), mx2(mx3(a, b, d0), d1));
}
template <typename X>
__device__ __forceinline__ X cell_flux(const CellCoef<X> &k, X cm2, X cm1, X c0, X cp1, X cp2, X dm4m, X dm4p)
{
    const X fbar = vfma(k.w[4], cp2, vfma(k.w[3], cp1, vfma(k.w[2], c0, vfma(k.w[1], cm1, vmul(k.w[0], cm2)))));
    const X dlm = vsub(c0, cm1), ful = vfma(k.alpha, dlm, c0), fmd = vmul(splat<X>(0.5), vsub(vadd(c0, cp1), dm4p));
    const X flc = vfma(splat<X>(4.0 / 3.0), dm4m, vfma(splat<X>(0.5), dlm, c0));
    const X v = mn3(mx3(fbar, mn3(c0, cp1, fmd), mn3(c0, ful, flc)), mx3(c0, cp1, fmd), mx3(c0, ful, flc));
    return flux_clamp(vmul(k.s, v), c0);
}
// periodic line in place
__device__ __forceinline__ float march_shift(float *p, long step, int L, const LineCoefT<float> &kc)
{
    const CellCoef<float> k = to_cell(kc);
    const float s0 = p[0], s1 = p[step], a = p[(long)(L - 3) * step];
    float cm2 = p[(long)(L - 2) * step], cm1 = p[(long)(L - 1) * step], c0 = s0, cp1 = s1, sum = 0.f;
    const float dm = cell_curv(cm2, cm1, s0);
    float d = cell_curv(cm1, s0, s1), q = minmod_curv(dm, d);
    float Fm = cell_flux(k, a, cm2, cm1, s0, s1, minmod_curv(cell_curv(a, cm2, cm1), dm), q); // face -1/2, donor c_{-1}
    auto face = [&](int i, float cp2) {
        const float dn = cell_curv(c0, cp1, cp2), qp = minmod_curv(d, dn);
        const float F = cell_flux(k, cm2, cm1, c0, cp1, cp2, q, qp);
        const float out = c0 + (Fm - F);
        p[(long)i * step] = out;
        sum += out;
        cm2 = cm1;
        cm1 = c0;
        c0 = cp1;
        cp1 = cp2;
        d = dn;
        q = qp;
        Fm = F;
    };
#pragma unroll 4
    for (int i = 0; i < L - 2; ++i) face(i, p[(long)(i + 2) * step]);
    face(L - 2, s0);
    face(L - 1, s1);
    return sum;
}
// The same walked from its last cell down, with every new value written N
// cells on (0 <= N <= kStash, N < L): each row is read once and written once, where marching
// in place and rotating the line afterwards (three reversals) read and wrote it three times.
// Row i + N has been read when cell i is done; the N values that wrap around to the first
// rows, still to be read, wait in `held`, and the last three cells, overwritten before the
// first ones need them, in registers.  The values are march_shift's, face by face.
// The values are what one line alone gives, and a pair's lines may shift by different N.
template <typename X> struct ShiftPut;
template <> struct ShiftPut<float> { // where the next cell down goes; past the line's end it wraps to row to - L
    int to;
    __device__ __forceinline__ void put(float *p, int step, int L, float *held, float v)
    {
        if (to < L) p[to * step] = v;
        else held[to - L] = v;
        --to;
    }
};
template <> struct ShiftPut<float2> {
    int to, to2;
    __device__ __forceinline__ void put(float2 *p, int step, int L, float2 *held, float2 v)
    {
        if (to == to2) {
            if (to < L) p[to * step] = v;
            else held[to - L] = v;
        } else {
            if (to < L) p[to * step].x = v.x;
            else held[to - L].x = v.x;
            if (to2 < L) p[to2 * step].y = v.y;
            else held[to2 - L].y = v.y;
        }
        --to;
        --to2;
    }
};
// rows of cells at p + r step (in X)
template <typename X>
__device__ __forceinline__ X shift_walk(X *p, int step, int L, ShiftPut<X> where, X *held, const CellCoef<X> &k)
{
    const X e3 = p[(L - 3) * step], e2 = p[(L - 2) * step], e1 = p[(L - 1) * step];
    const X s0 = p[0], s1 = p[step];
    X sum = splat<X>(0.0);
    // face i + 1/2 from its upper side: donor c0 = cell i, cm1 = i - 1, ... ; start at i = L - 1
    X cp1 = s0, c0 = e1, cm1 = e2, cm2 = e3;
    X d = cell_curv(cm1, c0, cp1), dm = cell_curv(cm2, cm1, c0); // curvatures of cells i, i - 1
    X q = minmod_curv(dm, d);                                    // at face i - 1/2
    X Fp = cell_flux(k, cm2, cm1, c0, cp1, s1, q, minmod_curv(d, cell_curv(c0, cp1, s1)));
    auto cell = [&](X cm3) { // the next cell i down, with cell i - 3
        const X dmm = cell_curv(cm3, cm2, cm1), qm = minmod_curv(dmm, dm);
        const X F = cell_flux(k, cm3, cm2, cm1, c0, cp1, qm, q); // face i - 1/2, donor cell i - 1
        const X out = vadd(c0, vsub(F, Fp));
        sum = vadd(sum, out);
        cp1 = c0;
        c0 = cm1;
        cm1 = cm2;
        cm2 = cm3;
        dm = dmm;
        q = qm;
        Fp = F;
        return out;
    };
    const X *below = p + (L - 4) * step; // cell i - 3
#pragma unroll 4
    for (int i = L - 1; i >= 3; --i, below -= step) where.put(p, step, L, held, cell(*below));
    where.put(p, step, L, held, cell(e1));
    where.put(p, step, L, held, cell(e2));
    where.put(p, step, L, held, cell(e3));
    return sum;
}
__device__ __forceinline__ float march_shift_down(float *p, int step, int L, int N, const LineCoefT<float> &k)
{
    float held[kStash];
    const float sum = shift_walk<float>(p, step, L, ShiftPut<float>{L - 1 + N}, held, to_cell(k));
    for (int j = 0; j < N; ++j) p[j * step] = held[j];
    return sum;
}
// two adjacent columns
__device__ __forceinline__ float2 march_shift_down(float2 *p, int step, int L, int N, int N2, const LineCoefT<float> &k,
                                                   const LineCoefT<float> &k2)
{
    float2 held[kStash];
    const float2 sum = shift_walk<float2>(p, step, L, ShiftPut<float2>{L - 1 + N, L - 1 + N2}, held, to_cell2(k, k2));
    for (int j = 0; j < N; ++j) p[j * step].x = held[j].x;
    for (int j = 0; j < N2; ++j) p[j * step].y = held[j].y;
    return sum;
}

} // namespace vk
