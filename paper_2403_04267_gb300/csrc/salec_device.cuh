// salec_device.cuh -- device helpers shared by the phase kernels (salec_kernels.cu) and
// the fused tile kernel (salec_fused.cu): block reductions, the absorbing strip's row
// mask, the cell geometry of uniform and non-uniform grids, and the dual-face fluxes of
// the momentum remap.
#pragma once

#include "salec_internal.cuh"

namespace salec {

__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// block-wide sum, result valid in thread 0 (blocks are whole warps, at most kMaxThreads)
static __device__ double block_sum(double v, double* sh)
{
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int nw = (blockDim.x * blockDim.y) >> 5;
    v = warp_sum(v);
    __syncthreads();
    if ((tid & 31) == 0) sh[tid >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (tid == 0)
        for (int w = 0; w < nw; ++w) s += sh[w];
    return s;
}

// The right absorbing strip acts on the rows whose reference (far-field) state holds
// material: the medium whose waves it absorbs.  Above the target the reference is void and
// damping toward it would remove ejecta, so there it does nothing (cells: row j; vertices:
// either adjacent cell row).
template <typename T>
__device__ __forceinline__ bool strip_row_c(const PtrsT<T>& p, int j) { return pos(p.rho_ref[j]); }
template <typename T>
__device__ __forceinline__ bool strip_row_v(const PtrsT<T>& p, int j, int nz)
{
    return (j > 0 && pos(p.rho_ref[j - 1])) || (j < nz && pos(p.rho_ref[j]));
}

// ---------------------------------------------------------------------------------
// Cell geometry per radian.  A non-uniform grid (UNI = false) takes a cell's volume and
// radial faces as a column entry times its row height: V = r_c dr dz, A_R = r_i dz; a
// uniform grid of dx cells (UNI = true) keeps one entry per column for every row, which
// spares the FP64 pipe those products.
// ---------------------------------------------------------------------------------
template <typename T, bool UNI>
struct Geo {
    static __device__ __forceinline__ T vol(const ParamsT<T>& P, int i, int j)
    {
        return UNI ? P.p.V[i] : P.p.A_Z[i] * P.p.dz[j];
    }
    static __device__ __forceinline__ T ivol(const ParamsT<T>& P, int i, int j)
    {
        return UNI ? P.p.invV[i] : P.p.invAZ[i] * P.p.idz[j];
    }
    // radial face area at r_i of row j
    static __device__ __forceinline__ T area_r(const ParamsT<T>& P, int i, int j)
    {
        return UNI ? P.p.A_R[i] : P.p.rR[i] * P.p.dz[j];
    }
    // net radial volume flux A_R(i+1) uR - A_R(i) uL of cell (i,j)
    static __device__ __forceinline__ T flux_r(const ParamsT<T>& P, int i, int j, T uL, T uR)
    {
        return UNI ? P.p.A_R[i + 1] * uR - P.p.A_R[i] * uL : P.p.dz[j] * (P.p.rR[i + 1] * uR - P.p.rR[i] * uL);
    }
    static __device__ __forceinline__ T idr(const ParamsT<T>& P, int i) { return UNI ? P.idx : P.p.idr[i]; }
    static __device__ __forceinline__ T idz(const ParamsT<T>& P, int j) { return UNI ? P.idx : P.p.idz[j]; }
    // the cell's length scale L = min(dr, dz) and 1 / L
    static __device__ __forceinline__ T len(const ParamsT<T>& P, int i, int j)
    {
        if (UNI) return P.dx;
        const T a = P.p.dr[i], b = P.p.dz[j];
        return a < b ? a : b;
    }
    static __device__ __forceinline__ T ilen(const ParamsT<T>& P, int i, int j)
    {
        if (UNI) return P.idx;
        const T a = P.p.idr[i], b = P.p.idz[j];
        return a > b ? a : b;
    }
    // derivatives of the cell's stress power V S:e with respect to its corner velocities:
    // V / (2 dr) for r-derivatives, V / (4 r_c) for the hoop strain rate
    static __device__ __forceinline__ T half_v_dr(const ParamsT<T>& P, int i, int j)
    {
        return UNI ? T(0.5) * P.p.A_Z[i] : T(0.5) * P.p.rc[i] * P.p.dz[j];
    }
    static __device__ __forceinline__ T quarter_v_rc(const ParamsT<T>& P, int i, int j)
    {
        return UNI ? T(0.25) * P.dx2 : T(0.25) * P.p.dr[i] * P.p.dz[j];
    }
};

// The Courant rate (|v| + c) / L of a cell only counts where it raises the running maximum,
// and in the FP64 form its two square roots and four vertex speeds are a third of phase 0's
// work on the FP64 pipe.  An upper bound in FP32 (from the high words, integer
// instructions) decides first: warps none of whose cells can exceed the maximum seen so far
// skip the FP64 evaluation.  The maximum that results is the same.
__host__ __device__ __forceinline__ float f32_of_bits(int b)
{
#ifdef __CUDA_ARCH__
    return __int_as_float(b);
#else
    float f;
    memcpy(&f, &b, 4);
    return f;
#endif
}
__host__ __device__ __forceinline__ float up_f32(double x)       // >= |x|; +inf for NaN and from 2^127 on
{
    const int h = high_word(x) & 0x7fffffff;
    if (h < 0x38200000) return 2.4e-38f;                         // below 2^-125 = 2.351e-38
    if (h >= 0x47e00000) return f32_of_bits(0x7f800000);
    return f32_of_bits(((h - 0x38000000) << 3) + 16);
}
__host__ __device__ __forceinline__ float down_f32(double x)     // <= x for x >= 0
{
    const int h = high_word(x);
    if (h < 0x38200000) return 0.0f;
    if (h >= 0x47e00000) return 1.7e38f;                         // from 2^127 = 1.701e38 on
    return f32_of_bits((h - 0x38000000) << 3);
}
__device__ __forceinline__ float up_w(double2 v)
{
    const float x = up_f32(v.x), y = up_f32(v.y);
    return __fmaf_ru(x, x, __fmul_ru(y, y));
}
__device__ __forceinline__ float up_w(float2) { return 0.0f; }
// whether (|v| + c) / L of a cell with squared sound speed c2 and corner velocities va.. vd may
// exceed `run` (the mixed form always evaluates: its square roots are cheap)
template <typename T, typename T2>
__device__ __forceinline__ bool rate_may_raise(T2 va, T2 vb, T2 vc, T2 vd, T c2, T ilen, bool scaled, double run)
{
    if (sizeof(T) == 4) return true;
    const float w = fmaxf(fmaxf(up_w(va), up_w(vb)), fmaxf(up_w(vc), up_w(vd)));
    float r = __fadd_ru(__fsqrt_ru(w), __fsqrt_ru(up_f32(double(c2))));
    if (scaled) r = __fmul_ru(r, up_f32(double(ilen)));
    return !(r <= down_f32(run));
}

// a / b with y close to 1 / b (a few units in the last place: on a non-uniform grid both y and b
// are products, each rounded): the quotient corrected by its remainder (Markstein, IBM J. Res.
// Dev. 34, 1990), three instructions on the FP64 pipe instead of a division's ten.  Exactly 1
// for a == b, otherwise within 0.5 + 2^-40 units in the last place of the true quotient; an
// infinite a gives infinity, as the division does.
__host__ __device__ __forceinline__ double div_by(double a, double b, double y)
{
    const double q = a * y, c = fma(fma(-q, b, a), y, q);
    return (high_word(q) & 0x7ff00000) == 0x7ff00000 ? q : c;
}
__device__ __forceinline__ float div_by(float a, float b, float) { return a / b; }

__device__ __forceinline__ bool finite_pos(double x) { return __double_as_longlong(x) > 0 && __double2hiint(x) < 0x7ff00000; }
__device__ __forceinline__ bool finite_pos(float x) { return __float_as_int(x) > 0 && __float_as_int(x) < 0x7f800000; }

// What a dual face carries: mass f, momentum f w and kinetic energy f |w|^2 / 2 with the
// upwind vertex velocity w.
template <typename T>
struct DualFace {
    T f, fr, fz, e;
};
// products rounded as written (never fused into a multiply-add with their later use), so
// that a face computed by either of its vertices, or read from the other, is the same
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
template <typename T>
__device__ __forceinline__ DualFace<T> dual_face(T f, typename VT<T>::T2 w)
{
    DualFace<T> d;
    d.f = f;
    d.fr = mul_rn(f, w.x);
    d.fz = mul_rn(f, w.y);
    d.e = mul_rn(mul_rn(T(0.5), f), add_rn(mul_rn(w.x, w.x), mul_rn(w.y, w.y)));
    return d;
}

// Net fluxes of a cell's remap: material volumes and masses, stress and damage contents,
// and the energy change of the inflows.
template <typename T, int NM>
struct Acc {
    T Vm[NM], Mm[NM], S[4];
    T dI;        // sum over inflows of (I_donor - I^L) * mass (the remap's energy change)
};

}  // namespace salec
