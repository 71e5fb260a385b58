// Device helpers of the kernels whose threads hold one species at two adjacent
// sites (lb_tiled.cuh, lb_patch.cu): stores of a pair in each storage format and
// the differences of Eq. (FFF) over a window of psi/rho pairs.
#pragma once

#include <type_traits>

#include "lb_common.cuh"

namespace lbhb {

// Stores of two adjacent columns of one species (8 bytes for FP32).
template <class T> struct Vec2;
template <> struct Vec2<float> {
    __device__ static void st(float* p, float a, float b) { *reinterpret_cast<float2*>(p) = make_float2(a, b); }
};
template <> struct Vec2<double> {
    __device__ static void st(double* p, double a, double b) { *reinterpret_cast<double2*>(p) = make_double2(a, b); }
};
template <> struct Vec2<__half> {
    // FP16 storage of shifted values: the caller subtracts the shift
    __device__ static void st(__half* p, float a, float b) { *reinterpret_cast<__half2*>(p) = __floats2half2_rn(a, b); }
};
// stochastically rounded FP16: stores with the thread's dither stream
template <> struct Vec2<half_sr> {
    __device__ static void st(half_sr* p, float a, float b, Dither& d)
    {
        const __half lo = half_sr_round(a, d), hi = half_sr_round(b, d);
        *reinterpret_cast<__half2*>(p) = __halves2half2(lo, hi);
    }
};
// paired and single stores of values already in the stored representation,
// dithered where the storage asks for it
template <class T, class C>
__device__ inline void st_pair(T* p, C a, C b, Dither& d)
{
    if constexpr (Store<T>::dithered)
        Vec2<T>::st(p, a, b, d);
    else
        Vec2<T>::st(p, a, b);
}
template <class T, class C>
__device__ inline void st_one(T* p, C v, Dither& d)
{
    if constexpr (std::is_same<T, half_sr>::value)
        p->h = half_sr_round(v, d);
    else if constexpr (std::is_same<T, __half>::value)
        *p = __float2half_rn(v);
    else
        *p = v;
}

// Element CI (0..5) of a window row of six columns held as three lane pairs.
template <int CI, class C>
__device__ __forceinline__ C win_at(const P2<C> (&row)[3])
{
    return (CI & 1) ? row[CI >> 1].b() : row[CI >> 1].a();
}

// g(r + c) - g(r - c) of Eq. (FFF) for both sites of a thread, c = (DX, DY):
// site o sits at column 2 + o of window row MID.  Pairs at an even column
// offset are the stored pairs (one packed subtraction); odd offsets straddle
// two pairs (two scalar subtractions).
template <int DX, int DY, int MID, int NR, class C>
__device__ __forceinline__ P2<C> pair_diff(const P2<C> (&w)[NR][3])
{
    constexpr int cp = 2 + DX, cm = 2 - DX;
    if constexpr ((DX & 1) == 0)
        return w[MID + DY][cp / 2] - w[MID - DY][cm / 2];
    else
        return P2<C>(win_at<cp>(w[MID + DY]) - win_at<cm>(w[MID - DY]),
                     win_at<cp + 1>(w[MID + DY]) - win_at<cm + 1>(w[MID - DY]));
}

// The half-stencil differences of psi (window rows k-2..k+2) and of the partner
// density rho_s' (rows k-1..k+1, belt 1 only), in the order of hs_dx / hs_dy.
template <class C>
__device__ __forceinline__ void window_diffs(const P2<C> (&v)[5][3], const P2<C> (&e)[3][3], P2<C> d[12],
                                             P2<C> de[4])
{
    d[0] = pair_diff<hs_dx(0), hs_dy(0), 2>(v);
    d[1] = pair_diff<hs_dx(1), hs_dy(1), 2>(v);
    d[2] = pair_diff<hs_dx(2), hs_dy(2), 2>(v);
    d[3] = pair_diff<hs_dx(3), hs_dy(3), 2>(v);
    d[4] = pair_diff<hs_dx(4), hs_dy(4), 2>(v);
    d[5] = pair_diff<hs_dx(5), hs_dy(5), 2>(v);
    d[6] = pair_diff<hs_dx(6), hs_dy(6), 2>(v);
    d[7] = pair_diff<hs_dx(7), hs_dy(7), 2>(v);
    d[8] = pair_diff<hs_dx(8), hs_dy(8), 2>(v);
    d[9] = pair_diff<hs_dx(9), hs_dy(9), 2>(v);
    d[10] = pair_diff<hs_dx(10), hs_dy(10), 2>(v);
    d[11] = pair_diff<hs_dx(11), hs_dy(11), 2>(v);
    de[0] = pair_diff<hs_dx(0), hs_dy(0), 1>(e);
    de[1] = pair_diff<hs_dx(1), hs_dy(1), 1>(e);
    de[2] = pair_diff<hs_dx(2), hs_dy(2), 1>(e);
    de[3] = pair_diff<hs_dx(3), hs_dy(3), 1>(e);
}

// Sum of the u_x of a 32-column group of one row by 32 / NW adjacent lanes of a
// warp, NW consecutive columns each (at(q): a lane's columns), in the first of
// them; one fixed order for every kernel that samples.  FP32 values are carried
// as an unevaluated (hi, lo) pair (error-free two-sum), ~2^-48 relative.
template <int NW, class At> __device__ __forceinline__ double group_sum(int lane, At at)
{
    constexpr int SEG = 32 / NW;
    using C = decltype(at(0));
    if constexpr (sizeof(C) == 4) {
        float hi = at(0), lo = 0.f;
#pragma unroll
        for (int q = 1; q < NW; ++q) {
            const float v = at(q);
            const float sum = __fadd_rn(hi, v);
            const float bp = __fsub_rn(sum, hi);
            lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(sum, bp)), __fsub_rn(v, bp)));
            hi = sum;
        }
#pragma unroll
        for (int o = SEG / 2; o > 0; o >>= 1) {
            const float h2 = __shfl_down_sync(0xffffffffu, hi, o, SEG);
            const float l2 = __shfl_down_sync(0xffffffffu, lo, o, SEG);
            const float sum = __fadd_rn(hi, h2);
            const float bp = __fsub_rn(sum, hi);
            const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(sum, bp)), __fsub_rn(h2, bp));
            hi = sum;
            lo = __fadd_rn(__fadd_rn(lo, l2), err);
        }
        return (double)hi + (double)lo;
    } else {
        double v = 0.0;
#pragma unroll
        for (int q = 0; q < NW; ++q) v += at(q);
#pragma unroll
        for (int o = SEG / 2; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, SEG);
        return v;
    }
}

}  // namespace lbhb
