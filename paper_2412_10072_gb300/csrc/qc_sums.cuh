// qc_sums.cuh -- device code shared by the solves from per-(interval, pair) sums.
#pragma once
#include "qc_jones.cuh"

namespace qc {

// sqrt(tn / td) < tol without the root and the division; 0 where there are no gains (td = 0).  A change of
// exactly zero is below any tolerance but zero, also one whose square underflows.
__device__ __forceinline__ bool converged(double tn, double td, double tol)
{
    return td > 0 && tn != 0 ? tn < tol * tol * td : 0.0 < tol;
}

// Transposed warp reduction of N = 4, 8 or 16 values per lane: each halving exchanges half of the
// values a lane holds; the lanes from 32 / N * i on end with the total of value i.  The sum over
// the lanes is carried as head and tail (Knuth's two-sum, one exact step per level), so the total over
// the antennas is as good as an FP64 sum of the lanes' terms: rounding the tree in FP32 alone is
// one unit in the last place of the whole right-hand side, which JHr = b - JHJ g turns into that
// much of the gains.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = a + b;
    const float z = s - a;
    e = (a - (s - z)) + (b - z);
}
// s + e += a b, the product's and the sum's rounding errors carried in e (Ogita, Rump and Oishi's
// compensated dot product); the multiplications are kept from being contracted into the sum
__device__ __forceinline__ void dot_add(float &s, float &e, float a, float b)
{
    const float p = __fmul_rn(a, b), r = __fmaf_rn(a, b, -p);
    float x;
    two_sum(s, p, s, x);
    e += r + x;
}
// a value as head and tail
struct HT { float hi, lo; };
__device__ __forceinline__ HT dot2(float a, float b, float c, float d)          // a b + c d
{
    const float p = __fmul_rn(a, b), r = __fmaf_rn(a, b, -p);
    const float q = __fmul_rn(c, d), t = __fmaf_rn(c, d, -q);
    HT v;
    float x;
    two_sum(p, q, v.hi, x);
    v.lo = (r + t) + x;
    return v;
}
__device__ __forceinline__ void dot_add(float &s, float &e, HT a, float b)
{
    dot_add(s, e, a.hi, b);
    e = fmaf(a.lo, b, e);
}
__device__ __forceinline__ HT neg(HT a) { return { -a.hi, -a.lo }; }

// the tails tail[N] of the values come in with them
template <int N> __device__ __forceinline__ double reduce_words(float (&h)[N], float (&t)[N], int lane)
{
    int o = 16;
#pragma unroll
    for (int n = N / 2; n >= 1; n >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float send = up ? h[i] : h[i + n], keep = up ? h[i + n] : h[i];
            const float ts = up ? t[i] : t[i + n];
            const float tail = (up ? t[i + n] : t[i]) + __shfl_xor_sync(0xffffffffu, ts, o);
            float e;
            two_sum(keep, __shfl_xor_sync(0xffffffffu, send, o), h[i], e);
            t[i] = tail + e;
        }
    }
#pragma unroll
    for (; o >= 1; o >>= 1) {
        const float tail = t[0] + __shfl_xor_sync(0xffffffffu, t[0], o);
        float e;
        two_sum(h[0], __shfl_xor_sync(0xffffffffu, h[0], o), h[0], e);
        t[0] = tail + e;
    }
    return (double)h[0] + (double)t[0];
}
template <int N> __device__ __forceinline__ double reduce_words(float (&h)[N], int lane)
{
    float t[N];
#pragma unroll
    for (int i = 0; i < N; ++i) t[i] = 0.f;
    return reduce_words<N>(h, t, lane);
}

// The contribution of one pair's plain diagonal sums S_kj (s), T_kj (t0, t1) to one of its antennas:
// h_k += sum_j |g_j|^2 S_kj into h[0], h[1] and b_k += sum_j g_j T_kj into h[4..7], with the other
// antenna's gains q = (g_XX, g_YY); the q side takes S_jk and conj(T_jk).
__device__ __forceinline__ void diag_pair_add(float4 sv, float4 t0, float4 t1, bool p_side, float4 q, float *h)
{
    const float sg = p_side ? 1.f : -1.f;
    const float s01 = p_side ? sv.y : sv.z, s10 = p_side ? sv.z : sv.y;
    const float2 u01 = p_side ? make_float2(t0.z, t0.w) : make_float2(t1.x, t1.y);
    const float2 u10 = p_side ? make_float2(t1.x, t1.y) : make_float2(t0.z, t0.w);
    const float n0 = fmaf(q.x, q.x, q.y * q.y), n1 = fmaf(q.z, q.z, q.w * q.w);
    h[0] += fmaf(n0, sv.x, n1 * s01);
    h[1] += fmaf(n0, s10, n1 * sv.w);
    h[4] += fmaf(q.x, t0.x, fmaf(-q.y, sg * t0.y, fmaf(q.z, u01.x, -q.w * (sg * u01.y))));
    h[5] += fmaf(q.x, sg * t0.y, fmaf(q.y, t0.x, fmaf(q.z, sg * u01.y, q.w * u01.x)));
    h[6] += fmaf(q.x, u10.x, fmaf(-q.y, sg * u10.y, fmaf(q.z, t1.z, -q.w * (sg * t1.w))));
    h[7] += fmaf(q.x, sg * u10.y, fmaf(q.y, u10.x, fmaf(q.z, sg * t1.w, q.w * t1.z)));
}

// The same with h as heads h and tails e, every product exact: a solve of few antennas has few pairs
// over which the roundings of plain products would average out.
__device__ __forceinline__ void diag_pair_add(float4 sv, float4 t0, float4 t1, bool p_side, float4 q, float *h, float *e)
{
    const float sg = p_side ? 1.f : -1.f;
    const float s01 = p_side ? sv.y : sv.z, s10 = p_side ? sv.z : sv.y;
    const float2 u01 = p_side ? make_float2(t0.z, t0.w) : make_float2(t1.x, t1.y);
    const float2 u10 = p_side ? make_float2(t1.x, t1.y) : make_float2(t0.z, t0.w);
    const HT n0 = dot2(q.x, q.x, q.y, q.y), n1 = dot2(q.z, q.z, q.w, q.w);
    const float qy = sg * q.y, qw = sg * q.w;
    dot_add(h[0], e[0], n0, sv.x);
    dot_add(h[0], e[0], n1, s01);
    dot_add(h[1], e[1], n0, s10);
    dot_add(h[1], e[1], n1, sv.w);
    // q conj(t) on the q side: the sign goes to the products with an imaginary part of t
    dot_add(h[4], e[4], q.x, t0.x);
    dot_add(h[4], e[4], -qy, t0.y);
    dot_add(h[4], e[4], q.z, u01.x);
    dot_add(h[4], e[4], -qw, u01.y);
    dot_add(h[5], e[5], sg * q.x, t0.y);
    dot_add(h[5], e[5], q.y, t0.x);
    dot_add(h[5], e[5], sg * q.z, u01.y);
    dot_add(h[5], e[5], q.w, u01.x);
    dot_add(h[6], e[6], q.x, u10.x);
    dot_add(h[6], e[6], -qy, u10.y);
    dot_add(h[6], e[6], q.z, t1.z);
    dot_add(h[6], e[6], -qw, t1.w);
    dot_add(h[7], e[7], sg * q.x, u10.y);
    dot_add(h[7], e[7], q.y, u10.x);
    dot_add(h[7], e[7], sg * q.z, t1.w);
    dot_add(h[7], e[7], q.w, t1.z);
}

} // namespace qc
