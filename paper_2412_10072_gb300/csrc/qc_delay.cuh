// qc_delay.cuh -- delay terms (QC_TERM_DELAY): gains parameterised per solution interval by
// a phase and a delay per correlation, evaluated at every channel,
//   g_c(nu) = exp(i (phi_c + 2 pi tau_c nu)),  parameters u = (phi_X, tau_X, phi_Y, tau_Y)
// (Scenario 2 of Section 2.4: each gain g_{n,s,a} is tied to a parameter u_{n,a} and the
// normal equations sum over samples, Eq. jhj_case2 and Eq. jhwr_case2).
//
// The accumulate kernels see a delay term as a diagonal term with one bin per (time
// interval, channel): its Jones table is evaluated at every channel, and they form the
// complex blocks JHJ_g, JHr_g of the diagonal entries per channel bin.  Within one channel
// bin the derivative dg/du is constant, so the chain rule of Eq. cp_jacobian applies to
// the per-channel sums exactly:
//   JHJ_u = sum over channels of 2 Re(J2^H JHJ_g J2),  JHr_u = sum of 2 Re(J2^H JHr_g),
//   J2 = d(g_X, g_Y)/du = [[i g_X, 2 pi nu i g_X, 0, 0], [0, 0, i g_Y, 2 pi nu i g_Y]].
// delay_update_kernel forms these 4x4 real blocks in FP64, solves them, updates the
// parameters, re-evaluates the channel table and tests convergence on the gains.
#pragma once
#include "qc_kernels.cuh"
#include "qc_sums.cuh"

namespace qc {

constexpr double DELAY_TWO_PI = 6.283185307179586476925286766559;

struct DelayArgs {
    int n_tint, n_fint, n_ant, n_chan;   // n_fint: parameter intervals along frequency
    const int *fmap;          // [n_chan] parameter interval of each channel
    const int2 *frange;       // [n_fint] first and last channel of each interval (x < 0: none)
    const double *nu;         // [n_chan] channel frequencies
    double *params;           // FP64 master [n_tint][n_fint][n_ant][4]
    float4 *tab;              // FP32 channel table [n_tint][n_ant][n_chan]: (g_X, g_Y)
    double omega_ref;         // 2 pi nu of the centre of the band: the streaming kernel's sums use
                              // omega' = 2 pi nu - omega_ref
};

// float32 parameters [n_tint][n_fint][n_ant][4] -> FP64 master copy
static __global__ void delay_params_in_kernel(long n, const float *src, double *params)
{
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        params[i] = (double)src[i];
}

__device__ __forceinline__ double2 delay_gain(double phi, double tau, double w)
{
    double s, c;
    sincos(phi + tau * w, &s, &c);
    return make_double2(c, s);
}

// Gain of one correlation, exp(i (phi + tau w)), in float: the phase is formed and reduced to
// [-pi, pi] in FP64, split into a float head and tail, and the head's sine and cosine
// (sincosf) corrected to first order by the tail, which keeps the float table within about
// one float rounding of the exact gain at FP32 cost (FP64 sincos is slow on this part).
__device__ __forceinline__ float2 delay_gain_f32(double phi, double tau, double w)
{
    const double th = phi + tau * w;
    const double r = th - DELAY_TWO_PI * rint(th * (1.0 / DELAY_TWO_PI));
    const float hi = (float)r, lo = (float)(r - (double)hi);
    float s, c;
    sincosf(hi, &s, &c);
    return make_float2(fmaf(-s, lo, c), fmaf(c, lo, s));
}

// |exp(i a) - exp(i b)|^2 = 4 sin^2((a - b) / 2), from the phase change d = a - b (formed in
// FP64 from the parameter changes; the sine of the reduced half angle in float)
__device__ __forceinline__ double delay_change2(double d)
{
    const double h = 0.5 * d;
    const double r = h - 0.5 * DELAY_TWO_PI * rint(h * (2.0 / DELAY_TWO_PI));
    const double sn = (double)sinf((float)r);
    return 4.0 * sn * sn;
}

// channel table from the FP64 parameters, one entry per (time interval, antenna, channel)
static __global__ void delay_tab_kernel(const DelayArgs a)
{
    const long n = (long)a.n_tint * a.n_ant * a.n_chan;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const int c = (int)(i % a.n_chan);
        const long ta = i / a.n_chan;
        const int ant = (int)(ta % a.n_ant), tint = (int)(ta / a.n_ant);
        const double *u = a.params + (((size_t)tint * a.n_fint + a.fmap[c]) * a.n_ant + ant) * 4;
        const double w = DELAY_TWO_PI * a.nu[c];
        const float2 gx = delay_gain_f32(u[0], u[1], w), gy = delay_gain_f32(u[2], u[3], w);
        a.tab[i] = make_float4(gx.x, gx.y, gy.x, gy.y);
    }
}

// FP64 master -> float32 parameters in the public layout
static __global__ void delay_params_out_kernel(long n, const double *params, float *dst)
{
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        dst[i] = (float)params[i];
}

struct DelayUpdArgs {
    DelayArgs d;
    double *acc;              // diagonal accumulators [n_tint * n_chan][n_ant][KG_DIAG] (read, then zeroed)
    int8_t *gain_flags;       // [n_tint][n_fint][n_ant]
    int *iters;               // [n_tint][n_fint]
    uint8_t *active;          // [n_tint * n_chan] channel bins
    const int *n_active_prev; // intervals active entering this iteration (0: nothing to do)
    int *n_active_next;       // incremented for every interval still active after it
    const long long *bin_nvis, *bin_nbytes;   // per channel bin
    unsigned long long *vis_iters, *acc_bytes;
    int k;                    // iteration (1-based)
    double alpha, tol;
    // a term solved from products (qc_delay_sums.cu): the h sums [bins][n_ant][6], the same for every
    // iteration (else null: they are in acc); the channel table is then left to the end of the solve
    const double *hsum;
    const float *omega, *omega_lo;   // [n_chan] omega' = 2 pi nu - omega_ref as head and tail (with hsum)
    const double2 *om_sums;   // [n_fint] sum of omega', of omega'^2 over the interval's channels (with hsum)
    double om_max;            // largest |omega'|
    int prod_bytes;           // bytes of a channel's products over the pairs (with hsum)
};

// One block per parameter interval (time interval x frequency interval), threads over antennas.
// SUMS = false: the accumulators are the complex diagonal blocks of every channel bin
// [n_tint * n_chan][n_ant][KG_DIAG] and activity is kept per channel bin; the chain rule is
// applied here, channel by channel.  SUMS = true: the streaming delay kernel has applied it
// per sample and left the 13 real sums of each (interval, antenna) [bins][n_ant][KG_SUMS]
// (h_XX, h_YY, h_XY times 1, omega', omega'^2; r_X, r_Y times 1, omega') with the centred
// omega' = omega - omega_ref; they are shifted back to omega here in FP64, so that a band of
// one frequency gives the exactly proportional phase and delay columns of the oracle (a
// singular block) rather than FP32 rounding; activity per interval.
constexpr int KG_SUMS = 16;

// Two real symmetric 2x2 systems [[a0, a1], [a1, a2]] (y0, y1) = (r0, r1) and [[c0, c1], [c1, c2]] (y2, y3) =
// (r2, r3) under block_solve's tests over the whole block-diagonal matrix (zero trace, zero
// determinant, reciprocal 1-norm condition number); returns 1 when singular.
__device__ __forceinline__ int delay_solve_pair(double a0, double a1, double a2, double c0, double c1, double c2, double r0,
                                                double r1, double r2, double r3, double (&y)[4])
{
    y[0] = y[1] = y[2] = y[3] = 0.0;
    if (!(a0 + a2 + c0 + c2 > 0)) return 1;
    const double da = a0 * a2 - a1 * a1, dc = c0 * c2 - c1 * c1;
    if (!(fabs(da) > 0) || !(fabs(dc) > 0)) return 1;
    const double ia = 1.0 / da, ic = 1.0 / dc;
    const double na = fmax(fabs(a0), fabs(a2)) + fabs(a1), nc = fmax(fabs(c0), fabs(c2)) + fabs(c1);
    if (!(1.0 / (fmax(na, nc) * fmax(na * fabs(ia), nc * fabs(ic))) >= 1e-12)) return 1;
    y[0] = (a2 * r0 - a1 * r1) * ia;
    y[1] = (a0 * r1 - a1 * r0) * ia;
    y[2] = (c2 * r2 - c1 * r3) * ic;
    y[3] = (c0 * r3 - c1 * r2) * ic;
    return 0;
}

__device__ __forceinline__ float4 delay_split(double a, double b)
{
    const float x = (float)a, y = (float)b;
    return make_float4(x, (float)(a - (double)x), y, (float)(b - (double)y));
}

// a + b om, each as head and tail, rounded to float once
__device__ __forceinline__ float delay_phase(float4 ab, float2 om)
{
    const float p = __fmul_rn(ab.z, om.x), r = __fmaf_rn(ab.z, om.x, -p);
    float s, e;
    two_sum(ab.x, p, s, e);
    return s + (e + (r + fmaf(ab.z, om.y, fmaf(ab.w, om.x, ab.y))));
}

// Counts and convergence of an interval, by the whole block (one thread adding up the counts of 512
// channels was 0.1 of the update's 0.13 ms on 75 intervals); tn, td (thread 0): the squared change
// of the gains and their squared norm.
template <bool SUMS>
__device__ __forceinline__ void delay_finish(const DelayUpdArgs &u, int bin, int2 fr, size_t cb0, double tn, double td)
{
    unsigned long long nv = 0, nb = 0;
    for (int c = fr.x + (int)threadIdx.x; c <= fr.y; c += blockDim.x) {
        nv += (unsigned long long)u.bin_nvis[cb0 + c];
        // from products: the samples once, then the products of the interval
        nb += u.hsum ? (unsigned long long)u.prod_bytes + (u.k == 1 ? (unsigned long long)u.bin_nbytes[cb0 + c] : 0ull)
                     : (unsigned long long)u.bin_nbytes[cb0 + c];
    }
    if (nv) atomicAdd(u.vis_iters, nv);
    if (nb) atomicAdd(u.acc_bytes, nb);
    if (threadIdx.x == 0) {
        const double delta = td > 0 ? sqrt(tn / td) : 0.0;
        if (u.iters) u.iters[bin] = u.k;
        if (delta < u.tol) {
            if (SUMS) u.active[bin] = 0;
            else
                for (int c = fr.x; c <= fr.y; ++c) u.active[cb0 + c] = 0;
        } else {
            atomicAdd(u.n_active_next, 1);
        }
    }
}

template <bool SUMS>
static __global__ void __launch_bounds__(128) delay_update_kernel(const DelayUpdArgs u)
{
    if (*u.n_active_prev == 0) return;
    const DelayArgs &d = u.d;
    const int bin = blockIdx.x;
    const int tint = bin / d.n_fint, fu = bin % d.n_fint;
    const int2 fr = d.frange[fu];
    const size_t cb0 = (size_t)tint * d.n_chan;            // first channel bin of the time interval
    if (fr.x < 0) {
        // no channel maps to this interval: no data, the parameters stay as they are
        if (u.k == 1) {
            for (int ant = threadIdx.x; ant < d.n_ant; ant += blockDim.x)
                if (u.gain_flags) u.gain_flags[(size_t)bin * d.n_ant + ant] = 1;
            if (threadIdx.x == 0 && u.iters) u.iters[bin] = 1;
        }
        return;
    }
    if (!u.active[SUMS ? (size_t)bin : cb0 + fr.x]) return;
    double num = 0, den = 0;
    for (int ant = threadIdx.x; ant < d.n_ant; ant += blockDim.x) {
        double *P = d.params + ((size_t)bin * d.n_ant + ant) * 4;
        const double u0 = P[0], u1 = P[1], u2 = P[2], u3 = P[3];
        double2 M[4][4], b[4], x[4];
        for (int i = 0; i < 4; ++i) {
            b[i] = make_double2(0.0, 0.0);
            for (int j = 0; j < 4; ++j) M[i][j] = make_double2(0.0, 0.0);
        }
        if (SUMS) {
            double *A = u.acc + ((size_t)bin * d.n_ant + ant) * KG_SUMS;
            double S[13];
            for (int i = 0; i < 13; ++i) { S[i] = A[i]; A[i] = 0.0; }
            if (u.hsum) {
                const double *H = u.hsum + ((size_t)bin * d.n_ant + ant) * 6;
                for (int i = 0; i < 6; ++i) S[i] = H[i];
            }
            // sum h w^k with w = w' + w0:  h w = h w' + w0 h,  h w^2 = h w'^2 + 2 w0 h w' + w0^2 h
            const double w0 = d.omega_ref;
            for (int base = 0; base <= 10; base += (base == 3 ? 7 : 3)) {
                const double s0 = S[base], s1 = S[base + 1], s2 = S[base + 2];
                S[base + 1] = s1 + w0 * s0;
                S[base + 2] = s2 + 2.0 * w0 * s1 + w0 * w0 * s0;
            }
            S[7] += w0 * S[6];
            S[9] += w0 * S[8];
            const int o2[2][2] = { { 0, 1 }, { 1, 2 } };    // power of omega of block entry (i, j)
            for (int i = 0; i < 2; ++i)
                for (int j = 0; j < 2; ++j) {
                    M[i][j].x = 2.0 * S[o2[i][j]];
                    M[2 + i][2 + j].x = 2.0 * S[3 + o2[i][j]];
                    M[i][2 + j].x = 2.0 * S[10 + o2[i][j]];
                    M[2 + j][i].x = 2.0 * S[10 + o2[i][j]];
                }
            b[0].x = 2.0 * S[6];
            b[1].x = 2.0 * S[7];
            b[2].x = 2.0 * S[8];
            b[3].x = 2.0 * S[9];
        }
        for (int c = fr.x; !SUMS && c <= fr.y; ++c) {
            double *A = u.acc + ((cb0 + c) * d.n_ant + ant) * KG_DIAG;
            const double h00 = A[0], h11 = A[1];
            const double2 h01 = make_double2(A[2], A[3]), j0 = make_double2(A[4], A[5]), j1 = make_double2(A[6], A[7]);
            for (int i = 0; i < KG_DIAG; ++i) A[i] = 0.0;
            const double w = DELAY_TWO_PI * d.nu[c];
            const double2 gx = delay_gain(u0, u1, w), gy = delay_gain(u2, u3, w);
            const double f[2] = { 1.0, w };
            // Re(conj(g_X) JHJ_g[X][Y] g_Y): the X-Y coupling (zero without a left factor)
            const double2 t = make_double2(gx.x * h01.x + gx.y * h01.y, gx.x * h01.y - gx.y * h01.x);
            const double xy = t.x * gy.x - t.y * gy.y;
            // Im(conj(g_c) JHr_g[c]) of each correlation
            const double rx = gx.x * j0.y - gx.y * j0.x, ry = gy.x * j1.y - gy.y * j1.x;
            for (int i = 0; i < 2; ++i) {
                for (int j = 0; j < 2; ++j) {
                    M[i][j].x += 2.0 * h00 * f[i] * f[j];
                    M[2 + i][2 + j].x += 2.0 * h11 * f[i] * f[j];
                    M[i][2 + j].x += 2.0 * xy * f[i] * f[j];
                    M[2 + j][i].x += 2.0 * xy * f[i] * f[j];
                }
                b[i].x += 2.0 * rx * f[i];
                b[2 + i].x += 2.0 * ry * f[i];
            }
        }
        int singular;
        if (SUMS && u.hsum) {
            // no coupling between X and Y: two real 2x2 solves
            double y[4];
            singular = delay_solve_pair(M[0][0].x, M[0][1].x, M[1][1].x, M[2][2].x, M[2][3].x, M[3][3].x, b[0].x, b[1].x,
                                        b[2].x, b[3].x, y);
            for (int e = 0; e < 4; ++e) x[e] = make_double2(y[e], 0.0);
        } else {
            singular = block_solve<4>(M, b, x);
        }
        if (!singular)
            for (int e = 0; e < 4; ++e) P[e] += u.alpha * x[e].x;
        if (u.gain_flags) u.gain_flags[(size_t)bin * d.n_ant + ant] = (int8_t)singular;
        if (SUMS) {
            // the parameter change, kept in the (already read) sums for the channel pass below
            double *A = u.acc + ((size_t)bin * d.n_ant + ant) * KG_SUMS;
            A[0] = P[0] - u0;
            A[1] = P[1] - u1;
            A[2] = P[2] - u2;
            A[3] = P[3] - u3;
            continue;
        }
        // re-evaluate the channel table; relative change of the gains over the interval's channels
        // (the gains have unit modulus: |g_new - g_old|^2 = 4 sin^2 of half the phase change,
        // |g_new|^2 = 1 per correlation)
        const double d0 = P[0] - u0, d1 = P[1] - u1, d2 = P[2] - u2, d3 = P[3] - u3;
        for (int c = fr.x; c <= fr.y; ++c) {
            const double w = DELAY_TWO_PI * d.nu[c];
            const float2 nx = delay_gain_f32(P[0], P[1], w), ny = delay_gain_f32(P[2], P[3], w);
            d.tab[((size_t)tint * d.n_ant + ant) * d.n_chan + c] = make_float4(nx.x, nx.y, ny.x, ny.y);
            num += delay_change2(d0 + d1 * w) + delay_change2(d2 + d3 * w);
            den += 2.0;
        }
    }
    if (SUMS && !u.hsum) return;       // delay_chan_kernel follows
    if (SUMS) {
        // the change of the gains, (antenna, channel) by (antenna, channel) over the block's threads: the
        // phase change of a channel from the FP64 changes as head and tail (an ulp of float, as an FP64
        // phase rounded to it; 64 antennas, 75 x 512: 10.5 ms a solve with FP64 phases)
        __syncthreads();
        const int nch = fr.y - fr.x + 1;
        for (int a0 = 0; a0 < d.n_ant; a0 += 128) {
            __shared__ float4 s_f[128][2];          // head and tail of the change at the centre, of its slope
            const int na = min(128, d.n_ant - a0);
            bool small = true;
            double e[4] = { 0, 0, 0, 0 };
            if ((int)threadIdx.x < na) {
                // about the band's centre: A0 + A1 w = (A0 + A1 w_ref) + A1 w'
                double *A = u.acc + ((size_t)bin * d.n_ant + a0 + threadIdx.x) * KG_SUMS;
                e[0] = A[0] + A[1] * d.omega_ref;
                e[1] = A[1];
                e[2] = A[2] + A[3] * d.omega_ref;
                e[3] = A[3];
                A[0] = A[1] = A[2] = A[3] = 0.0;
                s_f[threadIdx.x][0] = delay_split(e[0], e[1]);
                s_f[threadIdx.x][1] = delay_split(e[2], e[3]);
                // changes below 5e-4 over the whole interval (all but the first iterations): 4 sin^2 of half
                // the change is its square to 2e-8, and the sum over the channels is closed
                small = fabs(e[0]) + fabs(e[1]) * u.om_max < 5e-4 && fabs(e[2]) + fabs(e[3]) * u.om_max < 5e-4;
            }
            if (__syncthreads_and(small)) {
                if ((int)threadIdx.x < na) {
                    const double2 m = u.om_sums[fu];
                    num += e[0] * e[0] * nch + 2.0 * e[0] * e[1] * m.x + e[1] * e[1] * m.y;
                    num += e[2] * e[2] * nch + 2.0 * e[2] * e[3] * m.x + e[3] * e[3] * m.y;
                }
                continue;
            }
            for (int i = threadIdx.x; i < na * nch; i += blockDim.x) {
                const int ant = i / nch, c = fr.x + (i - ant * nch);
                const float2 om = make_float2(__ldg(u.omega + c), __ldg(u.omega_lo + c));
                const float4 x = s_f[ant][0], y = s_f[ant][1];
                const float px = delay_phase(x, om), py = delay_phase(y, om);
                if (fabsf(px) < 8.f && fabsf(py) < 8.f) {
                    const float s0 = sinf(0.5f * px), s1 = sinf(0.5f * py);
                    num += 4.0 * ((double)s0 * s0 + (double)s1 * s1);
                } else {
                    const double w = (double)om.x + (double)om.y;
                    num += delay_change2(((double)x.x + x.y) + ((double)x.z + x.w) * w) +
                           delay_change2(((double)y.x + y.y) + ((double)y.z + y.w) * w);
                }
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) den = 2.0 * d.n_ant * nch;
    }
    __shared__ double s_num[4], s_den[4];
    for (int dd = 16; dd > 0; dd >>= 1) {
        num += __shfl_down_sync(0xffffffffu, num, dd);
        den += __shfl_down_sync(0xffffffffu, den, dd);
    }
    const int wi = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { s_num[wi] = num; s_den[wi] = den; }
    __syncthreads();
    double tn = 0, td = 0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x + 31) / 32; ++i) { tn += s_num[i]; td += s_den[i]; }
    delay_finish<SUMS>(u, bin, fr, cb0, tn, td);
}

// The channel table and the change of the gains of the active intervals (SUMS without the products),
// an interval's (antenna, channel) pairs split over gridDim.y CTAs, the last of which tests
// convergence.  FP64 throughput bounds it (phases formed and reduced in FP64); one CTA an interval
// inside the update kept 64 of 152 SMs busy where there are 64 intervals: 490 us an iteration with 64
// antennas and 512 channels, 38 us the update and 166 us this like so.
static __global__ void __launch_bounds__(128) delay_chan_kernel(const DelayUpdArgs u)
{
    if (*u.n_active_prev == 0) return;
    const DelayArgs &d = u.d;
    const int bin = blockIdx.x, tint = bin / d.n_fint;
    const int2 fr = d.frange[bin % d.n_fint];
    if (fr.x < 0 || !u.active[bin]) return;
    const int nch = fr.y - fr.x + 1, n = d.n_ant * nch;
    const int per = (n + gridDim.y - 1) / gridDim.y, i0 = min(n, (int)blockIdx.y * per), i1 = min(n, i0 + per);
    double num = 0;
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        const int ant = i / nch, c = fr.x + (i - ant * nch);
        const double *P = d.params + ((size_t)bin * d.n_ant + ant) * 4;
        const double *A = u.acc + ((size_t)bin * d.n_ant + ant) * KG_SUMS;
        const double w = DELAY_TWO_PI * d.nu[c];
        const float2 nx = delay_gain_f32(P[0], P[1], w), ny = delay_gain_f32(P[2], P[3], w);
        d.tab[((size_t)tint * d.n_ant + ant) * d.n_chan + c] = make_float4(nx.x, nx.y, ny.x, ny.y);
        num += delay_change2(A[0] + A[1] * w) + delay_change2(A[2] + A[3] * w);
    }
    __shared__ double s_num[4];
    __shared__ bool s_last;
    for (int dd = 16; dd > 0; dd >>= 1) num += __shfl_down_sync(0xffffffffu, num, dd);
    if ((threadIdx.x & 31) == 0) s_num[threadIdx.x >> 5] = num;
    __syncthreads();                                  // every thread has read its changes
    // the interval's sum and the number of its CTAs that are done: spare words of the first antenna's sums
    double *A0 = u.acc + (size_t)bin * d.n_ant * KG_SUMS;
    unsigned long long *count = reinterpret_cast<unsigned long long *>(A0 + 14);
    if (threadIdx.x == 0) {
        atomicAdd(A0 + 13, s_num[0] + s_num[1] + s_num[2] + s_num[3]);
        __threadfence();
        s_last = atomicAdd(count, 1ull) == gridDim.y - 1;
    }
    __syncthreads();
    if (!s_last) return;
    double tn = 0;
    if (threadIdx.x == 0) {
        __threadfence();
        tn = atomicAdd(A0 + 13, 0.0);
        A0[13] = 0.0;
        *count = 0ull;
    }
    for (int ant = threadIdx.x; ant < d.n_ant; ant += blockDim.x) {
        double *A = u.acc + ((size_t)bin * d.n_ant + ant) * KG_SUMS;
        A[0] = A[1] = A[2] = A[3] = 0.0;
    }
    delay_finish<true>(u, bin, fr, (size_t)tint * d.n_chan, tn, 2.0 * n);
}

} // namespace qc

namespace qc {

// ---------------------------------------------------------------------------
// initial estimate of a delay term (Section 4.3, "Initial estimates"): the peak of the
// Fourier transform along frequency of the baselines that include the reference antenna
// ---------------------------------------------------------------------------

struct DelayInitArgs {
    int n_row, n_chan, n_ant, ref, n_tint, n_fint;
    const int4 *rows;          // [n_row] {ant1, ant2, time, baseline}
    const float4 *vis;         // [n_row][n_chan] x 2
    const float4 *model;       // [n_row][n_chan] x 2, or nullptr (FP16 model)
    const uint4 *model16;      // [n_row][n_chan], or nullptr
    const float *bl_scale;     // [n_bl] FP16 model scales
    const float4 *wf;          // [n_row][n_chan] weights, zero where flagged or autocorrelation
    const int *t_map;          // [n_time] time interval of each data time
    float2 *x;                 // [n_tint][n_ant][2][n_chan] spectra (zeroed before)
    const int4 *fint_info;     // [n_fint] {first channel, channels, N, log2 N}
    const double *fint_dnu;    // [n_fint] channel spacing
    const double *fint_nu0;    // [n_fint] frequency of the first channel
    float *params;             // [n_tint][n_fint][n_ant][4] out
};

// x[t][a][c][chan] += w d conj(m) of correlation c (XX, YY) over the rows on baselines with
// the reference antenna, conjugated for rows (ref, a).  One warp per row, lanes over channels.
static __global__ void delay_gather_kernel(const DelayInitArgs a)
{
    const int lane = threadIdx.x & 31;
    const long warp = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long n_warps = ((long)gridDim.x * blockDim.x) >> 5;
    for (long row = warp; row < a.n_row; row += n_warps) {
        const int4 r = a.rows[row];
        if (r.x == r.y || (r.x != a.ref && r.y != a.ref)) continue;
        const int ant = r.x == a.ref ? r.y : r.x;
        const bool flip = r.x == a.ref;
        float2 *xa = a.x + ((size_t)a.t_map[r.z] * a.n_ant + ant) * 2 * a.n_chan;
        for (int c = lane; c < a.n_chan; c += 32) {
            const size_t s = (size_t)row * a.n_chan + c;
            const float4 w = a.wf[s];
            if (w.x == 0.f && w.y == 0.f && w.z == 0.f && w.w == 0.f) continue;
            const J2 D = j_from(a.vis[2 * s], a.vis[2 * s + 1]);
            const J2 M = a.model ? j_from(a.model[2 * s], a.model[2 * s + 1]) : load_model16(a.model16[s], a.bl_scale[r.w]);
            float2 zx = cscale(cmulc(D.a, M.a), w.x), zy = cscale(cmulc(D.d, M.d), w.w);
            if (flip) { zx = cconj(zx); zy = cconj(zy); }
            atomicAdd(&xa[c].x, zx.x);
            atomicAdd(&xa[c].y, zx.y);
            atomicAdd(&xa[a.n_chan + c].x, zy.x);
            atomicAdd(&xa[a.n_chan + c].y, zy.y);
        }
    }
}

// One block per (time interval, frequency interval, antenna, correlation): the spectrum over
// the interval's channels, zero-padded to N (a power of two), transformed by a radix-2 FFT in
// shared memory, X_k = sum_c x_c exp(-2 pi i k c / N); the peak |X_k| (lowest signed k
// among equal values) gives tau = k / (N dnu) and phi = arg X_k - 2 pi tau nu_0.
static __global__ void __launch_bounds__(256) delay_peak_kernel(const DelayInitArgs a)
{
    extern __shared__ float2 fbuf[];
    const int corr = blockIdx.x & 1;
    const int rest = blockIdx.x >> 1;
    const int ant = rest % a.n_ant;
    const int bin = rest / a.n_ant;                         // tint * n_fint + fint
    const int fi = bin % a.n_fint, tint = bin / a.n_fint;
    float *out = a.params + ((size_t)bin * a.n_ant + ant) * 4 + 2 * corr;
    const int4 info = a.fint_info[fi];
    const int c0 = info.x, n_c = info.y, N = info.z, lg = info.w;
    const float2 *xs = a.x + (((size_t)tint * a.n_ant + ant) * 2 + corr) * a.n_chan + c0;
    if (ant == a.ref || n_c == 0) {
        if (threadIdx.x == 0) { out[0] = 0.f; out[1] = 0.f; }
        return;
    }
    if (n_c == 1) {
        if (threadIdx.x == 0) {
            const float2 v = xs[0];
            out[0] = (v.x != 0.f || v.y != 0.f) ? atan2f(v.y, v.x) : 0.f;
            out[1] = 0.f;
        }
        return;
    }
    for (int i = threadIdx.x; i < N; i += blockDim.x) fbuf[i] = make_float2(0.f, 0.f);
    __syncthreads();
    for (int c = threadIdx.x; c < n_c; c += blockDim.x) fbuf[__brev((unsigned)c) >> (32 - lg)] = xs[c];
    __syncthreads();
    for (int len = 2, lh = 0; len <= N; len <<= 1, ++lh) {
        const int half = len >> 1;
        for (int j = threadIdx.x; j < N / 2; j += blockDim.x) {
            const int grp = j >> lh, pos = j & (half - 1);
            const int i0 = grp * len + pos, i1 = i0 + half;
            float sn, cs;
            sincospif(-2.0f * (float)pos / (float)len, &sn, &cs);
            const float2 u = fbuf[i0], v = cmul(fbuf[i1], make_float2(cs, sn));
            fbuf[i0] = cadd(u, v);
            fbuf[i1] = csub(u, v);
        }
        __syncthreads();
    }
    float best = -1.f;
    int bk = 1 << 30;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const int ks = i < N / 2 ? i : i - N;
        const float m = cnorm2(fbuf[i]);
        if (m > best || (m == best && ks < bk)) { best = m; bk = ks; }
    }
    for (int d = 16; d > 0; d >>= 1) {
        const float om = __shfl_down_sync(0xffffffffu, best, d);
        const int ok = __shfl_down_sync(0xffffffffu, bk, d);
        if (om > best || (om == best && ok < bk)) { best = om; bk = ok; }
    }
    __shared__ float s_best[8];
    __shared__ int s_k[8];
    const int wi = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { s_best[wi] = best; s_k[wi] = bk; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i)
            if (s_best[i] > best || (s_best[i] == best && s_k[i] < bk)) { best = s_best[i]; bk = s_k[i]; }
        if (!(best > 0.f)) { out[0] = 0.f; out[1] = 0.f; return; }
        const float2 X = fbuf[bk >= 0 ? bk : bk + N];
        const double tau = (double)bk / ((double)N * a.fint_dnu[fi]);
        double phi = atan2((double)X.y, (double)X.x) - DELAY_TWO_PI * tau * a.fint_nu0[fi];
        phi -= DELAY_TWO_PI * floor(phi / DELAY_TWO_PI + 0.5);
        out[0] = (float)phi;
        out[1] = (float)tau;
    }
}

} // namespace qc
