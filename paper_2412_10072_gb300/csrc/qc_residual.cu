// qc_residual.cu -- chi^2 and the residual after calibration (Eq. min, Eq. baselineresidual), and MAD
// flagging of it (Section 4, "Additional features").
#include "qc_internal.h"

#include <algorithm>

namespace qc {

constexpr unsigned MAD_SENTINEL = 0x7f800001u;   // unused samples: after +inf, before the NaNs a sqrt gives

__device__ __forceinline__ int mad_digit(unsigned key, int level)
{
    return level == 0 ? (int)(key >> 20) : (level == 1 ? (int)(key >> 10) & 1023 : (int)key & 1023);
}
// the digits above a level
__device__ __forceinline__ unsigned mad_above(int level) { return level == 0 ? 0u : (level == 1 ? 0x7ff00000u : 0x7ffffc00u); }

// tot += the eight terms, summed as head and tail: exact to the last bits of the tail, two conversions to
// FP64 instead of eight.  Where the head overflows (or a term is infinite or NaN), term by term.
__device__ __forceinline__ void add_terms(double &tot, const float4 &a, const float4 &b)
{
    float s = a.x, e = 0.f;
    const float t[7] = { a.y, a.z, a.w, b.x, b.y, b.z, b.w };
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        float r;
        two_sum(s, t[i], s, r);
        e += r;
    }
    if (isfinite(s) && isfinite(e)) {
        tot += (double)s + (double)e;
    } else {
        tot += (double)a.x;
#pragma unroll
        for (int i = 0; i < 7; ++i) tot += (double)t[i];
    }
}

// A warp per row, two 32-channel chunks in flight: the chunks' data, model, weights and flags are
// loaded before the gains, whose table entries come from L1.  MAD: instead of chi^2 and the residual,
// the sample's key -- the bits of z = sqrt(sum_c w_c |r_c|^2), every operation rounded, in a fixed
// order, so that the residual (32 B a sample) is neither written nor read again.  (Counting the
// first digit here too doubled the kernel: most keys share a few bins; a pass over the keys, 4 B a
// sample, takes 65 us of the 1.3 ms.)  chi^2 is summed in FP64 per lane, the eight
// terms of two samples at a time (add_terms): converting every term to FP64 took longer than the
// memory (FP64 runs at 2 lanes a cycle and SM).  64 antennas, 60 x 509, residual written: 1.79 ms a call before, 1.52 now (the kernel
// 1.34, 5.2 TB/s).
template <bool M16, bool MAD, int NT>
static __global__ void __launch_bounds__(256, 2) residual_kernel(const ResArgs a, unsigned *__restrict__ keys, MadState *state)
{
    const Data &D = a.D;
    const Chain &C = a.C;
    __shared__ unsigned long long s_used;
    if constexpr (MAD) {
        if (threadIdx.x == 0) s_used = 0;
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const long warp = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long n_warps = ((long)gridDim.x * blockDim.x) >> 5;
    double tot = 0.0;
    unsigned used = 0;
    struct Samp { float4 d0, d1, m0, m1, w; bool ok; };
    for (long row = warp; row < D.n_row; row += n_warps) {
        const int4 meta = __ldg(D.rows + row);
        const size_t base = (size_t)row * D.n_chan;
        const bool cross = meta.x != meta.y;
        int tint[NT];
#pragma unroll
        for (int j = 0; j < NT; ++j) tint[j] = cross && j < C.n_terms ? __ldg(C.t[j].t_map + meta.z) : 0;
        const float sc = M16 && cross ? __ldg(D.bl_scale + meta.w) : 1.f;
        auto load = [&](int c) {
            Samp x;
            x.ok = false;
            if (c < D.n_chan && cross) {
                const size_t s = base + c;
                x.ok = !(D.flag && __ldg(D.flag + s));
                x.d0 = __ldcs(D.vis + 2 * s);
                x.d1 = __ldcs(D.vis + 2 * s + 1);
                if constexpr (M16) {
                    const uint4 h = __ldcs(D.model16 + s);
                    x.m0 = *reinterpret_cast<const float4 *>(&h);
                } else {
                    x.m0 = __ldcs(D.model + 2 * s);
                    x.m1 = __ldcs(D.model + 2 * s + 1);
                }
                x.w = __ldcs(D.weight + s);
            }
            return x;
        };
        float4 chi = make_float4(0, 0, 0, 0);     // the last sample's terms of chi^2
        auto finish = [&](int c, const Samp &x) {
            if constexpr (!MAD) chi = make_float4(0, 0, 0, 0);
            if (c >= D.n_chan) return;
            const size_t s = base + c;
            if (!x.ok) {
                if constexpr (MAD) {
                    keys[s] = MAD_SENTINEL;
                } else if (a.resid) {
                    __stcs(a.resid + 2 * s, make_float4(0, 0, 0, 0));
                    __stcs(a.resid + 2 * s + 1, make_float4(0, 0, 0, 0));
                }
                return;
            }
            J2 Cp = j_identity(), Cq = j_identity();
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                if (j >= C.n_terms) break;
                const DevTerm &T = C.t[j];
                const int fint = __ldg(T.f_map + c);
                Cp = j_mul(Cp, fetch_jones(T, C.n_ant, tint[j], fint, meta.x));
                Cq = j_mul(Cq, fetch_jones(T, C.n_ant, tint[j], fint, meta.y));
            }
            J2 M;
            if constexpr (M16) M = load_model16(*reinterpret_cast<const uint4 *>(&x.m0), sc);
            else M = j_from(x.m0, x.m1);
            const J2 V = j_mul_h(j_mul(Cp, M), Cq);
            const J2 Dm = j_from(x.d0, x.d1);
            J2 r;
            r.a = csub(Dm.a, V.a); r.b = csub(Dm.b, V.b); r.c = csub(Dm.c, V.c); r.d = csub(Dm.d, V.d);
            const float4 w = x.w;
            if constexpr (MAD) {
                const float t0 = __fadd_rn(__fmul_rn(r.a.x, r.a.x), __fmul_rn(r.a.y, r.a.y));
                const float t1 = __fadd_rn(__fmul_rn(r.b.x, r.b.x), __fmul_rn(r.b.y, r.b.y));
                const float t2 = __fadd_rn(__fmul_rn(r.c.x, r.c.x), __fmul_rn(r.c.y, r.c.y));
                const float t3 = __fadd_rn(__fmul_rn(r.d.x, r.d.x), __fmul_rn(r.d.y, r.d.y));
                float acc = __fmul_rn(w.x, t0);
                acc = __fadd_rn(acc, __fmul_rn(w.y, t1));
                acc = __fadd_rn(acc, __fmul_rn(w.z, t2));
                acc = __fadd_rn(acc, __fmul_rn(w.w, t3));
                keys[s] = __float_as_uint(__fsqrt_rn(acc));
                ++used;
            } else {
                chi = make_float4(__fmul_rn(w.x, cnorm2(r.a)), __fmul_rn(w.y, cnorm2(r.b)), __fmul_rn(w.z, cnorm2(r.c)),
                                  __fmul_rn(w.w, cnorm2(r.d)));
                if (a.resid) {
                    __stcs(a.resid + 2 * s, make_float4(r.a.x, r.a.y, r.b.x, r.b.y));
                    __stcs(a.resid + 2 * s + 1, make_float4(r.c.x, r.c.y, r.d.x, r.d.y));
                }
            }
        };
        for (int c = lane; c - lane < D.n_chan; c += 64) {
            const Samp x0 = load(c);
            const Samp x1 = load(c + 32);
            finish(c, x0);
            const float4 t0 = chi;
            finish(c + 32, x1);
            if constexpr (!MAD) add_terms(tot, t0, chi);
        }
    }
    if constexpr (MAD) {
        for (int d = 16; d > 0; d >>= 1) used += __shfl_down_sync(0xffffffffu, used, d);
        if (lane == 0 && used) atomicAdd(&s_used, (unsigned long long)used);
        __syncthreads();
        if (threadIdx.x == 0 && s_used) atomicAdd(&state->n_used, s_used);
    } else {
        for (int d = 16; d > 0; d >>= 1) tot += __shfl_down_sync(0xffffffffu, tot, d);
        __shared__ double part[8];
        if (lane == 0) part[threadIdx.x >> 5] = tot;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0;
            for (int i = 0; i < (int)blockDim.x / 32; ++i) t += part[i];
            atomicAdd(a.chi2, t);
        }
    }
}

// key of |z - med| for a used sample (the sentinel stays)
__device__ __forceinline__ unsigned mad_dev(unsigned key, float med)
{
    return key == MAD_SENTINEL ? key : __float_as_uint(fabsf(__fsub_rn(__uint_as_float(key), med)));
}

// The bin of hist (n <= 2048) that holds rank k, and the rank inside it; a block of 256 threads.
__device__ __forceinline__ void mad_find(const unsigned *hist, int n, unsigned long long k, int *s_bin,
                                         unsigned long long *s_rank, unsigned long long *s_part)
{
    const int tid = threadIdx.x, per = n / 256;
    unsigned long long sum = 0;
    for (int i = 0; i < per; ++i) sum += hist[tid * per + i];
    s_part[tid] = sum;
    __syncthreads();
    if (tid < 32) {
        // exclusive scan of the 256 shares by one warp, eight a lane
        unsigned long long v[8], run = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) { v[i] = s_part[tid * 8 + i]; run += v[i]; }
        unsigned long long inc = run;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long o = __shfl_up_sync(0xffffffffu, inc, d);
            if (tid >= d) inc += o;
        }
        unsigned long long ex = inc - run;
#pragma unroll
        for (int i = 0; i < 8; ++i) { s_part[tid * 8 + i] = ex; ex += v[i]; }
    }
    __syncthreads();
    unsigned long long cum = s_part[tid];
    if (k >= cum && k < cum + sum)
        for (int i = 0; i < per; ++i) {
            const unsigned h = hist[tid * per + i];
            if (k < cum + h) {
                *s_bin = tid * per + i;
                *s_rank = k - cum;
                break;
            }
            cum += h;
        }
    __syncthreads();
}

// After level `level` of statistic `dev` (0 median, 1 MAD): its digit, and the next level's empty
// histogram; the last level leaves the median or the threshold.
static __global__ void __launch_bounds__(256) mad_pick_kernel(MadState *s, int dev, int level, float factor)
{
    __shared__ int s_bin;
    __shared__ unsigned long long s_rank, s_part[256];
    if (s->n_used == 0) {
        if (threadIdx.x == 0) s->thr = INFINITY;
        return;
    }
    const unsigned long long k = level == 0 ? (s->n_used - 1) / 2 : s->k;
    mad_find(s->hist, level == 0 ? 2048 : 1024, k, &s_bin, &s_rank, s_part);
    for (int i = threadIdx.x; i < 2048; i += blockDim.x) s->hist[i] = 0;
    if (threadIdx.x == 0) {
        unsigned p = level == 0 ? 0u : s->prefix;
        p |= (unsigned)s_bin << (level == 0 ? 20 : (level == 1 ? 10 : 0));
        s->prefix = p;
        s->k = s_rank;
        if (level == MAD_LEVELS - 1) {
            // the sentinel's place in the order is that of an infinite value
            const float v = p == MAD_SENTINEL ? INFINITY : __uint_as_float(p);
            if (dev) s->thr = __fmul_rn(factor, v);
            else s->med = v;
        }
    }
}

// histogram of digit `level` of the keys (dev: of |z - med|) whose digits above equal the prefix
static __global__ void __launch_bounds__(256) mad_hist_kernel(long n, const unsigned *__restrict__ keys, MadState *s, int dev,
                                                              int level)
{
    __shared__ unsigned h[2048];
    if (s->n_used == 0) return;
    const float med = s->med;
    const unsigned above = mad_above(level), prefix = s->prefix & above;
    for (int t = threadIdx.x; t < 2048; t += blockDim.x) h[t] = 0;
    __syncthreads();
    auto one = [&](unsigned key) {
        const unsigned k = dev ? mad_dev(key, med) : key;
        if ((k & above) == prefix) atomicAdd(&h[mad_digit(k, level) & 2047], 1u);
    };
    const long n4 = n / 4, step = (long)gridDim.x * blockDim.x, t0 = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const uint4 *k4 = reinterpret_cast<const uint4 *>(keys);
    for (long i = t0; i < n4; i += 2 * step) {
        const uint4 a = __ldg(k4 + i);
        const bool two = i + step < n4;
        const uint4 b = two ? __ldg(k4 + i + step) : a;
        one(a.x); one(a.y); one(a.z); one(a.w);
        if (two) { one(b.x); one(b.y); one(b.z); one(b.w); }
    }
    for (long i = 4 * n4 + t0; i < n; i += step) one(__ldg(keys + i));
    __syncthreads();
    for (int t = threadIdx.x; t < 2048; t += blockDim.x)
        if (h[t]) atomicAdd(&s->hist[t], h[t]);
}

__device__ __forceinline__ bool mad_is_out(unsigned key, float med, float thr)
{
    return key != MAD_SENTINEL && __uint_as_float(mad_dev(key, med)) > thr;
}

static __global__ void __launch_bounds__(256) mad_flag_kernel(long n, const unsigned *__restrict__ keys, MadState *s,
                                                              uint8_t *__restrict__ out)
{
    const float med = s->med, thr = s->thr;
    const bool none = s->n_used == 0;
    unsigned cnt = 0;
    const bool al = ((uintptr_t)out & 3) == 0;         // the caller's array: words where it is aligned
    const long n4 = al ? n / 4 : 0, step = (long)gridDim.x * blockDim.x;
    const long t0 = (long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long i = t0; i < n4; i += step) {
        const uint4 k = __ldg(reinterpret_cast<const uint4 *>(keys) + i);
        uchar4 f = make_uchar4(0, 0, 0, 0);
        if (!none) {
            f.x = mad_is_out(k.x, med, thr);
            f.y = mad_is_out(k.y, med, thr);
            f.z = mad_is_out(k.z, med, thr);
            f.w = mad_is_out(k.w, med, thr);
        }
        reinterpret_cast<uchar4 *>(out)[i] = f;
        cnt += f.x + f.y + f.z + f.w;
    }
    for (long i = 4 * n4 + t0; i < n; i += step) {
        const uint8_t f = !none && mad_is_out(__ldg(keys + i), med, thr) ? 1 : 0;
        out[i] = f;
        cnt += f;
    }
    for (int d = 16; d > 0; d >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, d);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(&s->n_flagged, (unsigned long long)cnt);
}

// Per-baseline mode: one block per unordered antenna pair walks the rows of its strips (one per
// orientation); the two statistics by the same digits with the histogram in shared memory.  A
// pair's keys (4 B x its samples) stay in L2 from the second of the seven walks on.
static __global__ void __launch_bounds__(256) mad_group_kernel(const int2 *groups, const int *strip_off,
                                                               const int *strip_rows, int n_chan,
                                                               const unsigned *__restrict__ keys, float factor, MadState *st,
                                                               uint8_t *__restrict__ out)
{
    __shared__ unsigned hist[2048];
    __shared__ int s_bin;
    __shared__ unsigned long long s_rank, s_part[256], s_used;
    const int2 g = groups[blockIdx.x];
    const int a0 = strip_off[g.x], n0 = strip_off[g.x + 1] - a0;
    const int b0 = g.y >= 0 ? strip_off[g.y] : 0, n1 = g.y >= 0 ? strip_off[g.y + 1] - b0 : 0;
    const long n = (long)(n0 + n1) * n_chan;
    const int dr = (int)(blockDim.x / n_chan), dc = (int)blockDim.x - dr * n_chan;
    // f(position in the arrays) for every sample of the pair
    auto walk = [&](auto &&f) {
        int r = (int)threadIdx.x / n_chan, c = (int)threadIdx.x - r * n_chan;
#pragma unroll 4
        for (long i = threadIdx.x; i < n; i += blockDim.x) {
            const int row = __ldg(strip_rows + (r < n0 ? a0 + r : b0 + r - n0));
            f((size_t)row * n_chan + c);
            c += dc;
            r += dr;
            if (c >= n_chan) { c -= n_chan; ++r; }
        }
    };
    if (threadIdx.x == 0) s_used = 0;
    float med = 0.f, thr = INFINITY;
    for (int dev = 0; dev < 2; ++dev) {
        unsigned prefix = 0;
        unsigned long long k = 0;
        for (int level = 0; level < MAD_LEVELS; ++level) {
            for (int t = threadIdx.x; t < 2048; t += blockDim.x) hist[t] = 0;
            __syncthreads();
            const unsigned above = mad_above(level);
            unsigned used = 0;
            walk([&](size_t s) {
                const unsigned key = __ldg(keys + s);
                used += key != MAD_SENTINEL;
                const unsigned v = dev ? mad_dev(key, med) : key;
                // unused samples are left out: the statistics are over the pair's used samples
                if (key != MAD_SENTINEL && (v & above) == prefix) atomicAdd(&hist[mad_digit(v, level) & 2047], 1u);
            });
            if (dev == 0 && level == 0) {
                for (int d = 16; d > 0; d >>= 1) used += __shfl_down_sync(0xffffffffu, used, d);
                if ((threadIdx.x & 31) == 0) atomicAdd(&s_used, (unsigned long long)used);
            }
            __syncthreads();
            if (s_used == 0) break;
            if (level == 0) k = (s_used - 1) / 2;
            mad_find(hist, level == 0 ? 2048 : 1024, k, &s_bin, &s_rank, s_part);
            prefix |= (unsigned)s_bin << (level == 0 ? 20 : (level == 1 ? 10 : 0));
            k = s_rank;
            __syncthreads();
        }
        if (s_used == 0) break;
        if (dev == 0) med = __uint_as_float(prefix);
        else thr = __fmul_rn(factor, __uint_as_float(prefix));
    }
    unsigned cnt = 0;
    walk([&](size_t s) {
        const uint8_t f = mad_is_out(__ldg(keys + s), med, thr) ? 1 : 0;
        out[s] = f;
        cnt += f;
    });
    for (int d = 16; d > 0; d >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, d);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(&st->n_flagged, (unsigned long long)cnt);
}

} // namespace qc

static int rows_grid(long rows, int sm_count, int per_sm)
{
    return (int)std::max(1L, std::min((rows + 7) / 8, (long)sm_count * per_sm));
}

template <bool MAD, int NT>
static cudaError_t launch_rows(const qc::ResArgs &a, bool m16, unsigned *keys, qc::MadState *state, int sm_count,
                               cudaStream_t st)
{
    const int grid = rows_grid(a.D.n_row, sm_count, 8);
    if (m16) qc::residual_kernel<true, MAD, NT><<<grid, 256, 0, st>>>(a, keys, state);
    else qc::residual_kernel<false, MAD, NT><<<grid, 256, 0, st>>>(a, keys, state);
    return cudaGetLastError();
}

// chains of up to two terms have their own instances: the code of the further terms costs registers
cudaError_t residual_launch(const qc::ResArgs &a, bool m16, int sm_count, cudaStream_t st)
{
    return a.C.n_terms <= 2 ? launch_rows<false, 2>(a, m16, nullptr, nullptr, sm_count, st)
                            : launch_rows<false, qc::MAXT>(a, m16, nullptr, nullptr, sm_count, st);
}

cudaError_t mad_keys_launch(const qc::ResArgs &a, bool m16, unsigned *keys, qc::MadState *state, int sm_count,
                            cudaStream_t st)
{
    return a.C.n_terms <= 2 ? launch_rows<true, 2>(a, m16, keys, state, sm_count, st)
                            : launch_rows<true, qc::MAXT>(a, m16, keys, state, sm_count, st);
}

cudaError_t mad_global_launch(long n, const unsigned *keys, float factor, qc::MadState *state, uint8_t *out, int sm_count,
                              cudaStream_t st)
{
    const int grid = (int)std::max(1L, std::min((n / 4 + 255) / 256, (long)sm_count * 8));
    for (int dev = 0; dev < 2; ++dev)
        for (int level = 0; level < qc::MAD_LEVELS; ++level) {
            qc::mad_hist_kernel<<<grid, 256, 0, st>>>(n, keys, state, dev, level);
            qc::mad_pick_kernel<<<1, 256, 0, st>>>(state, dev, level, factor);
        }
    qc::mad_flag_kernel<<<grid, 256, 0, st>>>(n, keys, state, out);
    return cudaGetLastError();
}

cudaError_t mad_group_launch(int n_groups, const int2 *groups, const int *strip_off, const int *strip_rows, int n_chan,
                             const unsigned *keys, float factor, qc::MadState *state, uint8_t *out, cudaStream_t st)
{
    if (n_groups == 0) return cudaSuccess;
    qc::mad_group_kernel<<<n_groups, 256, 0, st>>>(groups, strip_off, strip_rows, n_chan, keys, factor, state, out);
    return cudaGetLastError();
}
