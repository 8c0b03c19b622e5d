// qc_delay_sums.cu -- the solve of a delay term from products formed once (not in the paper).
//
// The gains of a delay term have unit modulus, so with the other term fixed and X = O_p M O_q^H (the
// other term folded into the model) the blocks of one sample are
//   h_p,k = sum_j w_kj |X_kj|^2 |g_q,j|^2 = sum_j w_kj |X_kj|^2              (no gains in it), and
//   Im(conj(g_p,k) JHr_p,k) = sum_j Im z_kj,   z_kj = conj(g_p,k) g_q,j w_kj conj(X_kj) D_kj
// (the terms h |g_p|^2 are real), for antenna q h_q,j = sum_k w_kj |X_kj|^2 and -sum_k Im z_kj.  One pass
// over the samples forms
//   T[time interval][pair][channel]_kj = sum w_kj conj(X_kj) D_kj   (four complex FP32, 32 B), and
//   H[interval][antenna] = sum h (1, omega', omega'^2) per correlation (FP64),
// and every iteration reads T alone: 32 B a sample and about 45 instructions instead of 80 B and
// about 300.
#include "qc_internal.h"

#include <algorithm>

namespace qc {

constexpr unsigned WARP_ALL = 0xffffffffu;

struct HsumLayout {
    static constexpr int KR = KG_HSUM, KG = KG_HSUM;
    __device__ static constexpr int g(int i) { return i; }
};

__device__ __forceinline__ void red_add_v4(float4 *p, float4 v)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(__cvta_generic_to_global(p)), "f"(v.x),
                 "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

// The pass: each warp walks units (a block of rows of one baseline strip, its 32-channel chunks
// inside each row or, with chunk_major, its rows inside one chunk), DEPTH - 1 steps ahead through a
// cp.async ring.  A lane (one channel) keeps T of its slot until the time interval or chunk
// changes (then added to the slot, in FP64 where the slot takes several additions) and H until its
// parameter interval or the pair changes.  HBM-bound: it reads the samples once and writes T (80 +
// 32 B a sample with one integration an interval).
template <int OK, bool M16>
static __global__ void __launch_bounds__(128, 4) delay_sums_pass_kernel(const DelaySumsArgs a)
{
    constexpr int V4 = M16 ? 4 : 5, DEPTH = 4;
    extern __shared__ float4 s_ring[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    float4 *ring = s_ring + (size_t)wib * DEPTH * (V4 * 32 + 2);
    const int n_chan = a.n_chan;
    const int groups = a.chunk_major ? a.n_chunks : 1;
    const long n_units = (long)a.n_strips * a.n_rb * groups;
    const long stride = ((long)gridDim.x * blockDim.x) >> 5;
    // issue cursor
    long unit = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int k0 = 0, k1 = 0, k = 0, ch = 0, ch0 = 0, ch1 = 0;
    // the current row's entry, loaded a step before its copies are issued (their addresses depend on it)
    int4 mr = make_int4(-1, 0, 0, 0);
    float msc = 0.f;
    auto load_row = [&]() {
        mr = __ldg(a.mrows + k);
        if constexpr (M16) msc = __ldg(a.mscale + k);
    };
    auto unit_start = [&]() {
        for (; unit < n_units; unit += stride) {
            const int g = (int)(unit % groups);
            const long sr = unit / groups;
            const int s = (int)(sr / a.n_rb), b = (int)(sr % a.n_rb);
            ch0 = a.chunk_major ? g : 0;
            ch1 = a.chunk_major ? g + 1 : a.n_chunks;
            const int kb = __ldg(a.strip_off + s);
            k0 = kb + b * a.rb;
            k1 = min(__ldg(a.strip_off + s + 1), k0 + a.rb);
            if (k0 < k1) break;
        }
        k = k0;
        ch = ch0;
        if (unit < n_units) load_row();
    };
    unit_start();
    int is = 0;
    auto issue = [&]() {
        float4 *stage = ring + (size_t)is * (V4 * 32 + 2);
        if (++is == DEPTH) is = 0;
        int4 m0 = make_int4(-1, 0, 0, 0), m1 = make_int4(0, 0, 0, 0);
        if (unit < n_units) {
            const int c = ch * 32 + lane;
            const bool rd = mr.x >= 0 && c < n_chan;
            const size_t s = rd ? (size_t)mr.x * n_chan + c : 0;
            const uint32_t nb = rd ? 16u : 0u;
            cp_async16(stage + lane, a.vis + 2 * s, nb);
            cp_async16(stage + 32 + lane, a.vis + 2 * s + 1, nb);
            cp_async16(stage + 64 + lane, a.wf + s, nb);
            if constexpr (M16) {
                cp_async16(stage + 96 + lane, a.model16 + s, nb);
            } else {
                cp_async16(stage + 96 + lane, a.model + 2 * s, nb);
                cp_async16(stage + 128 + lane, a.model + 2 * s + 1, nb);
            }
            m0 = make_int4(__ldg(a.t_map + mr.y), ch, mr.z, mr.w);
            if constexpr (OK != KIND_NONE) m1.x = __ldg(a.to.t_map + mr.y);
            if constexpr (M16) m1.y = __float_as_int(msc);
        }
        if (lane == 0) {
            reinterpret_cast<int4 *>(stage + V4 * 32)[0] = m0;
            reinterpret_cast<int4 *>(stage + V4 * 32)[1] = m1;
        }
        cp_async_commit();
        if (unit < n_units) {
            bool done;
            const int kp = k;
            if (a.chunk_major) done = ++k == k1;
            else { if (++ch == ch1) { ch = ch0; ++k; } done = k >= k1; }
            if (done) {
                unit += stride;
                unit_start();
            } else if (k != kp) {
                load_row();
            }
        }
    };
#pragma unroll
    for (int d = 0; d < DEPTH - 1; ++d) issue();

    Acc<KG_HSUM, false> Hp, Hq;
    Hp.zero();
    Hq.zero();
    float t[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) t[i] = 0.f;
    long cur_slot = -1;
    int cur_key = -1, cur_pq = -1, stage_c = 0;
    auto write_slot = [&]() {
        if (cur_slot >= 0) {
            float4 *dst = a.T + (size_t)cur_slot * 64 + lane;
            const float4 lo = make_float4(t[0], t[1], t[2], t[3]), hi = make_float4(t[4], t[5], t[6], t[7]);
            if (a.store) {
                dst[0] = lo;
                dst[32] = hi;
            } else if (a.T64) {
                double *d = a.T64 + ((size_t)cur_slot * 64 + lane) * 4;
#pragma unroll
                for (int i = 0; i < 8; ++i) atomicAdd(d + (i < 4 ? i : 128 + i - 4), (double)t[i]);
            } else {
                red_add_v4(dst, lo);
                red_add_v4(dst + 32, hi);
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = 0.f;
    };
    for (;;) {
        __syncwarp();                       // every lane is done with the stage about to be refilled
        issue();
        cp_async_wait<DEPTH - 1>();
        __syncwarp();
        const float4 *st = ring + (size_t)stage_c * (V4 * 32 + 2);
        if (++stage_c == DEPTH) stage_c = 0;
        const int4 m0 = reinterpret_cast<const int4 *>(st + V4 * 32)[0];
        const int4 m1 = reinterpret_cast<const int4 *>(st + V4 * 32)[1];
        if (m0.x < 0) break;
        const int c = m0.y * 32 + lane, pq = m0.w;
        const bool in = c < n_chan;
        const int cc = in ? c : n_chan - 1;
        const long slot = ((long)m0.x * a.n_chunks + m0.y) * a.n_up + (m0.z & 0x7fffffff);
        if (slot != cur_slot) { write_slot(); cur_slot = slot; }
        const int key = in ? m0.x * a.n_fint + __ldg(a.fmap + cc) : -1;
        if (__any_sync(WARP_ALL, key != cur_key || pq != cur_pq)) {
            // lanes past the last channel keep a key of -1: a flush covers their empty sums
            if (__any_sync(WARP_ALL, cur_key >= 0))
                flush_pair<KG_HSUM, KG_HSUM, HsumLayout>(Hp, Hq, cur_key, cur_pq, lane, a.active, a.hsum, a.n_ant);
            cur_key = key;
            cur_pq = pq;
        }
        float4 w = st[64 + lane];
        if (w.x != 0.f || w.y != 0.f || w.z != 0.f || w.w != 0.f) {
            J2 D = j_from(st[lane], st[32 + lane]);
            const bool conj = m0.z < 0;     // the row is (q, p): D -> D^H, M -> M^H, w permuted
            const int p = pq & 0xffff, q = (int)((unsigned)pq >> 16);
            J2 X;
            if constexpr (M16) X = load_model16(*reinterpret_cast<const uint4 *>(st + 96 + lane), __int_as_float(m1.y));
            else X = j_from(st[96 + lane], st[128 + lane]);
            if (conj) X = j_herm(X);
            if constexpr (OK != KIND_NONE) {
                const int fo = __ldg(a.to.f_map + cc);
                const J2 Op = fetch_k<OK>(a.to, a.n_ant, m1.x, fo, p);
                const J2 Oq = fetch_k<OK>(a.to, a.n_ant, m1.x, fo, q);
                if constexpr (OK == KIND_DIAG) X = j_muld(j_dmul(Op.a, Op.d, X), cconj(Oq.a), cconj(Oq.d));
                else X = j_mul_h(j_mul(Op, X), Oq);
            }
            if (conj) {
                D = j_herm(D);
                w = make_float4(w.x, w.z, w.y, w.w);
            }
            const float2 wd[4] = { cscale(D.a, w.x), cscale(D.b, w.y), cscale(D.c, w.z), cscale(D.d, w.w) };
            const float2 x[4] = { X.a, X.b, X.c, X.d };
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 v = cfma_conj(x[i], wd[i], make_float2(t[2 * i], t[2 * i + 1]));
                t[2 * i] = v.x;
                t[2 * i + 1] = v.y;
            }
            const float s0 = w.x * cnorm2(x[0]), s1 = w.y * cnorm2(x[1]), s2 = w.z * cnorm2(x[2]), s3 = w.w * cnorm2(x[3]);
            const float om = __ldg(a.omega + cc), om2 = om * om;
            const float hp0 = s0 + s1, hp1 = s2 + s3, hq0 = s0 + s2, hq1 = s1 + s3;
            Hp.s[0] += hp0;
            Hp.s[1] = fmaf(hp0, om, Hp.s[1]);
            Hp.s[2] = fmaf(hp0, om2, Hp.s[2]);
            Hp.s[3] += hp1;
            Hp.s[4] = fmaf(hp1, om, Hp.s[4]);
            Hp.s[5] = fmaf(hp1, om2, Hp.s[5]);
            Hq.s[0] += hq0;
            Hq.s[1] = fmaf(hq0, om, Hq.s[1]);
            Hq.s[2] = fmaf(hq0, om2, Hq.s[2]);
            Hq.s[3] += hq1;
            Hq.s[4] = fmaf(hq1, om, Hq.s[4]);
            Hq.s[5] = fmaf(hq1, om2, Hq.s[5]);
        }
    }
    write_slot();
    if (__any_sync(WARP_ALL, cur_key >= 0))
        flush_pair<KG_HSUM, KG_HSUM, HsumLayout>(Hp, Hq, cur_key, cur_pq, lane, a.active, a.hsum, a.n_ant);
    cp_async_wait<0>();
}

// FP64 products to the FP32 ones that the iterations read (four a thread)
static __global__ void delay_round_kernel(long n4, const double2 *__restrict__ src, float4 *__restrict__ dst)
{
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (long)gridDim.x * blockDim.x) {
        const double2 a = src[2 * i], b = src[2 * i + 1];
        dst[i] = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
    }
}

// One iteration's right-hand sides: a CTA per (time interval, 32-channel chunk), lanes over the
// channels.  The antennas' gains at those channels are evaluated once into shared memory; the pairs
// are walked in 8 x 8 tiles of antennas handed out to the warps, so that the eight q sums of a row of
// a tile stay in registers and only their totals go to the shared sums (FP64: the FP32 terms of 8
// pairs at most).  T streams at 1 KB a pair with eight 16-byte loads a lane in flight; nothing else
// comes from DRAM.
constexpr int DT = 8;                       // antennas of a tile's side

static __global__ void __launch_bounds__(256, 2) delay_sums_iter_kernel(const DelaySumsArgs a)
{
    if (__ldg(a.n_active) == 0) return;
    extern __shared__ float4 s_gains[];     // [n_ant][32] (g_X, g_Y)
    double *s_r = reinterpret_cast<double *>(s_gains + (size_t)a.n_ant * 32);   // [n_ant][2][32] r_X, r_Y
    __shared__ int s_tile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int tint = blockIdx.x / a.n_chunks, chunk = blockIdx.x % a.n_chunks, na = a.n_ant;
    const int c = min(chunk * 32 + lane, a.n_chan - 1);
    const bool in = chunk * 32 + lane < a.n_chan;
    const int bin = tint * a.n_fint + __ldg(a.fmap + c);
    const bool act = in && a.active[bin];
    if (!__any_sync(WARP_ALL, act)) return; // the same in every warp: converged intervals read nothing
    {
        const double w = DELAY_TWO_PI * a.nu[c];
        for (int i = warp; i < na; i += nw) {
            const double *u = a.params + ((size_t)bin * na + i) * 4;
            const float2 gx = delay_gain_f32(u[0], u[1], w), gy = delay_gain_f32(u[2], u[3], w);
            s_gains[i * 32 + lane] = make_float4(gx.x, gx.y, gy.x, gy.y);
            s_r[i * 64 + lane] = s_r[i * 64 + 32 + lane] = 0.0;
        }
    }
    if (threadIdx.x == 0) s_tile = 0;
    __syncthreads();
    const float4 *T = a.T + ((size_t)blockIdx.x * a.n_up) * 64 + lane;
    const int nb = (na + DT - 1) / DT, n_tile = nb * (nb + 1) / 2;
    for (;;) {
        int tile = 0;
        if (lane == 0) tile = atomicAdd(&s_tile, 1);
        tile = __shfl_sync(WARP_ALL, tile, 0);
        if (tile >= n_tile) break;
        int pb = 0;
        while (tile >= nb - pb) { tile -= nb - pb; ++pb; }
        const int q0 = (pb + tile) * DT, p_end = min(na, (pb + 1) * DT);
        float2 rq[DT];
#pragma unroll
        for (int j = 0; j < DT; ++j) rq[j] = make_float2(0.f, 0.f);
        for (int p = pb * DT; p < p_end; ++p) {
            const int ql = q0 + (lane & (DT - 1));
            const int up_l = ql > p && ql < na ? __ldg(a.upair + (size_t)p * na + ql) : -1;
            const float4 gp = s_gains[p * 32 + lane];
            float2 rp = make_float2(0.f, 0.f);
#pragma unroll
            for (int h = 0; h < DT; h += 4) {
                float4 t0[4], t1[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int up = __shfl_sync(WARP_ALL, up_l, h + j);
                    t0[j] = t1[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (up >= 0) {
                        t0[j] = __ldcg(T + (size_t)up * 64);
                        t1[j] = __ldcg(T + (size_t)up * 64 + 32);
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 gq = s_gains[min(q0 + h + j, na - 1) * 32 + lane];
                    // Im(conj(g_p,k) T_kj g_q,j)
                    const float2 a00 = make_float2(fmaf(gp.x, t0[j].x, gp.y * t0[j].y), fmaf(gp.x, t0[j].y, -gp.y * t0[j].x));
                    const float2 a01 = make_float2(fmaf(gp.x, t0[j].z, gp.y * t0[j].w), fmaf(gp.x, t0[j].w, -gp.y * t0[j].z));
                    const float2 a10 = make_float2(fmaf(gp.z, t1[j].x, gp.w * t1[j].y), fmaf(gp.z, t1[j].y, -gp.w * t1[j].x));
                    const float2 a11 = make_float2(fmaf(gp.z, t1[j].z, gp.w * t1[j].w), fmaf(gp.z, t1[j].w, -gp.w * t1[j].z));
                    const float z00 = fmaf(a00.x, gq.y, a00.y * gq.x), z01 = fmaf(a01.x, gq.w, a01.y * gq.z);
                    const float z10 = fmaf(a10.x, gq.y, a10.y * gq.x), z11 = fmaf(a11.x, gq.w, a11.y * gq.z);
                    rp.x += z00 + z01;
                    rp.y += z10 + z11;
                    rq[h + j].x -= z00 + z10;
                    rq[h + j].y -= z01 + z11;
                }
            }
            atomicAdd(&s_r[p * 64 + lane], (double)rp.x);
            atomicAdd(&s_r[p * 64 + 32 + lane], (double)rp.y);
        }
#pragma unroll
        for (int j = 0; j < DT; ++j)
            if (q0 + j < na) {
                atomicAdd(&s_r[(q0 + j) * 64 + lane], (double)rq[j].x);
                atomicAdd(&s_r[(q0 + j) * 64 + 32 + lane], (double)rq[j].y);
            }
    }
    __syncthreads();
    // sums over the chunk's channels of r (1, omega'), per parameter interval
    const float om = __ldg(a.omega + c);
    const unsigned acts = __ballot_sync(WARP_ALL, act);
    const int b0 = __shfl_sync(WARP_ALL, bin, __ffs(acts) - 1);
    const bool one = __all_sync(WARP_ALL, !act || bin == b0);
    for (int i = warp; i < na; i += nw) {
        const double rx = act ? s_r[i * 64 + lane] : 0.0, ry = act ? s_r[i * 64 + 32 + lane] : 0.0;
        const double w[4] = { rx, rx * om, ry, ry * om };
        float v[4], tail[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            v[e] = (float)w[e];
            tail[e] = isfinite(v[e]) ? (float)(w[e] - (double)v[e]) : 0.f;
        }
        if (one) {
            const double tot = reduce_words<4>(v, tail, lane);
            if ((lane & 7) == 0) atomicAdd(a.acc + ((size_t)b0 * na + i) * KG_SUMS + 6 + (lane >> 3), tot);
        } else if (act) {
#pragma unroll
            for (int e = 0; e < 4; ++e) atomicAdd(a.acc + ((size_t)bin * na + i) * KG_SUMS + 6 + e, w[e]);
        }
    }
}

} // namespace qc

template <int OK, bool M16>
static cudaError_t launch_dsum_pass(const qc::DelaySumsArgs &a, int sm_count, cudaStream_t st)
{
    constexpr int V4 = M16 ? 4 : 5, DEPTH = 4;
    const int smem = 4 * DEPTH * (V4 * 32 + 2) * (int)sizeof(float4);
    const void *fn = (const void *)qc::delay_sums_pass_kernel<OK, M16>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    int occ = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, 128, smem);
    if (e != cudaSuccess) return e;
    const long units = (long)a.n_strips * a.n_rb * (a.chunk_major ? a.n_chunks : 1);
    const int grid = (int)std::max(1L, std::min((long)sm_count * std::max(1, occ), (units + 3) / 4));
    qc::delay_sums_pass_kernel<OK, M16><<<grid, 128, smem, st>>>(a);
    return cudaGetLastError();
}

template <int OK> static cudaError_t launch_dsum_pass_ok(const qc::DelaySumsArgs &a, int sm_count, cudaStream_t st)
{
    return a.model16 ? launch_dsum_pass<OK, true>(a, sm_count, st) : launch_dsum_pass<OK, false>(a, sm_count, st);
}

cudaError_t dsum_launch_pass(const qc::DelaySumsArgs &a, int ok, int sm_count, cudaStream_t st)
{
    if (ok == qc::KIND_NONE) return launch_dsum_pass_ok<qc::KIND_NONE>(a, sm_count, st);
    if (ok == qc::KIND_DIAG) return launch_dsum_pass_ok<qc::KIND_DIAG>(a, sm_count, st);
    return launch_dsum_pass_ok<qc::KIND_FULL>(a, sm_count, st);
}

cudaError_t dsum_launch_round(size_t words, const double *src, float4 *dst, int sm_count, cudaStream_t st)
{
    const long n4 = (long)(words / 4);
    const int grid = (int)std::max(1L, std::min((n4 + 255) / 256, (long)sm_count * 16));
    qc::delay_round_kernel<<<grid, 256, 0, st>>>(n4, (const double2 *)src, dst);
    return cudaGetLastError();
}

cudaError_t dsum_launch_iter(const qc::DelaySumsArgs &a, cudaStream_t st)
{
    const int smem = a.n_ant * 32 * (int)(sizeof(float4) + 2 * sizeof(double));
    const cudaError_t e = cudaFuncSetAttribute(qc::delay_sums_iter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    qc::delay_sums_iter_kernel<<<a.n_tint * a.n_chunks, 256, smem, st>>>(a);
    return cudaGetLastError();
}
