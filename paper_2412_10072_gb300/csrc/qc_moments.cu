// qc_moments.cu -- the solve of one term from per-(interval, antenna pair) sums (not in the paper).
//
// While one term of a chain is solved the others are fixed, so every sample of a baseline
// (p, q) in a solution interval enters J^H W J and J^H W r (Eq. jhj_entry_simplified,
// Eq. jhr_entry_simplified) through sums that do not depend on the solved gains.  The sums are
// kept per unordered pair p < q (a row with ant1 > ant2 enters through its conjugate baseline:
// D -> D^H, M -> M^H, the cross-hand weights swapped, p and q exchanged); kj = 2k + j indexes the
// weight and data of correlation (k, j).
//
// Full form: the solved term G is full-Jones with no term to its left.  With X = R_p M R_q^H, R the
// term to its right (X = M when there is none), and u = 2l + m indexing X_lm:
//     S[kj][u][v] = sum w_kj conj(X_u) X_v,  T[kj][u] = sum w_kj conj(X_u) D_kj    (96 words of 100)
//     JHJ_p[(k,l),(k,l')] += sum_j sum_m sum_m' G_q,jm conj(G_q,jm') S[kj][(l,m)][(l',m')]
//     b_p[(k,l)]          += sum_j sum_m G_q,jm T[kj][(l,m)]
//     JHJ_q[(k,l),(k,l')] += sum_j sum_m sum_m' G_p,jm conj(G_p,jm') conj(S[jk][(m,l)][(m',l')])
//     b_q[(k,l)]          += sum_j sum_m G_p,jm conj(T[jk][(m,l)])
// E form: the solved term g (diagonal or phase-only) has a full term L to its left.  With
// E_kj,ab = L_p,ka M_ab conj(L_q,jb) and u = 2a + b:
//     S'[u][v] = sum sum_kj w_kj conj(E_kj,u) E_kj,v,  T'[u] = sum sum_kj w_kj conj(E_kj,u) D_kj
//                                                                                  (24 words of 28)
//     JHJ_p[a][a'] += sum_b sum_b' g_q,b conj(g_q,b') S'[(a,b)][(a',b')],  b_p[a] += sum_b g_q,b T'[(a,b)]
//     JHJ_q[b][b'] += sum_a sum_a' g_p,a conj(g_p,a') conj(S'[(a,b)][(a',b')]),
//     b_q[b]       += sum_a g_p,a conj(T'[(a,b)])
// Plain diagonal form: any other diagonal or phase-only solved term (the other term diagonal, or to
// its right).  With X = O_p M O_q^H: S_kj = sum w_kj |X_kj|^2, T_kj = sum w_kj conj(X_kj) D_kj (12 words),
//     JHJ_p[k][k] += sum_j |g_q,j|^2 S_kj,  b_p[k] += sum_j g_q,j T_kj,  and conjugated for q.
// In all of them JHr = b - JHJ vec(g).  One pass over the data per term solve forms the sums
// (mom_pass_kernel): FP32 register sums of a lane's 8 samples (short forms, kept as head and tail beyond
// that) or 16 to 32 (full form), added up over the lanes with the last levels' rounding kept, and
// then to the slots, exactly where a slot takes one addition and in FP64 where it takes several.
// The intervals are independent from there on, so one CTA per interval runs all of its iterations
// (mom_iterate_kernel): an iteration reads 400, 112 or 96 B per (interval, pair) and side out of L2
// (800 and 224 B with tails) instead of 80 B per sample out of HBM, with no launch in between; the
// products and sums over the pairs are compensated.  Error of the gains against FP64 (rms, relative;
// rounding the result alone 2.4e-8), then the iterations on the samples: 7 antennas, 4 x 4 intervals
// 3.8e-8 and 3.8e-8, one interval of 150 x 512 3.1e-8 and 3.0e-8, full-Jones 2.7e-8 and 2.6e-8; 20
// antennas 3.6e-8 and 3.9e-8; 64 antennas, G and B, 3.0e-8 and 3.0e-8.  Time, two-term chain (64
// antennas, 300 x 512, three epochs of 20 iterations a term): 660 ms on the samples, 46.2 ms from sums; 27
// antennas, 61 x 131, intervals of 5 x 17: 3.78 and 0.37 ms; 7 antennas, 60 x 16: 1.02 and 0.23 ms.
#include "qc_internal.h"

#include <algorithm>
#include <type_traits>

namespace qc {

constexpr unsigned FULL_MASK = 0xffffffffu;

// (re, im) += conj(x) y, four fused multiply-adds
__device__ __forceinline__ void cacc_conj(float &re, float &im, float2 x, float2 y)
{
    re = fmaf(x.x, y.x, fmaf(x.y, y.y, re));
    im = fmaf(x.x, y.y, fmaf(-x.y, y.x, im));
}

// One sample's terms added to a lane's register sums, full form (one lane per sample; words as
// the slot: S[kj] at 16 kj, T[kj] at MOM_T + 8 kj; all indices compile-time constants after
// unrolling; X = R_p M R_q^H).
constexpr int MOM_FW = 96;
__device__ __forceinline__ void mom_add(float (&acc)[MOM_FW], const J2 &D, const J2 &X, float4 w)
{
    const float2 x[4] = { X.a, X.b, X.c, X.d };
    const float2 d[4] = { D.a, D.b, D.c, D.d };
    const float wv[4] = { w.x, w.y, w.z, w.w };
    float diag[4];
    float2 off[6];
#pragma unroll
    for (int u = 0; u < 4; ++u) diag[u] = cnorm2(x[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = u + 1; v < 4; ++v) off[mom_pair(u, v)] = cmulc(x[v], x[u]);   // conj(x_u) x_v
#pragma unroll
    for (int kj = 0; kj < 4; ++kj) {
        const int s = 16 * kj;
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[s + u] = fmaf(wv[kj], diag[u], acc[s + u]);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            acc[s + 4 + 2 * i] = fmaf(wv[kj], off[i].x, acc[s + 4 + 2 * i]);
            acc[s + 5 + 2 * i] = fmaf(wv[kj], off[i].y, acc[s + 5 + 2 * i]);
        }
        const float2 wd = cscale(d[kj], wv[kj]);
        const int t = MOM_T + 8 * kj;
#pragma unroll
        for (int u = 0; u < 4; ++u) cacc_conj(acc[t + 2 * u], acc[t + 2 * u + 1], x[u], wd);   // conj(x_u) w d
    }
}

// The diagonal form, one lane per sample: register words [0, 16) S' packed as the full form's
// S blocks, [16, 24) T'.
constexpr int MOM_EW = 24;

// The plain diagonal form: X_kj = R_p,k M_kj conj(R_q,j) for a diagonal fixed term on either side
// (or R_p M R_q^H for a full one on the right): words [0, 4) S_kj = sum w |X_kj|^2, [4, 12) T_kj =
// sum w conj(X_kj) D_kj.
__device__ __forceinline__ void mom_add_d(float (&acc)[MOM_D], const J2 &D, const J2 &X, float4 w)
{
    const float2 x[4] = { X.a, X.b, X.c, X.d };
    const float2 d[4] = { D.a, D.b, D.c, D.d };
    const float wv[4] = { w.x, w.y, w.z, w.w };
#pragma unroll
    for (int kj = 0; kj < 4; ++kj) {
        acc[kj] = fmaf(wv[kj], cnorm2(x[kj]), acc[kj]);
        cacc_conj(acc[4 + 2 * kj], acc[5 + 2 * kj], x[kj], cscale(d[kj], wv[kj]));
    }
}

// E form: with E_kj,ab = L_p,ka M_ab conj(L_q,jb), every product conj(E_kj,ab) E_kj,a'b' is conj(M_ab)
// M_a'b' times a factor of L alone, so the four correlations are summed in those factors first,
//   K[(a,b)][(a',b')] = sum_k P_k[a][a'] sum_j w_kj Q_j[b][b'],
//   P_k[a][a'] = conj(L_p,ka) L_p,ka',  Q_j[b][b'] = L_q,jb conj(L_q,jb'),
// S' += conj(M_ab) M_a'b' K, and T' += conj(M_ab) (L_p^H (w D) L_q)_ab.  Forming the E_kj and adding their
// products one by one takes 390 instructions a sample, this 236, and each word of the sums is
// rounded once or twice a sample instead of eight times.
__device__ __forceinline__ void mom_add_e(float (&acc)[MOM_EW], const J2 &D, const J2 &M, const J2 &Lp,
                                          const J2 &Lq, float4 w)
{
    const float2 m[4] = { M.a, M.b, M.c, M.d };       // M_ab at 2a + b
    const float2 lp[4] = { Lp.a, Lp.b, Lp.c, Lp.d };  // L_p,ka at 2k + a
    const float2 lq[4] = { Lq.a, Lq.b, Lq.c, Lq.d };
    const float wv[4] = { w.x, w.y, w.z, w.w };
    float kd[4] = { 0.f, 0.f, 0.f, 0.f };             // K on the diagonal
    float2 ko[6];                                     // K[u][v] at mom_pair(u, v)
#pragma unroll
    for (int i = 0; i < 6; ++i) ko[i] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float w0 = wv[2 * k], w1 = wv[2 * k + 1];
        const float r0 = fmaf(w0, cnorm2(lq[0]), w1 * cnorm2(lq[2]));      // sum_j w_kj Q_j[0][0]
        const float r1 = fmaf(w0, cnorm2(lq[1]), w1 * cnorm2(lq[3]));
        const float2 qa = cmulc(lq[0], lq[1]), qb = cmulc(lq[2], lq[3]);
        const float2 r01 = make_float2(fmaf(w0, qa.x, w1 * qb.x), fmaf(w0, qa.y, w1 * qb.y));
        const float p0 = cnorm2(lp[2 * k]), p1 = cnorm2(lp[2 * k + 1]);
        const float2 p01 = cmulc(lp[2 * k + 1], lp[2 * k]);                // conj(L_k0) L_k1
        kd[0] = fmaf(p0, r0, kd[0]);
        kd[1] = fmaf(p0, r1, kd[1]);
        kd[2] = fmaf(p1, r0, kd[2]);
        kd[3] = fmaf(p1, r1, kd[3]);
        ko[0] = make_float2(fmaf(p0, r01.x, ko[0].x), fmaf(p0, r01.y, ko[0].y));       // (00)(01)
        ko[5] = make_float2(fmaf(p1, r01.x, ko[5].x), fmaf(p1, r01.y, ko[5].y));       // (10)(11)
        ko[1] = make_float2(fmaf(r0, p01.x, ko[1].x), fmaf(r0, p01.y, ko[1].y));       // (00)(10)
        ko[4] = make_float2(fmaf(r1, p01.x, ko[4].x), fmaf(r1, p01.y, ko[4].y));       // (01)(11)
        // (00)(11): p01 r01;  (01)(10): p01 conj(r01)
        ko[2] = make_float2(fmaf(p01.x, r01.x, fmaf(-p01.y, r01.y, ko[2].x)),
                            fmaf(p01.x, r01.y, fmaf(p01.y, r01.x, ko[2].y)));
        ko[3] = make_float2(fmaf(p01.x, r01.x, fmaf(p01.y, r01.y, ko[3].x)),
                            fmaf(-p01.x, r01.y, fmaf(p01.y, r01.x, ko[3].y)));
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        acc[u] = fmaf(cnorm2(m[u]), kd[u], acc[u]);
#pragma unroll
        for (int v = u + 1; v < 4; ++v) {
            const int i = mom_pair(u, v);
            const float2 z = cmulc(m[v], m[u]);                             // conj(M_u) M_v
            acc[4 + 2 * i] = fmaf(z.x, ko[i].x, fmaf(-z.y, ko[i].y, acc[4 + 2 * i]));
            acc[5 + 2 * i] = fmaf(z.x, ko[i].y, fmaf(z.y, ko[i].x, acc[5 + 2 * i]));
        }
    }
    J2 wd;
    wd.a = cscale(D.a, w.x); wd.b = cscale(D.b, w.y);
    wd.c = cscale(D.c, w.z); wd.d = cscale(D.d, w.w);
    const J2 z = j_mul(j_herm(Lp), j_mul(wd, Lq));
    const float2 zv[4] = { z.a, z.b, z.c, z.d };
#pragma unroll
    for (int u = 0; u < 4; ++u) cacc_conj(acc[16 + 2 * u], acc[17 + 2 * u], m[u], zv[u]);
}

// One word of a slot, x + tail.  A slot that takes one addition (mom64 null) keeps it as head and
// tail, both exact (many antennas: rounded to the head, tail null); where a slot is added to several times the additions are FP64, split into head and tail at the
// end (mom_split_kernel).  FP32 additions there grew the gains' error with the interval: 2.0e-7 for
// one interval of 7 antennas over 150 x 512, 3.0e-8 like this.
__device__ __forceinline__ void slot_add(const MomArgs &a, size_t i, float x, float tail)
{
    if (a.mom64) {
        atomicAdd(a.mom64 + i, (double)x + (double)tail);
    } else {
        const float h = x + tail, l = tail - (h - x);
        atomicAdd(a.mom + i, h);
        if (a.tail && isfinite(h) && l != 0.f) atomicAdd(a.tail + i, l);   // an infinite or NaN head has no tail
    }
}

// Add the warp's register sums (NW words, the slot's order; heads acc, tails lo(v)) to the sums of each
// lane's key (-1: nothing, sums of zero) and zero them:
//  - one key for the warp: a reduce-scatter of 32 words at a time (after the halvings at lane
//    offsets 16 .. 1 lane L holds word L of the group), then one coalesced access per group; the
//    last three levels, whose roundings no longer average out, carry their tails;
//  - 32 distinct keys: each lane adds its own words;
//  - otherwise: a segmented reduction per word over the run of equal keys (channel intervals
//    are contiguous, so a run is a range of lanes), stopped at parts of a quarter of the longest run,
//    whose first lanes add them (to FP64 slots, see slots_once).
template <int NW, typename LO>
__device__ __forceinline__ void mom_flush(float (&acc)[NW], LO &&lo, int key, int lane, const MomArgs &a)
{
    constexpr int F = (NW + 31) / 32, P = 32;    // groups of 32 words, one exchange tree each
    constexpr int stride = NW == MOM_FW ? MOM_N : (NW == MOM_EW ? MOM_E : MOM_D);
    const int k0 = __reduce_max_sync(FULL_MASK, key);
    if (__all_sync(FULL_MASK, key == k0 || key < 0)) {
        if (k0 >= 0) {
            // in place, group by group: after the halving at offset o the live words are [0 .. h)
            const size_t at = (size_t)k0 * stride + lane;
#pragma unroll
            for (int v = 0; v < NW; ++v) acc[v] += lo(v);
#pragma unroll
            for (int f = 0; f < F; ++f) {
                float t[4] = { 0.f, 0.f, 0.f, 0.f };
#pragma unroll
                for (int h = P / 2, o = 16; o >= 1; h >>= 1, o >>= 1) {
                    const bool up = (lane & o) != 0;
#pragma unroll
                    for (int i = 0; i < h; ++i) {
                        const float w0 = 32 * f + i < NW ? acc[32 * f + i] : 0.f;
                        const float w1 = 32 * f + i + h < NW ? acc[32 * f + i + h] : 0.f;
                        const float send = up ? w0 : w1;
                        const float keep = up ? w1 : w0;
                        if (32 * f + i >= NW) continue;
                        const float got = __shfl_xor_sync(FULL_MASK, send, o);
                        if (h > 4) {
                            acc[32 * f + i] = keep + got;
                        } else {
                            float e;
                            two_sum(keep, got, acc[32 * f + i], e);
                            if (h < 4) {
                                const float ts = up ? t[i] : t[i + h];
                                e += (up ? t[i + h] : t[i]) + __shfl_xor_sync(FULL_MASK, ts, o);
                            }
                            t[i] = e;
                        }
                    }
                }
                if (32 * f + lane < NW) slot_add(a, at + 32 * f, acc[32 * f], t[0]);
            }
        }
    } else {
        const unsigned m = __match_any_sync(FULL_MASK, key);
        const size_t at = (size_t)(key >= 0 ? key : 0) * stride;
        const int len = key >= 0 ? __popc(m) : 0;
        const int longest = __reduce_max_sync(FULL_MASK, len);
        if (longest <= 1) {
            if (key >= 0) {
#pragma unroll
                for (int v = 0; v < NW; ++v) slot_add(a, at + v, acc[v], lo(v));
            }
        } else {
            const int first = __ffs(m) - 1, end = 32 - __clz(m);
            // lanes of a part: the largest power of two up to a quarter of the longest run
            const int step = 1 << (31 - __clz(max(1, longest >> 2)));
            const int part_end = min(end, first + ((lane - first) / step + 1) * step);
            const bool head = key >= 0 && (lane - first) % step == 0;
#pragma unroll
            for (int v = 0; v < NW; ++v) {
                float x = acc[v] + lo(v);
                for (int d = 1; d < step; d <<= 1) {
                    const float o = __shfl_down_sync(FULL_MASK, x, d);
                    if (lane + d < part_end) x += o;
                }
                if (head) slot_add(a, at + v, x, 0.f);
            }
        }
    }
#pragma unroll
    for (int v = 0; v < NW; ++v) acc[v] = 0.f;
}

// FP64 slots to heads and tails
static __global__ void mom_split_kernel(long n2, const double2 *__restrict__ src, float2 *__restrict__ dst,
                                        float2 *__restrict__ tail)
{
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += (long)gridDim.x * blockDim.x) {
        const double2 v = src[i];
        const float2 h = make_float2((float)v.x, (float)v.y);
        dst[i] = h;
        if (tail) tail[i] = make_float2(isfinite(h.x) ? (float)(v.x - (double)h.x) : 0.f,
                                        isfinite(h.y) ? (float)(v.y - (double)h.y) : 0.f);
    }
}

// The rows of the baseline strips in strip order, as the pass reads them: {row (-1: no usable
// sample), time, pair | conj << 31, p | q << 16} with (p, q) the baseline as the sums orient it.
static __global__ void mom_rows_kernel(long n, const int *strip_rows, const int4 *rows, const uint8_t *row_live,
                                       const int *up_of_bl, const float *bl_scale, int4 *out, float *scale)
{
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int row = strip_rows[k];
    const int4 r = rows[row];
    const bool conj = r.x > r.y;
    const int p = conj ? r.y : r.x, q = conj ? r.x : r.y;
    out[k] = make_int4(row_live[row] ? row : -1, r.z, (int)((unsigned)up_of_bl[r.w] | (conj ? 0x80000000u : 0u)),
                       p | (q << 16));
    if (scale) scale[k] = bl_scale[r.w];
}

// The strips without their rows of no usable sample (one warp per strip): the entries kept, from the
// strip's offset on, and where they end.
static __global__ void mom_live_kernel(int n_strips, const int *strip_off, const int4 *rows, const float *scale, int4 *live,
                                       float *live_scale, int *strip_end)
{
    const int s = (int)(((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (s >= n_strips) return;
    const int k1 = strip_off[s + 1];
    int at = strip_off[s];
    for (int k0 = at; k0 < k1; k0 += 32) {
        const int k = k0 + lane;
        const int4 r = k < k1 ? rows[k] : make_int4(-1, 0, 0, 0);
        const unsigned m = __ballot_sync(FULL_MASK, r.x >= 0);
        if (r.x >= 0) {
            const int to = at + __popc(m & ((1u << lane) - 1));
            live[to] = r;
            if (live_scale) live_scale[to] = scale[k];
        }
        at += __popc(m);
    }
    if (lane == 0) strip_end[s] = at;
}

template <int K>
__device__ __forceinline__ J2 fac_jones(const float4 *o)
{
    if constexpr (K == KIND_FULL) return j_from(o[0], o[1]);
    else if constexpr (K == KIND_DIAG) return j_diag(o[0]);
    else return j_identity();
}

// Shape of a warp's ring of the pass (one lane per sample, 32-channel chunks): per stage, in
// float4 units, the chunk's data quads d0 [0, 32), d1 [32, 64), model quads m0 [64, 96) and m1
// (FP16 model: one word), folded weights w, then the fixed term's table entries for p and for
// q (NO float4 each, per channel, or only the first one when the chunk lies in one of the term's
// frequency intervals), the lanes' keys (32 ints) and one int4 of meta data.
template <int FORM, int OK, bool M16> struct MomRing {
    static constexpr int NO = OK == KIND_FULL ? 2 : (OK == KIND_DIAG ? 1 : 0);
    static constexpr int OFF_W = M16 ? 96 : 128;
    static constexpr int OFF_OP = OFF_W + 32, OFF_OQ = OFF_OP + 32 * NO, OFF_KEY = OFF_OQ + 32 * NO;
    static constexpr int OFF_META = OFF_KEY + 8;
    static constexpr int STAGE = OFF_META + 1;               // float4 per stage
    // three CTAs of 4 warps per SM (the full form's 96 register sums fit 168 registers); ring
    // depth as the shared memory of three CTAs allows
    static constexpr int PER_SM = 3;
    static constexpr int DEPTH = NO == 2 ? 3 : (NO == 1 ? 4 : 6);
    static constexpr size_t SMEM = (size_t)4 * DEPTH * STAGE * sizeof(float4);
    // A lane's sums over a long strip are FP32 sums of terms of one sign, whose rounding grows with
    // the number of terms and moves the fixed point of all antennas the same way.  The short slots keep a
    // head and a tail that take the sums every LIFT steps, the rounding of the head going to the
    // tail (kept in shared memory where the registers are taken); the full form, which has neither,
    // goes to its slot every 32 steps (16 with the FP16 model).
    static constexpr bool TWO_LEVEL = FORM != FORM_FULL;
    static constexpr bool TAIL_SMEM = FORM == FORM_E;
    static constexpr int LIFT = 8;
    static constexpr int FLUSH_EVERY = TWO_LEVEL ? 1 << 30 : mom_flush_every(M16);
    static constexpr size_t TAIL = TAIL_SMEM ? (size_t)128 * MOM_EW * sizeof(float) : 0;
    // integrations whose time maps fit beside the rings (and tails) of three CTAs
    static constexpr int MAX_STAGED = TAIL_SMEM ? 512 : 1024;
};

constexpr int MOM_END = 2;       // meta: the warp's steps have run out (bit 0: conjugate baseline)

// The issuing side of a warp: its steps in order, unit by unit (grid stride; a unit is a block
// of rb rows of one baseline strip x a group of chunks), each copied into a ring stage by
// cp.async (zero-filled past the last channel).  Rows without usable data are not in the table.  What
// belongs to a row is computed once a row: row-major units take all chunks of it one after the
// other, and the bookkeeping of a step was as long as its arithmetic.
template <int FORM, int OK, bool M16> struct MomCursor {
    using R = MomRing<FORM, OK, M16>;
    long unit, n_units, stride;
    int n_groups;
    int k0, k1, ch0, ch1, k, ch;
    bool cm;
    // the next row's entry, loaded when the cursor reaches the row (a step before its first use)
    int4 mr = make_int4(-1, 0, 0, 0);
    float msc = 0.f;
    bool fresh = false;                   // mr has not been turned into the values below
    size_t base = 0;                      // first sample of the row
    int key0 = 0, tab_p = 0, tab_q = 0, meta = 0;   // key, table entries (first interval), conjugate flag
    const int *tmap_n, *tmap_o;           // time maps of the solved and the fixed term (shared memory)
    // frequency intervals of the lane's channel (fixed term: of the chunk's first channel where one
    // stands for all), loaded when the cursor reaches the chunk, a step before their use
    int fn = 0, fo = 0;

    __device__ __forceinline__ void load_chunk(const MomArgs &a, int lane)
    {
        const int c = min(ch * 32 + lane, a.n_chan - 1);
        if (a.tn_map == MAP_ANY || a.tn_map == MAP_CHUNK) fn = __ldg(a.tn.f_map + c);
        if constexpr (R::NO > 0) {
            if (a.to_map == MAP_CHUNK) fo = __ldg(a.to.f_map + ch * 32);
            else if (a.to_map == MAP_ANY) fo = __ldg(a.to.f_map + c);
        }
    }

    __device__ __forceinline__ void load_row(const MomArgs &a)
    {
        mr = __ldg(a.mrows + k);
        if constexpr (M16) msc = __ldg(a.mscale + k);
        fresh = true;
    }

    __device__ __forceinline__ void bounds(const MomArgs &a, int lane)
    {
        // the first unit from here on with rows (or none: unit >= n_units)
        for (; unit < n_units; unit += stride) {
            const int g = (int)(unit % n_groups);
            const long sr = unit / n_groups;
            const int s = (int)(sr / a.n_rb), b = (int)(sr % a.n_rb);
            ch0 = g * a.group;
            ch1 = min(a.n_chunks, ch0 + a.group);
            const int kb = __ldg(a.strip_off + s);
            k0 = kb + b * a.rb;
            k1 = min(__ldg(a.strip_end + s), k0 + a.rb);
            if (k0 < k1) break;
        }
        k = k0;
        ch = ch0;
        if (unit < n_units) {
            load_row(a);
            load_chunk(a, lane);
        }
    }

    __device__ __forceinline__ void start(const MomArgs &a, int lane, long first, long step, const int *tn, const int *to)
    {
        tmap_n = tn;
        tmap_o = to;
        n_groups = (a.n_chunks + a.group - 1) / a.group;
        n_units = (long)a.n_strips * a.n_rb * n_groups;
        stride = step;
        unit = first;
        cm = a.chunk_major != 0;
        bounds(a, lane);
    }

    __device__ __forceinline__ void advance(const MomArgs &a, int lane)
    {
        if (cm) {
            // chunk-major units hold one chunk
            if (++k < k1) { load_row(a); return; }
        } else {
            if (++ch < ch1) { load_chunk(a, lane); return; }
            ch = ch0;
            if (++k < k1) {
                load_row(a);
                if (ch1 - ch0 > 1) load_chunk(a, lane);
                return;
            }
        }
        unit += stride;
        bounds(a, lane);
    }

    __device__ __forceinline__ void issue(const MomArgs &a, int lane, float4 *stage)
    {
        if (unit >= n_units) {
            if (lane == 0) reinterpret_cast<int *>(stage + R::OFF_META)[0] = MOM_END;
            cp_async_commit();
            return;
        }
        if (fresh) {
            fresh = false;
            base = (size_t)mr.x * a.n_chan;
            key0 = tmap_n[mr.y] * a.tn.n_fint * a.n_up + (mr.z & 0x7fffffff);
            meta = mr.z < 0 ? 1 : 0;
            if constexpr (R::NO > 0) {
                const int t = tmap_o[mr.y] * a.n_ant;
                tab_p = (t + (mr.w & 0xffff)) * a.to.n_fint;
                tab_q = (t + (mr.w >> 16)) * a.to.n_fint;
            }
        }
        const int c = ch * 32 + lane;
        const bool in = c < a.n_chan;
        const size_t i = in ? base + c : 0;
        const uint32_t nb = in ? 16u : 0u;
        cp_async16(stage + lane, a.vis + 2 * i, nb);
        cp_async16(stage + 32 + lane, a.vis + 2 * i + 1, nb);
        if constexpr (M16) {
            cp_async16(stage + 64 + lane, a.model16 + i, nb);
        } else {
            cp_async16(stage + 64 + lane, a.model + 2 * i, nb);
            cp_async16(stage + 96 + lane, a.model + 2 * i + 1, nb);
        }
        cp_async16(stage + R::OFF_W + lane, a.wf + i, nb);
        int flags = meta;
        if constexpr (R::NO > 0) {
            // the fixed term's entries: one per chunk where the chunk lies in one of its frequency intervals
            const int fi = a.to_map == MAP_IDENTITY ? (in ? c : 0) : fo;
            const bool uni = a.to_map == MAP_ONE || a.to_map == MAP_CHUNK ||
                             (a.to_map == MAP_ANY && __all_sync(FULL_MASK, fi == __shfl_sync(FULL_MASK, fi, 0)));
            if (uni) {
                flags |= 4;
                if (lane < 2 * R::NO) {
                    const int side = lane / R::NO, part = lane % R::NO;
                    cp_async16(stage + (side ? R::OFF_OQ : R::OFF_OP) + part,
                               a.to.tab + (size_t)R::NO * ((side ? tab_q : tab_p) + fi) + part, 16u);
                }
            } else {
#pragma unroll
                for (int part = 0; part < R::NO; ++part) {
                    cp_async16(stage + R::OFF_OP + R::NO * lane + part, a.to.tab + (size_t)R::NO * (tab_p + fi) + part, nb);
                    cp_async16(stage + R::OFF_OQ + R::NO * lane + part, a.to.tab + (size_t)R::NO * (tab_q + fi) + part, nb);
                }
            }
        }
        int key = key0;
        if (a.tn_map == MAP_IDENTITY) key += c * a.n_up;
        else key += fn * a.n_up;
        reinterpret_cast<int *>(stage + R::OFF_KEY)[lane] = in ? key : -1;
        if (lane == 0) {
            reinterpret_cast<int *>(stage + R::OFF_META)[0] = flags;
            if constexpr (M16) reinterpret_cast<float *>(stage + R::OFF_META)[1] = msc;
        }
        cp_async_commit();
        advance(a, lane);
    }
};

// One pass: warps walk units of a baseline strip (the rows of one ordered baseline in time
// order): blocks of rb rows x groups of 32-channel chunks, a row's chunks inside each row or,
// with chunk_major, the rows inside each chunk (an interval several times long then keeps its
// keys).  Each warp streams its steps through a ring of DEPTH cp.async stages in shared memory,
// DEPTH - 1 steps ahead of the arithmetic, which adds each lane's sample to its register sums;
// the sums are flushed when any lane's (interval, pair) key changes.  The fixed term is L
// (diagonal form) or R (full form) of kind OK.
template <int FORM, int OK, bool M16>
static __global__ void __launch_bounds__(128, MomRing<FORM, OK, M16>::PER_SM) mom_pass_kernel(const MomArgs a)
{
    using R = MomRing<FORM, OK, M16>;
    constexpr int NW = FORM == FORM_FULL ? MOM_FW : (FORM == FORM_E ? MOM_EW : MOM_D);
    if (a.n_active && __ldg(a.n_active) == 0) return;
    extern __shared__ float4 mom_ring[];
    const int lane = threadIdx.x & 31;
    float4 *ring = mom_ring + (size_t)(threadIdx.x >> 5) * R::DEPTH * R::STAGE;
    float acc[NW], hi[R::TWO_LEVEL ? NW : 1], lo_reg[R::TWO_LEVEL && !R::TAIL_SMEM ? NW : 1];
    float *lo_smem = reinterpret_cast<float *>(mom_ring + (size_t)4 * R::DEPTH * R::STAGE) + threadIdx.x;
    auto tail = [&](int v) -> float & {
        if constexpr (R::TAIL_SMEM) return lo_smem[128 * v];
        else return lo_reg[R::TWO_LEVEL ? v : 0];
    };
#pragma unroll
    for (int v = 0; v < NW; ++v) {
        acc[v] = 0.f;
        if constexpr (R::TWO_LEVEL) { hi[v] = 0.f; tail(v) = 0.f; }
    }
    auto lift = [&]() {
        if constexpr (R::TWO_LEVEL) {
#pragma unroll
            for (int v = 0; v < NW; ++v) {
                float e;
                two_sum(hi[v], acc[v], hi[v], e);
                tail(v) += e;
                acc[v] = 0.f;
            }
        }
    };
    const int *tmap_n = a.tn.t_map, *tmap_o = a.to.t_map;
    if (a.stage_maps) {
        int *s_map = reinterpret_cast<int *>(reinterpret_cast<char *>(mom_ring) + R::SMEM + R::TAIL);
        for (int i = threadIdx.x; i < a.n_time; i += blockDim.x) {
            s_map[i] = __ldg(a.tn.t_map + i);
            s_map[a.n_time + i] = __ldg(a.to.t_map + i);
        }
        __syncthreads();
        tmap_n = s_map;
        tmap_o = s_map + a.n_time;
    }
    MomCursor<FORM, OK, M16> cur;
    cur.start(a, lane, ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5, ((long)gridDim.x * blockDim.x) >> 5, tmap_n, tmap_o);
    int is = 0;
#pragma unroll
    for (int d = 0; d < R::DEPTH - 1; ++d) {
        cur.issue(a, lane, ring + (size_t)is * R::STAGE);
        if (++is == R::DEPTH) is = 0;
    }
    auto add = [&](const float4 *st, int meta) {
        float4 w = st[R::OFF_W + lane], d0, d1, m0, m1;
        auto load = [&]() {
            d0 = st[lane];
            d1 = st[32 + lane];
            m0 = st[64 + lane];
            if constexpr (!M16) m1 = st[96 + lane];
        };
        // all loads of the sample together, one shared-memory latency for the step (with the keys read
        // ahead 1.77 -> 1.66 ms a pass for the left-full form on 64 antennas, 85 x 512; the full form
        // gains nothing from it and has no registers to spare)
        if constexpr (FORM != FORM_FULL) load();
        // any weight other than +-0
        if ((__float_as_uint(w.x) | __float_as_uint(w.y) | __float_as_uint(w.z) | __float_as_uint(w.w)) & 0x7fffffffu) {
            if constexpr (FORM == FORM_FULL) load();
            J2 D = j_from(d0, d1), M;
            if constexpr (M16)
                M = load_model16(make_uint4(__float_as_uint(m0.x), __float_as_uint(m0.y), __float_as_uint(m0.z),
                                            __float_as_uint(m0.w)),
                                 reinterpret_cast<const float *>(st + R::OFF_META)[1]);
            else
                M = j_from(m0, m1);
            if (meta & 1) {                    // the conjugate baseline: D -> D^H, M -> M^H, w permuted
                D = j_herm(D);
                M = j_herm(M);
                w = make_float4(w.x, w.z, w.y, w.w);
            }
            const int oc = (meta & 4) ? 0 : lane * R::NO;
            if constexpr (FORM != FORM_E) {
                if constexpr (OK == KIND_DIAG) {
                    const float4 rp = st[R::OFF_OP + oc], rq = st[R::OFF_OQ + oc];
                    M = j_muld(j_dmul(make_float2(rp.x, rp.y), make_float2(rp.z, rp.w), M),
                               make_float2(rq.x, -rq.y), make_float2(rq.z, -rq.w));
                } else if constexpr (OK == KIND_FULL) {
                    M = j_mul_h(j_mul(fac_jones<OK>(st + R::OFF_OP + oc), M), fac_jones<OK>(st + R::OFF_OQ + oc));
                }
                if constexpr (FORM == FORM_FULL) mom_add(acc, D, M, w);
                else mom_add_d(acc, D, M, w);
            } else {
                mom_add_e(acc, D, M, fac_jones<OK>(st + R::OFF_OP + oc), fac_jones<OK>(st + R::OFF_OQ + oc), w);
            }
        }
    };
    // runs of steps with unchanged keys: the inner loop only adds; a key change leaves it to
    // flush the sums, then adds the step that changed the key
    int key_cur = -1, stage = 0, next = 0, run = 0;
    bool done = false;
    // the key and flags of a step are read a step ahead (they were written with its issue, DEPTH - 1
    // steps ago), so that the loop's decisions wait on no load.  Not in the full form, whose registers
    // are all taken: 1.87 ms a pass with, 1.80 without (64 antennas, 85 x 512)
    constexpr bool AHEAD = FORM != FORM_FULL;
    auto peek = [&](int s, int &m, int &k) {
        const float4 *p = ring + (size_t)s * R::STAGE;
        m = reinterpret_cast<const int *>(p + R::OFF_META)[0];
        k = reinterpret_cast<const int *>(p + R::OFF_KEY)[lane];
    };
    int meta_next = 0, key_next = -1;
    if constexpr (AHEAD) {
        __syncwarp();
        peek(0, meta_next, key_next);
    }
    for (;;) {
        const float4 *st;
        int meta = 0, key = -1;
        for (;;) {
            __syncwarp();                      // every lane is done with the stage about to be refilled
            cur.issue(a, lane, ring + (size_t)is * R::STAGE);
            if (++is == R::DEPTH) is = 0;
            cp_async_wait<R::DEPTH - 1>();
            __syncwarp();
            st = ring + (size_t)stage * R::STAGE;
            next = stage + 1 == R::DEPTH ? 0 : stage + 1;
            if constexpr (AHEAD) {
                meta = meta_next;
                key = key_next;
                peek(next, meta_next, key_next);
            } else {
                peek(stage, meta, key);
            }
            if (meta & MOM_END) { done = true; break; }
            // lanes past the last channel keep the key they had: they add nothing
            if (__any_sync(FULL_MASK, key != key_cur && key >= 0) || ++run == R::FLUSH_EVERY) break;
            if (R::TWO_LEVEL && run % R::LIFT == 0) lift();
            add(st, meta);
            stage = next;
        }
        if constexpr (R::TWO_LEVEL) {
            lift();
            mom_flush<NW>(hi, tail, key_cur, lane, a);
#pragma unroll
            for (int v = 0; v < NW; ++v) tail(v) = 0.f;
        } else {
            mom_flush<NW>(acc, [](int) { return 0.f; }, key_cur, lane, a);
        }
        if (done) break;
        run = 0;
        key_cur = key;
        add(st, meta);
        stage = next;
    }
    cp_async_wait<0>();
}

// gains of an antenna in a bin as complex FP64 entries (row-major; phase-only: diag(e^{i phi}))
__device__ __forceinline__ void gains_of(int type, const double *params, size_t pidx, double2 G[4])
{
    if (type == QC_TERM_PHASE) {
        double sn, cs;
        sincos(params[2 * pidx], &sn, &cs);
        G[0] = make_double2(cs, sn);
        sincos(params[2 * pidx + 1], &sn, &cs);
        G[3] = make_double2(cs, sn);
        G[1] = G[2] = make_double2(0.0, 0.0);
    } else {
        const double2 *P = reinterpret_cast<const double2 *>(params) + 4 * pidx;
#pragma unroll
        for (int e = 0; e < 4; ++e) G[e] = P[e];
    }
}

// One antenna's normal equations from its pairs, the register sums of a lane: per block k the
// Hermitian 2x2 [[h00, h01], [conj(h01), h11]] and b[2] (the full form has two blocks, rows
// (k, 0), (k, 1) of G; the other forms one, over g_XX and g_YY).
constexpr int NE_WORDS = 8;      // h00, h11, Re h01, Im h01, b0, b1 of one block
template <int FORM> struct NormSums {
    static constexpr int NB = FORM == FORM_FULL ? 2 : 1;
    static constexpr int NWORD = NB * NE_WORDS;
};

// The pair's contribution of one 4x4 block S (16 packed words), T (8 words) with the other
// antenna's gain row (g0, g1): with u = 2l + m,
//   h[l][l2] += sum_m sum_m2 g_m conj(g_m2) S[(l,m)][(l2,m2)],  b[l] += sum_m g_m T[(l,m)].
// The q side takes conj(S[(m,l)][(m2,l2)]) and conj(T[(m,l)]): indices 1 and 2 exchanged, conjugated.
// EXACT: exact products, h heads and e tails of the sums (few antennas have few pairs over which the
// roundings of plain products average out); else plain, e unused.
template <bool EXACT>
__device__ __forceinline__ void pair_block(const float4 *__restrict__ sv, const float4 *__restrict__ tv, bool p_side,
                                           float2 g0, float2 g1, float *h, float *e)
{
    const float4 a0 = __ldg(sv), a1 = __ldg(sv + 1), a2 = __ldg(sv + 2), a3 = __ldg(sv + 3);
    const float4 t0 = __ldg(tv), t1 = __ldg(tv + 1);
    const float sg = p_side ? 1.f : -1.f;
    const float d1 = p_side ? a0.y : a0.z, d2 = p_side ? a0.z : a0.y;
    float2 s01 = p_side ? make_float2(a1.x, a1.y) : make_float2(a1.z, a1.w);
    float2 s02 = p_side ? make_float2(a1.z, a1.w) : make_float2(a1.x, a1.y);
    float2 s03 = make_float2(a2.x, a2.y);
    const float2 s12 = make_float2(a2.z, a2.w);             // its own conjugate transpose on the q side
    float2 s13 = p_side ? make_float2(a3.x, a3.y) : make_float2(a3.z, a3.w);
    float2 s23 = p_side ? make_float2(a3.z, a3.w) : make_float2(a3.x, a3.y);
    s01.y *= sg; s02.y *= sg; s03.y *= sg; s13.y *= sg; s23.y *= sg;
    float2 u0 = make_float2(t0.x, t0.y), u3 = make_float2(t1.z, t1.w);
    float2 u1 = p_side ? make_float2(t0.z, t0.w) : make_float2(t1.x, t1.y);
    float2 u2 = p_side ? make_float2(t1.x, t1.y) : make_float2(t0.z, t0.w);
    u0.y *= sg; u1.y *= sg; u2.y *= sg; u3.y *= sg;
    if constexpr (EXACT) {
        const HT n0 = dot2(g0.x, g0.x, g0.y, g0.y), n1 = dot2(g1.x, g1.x, g1.y, g1.y);
        const HT xr = dot2(g0.x, g1.x, g0.y, g1.y), xi = dot2(g0.y, g1.x, -g0.x, g1.y);   // g_0 conj(g_1)
        const HT xr2 = { 2.f * xr.hi, 2.f * xr.lo }, xi2 = { -2.f * xi.hi, -2.f * xi.lo };
        dot_add(h[0], e[0], n0, a0.x);
        dot_add(h[0], e[0], n1, d1);
        dot_add(h[0], e[0], xr2, s01.x);
        dot_add(h[0], e[0], xi2, s01.y);
        dot_add(h[1], e[1], n0, d2);
        dot_add(h[1], e[1], n1, a0.w);
        dot_add(h[1], e[1], xr2, s23.x);
        dot_add(h[1], e[1], xi2, s23.y);
        // n0 S02 + n1 S13 + x S03 + conj(x) S12
        dot_add(h[2], e[2], n0, s02.x);
        dot_add(h[2], e[2], n1, s13.x);
        dot_add(h[2], e[2], xr, s03.x);
        dot_add(h[2], e[2], xr, s12.x);
        dot_add(h[2], e[2], xi, s12.y);
        dot_add(h[2], e[2], neg(xi), s03.y);
        dot_add(h[3], e[3], n0, s02.y);
        dot_add(h[3], e[3], n1, s13.y);
        dot_add(h[3], e[3], xr, s03.y);
        dot_add(h[3], e[3], xr, s12.y);
        dot_add(h[3], e[3], xi, s03.x);
        dot_add(h[3], e[3], neg(xi), s12.x);
        dot_add(h[4], e[4], g0.x, u0.x);
        dot_add(h[4], e[4], -g0.y, u0.y);
        dot_add(h[4], e[4], g1.x, u1.x);
        dot_add(h[4], e[4], -g1.y, u1.y);
        dot_add(h[5], e[5], g0.x, u0.y);
        dot_add(h[5], e[5], g0.y, u0.x);
        dot_add(h[5], e[5], g1.x, u1.y);
        dot_add(h[5], e[5], g1.y, u1.x);
        dot_add(h[6], e[6], g0.x, u2.x);
        dot_add(h[6], e[6], -g0.y, u2.y);
        dot_add(h[6], e[6], g1.x, u3.x);
        dot_add(h[6], e[6], -g1.y, u3.y);
        dot_add(h[7], e[7], g0.x, u2.y);
        dot_add(h[7], e[7], g0.y, u2.x);
        dot_add(h[7], e[7], g1.x, u3.y);
        dot_add(h[7], e[7], g1.y, u3.x);
    } else {
        const float n0 = cnorm2(g0), n1 = cnorm2(g1);
        const float2 x = cmulc(g0, g1);                         // g_0 conj(g_1)
        h[0] += fmaf(n0, a0.x, fmaf(n1, d1, 2.f * fmaf(x.x, s01.x, -x.y * s01.y)));
        h[1] += fmaf(n0, d2, fmaf(n1, a0.w, 2.f * fmaf(x.x, s23.x, -x.y * s23.y)));
        // n0 S02 + n1 S13 + x S03 + conj(x) S12
        h[2] += fmaf(n0, s02.x, fmaf(n1, s13.x, fmaf(x.x, s03.x + s12.x, x.y * (s12.y - s03.y))));
        h[3] += fmaf(n0, s02.y, fmaf(n1, s13.y, fmaf(x.x, s03.y + s12.y, x.y * (s03.x - s12.x))));
        h[4] += fmaf(g0.x, u0.x, fmaf(-g0.y, u0.y, fmaf(g1.x, u1.x, -g1.y * u1.y)));
        h[5] += fmaf(g0.x, u0.y, fmaf(g0.y, u0.x, fmaf(g1.x, u1.y, g1.y * u1.x)));
        h[6] += fmaf(g0.x, u2.x, fmaf(-g0.y, u2.y, fmaf(g1.x, u3.x, -g1.y * u3.y)));
        h[7] += fmaf(g0.x, u2.y, fmaf(g0.y, u2.x, fmaf(g1.x, u3.y, g1.y * u3.x)));
    }
}

// The contribution of pair (a, o) to antenna a's register sums; gains of o from g (full: the two
// float4 of its table entry; else one, (g_XX, g_YY)).
template <int FORM, bool EXACT>
__device__ __forceinline__ void pair_add(const float *__restrict__ slot, bool p_side, const float4 *g, float *h,
                                         float *e)
{
    const float4 *s = reinterpret_cast<const float4 *>(slot);
    if constexpr (FORM == FORM_FULL) {
        // rows j of G_o; a diagonal term's table entry is diag(g_XX, g_YY)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int blk = p_side ? 2 * k + j : 2 * j + k;
                pair_block<EXACT>(s + 4 * blk, s + MOM_T / 4 + 2 * blk, p_side, make_float2(g[j].x, g[j].y),
                           make_float2(g[j].z, g[j].w), h + NE_WORDS * k, e + NE_WORDS * k);
            }
    } else if constexpr (FORM == FORM_E) {
        pair_block<EXACT>(s, s + MOM_ET / 4, p_side, make_float2(g[0].x, g[0].y), make_float2(g[0].z, g[0].w), h, e);
    } else {
        if constexpr (EXACT) diag_pair_add(__ldg(s), __ldg(s + 1), __ldg(s + 2), p_side, g[0], h, e);
        else diag_pair_add(__ldg(s), __ldg(s + 1), __ldg(s + 2), p_side, g[0], h);
    }
}

// One warp: antenna a's normal equations of an interval over the other antennas (lanes), in FP32;
// the totals to out[NWORD].  Antenna o's gains (full: two float4, else one) at gains + o * gstride.
// TAIL: the slots' tails as well (the sums are linear in the slots: the tails' plain sums go to e).
template <int FORM, bool TAIL>
__device__ __forceinline__ void antenna_sums(const MomNormArgs &A, size_t bin_off, int a, int lane,
                                             const float4 *gains, size_t gstride, double *out)
{
    constexpr int N = NormSums<FORM>::NWORD;
    float h[N], e[N];
#pragma unroll
    for (int i = 0; i < N; ++i) h[i] = e[i] = 0.f;
    for (int o = lane; o < A.n_ant; o += 32) {
        if (o == a) continue;
        const int up = __ldg(A.upair + (size_t)a * A.n_ant + o);
        if (up < 0) continue;
        float4 g[2];
        g[0] = gains[o * gstride];
        if constexpr (FORM == FORM_FULL) g[1] = gains[o * gstride + 1];
        const size_t at = bin_off + (size_t)up * mom_words(FORM);
        pair_add<FORM, true>(A.mom + at, a < o, g, h, e);                          // the smaller index is the sums' p
        if constexpr (TAIL) pair_add<FORM, false>(A.tail + at, a < o, g, e, nullptr);
    }
    const double v = reduce_words<N>(h, e, lane);
    if (lane % (32 / N) == 0) out[lane / (32 / N)] = v;
}

// Per-iteration form (more antennas than the one-launch kernel takes, divergence flagging, an
// allreduce before the update): one warp per (interval, antenna); JHr = b - JHJ vec(G_a) in FP64,
// written in the update kernel's accumulator layout.
template <int FORM, bool TAIL>
static __global__ void __launch_bounds__(128) mom_normal_kernel(const MomNormArgs A)
{
    constexpr int N = NormSums<FORM>::NWORD, NF4 = FORM == FORM_FULL ? 2 : 1;
    if (__ldg(A.n_active) == 0) return;
    __shared__ double s_out[4][N];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long w = (long)blockIdx.x * 4 + warp;
    if (w >= (long)A.n_bins * A.n_ant) return;
    const int bin = (int)(w / A.n_ant), a = (int)(w % A.n_ant);
    if (!A.active[bin]) return;
    const int tint = bin / A.n_fint, fint = bin - tint * A.n_fint;
    const size_t bin_off = (size_t)bin * A.n_up * mom_words(FORM), gstride = (size_t)NF4 * A.n_fint;
    const float4 *gains = A.tab + NF4 * ((size_t)tint * A.n_ant * A.n_fint + fint);
    antenna_sums<FORM, TAIL>(A, bin_off, a, lane, gains, gstride, s_out[warp]);
    __syncwarp();
    if (lane != 0) return;
    double2 G[4];
    gains_of(A.type, A.params, (size_t)bin * A.n_ant + a, G);
    double *out = A.acc + ((size_t)bin * A.n_ant + a) * (FORM == FORM_FULL ? KG_FULL : KG_DIAG);
    if constexpr (FORM == FORM_FULL)
        for (int i = 4; i < 16; ++i) out[i] = 0.0;                  // no coupling between the rows of G
#pragma unroll
    for (int k = 0; k < N / NE_WORDS; ++k) {
        const double *x = s_out[warp] + NE_WORDS * k;
        const double h00 = x[0], h11 = x[1], hx = x[2], hy = x[3];
        const double2 g0 = FORM == FORM_FULL ? G[2 * k] : G[0], g1 = FORM == FORM_FULL ? G[2 * k + 1] : G[3];
        out[2 * k] = h00;
        out[2 * k + 1] = h11;
        double *off = out + (FORM == FORM_FULL ? (k ? 14 : 4) : 2);
        off[0] = hx;
        off[1] = hy;
        double *r = out + (FORM == FORM_FULL ? 16 + 4 * k : 4);
        r[0] = x[4] - (h00 * g0.x + (hx * g1.x - hy * g1.y));
        r[1] = x[5] - (h00 * g0.y + (hx * g1.y + hy * g1.x));
        r[2] = x[6] - ((hx * g0.x + hy * g0.y) + h11 * g1.x);
        r[3] = x[7] - ((hx * g0.y - hy * g0.x) + h11 * g1.y);
    }
}

// Solve the Hermitian 2x2 blocks [[h00, h01], [conj(h01), h11]] x = r of one antenna in FP64 with
// block_solve's singularity tests over the whole block-diagonal matrix (zero trace, zero
// determinant, 1-norm condition number above 1e12); returns 1 when singular.  FP64 runs at two
// lanes a cycle and SM with long latencies, and this chain is most of an iteration on few antennas:
// one division a block, the condition number tested without one, |h01| (for that test alone)
// from an FP32 root where FP32 holds it.
__device__ __forceinline__ double root_of(double v)
{
    return v > 1e-30 && v < 1e30 ? (double)sqrtf((float)v) : sqrt(v);
}
template <int NB, bool OFF>
__device__ __forceinline__ int solve_blocks(const double (&h00)[NB], const double (&h11)[NB], const double2 (&h01)[NB],
                                            const double2 (&r)[2 * NB], double2 (&x)[2 * NB])
{
    double trace = 0, anorm = 0, inorm = 0;
#pragma unroll
    for (int k = 0; k < NB; ++k) trace += h00[k] + h11[k];
    if (!(trace > 0)) return 1;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
        const double o2 = OFF ? h01[k].x * h01[k].x + h01[k].y * h01[k].y : 0.0;
        const double det = h00[k] * h11[k] - o2;
        if (!(fabs(det) > 0)) return 1;
        const double rd = 1.0 / det;
        const double big = fmax(fabs(h00[k]), fabs(h11[k])) + (OFF ? root_of(o2) : 0.0);
        anorm = fmax(anorm, big);
        inorm = fmax(inorm, big * fabs(rd));
        const double2 r0 = r[2 * k], r1 = r[2 * k + 1], z = h01[k];
        if constexpr (OFF) {
            x[2 * k] = make_double2((h11[k] * r0.x - (z.x * r1.x - z.y * r1.y)) * rd,
                                    (h11[k] * r0.y - (z.x * r1.y + z.y * r1.x)) * rd);
            x[2 * k + 1] = make_double2((h00[k] * r1.x - (z.x * r0.x + z.y * r0.y)) * rd,
                                        (h00[k] * r1.y - (z.x * r0.y - z.y * r0.x)) * rd);
        } else {
            const double a = h11[k] * rd, b = h00[k] * rd;
            x[2 * k] = make_double2(a * r0.x, a * r0.y);
            x[2 * k + 1] = make_double2(b * r1.x, b * r1.y);
        }
    }
    return !(anorm * inorm <= 1e12);
}

// Every iteration of one solution interval in one CTA: intervals are independent of each other once
// their sums are formed, so nothing has to be exchanged between CTAs and no launch, graph node
// or grid-wide counter stands between two iterations.  Per iteration the warps form the antennas'
// normal equations from the sums (L2), one thread per antenna solves and updates in FP64 exactly as
// update_kernel does, and the FP64 relative change of the interval ends the loop.
template <int FORM, bool TAIL>
static __global__ void __launch_bounds__(512, 1) mom_iterate_kernel(const MomIterArgs a)
{
    constexpr bool GFULL = FORM == FORM_FULL;
    constexpr int N = NormSums<FORM>::NWORD, NB = GFULL ? 2 : 1, NF4 = NB;
    extern __shared__ float4 s_mem[];
    const MomNormArgs &A = a.n;
    float4 *g32 = s_mem;                                                       // [n_ant][NF4]
    double *sums = reinterpret_cast<double *>(s_mem + (size_t)A.n_ant * NF4);  // [n_ant][N]
    double2 *g64 = reinterpret_cast<double2 *>(sums + (size_t)A.n_ant * N);    // [n_ant][2 NB] the FP64 master
    const bool phase = !GFULL && A.type == QC_TERM_PHASE;
    __shared__ double s_num[16], s_den[16];
    __shared__ int s_done;
    const int bin = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const int tint = bin / A.n_fint, fint = bin - tint * A.n_fint;
    const size_t bin_off = (size_t)bin * A.n_up * mom_words(FORM);
    auto tab_at = [&](int i) { return a.tab + NF4 * (((size_t)tint * A.n_ant + i / NF4) * A.n_fint + fint) + i % NF4; };
    for (int i = tid; i < A.n_ant * NF4; i += blockDim.x) g32[i] = *tab_at(i);
    // phase-only: (phi_X, phi_Y) in the first entry; diagonal: entries 0 and 3 of the four kept
    const double2 *P0 = reinterpret_cast<const double2 *>(a.params) + (size_t)bin * A.n_ant * (phase ? 1 : 4);
    for (int i = tid; i < A.n_ant * 2 * NB; i += blockDim.x) {
        const int ant = i / (2 * NB), e = i % (2 * NB);
        if (phase) { if (e == 0) g64[2 * ant] = P0[ant]; }
        else g64[i] = P0[4 * ant + (GFULL ? e : 3 * e)];
    }
    __syncthreads();
    int k = 1;
    for (;; ++k) {
        for (int ant = warp; ant < A.n_ant; ant += nw)
            antenna_sums<FORM, TAIL>(A, bin_off, ant, lane, g32, NF4, sums + (size_t)ant * N);
        __syncthreads();
        const double alpha = a.alternate ? ((k % 2 == 0) ? 0.5 : 1.0) : a.damping;
        double num = 0, den = 0;
        for (int ant = tid; ant < A.n_ant; ant += blockDim.x) {
            const double *h = sums + (size_t)ant * N;
            double2 old[2 * NB], now[2 * NB], r[2 * NB], x[2 * NB], h01[NB];
            double h00[NB], h11[NB];
            double2 *G = g64 + (size_t)ant * 2 * NB;
            if (phase) {
                sincos(G[0].x, &old[0].y, &old[0].x);
                sincos(G[0].y, &old[1].y, &old[1].x);
            } else {
#pragma unroll
                for (int e = 0; e < 2 * NB; ++e) old[e] = G[e];
            }
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const double *w = h + NE_WORDS * b;
                h00[b] = w[0];
                h11[b] = w[1];
                h01[b] = FORM == FORM_D ? make_double2(0, 0) : make_double2(w[2], w[3]);
                const double2 g0 = old[2 * b], g1 = old[2 * b + 1], z = h01[b];
                r[2 * b] = make_double2(w[4] - (h00[b] * g0.x + (z.x * g1.x - z.y * g1.y)),
                                        w[5] - (h00[b] * g0.y + (z.x * g1.y + z.y * g1.x)));
                r[2 * b + 1] = make_double2(w[6] - ((z.x * g0.x + z.y * g0.y) + h11[b] * g1.x),
                                            w[7] - ((z.x * g0.y - z.y * g0.x) + h11[b] * g1.y));
            }
            int singular;
            if (phase) {
                // chain rule with dg/dphi = i g (Scenario 1): 2 Re(conj(g_u) g_v JHJ), 2 Im(conj(g_u) JHr)
                const double2 g0 = old[0], g1 = old[1], z = h01[0];
                const double2 c = make_double2(g0.x * g1.x + g0.y * g1.y, g0.x * g1.y - g0.y * g1.x);
                double m0[1] = { 2.0 * (g0.x * g0.x + g0.y * g0.y) * h00[0] };
                double m1[1] = { 2.0 * (g1.x * g1.x + g1.y * g1.y) * h11[0] };
                double2 mo[1] = { make_double2(2.0 * (c.x * z.x - c.y * z.y), 0.0) }, rb[2], xb[2];
                rb[0] = make_double2(2.0 * (g0.x * r[0].y - g0.y * r[0].x), 0.0);
                rb[1] = make_double2(2.0 * (g1.x * r[1].y - g1.y * r[1].x), 0.0);
                singular = solve_blocks<1, FORM != FORM_D>(m0, m1, mo, rb, xb);
                double2 phi = G[0];
                if (!singular) { phi.x += alpha * xb[0].x; phi.y += alpha * xb[1].x; }
                G[0] = phi;
                sincos(phi.x, &now[0].y, &now[0].x);
                sincos(phi.y, &now[1].y, &now[1].x);
            } else {
                singular = solve_blocks<NB, FORM != FORM_D>(h00, h11, h01, r, x);
#pragma unroll
                for (int e = 0; e < 2 * NB; ++e) {
                    now[e] = singular ? old[e] : make_double2(old[e].x + alpha * x[e].x, old[e].y + alpha * x[e].y);
                    G[e] = now[e];
                }
            }
            a.gain_flags[(size_t)bin * A.n_ant + ant] = (int8_t)singular;
#pragma unroll
            for (int f = 0; f < NF4; ++f)
                g32[NF4 * ant + f] = make_float4((float)now[2 * f].x, (float)now[2 * f].y, (float)now[2 * f + 1].x,
                                                 (float)now[2 * f + 1].y);
#pragma unroll
            for (int e = 0; e < 2 * NB; ++e) {
                const double dx = now[e].x - old[e].x, dy = now[e].y - old[e].y;
                num += dx * dx + dy * dy;
                den += now[e].x * now[e].x + now[e].y * now[e].y;
            }
        }
        for (int d = 16; d > 0; d >>= 1) {
            num += __shfl_down_sync(FULL_MASK, num, d);
            den += __shfl_down_sync(FULL_MASK, den, d);
        }
        if (lane == 0) { s_num[warp] = num; s_den[warp] = den; }
        __syncthreads();
        if (tid == 0) {
            double tn = 0, td = 0;
            for (int i = 0; i < nw; ++i) { tn += s_num[i]; td += s_den[i]; }
            const bool conv = converged(tn, td, a.tol);
            if (!conv) atomicAdd(a.cnt + k, 1);                      // still active after iteration k
            s_done = conv || k == a.max_iter;
        }
        __syncthreads();
        if (s_done) break;
    }
    for (int i = tid; i < A.n_ant * NF4; i += blockDim.x) *tab_at(i) = g32[i];
    double2 *P1 = reinterpret_cast<double2 *>(a.params) + (size_t)bin * A.n_ant * (phase ? 1 : 4);
    for (int i = tid; i < A.n_ant * 2 * NB; i += blockDim.x) {
        const int ant = i / (2 * NB), e = i % (2 * NB);
        if (phase) { if (e == 0) P1[ant] = g64[2 * ant]; }
        else P1[4 * ant + (GFULL ? e : 3 * e)] = g64[i];
    }
    if (tid == 0) {
        a.iters[bin] = k;
        atomicAdd(a.vis_iters, (unsigned long long)a.bin_nvis[bin] * k);
        atomicAdd(a.acc_bytes, (unsigned long long)(a.bin_nbytes[bin] + a.iter_bytes * k));
    }
}

// algorithmic bytes: the pass reads every sample of the bins once (their streaming bytes);
// an iteration reads each bin's sums twice (once per side) and writes its accumulators
static __global__ void mom_bytes_kernel(int n_bins, const long long *bin_nbytes, long long per_iter,
                                        long long *iter_nbytes, unsigned long long *acc_bytes)
{
    unsigned long long s = 0;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < n_bins; b += gridDim.x * blockDim.x) {
        s += (unsigned long long)bin_nbytes[b];
        iter_nbytes[b] = per_iter;
    }
    for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(acc_bytes, s);
}

} // namespace qc

template <int FORM, int OK, bool M16>
static cudaError_t launch_pass(const qc::MomArgs &a, int sm_count, cudaStream_t st)
{
    using R = qc::MomRing<FORM, OK, M16>;
    // the raised shared-memory limit belongs to the device's copy of the kernel: set on every launch
    qc::MomArgs b = a;
    b.stage_maps = a.n_time <= R::MAX_STAGED;
    const int smem = (int)(R::SMEM + R::TAIL) + (b.stage_maps ? 2 * a.n_time * (int)sizeof(int) : 0);
    const cudaError_t e = cudaFuncSetAttribute(qc::mom_pass_kernel<FORM, OK, M16>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const int block = 128;
    const int n_groups = (a.n_chunks + a.group - 1) / a.group;
    const long units = (long)a.n_strips * a.n_rb * n_groups;
    const int grid = (int)std::max(1L, std::min((long)sm_count * R::PER_SM, (units * 32 + block - 1) / block));
    qc::mom_pass_kernel<FORM, OK, M16><<<grid, block, smem, st>>>(b);
    return cudaGetLastError();
}

// the pass kernel of a form and fixed-term kind (ok: KIND_* of the term to the right in the full
// form, of the one to the left in the E form, of either in the plain diagonal form)
template <bool M16>
static cudaError_t launch_pass_any(const qc::MomArgs &a, int form, int ok, int sm_count, cudaStream_t st)
{
    using namespace qc;
    if (form == FORM_FULL) {
        if (ok == KIND_NONE) return launch_pass<FORM_FULL, KIND_NONE, M16>(a, sm_count, st);
        if (ok == KIND_DIAG) return launch_pass<FORM_FULL, KIND_DIAG, M16>(a, sm_count, st);
        return launch_pass<FORM_FULL, KIND_FULL, M16>(a, sm_count, st);
    }
    if (form == FORM_E) return ok == KIND_FULL ? launch_pass<FORM_E, KIND_FULL, M16>(a, sm_count, st) : cudaErrorInvalidValue;
    if (ok == KIND_NONE) return launch_pass<FORM_D, KIND_NONE, M16>(a, sm_count, st);
    if (ok == KIND_DIAG) return launch_pass<FORM_D, KIND_DIAG, M16>(a, sm_count, st);
    return launch_pass<FORM_D, KIND_FULL, M16>(a, sm_count, st);
}

cudaError_t mom_launch_pass(const qc::MomArgs &a, int form, int ok, int sm_count, cudaStream_t st)
{
    return a.model16 ? launch_pass_any<true>(a, form, ok, sm_count, st) : launch_pass_any<false>(a, form, ok, sm_count, st);
}

cudaError_t mom_launch_split(size_t words, const double *src, float *dst, float *tail, int sm_count, cudaStream_t st)
{
    const long n2 = (long)(words / 2);              // a slot is a whole number of 16-byte vectors
    const int grid = (int)std::max(1L, std::min((n2 + 255) / 256, (long)sm_count * 16));
    qc::mom_split_kernel<<<grid, 256, 0, st>>>(n2, (const double2 *)src, (float2 *)dst, (float2 *)tail);
    return cudaGetLastError();
}

cudaError_t mom_launch_bytes(int n_bins, const long long *bin_nbytes, long long per_iter, long long *iter_nbytes,
                             unsigned long long *acc_bytes, cudaStream_t st)
{
    qc::mom_bytes_kernel<<<(n_bins + 255) / 256, 256, 0, st>>>(n_bins, bin_nbytes, per_iter, iter_nbytes, acc_bytes);
    return cudaGetLastError();
}

template <int FORM> static cudaError_t launch_normal(const qc::MomNormArgs &a, cudaStream_t st)
{
    const unsigned grid = (unsigned)(((long)a.n_bins * a.n_ant + 3) / 4);
    if (a.tail) qc::mom_normal_kernel<FORM, true><<<grid, 128, 0, st>>>(a);
    else qc::mom_normal_kernel<FORM, false><<<grid, 128, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t mom_launch_normal(const qc::MomNormArgs &a, cudaStream_t st)
{
    if (a.form == qc::FORM_FULL) return launch_normal<qc::FORM_FULL>(a, st);
    if (a.form == qc::FORM_E) return launch_normal<qc::FORM_E>(a, st);
    return launch_normal<qc::FORM_D>(a, st);
}

template <int FORM, bool TAIL> static cudaError_t launch_iterate(const qc::MomIterArgs &a, int sm_count, cudaStream_t st)
{
    // a warp an antenna and round: 16 warps where every interval has an SM to itself, else two CTAs of 8;
    // fewer for few antennas, unless a turn is long (the forms with 4x4 blocks) or all of them have one (10
    // antennas, full and left-full form, 120 intervals: 0.70 ms with 4 warps, 0.58 with 10; 7 antennas, 60
    // intervals: 0.27 with 2, 0.24 with 7; 16 antennas, plain diagonal form: 0.32 with 4, 0.33 with 16)
    const int n_ant = a.n.n_ant;
    const bool alone = a.n.n_bins <= sm_count;
    const int block = alone && (FORM != qc::FORM_D || n_ant <= 8) ? 32 * std::min(16, std::max(2, n_ant))
                      : n_ant > 16                                ? (alone ? 512 : 256)
                                                                  : (n_ant > 8 ? 128 : 64);
    constexpr int NB = FORM == qc::FORM_FULL ? 2 : 1;
    const size_t smem = (size_t)n_ant * (NB * sizeof(float4) + qc::NormSums<FORM>::NWORD * sizeof(double) + 2 * NB * sizeof(double2));
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(qc::mom_iterate_kernel<FORM, TAIL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)smem);
        if (e != cudaSuccess) return e;
    }
    qc::mom_iterate_kernel<FORM, TAIL><<<a.n.n_bins, block, smem, st>>>(a);
    return cudaGetLastError();
}

template <int FORM> static cudaError_t launch_iterate(const qc::MomIterArgs &a, int sm_count, cudaStream_t st)
{
    return a.n.tail ? launch_iterate<FORM, true>(a, sm_count, st) : launch_iterate<FORM, false>(a, sm_count, st);
}

cudaError_t mom_launch_iterate(const qc::MomIterArgs &a, int sm_count, cudaStream_t st)
{
    if (a.n.form == qc::FORM_FULL) return launch_iterate<qc::FORM_FULL>(a, sm_count, st);
    if (a.n.form == qc::FORM_E) return launch_iterate<qc::FORM_E>(a, sm_count, st);
    return launch_iterate<qc::FORM_D>(a, sm_count, st);
}

cudaError_t mom_launch_rows(long n, const int *strip_rows, const int4 *rows, const uint8_t *row_live,
                            const int *up_of_bl, const float *bl_scale, int4 *out, float *scale, int n_strips,
                            const int *strip_off, int4 *live, float *live_scale, int *strip_end, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    qc::mom_rows_kernel<<<(int)((n + 255) / 256), 256, 0, st>>>(n, strip_rows, rows, row_live, up_of_bl, bl_scale, out,
                                                               scale);
    qc::mom_live_kernel<<<(n_strips + 7) / 8, 256, 0, st>>>(n_strips, strip_off, out, scale, live, live_scale, strip_end);
    return cudaGetLastError();
}

