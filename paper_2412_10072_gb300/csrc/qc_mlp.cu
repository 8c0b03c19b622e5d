// qc_mlp.cu -- learned warm start for the batched solver: per-antenna features,
// a 3 x 128 GELU multilayer perceptron (forward, backward, Adam) and the
// selection of initial gains.
//
// The paper's solvers start from initial estimates where a term allows it
// (Section 4.3, "Initial estimates"); here a small network predicts each
// interval's diagonal gains from per-antenna summaries of its data, and
// Algorithm 1 still iterates to tolerance from there.  All arithmetic is
// FP32 on the CUDA cores (the layers are 128 wide: tensor cores would not be
// fed), with exact-erf GELU.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <string>

#include "../../include/qc.h"
#include "qc_jones.cuh"

namespace {

using namespace qc;

constexpr int IN = QC_MLP_IN, HID = QC_MLP_HIDDEN, OUT = QC_MLP_OUT;
constexpr int SKIP = 6;           // first input feature passed straight to the outputs
// parameter offsets inside the flat float buffer
constexpr int W1 = 0, B1 = W1 + HID * IN, W2 = B1 + HID, B2 = W2 + HID * HID, W3 = B2 + HID, B3 = W3 + HID * HID,
              W4 = B3 + HID, B4 = W4 + OUT * HID, NPARAM = B4 + OUT;
static_assert(NPARAM == QC_MLP_NPARAM, "parameter count");

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_d(float z)
{
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// ---------------------------------------------------------------------------
// forward: y = x[6..9] + W4 g(W3 g(W2 g(W1 x + b1) + b2) + b3) + b4,  g = GELU
// (the skip term passes the previous-interval gain features straight through,
// so the layers learn the correction to them)
// ---------------------------------------------------------------------------

// Both kernels take tiles of 32 rows and keep the two 128 x 128 matrices in shared memory with rows of
// 132 floats, which makes every 16-byte access below conflict-free: eight lanes of a quarter of a
// warp touch eight matrix rows 4 banks apart, or 128 contiguous bytes.  A warp computes 16 rows x 32
// columns of a layer, a thread 4 x 4, from float4s along the summed index: 64 FMAs for eight 16-byte
// shared loads of one wavefront each, so the FMA pipe and not shared memory is the limit.  (One
// thread's four columns a matrix row apart, read word by word, put all lanes on one bank.)  32
// rows give 128 tiles for the usual mini-batch of 4096 rows on 152 SMs.  Training step, 4096
// rows: 315 us before, 81 us now (forward 23, backward 60 of them on the device).
constexpr int TR = 32;            // rows per CTA tile
constexpr int FT = 256;           // threads
constexpr int LD = HID + 4;       // row stride of matrices and activations in shared memory
constexpr int LD1 = IN + 1;       // row stride of W1 and of the input tile

// rows x HID floats from global memory (row-major) to shared rows of LD floats
__device__ __forceinline__ void stage_rows(float *dst, const float *__restrict__ src, int rows)
{
    if (((uintptr_t)src & 15) == 0) {
        for (int i = threadIdx.x; i < rows * (HID / 4); i += blockDim.x) {
            const int r = i / (HID / 4), c = i % (HID / 4);
            *reinterpret_cast<float4 *>(dst + r * LD + 4 * c) = __ldg(reinterpret_cast<const float4 *>(src) + i);
        }
    } else {
        for (int i = threadIdx.x; i < rows * HID; i += blockDim.x) dst[(i / HID) * LD + i % HID] = __ldg(src + i);
    }
}

// the thread's rows and columns of a layer's 32 x 128 outputs
struct TileMap {
    int r0, c0;                   // first row (then +4 i), first column
    __device__ __forceinline__ TileMap()
    {
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        r0 = 16 * (w & 1) + (lane >> 3);
        c0 = 32 * (w >> 1) + (lane & 7);
    }
};

__device__ __forceinline__ float at4(const float4 &v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// out = GELU(in W^T + b) for the tile (sums over k in ascending order from the bias); z (nullable)
// receives the pre-activations
__device__ __forceinline__ void dense_tile(const float *in, const float *W, const float *__restrict__ b, float *out,
                                           float *z, long row0, int nr)
{
    const TileMap m;              // columns c0 + 8 j
    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float bj = __ldg(b + m.c0 + 8 * j);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i][j] = bj;
    }
#pragma unroll 2
    for (int k = 0; k < HID; k += 4) {
        float4 x[4], w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float4 *>(in + (m.r0 + 4 * i) * LD + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const float4 *>(W + (m.c0 + 8 * j) * LD + k);
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(at4(x[i], e), at4(w[j], e), acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = m.r0 + 4 * i;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (z && r < nr) z[(size_t)(row0 + r) * 3 * HID + m.c0 + 8 * j] = acc[i][j];
            out[r * LD + m.c0 + 8 * j] = gelu(acc[i][j]);
        }
    }
}

__global__ void __launch_bounds__(FT, 1) mlp_forward_kernel(const float *__restrict__ P, const float *__restrict__ x,
                                                            long n, float *__restrict__ y, float *__restrict__ z)
{
    extern __shared__ __align__(16) float sm[];
    float *w2 = sm, *w3 = w2 + HID * LD, *h0 = w3 + HID * LD, *h1 = h0 + TR * LD, *w4 = h1 + TR * LD;
    float *w1 = w4 + OUT * HID, *xs = w1 + HID * LD1;
    stage_rows(w2, P + W2, HID);
    stage_rows(w3, P + W3, HID);
    for (int i = threadIdx.x; i < HID * IN; i += blockDim.x) w1[(i / IN) * LD1 + i % IN] = __ldg(P + W1 + i);
    for (int i = threadIdx.x; i < OUT * HID; i += blockDim.x) w4[i] = __ldg(P + W4 + i);
    for (long row0 = (long)blockIdx.x * TR; row0 < n; row0 += (long)gridDim.x * TR) {
        const int nr = (int)min((long)TR, n - row0);
        __syncthreads();
        for (int i = threadIdx.x; i < TR * IN; i += blockDim.x) {
            const int r = i / IN;
            xs[r * LD1 + i % IN] = r < nr ? __ldg(x + row0 * IN + i) : 0.f;
        }
        __syncthreads();
        {
            const TileMap m;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = m.c0 + 8 * j;
                const float bj = __ldg(P + B1 + c);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = m.r0 + 4 * i;
                    float s = bj;
#pragma unroll
                    for (int k = 0; k < IN; ++k) s = fmaf(xs[r * LD1 + k], w1[c * LD1 + k], s);
                    if (z && r < nr) z[(size_t)(row0 + r) * 3 * HID + c] = s;
                    h0[r * LD + c] = gelu(s);
                }
            }
        }
        __syncthreads();
        dense_tile(h0, w2, P + B2, h1, z ? z + HID : nullptr, row0, nr);
        __syncthreads();
        dense_tile(h1, w3, P + B3, h0, z ? z + 2 * HID : nullptr, row0, nr);
        __syncthreads();
        // one thread per output (32 rows x 4): h0's rows are 4 banks apart, w4 is a broadcast
        if (threadIdx.x < TR * OUT) {
            const int r = threadIdx.x % TR, j = threadIdx.x / TR;
            float s = __ldg(P + B4 + j) + xs[r * LD1 + SKIP + j];
#pragma unroll 8
            for (int k = 0; k < HID; k += 4) {
                const float4 h = *reinterpret_cast<const float4 *>(h0 + r * LD + k);
                const float4 w = *reinterpret_cast<const float4 *>(w4 + j * HID + k);
                s = fmaf(h.x, w.x, s);
                s = fmaf(h.y, w.y, s);
                s = fmaf(h.z, w.z, s);
                s = fmaf(h.w, w.w, s);
            }
            if (r < nr) y[(row0 + r) * OUT + j] = s;
        }
    }
}

// ---------------------------------------------------------------------------
// backward of the mean squared error over n rows x OUT outputs
// ---------------------------------------------------------------------------

// dst = (d W) * gelu'(z) for the tile: the deltas of a layer from those of the next one
__device__ __forceinline__ void delta_tile(const float *d, const float *W, const float *__restrict__ z, float *dst,
                                           long row0, int nr)
{
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r0 = 16 * (w & 1) + (lane >> 3), c0 = 32 * (w >> 1) + 4 * (lane & 7);   // columns c0 .. c0 + 3
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll 2
    for (int k = 0; k < HID; k += 4) {
        float4 x[4], v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float4 *>(d + (r0 + 4 * i) * LD + k);
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = *reinterpret_cast<const float4 *>(W + (k + e) * LD + c0);
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(at4(x[i], e), at4(v[e], j), acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = r0 + 4 * i;
        float o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            o[j] = r < nr ? acc[i][j] * gelu_d(__ldg(z + (size_t)(row0 + r) * 3 * HID + c0 + j)) : 0.f;
        *reinterpret_cast<float4 *>(dst + r * LD + c0) = make_float4(o[0], o[1], o[2], o[3]);
    }
}

// the thread's 8 x 8 part of a 128 x 128 weight gradient: rows j0 .. j0 + 7, columns k0 .. k0 + 3 and
// k0 + 32 .. k0 + 35
struct GradMap {
    int j0, k0;
    __device__ __forceinline__ GradMap()
    {
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        j0 = 32 * (w >> 1) + 8 * (lane >> 3);
        k0 = 64 * (w & 1) + 4 * (lane & 7);
    }
};

// acc += d^T a over the tile's rows (64 FMAs for four 16-byte shared loads)
__device__ __forceinline__ void grad_tile(float (&acc)[8][8], const float *d, const float *a)
{
    const GradMap m;
#pragma unroll 2
    for (int r = 0; r < TR; ++r) {
        const float4 d0 = *reinterpret_cast<const float4 *>(d + r * LD + m.j0);
        const float4 d1 = *reinterpret_cast<const float4 *>(d + r * LD + m.j0 + 4);
        const float4 a0 = *reinterpret_cast<const float4 *>(a + r * LD + m.k0);
        const float4 a1 = *reinterpret_cast<const float4 *>(a + r * LD + m.k0 + 32);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float dj = j < 4 ? at4(d0, j) : at4(d1, j - 4);
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[j][k] = fmaf(dj, k < 4 ? at4(a0, k) : at4(a1, k - 4), acc[j][k]);
        }
    }
}

__device__ __forceinline__ void grad_add(float *G, const float (&acc)[8][8])
{
    const GradMap m;
    const bool al = ((uintptr_t)G & 15) == 0;
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float *p = G + (m.j0 + j) * HID + m.k0 + 32 * h;
            const float *v = &acc[j][4 * h];
            if (al) {
                asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(__cvta_generic_to_global(p)), "f"(v[0]),
                             "f"(v[1]), "f"(v[2]), "f"(v[3])
                             : "memory");
            } else {
                for (int e = 0; e < 4; ++e) atomicAdd(p + e, v[e]);
            }
        }
}

// A CTA keeps its part of every gradient in registers over all of its tiles (the two 128 x 128
// matrices 64 words a thread each) and adds it to the result once.
__global__ void __launch_bounds__(FT, 1) mlp_backward_kernel(const float *__restrict__ P, const float *__restrict__ x,
                                                             const float *__restrict__ z, const float *__restrict__ y,
                                                             const float *__restrict__ target, long n,
                                                             float *__restrict__ G, double *__restrict__ loss)
{
    extern __shared__ __align__(16) float sm[];
    float *w2 = sm, *w3 = w2 + HID * LD;
    float *a1 = w3 + HID * LD, *a2 = a1 + TR * LD, *a3 = a2 + TR * LD;      // activations
    float *dA = a3 + TR * LD, *dB = dA + TR * LD;                            // deltas
    float *w4 = dB + TR * LD, *dout = w4 + OUT * HID, *xs = dout + TR * OUT;
    __shared__ double red[FT / 32];
    const int tid = threadIdx.x;
    stage_rows(w2, P + W2, HID);
    stage_rows(w3, P + W3, HID);
    for (int i = tid; i < OUT * HID; i += blockDim.x) w4[i] = __ldg(P + W4 + i);
    const float scale = 2.f / (float)((double)n * OUT);
    double lsum = 0;
    float g2[8][8], g3[8][8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int k = 0; k < 8; ++k) { g2[j][k] = 0.f; g3[j][k] = 0.f; }
    float g1[HID * IN / FT], g4[OUT * HID / FT], gb[2], gb4 = 0.f;   // W1, W4, b1..b3, b4
#pragma unroll
    for (int i = 0; i < HID * IN / FT; ++i) g1[i] = 0.f;
#pragma unroll
    for (int i = 0; i < OUT * HID / FT; ++i) g4[i] = 0.f;
    gb[0] = gb[1] = 0.f;
    // bias sums: thread t < 128 takes b3[t] then b1[t], the others b2[t - 128]
    auto bias = [&](const float *d, int slot) {
        const int c = tid & (HID - 1);
        float s = 0.f;
#pragma unroll 8
        for (int r = 0; r < TR; ++r) s += d[r * LD + c];
        gb[slot] += s;
    };
    for (long row0 = (long)blockIdx.x * TR; row0 < n; row0 += (long)gridDim.x * TR) {
        const int nr = (int)min((long)TR, n - row0);
        __syncthreads();
        for (int i = tid; i < TR * HID; i += blockDim.x) {
            const int r = i / HID, k = i % HID;
            const bool ok = r < nr;
            const float *zr = z + (size_t)(row0 + r) * 3 * HID;
            a1[r * LD + k] = ok ? gelu(__ldg(zr + k)) : 0.f;
            a2[r * LD + k] = ok ? gelu(__ldg(zr + HID + k)) : 0.f;
            a3[r * LD + k] = ok ? gelu(__ldg(zr + 2 * HID + k)) : 0.f;
        }
        for (int i = tid; i < TR * IN; i += blockDim.x) {
            const int r = i / IN;
            xs[r * LD1 + i % IN] = r < nr ? __ldg(x + row0 * IN + i) : 0.f;
        }
        if (tid < TR * OUT) {
            const int r = tid / OUT;
            float d = 0.f;
            if (r < nr) {
                const float e = __ldg(y + row0 * OUT + tid) - __ldg(target + row0 * OUT + tid);
                lsum += (double)e * e;
                d = scale * e;
            }
            dout[tid] = d;
        }
        __syncthreads();
        // output layer: its gradient, and delta 3 = (d_out W4) * gelu'(z3) into dA
#pragma unroll
        for (int i = 0; i < OUT * HID / FT; ++i) {
            const int e = tid + FT * i, j = e / HID, k = e % HID;
            float s = 0.f;
#pragma unroll 8
            for (int r = 0; r < TR; ++r) s = fmaf(dout[r * OUT + j], a3[r * LD + k], s);
            g4[i] += s;
        }
        if (tid < OUT) {
            float s = 0.f;
            for (int r = 0; r < TR; ++r) s += dout[r * OUT + tid];
            gb4 += s;
        }
        for (int i = tid; i < TR * HID; i += blockDim.x) {
            const int r = i / HID, k = i % HID;
            float s = 0.f;
#pragma unroll
            for (int j = 0; j < OUT; ++j) s = fmaf(dout[r * OUT + j], w4[j * HID + k], s);
            dA[r * LD + k] = r < nr ? s * gelu_d(__ldg(z + (size_t)(row0 + r) * 3 * HID + 2 * HID + k)) : 0.f;
        }
        __syncthreads();
        grad_tile(g3, dA, a2);
        if (tid < HID) bias(dA, 0);
        delta_tile(dA, w3, z + HID, dB, row0, nr);
        __syncthreads();
        grad_tile(g2, dB, a1);
        if (tid >= HID) bias(dB, 0);
        delta_tile(dB, w2, z, dA, row0, nr);
        __syncthreads();
        if (tid < HID) bias(dA, 1);
#pragma unroll
        for (int i = 0; i < HID * IN / FT; ++i) {
            const int e = tid + FT * i, j = e / IN, k = e % IN;
            float s = 0.f;
#pragma unroll 8
            for (int r = 0; r < TR; ++r) s = fmaf(dA[r * LD + j], xs[r * LD1 + k], s);
            g1[i] += s;
        }
    }
    grad_add(G + W3, g3);
    grad_add(G + W2, g2);
#pragma unroll
    for (int i = 0; i < HID * IN / FT; ++i) atomicAdd(G + W1 + tid + FT * i, g1[i]);
#pragma unroll
    for (int i = 0; i < OUT * HID / FT; ++i) atomicAdd(G + W4 + tid + FT * i, g4[i]);
    if (tid < HID) {
        atomicAdd(G + B3 + tid, gb[0]);
        atomicAdd(G + B1 + tid, gb[1]);
    } else {
        atomicAdd(G + B2 + tid - HID, gb[0]);
    }
    if (tid < OUT) atomicAdd(G + B4 + tid, gb4);
    for (int d = 16; d > 0; d >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, d);
    if ((tid & 31) == 0) red[tid >> 5] = lsum;
    __syncthreads();
    if (tid == 0) {
        double t = 0;
        for (int i = 0; i < (int)blockDim.x / 32; ++i) t += red[i];
        atomicAdd(loss, t / ((double)n * OUT));
    }
}

__global__ void mlp_zero_kernel(float *grad, double *loss)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NPARAM) grad[i] = 0.f;
    if (i == 0) *loss = 0.0;
}

__global__ void adam_kernel(float *p, const float *g, float *m, float *v, int n, float lr, float b1, float b2,
                            float eps, float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

thread_local std::string g_mlp_error;

int cerr(cudaError_t e, const char *what)
{
    g_mlp_error = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? QC_ENOMEM : QC_ECUDA;
}

size_t fwd_smem() { return sizeof(float) * (2 * HID * LD + 2 * TR * LD + OUT * HID + HID * LD1 + TR * LD1); }
size_t bwd_smem() { return sizeof(float) * (2 * HID * LD + 5 * TR * LD + OUT * HID + TR * OUT + TR * LD1); }

int sm_count()
{
    int dev = 0, n = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n;
}

} // namespace

extern "C" int qc_mlp_forward(const float *params, const float *x, int64_t n, float *y, float *z, void *stream)
{
    g_mlp_error.clear();
    if (!params || !x || !y || n < 0) { g_mlp_error = "invalid arguments"; return QC_EINVAL; }
    if (n == 0) return QC_OK;
    cudaError_t e = cudaFuncSetAttribute(mlp_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fwd_smem());
    if (e != cudaSuccess) return cerr(e, "cudaFuncSetAttribute");
    const long tiles = (n + TR - 1) / TR;
    const int grid = (int)std::min<long>(tiles, (long)sm_count());
    mlp_forward_kernel<<<grid, FT, fwd_smem(), (cudaStream_t)stream>>>(params, x, n, y, z);
    e = cudaGetLastError();
    return e == cudaSuccess ? QC_OK : cerr(e, "mlp forward");
}

extern "C" int qc_mlp_backward(const float *params, const float *x, const float *z, const float *y, const float *target,
                               int64_t n, float *grad, double *loss, void *stream)
{
    g_mlp_error.clear();
    if (!params || !x || !z || !y || !target || !grad || !loss || n < 1) { g_mlp_error = "invalid arguments"; return QC_EINVAL; }
    cudaStream_t st = (cudaStream_t)stream;
    mlp_zero_kernel<<<(NPARAM + 255) / 256, 256, 0, st>>>(grad, loss);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mlp_backward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bwd_smem());
    if (e != cudaSuccess) return cerr(e, "mlp backward setup");
    const long tiles = (n + TR - 1) / TR;
    const int grid = (int)std::min<long>(tiles, (long)sm_count());
    mlp_backward_kernel<<<grid, FT, bwd_smem(), st>>>(params, x, z, y, target, n, grad, loss);
    e = cudaGetLastError();
    return e == cudaSuccess ? QC_OK : cerr(e, "mlp backward");
}

extern "C" int qc_mlp_adam(float *params, const float *grad, float *m, float *v, float lr, float beta1, float beta2,
                           float eps, int32_t step, void *stream)
{
    g_mlp_error.clear();
    if (!params || !grad || !m || !v || step < 1) { g_mlp_error = "invalid arguments"; return QC_EINVAL; }
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    adam_kernel<<<(NPARAM + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params, grad, m, v, NPARAM, lr, beta1, beta2,
                                                                         eps, c1, c2);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? QC_OK : cerr(e, "adam");
}

extern "C" const char *qc_mlp_last_error(void) { return g_mlp_error.c_str(); }
