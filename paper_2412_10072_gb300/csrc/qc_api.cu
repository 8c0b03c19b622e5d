// qc_api.cu -- host side of libqc: validation, device staging, the chain
// schedule of epochs x terms x iterations (Section 4.3 of arxiv 2412.10072)
// and CUDA-graph replay of each term's iteration loop.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <memory>
#include <string>
#include <vector>

#include "../../include/qc.h"
#include "qc_internal.h"
#include "qc_kernels.cuh"

using namespace qc;

namespace {

thread_local std::string g_create_error;

__global__ void bl_scale_kernel(const float4 *model, const int4 *rows, int n_row, int n_chan, unsigned *scale_bits)
{
    const long n = (long)n_row * n_chan;
    for (long s = (long)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (long)gridDim.x * blockDim.x) {
        const int row = (int)(s / n_chan);
        const int4 meta = rows[row];
        if (meta.x == meta.y) continue;
        const float4 a = model[2 * s], b = model[2 * s + 1];
        float m = fmaxf(fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), fabsf(a.w))),
                        fmaxf(fmaxf(fabsf(b.x), fabsf(b.y)), fmaxf(fabsf(b.z), fabsf(b.w))));
        if (!(m <= 3.0e38f)) m = 0.f;           // non-finite (flagged garbage) does not set the scale
        atomicMax(scale_bits + meta.w, __float_as_uint(m));
    }
}

__global__ void pack16_kernel(const float4 *model, const int4 *rows, int n_row, int n_chan, const float *scale,
                              uint4 *out)
{
    const long n = (long)n_row * n_chan;
    for (long s = (long)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (long)gridDim.x * blockDim.x) {
        const int row = (int)(s / n_chan);
        const int4 meta = rows[row];
        const float sc = meta.x == meta.y ? 1.f : scale[meta.w];
        const float inv = sc > 0.f ? 1.f / sc : 0.f;
        const float4 a = model[2 * s], b = model[2 * s + 1];
        __half2 h0 = __floats2half2_rn(a.x * inv, a.y * inv), h1 = __floats2half2_rn(a.z * inv, a.w * inv);
        __half2 h2 = __floats2half2_rn(b.x * inv, b.y * inv), h3 = __floats2half2_rn(b.z * inv, b.w * inv);
        uint4 o;
        o.x = *reinterpret_cast<unsigned *>(&h0);
        o.y = *reinterpret_cast<unsigned *>(&h1);
        o.z = *reinterpret_cast<unsigned *>(&h2);
        o.w = *reinterpret_cast<unsigned *>(&h3);
        out[s] = o;
    }
}

__global__ void fix_scale_kernel(unsigned *bits, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const float v = __uint_as_float(bits[i]);
        reinterpret_cast<float *>(bits)[i] = v > 0.f ? v : 1.f;
    }
}

// user gains [n_tint][n_fint][n_ant][4] (complex64) or phases [..][2] (float32)
// -> FP64 master parameters and FP32 kernel table [n_tint][n_ant][n_fint]
__global__ void gains_in_kernel(int type, int n_tint, int n_fint, int n_ant, const void *src, double *params,
                                float4 *tab)
{
    const long n = (long)n_tint * n_fint * n_ant;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const int ant = (int)(i % n_ant);
        const long bin = i / n_ant;
        const int tint = (int)(bin / n_fint), fint = (int)(bin % n_fint);
        const size_t t = ((size_t)tint * n_ant + ant) * n_fint + fint;
        if (type == 2) {
            const float *ph = (const float *)src + 2 * i;
            params[2 * i] = ph[0];
            params[2 * i + 1] = ph[1];
            double s0, c0, s1, c1;
            sincos((double)ph[0], &s0, &c0);
            sincos((double)ph[1], &s1, &c1);
            tab[t] = make_float4((float)c0, (float)s0, (float)c1, (float)s1);
            continue;
        }
        const float2 *g = (const float2 *)src + 4 * i;
        double2 *P = reinterpret_cast<double2 *>(params) + 4 * i;
        for (int e = 0; e < 4; ++e) P[e] = make_double2(g[e].x, g[e].y);
        if (type == 0) { P[1] = make_double2(0, 0); P[2] = make_double2(0, 0); }
        if (type == 1) {
            tab[2 * t] = make_float4(g[0].x, g[0].y, g[1].x, g[1].y);
            tab[2 * t + 1] = make_float4(g[2].x, g[2].y, g[3].x, g[3].y);
        } else {
            tab[t] = make_float4(g[0].x, g[0].y, g[3].x, g[3].y);
        }
    }
}

__global__ void gains_out_kernel(int type, long n, const double *params, void *dst)
{
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        if (type == 2) {
            float *ph = (float *)dst + 2 * i;
            ph[0] = (float)params[2 * i];
            ph[1] = (float)params[2 * i + 1];
            continue;
        }
        float2 *g = (float2 *)dst + 4 * i;
        const double2 *P = reinterpret_cast<const double2 *>(params) + 4 * i;
        for (int e = 0; e < 4; ++e) g[e] = make_float2((float)P[e].x, (float)P[e].y);
        if (type == 0) { g[1] = make_float2(0.f, 0.f); g[2] = make_float2(0.f, 0.f); }
    }
}

__global__ void bin_bytes_kernel(int n, const long long *nvis, const long long *nunflag, long long b_flag,
                                 long long b_unflag, long long *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = nvis[i] * b_flag + nunflag[i] * b_unflag;
}

__global__ void init_term_kernel(int n_bins, uint8_t *active, int *cnt, int n_cnt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_bins) active[i] = 1;
    if (i < n_cnt) cnt[i] = i == 0 ? n_bins : 0;
}

template <typename T> size_t nbytes(size_t n) { return n * sizeof(T); }

int grid_for(long n, int block, int sm)
{
    long g = (n + block - 1) / block;
    return (int)std::max(1L, std::min(g, (long)sm * 32));
}

} // namespace

// ---------------------------------------------------------------------------
// context
// ---------------------------------------------------------------------------

qc_ctx::~qc_ctx()
{
    for (auto &b : tb) if (b.exec) cudaGraphExecDestroy(b.exec);
    for (void *p : owned) qc_dev_free(p);
    if (pin_ptr) cudaFreeHost(pin_ptr);
    if (pin_next) cudaFreeHost(pin_next);
    for (auto e : events) cudaEventDestroy(e);
    for (auto e : sums_events) cudaEventDestroy(e);
    if (own_stream) cudaStreamDestroy(own_stream);
}

void qc_ctx::pin_begin()
{
    pin_used = pin_want = 0;
    pin_outs.clear();
    pin_open = true;
}

// A call that ends before pin_end has its copies finished here, while its stream still exists: the stream
// is the caller's, and nothing keeps its handle beyond the call.
PinScope::~PinScope()
{
    if (!c->pin_open) return;
    cudaStreamSynchronize(st);
    c->pin_outs.clear();
    c->pin_open = false;
}

void *qc_ctx::pin_get(size_t bytes)
{
    bytes = (bytes + 63) / 64 * 64;
    pin_want += bytes;
    if (pin_used + bytes > pin_size) return nullptr;
    void *p = pin_ptr + pin_used;
    pin_used += bytes;
    return p;
}

// Room for what this call has asked for and will ask for (`more`), for the calls to come: allocated (0.1 ms)
// by a solve once its iterations are on the stream, which hide it; a call that finds no room copies directly.
void qc_ctx::pin_reserve(size_t more)
{
    const size_t want = pin_want + more, size = (want + (64u << 10) - 1) / (64u << 10) * (64u << 10);
    if (want <= pin_size || size > PIN_MAX || pin_next) return;
    void *p = nullptr;
    if (cudaHostAlloc(&p, size, cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    pin_next = (char *)p;
    pin_next_size = size;
}

cudaError_t qc_ctx::to_device(void *dst, const void *src, size_t bytes, cudaStream_t st)
{
    void *p = pin_get(bytes);
    if (p) memcpy(p, src, bytes);
    return cudaMemcpyAsync(dst, p ? p : src, bytes, cudaMemcpyHostToDevice, st);
}

cudaError_t qc_ctx::to_host(void *dst, const void *src, size_t bytes, cudaStream_t st)
{
    void *p = pin_get(bytes);
    if (p) pin_outs.push_back({ dst, p, bytes });
    return cudaMemcpyAsync(p ? p : dst, src, bytes, cudaMemcpyDeviceToHost, st);
}

void qc_ctx::pin_end()
{
    for (const PinOut &o : pin_outs) memcpy(o.dst, o.src, o.bytes);
    pin_outs.clear();
    pin_open = false;
    if (pin_next) {                 // nothing of the old block is in flight any more
        if (pin_ptr) cudaFreeHost(pin_ptr);
        pin_ptr = pin_next;
        pin_size = pin_next_size;
        pin_next = nullptr;
    }
}

int qc_ctx::fail(int code, const std::string &msg)
{
    err = msg;
    return code;
}

int qc_ctx::cuda_fail(cudaError_t e, const char *what)
{
    err = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? QC_ENOMEM : QC_ECUDA;
}

namespace {
std::atomic<long long> g_alloc_countdown{0};   // > 0: the allocation that brings it to 0 fails
std::atomic<long long> g_live_allocs{0};
std::atomic<long long> g_free_bytes{-1};       // >= 0: what qc_dev_spare takes for the free memory
std::atomic<unsigned long long> g_wait_limit_ns{2000000000ull};
std::atomic<int> g_wait_stall{-1};
} // namespace

cudaError_t qc_dev_malloc(void **p, size_t bytes)
{
    *p = nullptr;
    long long c = g_alloc_countdown.load();
    while (c > 0 && !g_alloc_countdown.compare_exchange_weak(c, c - 1)) {}
    if (c == 1) return cudaErrorMemoryAllocation;      // injected on the host: cudaMalloc is not called
    const cudaError_t e = cudaMalloc(p, std::max<size_t>(bytes, 16));
    if (e == cudaSuccess) ++g_live_allocs;
    return e;
}

// Whether `bytes` more of workspace that a route can do without leave as much again for the caller's own
// allocations.
bool qc_dev_spare(size_t bytes)
{
    size_t avail = 0, total = 0;
    const long long forced = g_free_bytes.load();
    if (forced >= 0) avail = (size_t)forced;
    else if (cudaMemGetInfo(&avail, &total) != cudaSuccess) { cudaGetLastError(); return true; }
    return bytes <= avail / 2;
}

void qc_dev_free(void *p)
{
    if (!p) return;
    cudaFree(p);
    --g_live_allocs;
}

uint64_t qc_wait_limit_ns() { return g_wait_limit_ns.load(); }
int qc_wait_stall_stage() { return g_wait_stall.load(); }

extern "C" void qc_test_fail_alloc(int64_t n) { g_alloc_countdown.store(n > 0 ? n : 0); }
extern "C" void qc_test_free_bytes(int64_t bytes) { g_free_bytes.store(bytes >= 0 ? bytes : -1); }
extern "C" int64_t qc_test_live_allocs(void) { return g_live_allocs.load(); }
extern "C" void qc_test_wait_limit(int64_t limit_ns, int32_t stall_stage)
{
    g_wait_limit_ns.store(limit_ns > 0 ? (unsigned long long)limit_ns : 2000000000ull);
    g_wait_stall.store(stall_stage >= 0 ? stall_stage : -1);
}

void *qc_ctx::alloc(size_t bytes, cudaError_t *e)
{
    void *p = nullptr;
    *e = qc_dev_malloc(&p, bytes);
    if (*e == cudaSuccess) owned.push_back(p);
    return p;
}

void qc_ctx::release(void *p)
{
    auto it = std::find(owned.begin(), owned.end(), p);
    if (it != owned.end()) { qc_dev_free(p); owned.erase(it); }
}

void qc_ctx::drop(Buf &b)
{
    if (b.ptr) release(b.ptr);
    b = Buf();
}

int qc_ctx::ensure(Buf &b, size_t bytes)
{
    if (b.bytes >= bytes && b.ptr) return QC_OK;
    if (b.ptr) release(b.ptr);
    cudaError_t e;
    b.ptr = alloc(bytes, &e);
    b.bytes = b.ptr ? std::max<size_t>(bytes, 16) : 0;
    if (e != cudaSuccess) { b.ptr = nullptr; return cuda_fail(e, "cudaMalloc"); }
    return QC_OK;
}

#define CK(call)                                          \
    do {                                                  \
        cudaError_t e_ = (call);                          \
        if (e_ != cudaSuccess) return c->cuda_fail(e_, #call); \
    } while (0)

extern "C" int qc_create(const qc_problem *p, qc_ctx **out)
{
    g_create_error.clear();
    if (!out) { g_create_error = "out is NULL"; return QC_EINVAL; }
    *out = nullptr;
    auto bad = [](const char *m) { g_create_error = m; return QC_EINVAL; };
    if (!p) return bad("problem is NULL");
    if (p->n_corr != 4) return bad("n_corr must be 4");
    if (p->n_dir < 1 || p->n_dir > QC_MAX_DIRS) return bad("n_dir must be in [1, QC_MAX_DIRS]");
    if (p->n_dir > 1 && p->model_fp16) return bad("the float16 model takes one direction (n_dir = 1)");
    if (p->n_row < 0 || p->n_chan < 1 || p->n_ant < 2 || p->n_time < 1) return bad("invalid sizes");
    if ((long long)p->n_row * p->n_chan > (1LL << 40)) return bad("problem too large");
    if (!p->data || !p->model || !p->weight) return bad("data, model and weight are required");
    if (!p->ant1 || !p->ant2 || !p->time_idx) return bad("ant1, ant2 and time_idx are required (host arrays)");
    if (p->memory != QC_MEM_HOST && p->memory != QC_MEM_DEVICE) return bad("memory must be QC_MEM_HOST or QC_MEM_DEVICE");
    for (int r = 0; r < p->n_row; ++r) {
        if (p->ant1[r] < 0 || p->ant1[r] >= p->n_ant || p->ant2[r] < 0 || p->ant2[r] >= p->n_ant)
            return bad("antenna index out of range");
        if (p->time_idx[r] < 0 || p->time_idx[r] >= p->n_time) return bad("time index out of range");
    }
    if (p->memory == QC_MEM_DEVICE) {
        for (const void *ptr : { p->data, p->model, (const void *)p->weight })
            if (((uintptr_t)ptr) % 16) return bad("device data/model/weight must be 16-byte aligned");
    }

    std::unique_ptr<qc_ctx> c(new qc_ctx());
    c->n_row = p->n_row;
    c->n_chan = p->n_chan;
    c->n_ant = p->n_ant;
    c->n_time = p->n_time;
    c->n_dir = p->n_dir;
    c->m16 = p->model_fp16 != 0;
    c->has_flag = p->flag != nullptr;
    {
        cudaError_t e = cudaGetDevice(&c->dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, c->dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->dev);
        if (e == cudaSuccess)
            e = cudaDeviceGetAttribute(&c->smem_per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, c->dev);
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->own_stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) { g_create_error = std::string("CUDA init: ") + cudaGetErrorString(e); return QC_ECUDA; }
    }
    // rows {ant1, ant2, time, baseline id}; strips: rows of one (ant1, ant2) pair in time order
    const int na = p->n_ant;
    std::vector<int> bl_of_pair((size_t)na * na, -1);
    std::vector<int4> rows(p->n_row);
    int n_bl = 0;
    for (int r = 0; r < p->n_row; ++r) {
        const int a1 = p->ant1[r], a2 = p->ant2[r];
        int bl = 0;
        if (a1 != a2) {
            int &slot = bl_of_pair[(size_t)a1 * na + a2];
            if (slot < 0) slot = n_bl++;
            bl = slot;
        }
        rows[r] = make_int4(a1, a2, p->time_idx[r], bl);
    }
    c->n_bl = n_bl;
    std::vector<int> strip_off(n_bl + 1, 0), strip_rows;
    for (int r = 0; r < p->n_row; ++r) if (rows[r].x != rows[r].y) strip_off[rows[r].w + 1]++;
    for (int b = 0; b < n_bl; ++b) strip_off[b + 1] += strip_off[b];
    strip_rows.resize(strip_off[n_bl]);
    {
        std::vector<int> fill(strip_off.begin(), strip_off.end() - 1);
        for (int r = 0; r < p->n_row; ++r) if (rows[r].x != rows[r].y) strip_rows[fill[rows[r].w]++] = r;
        for (int b = 0; b < n_bl; ++b)
            std::stable_sort(strip_rows.begin() + strip_off[b], strip_rows.begin() + strip_off[b + 1],
                             [&](int x, int y) { return rows[x].z < rows[y].z; });
    }
    c->n_strips = n_bl;
    c->n_strip_rows = (long)strip_rows.size();
    for (int b = 0; b < n_bl; ++b) c->max_strip_rows = std::max(c->max_strip_rows, strip_off[b + 1] - strip_off[b]);
    c->full_grid = n_bl > 0;
    for (int b = 0; b < n_bl && c->full_grid; ++b) {
        c->full_grid = strip_off[b + 1] - strip_off[b] == p->n_time;
        for (int k = strip_off[b]; k < strip_off[b + 1] && c->full_grid; ++k)
            c->full_grid = rows[strip_rows[k]].z == k - strip_off[b];
    }
    cudaError_t e;
    qc_ctx *cc = c.get();
    auto dalloc = [&](size_t bytes) -> void * { return cc->alloc(bytes, &e); };
#define DALLOC(dst, T, n)                                                                    \
    do {                                                                                     \
        dst = (T *)dalloc(nbytes<T>(n));                                                     \
        if (e != cudaSuccess) { g_create_error = "cudaMalloc failed"; return e == cudaErrorMemoryAllocation ? QC_ENOMEM : QC_ECUDA; } \
    } while (0)
#define HCOPY(dst, src, bytes)                                                               \
    do {                                                                                     \
        e = cudaMemcpy(dst, src, bytes, cudaMemcpyHostToDevice);                             \
        if (e != cudaSuccess) { g_create_error = std::string("H2D copy: ") + cudaGetErrorString(e); return QC_ECUDA; } \
    } while (0)
    DALLOC(c->d_rows, int4, std::max(1, p->n_row));
    if (p->n_row) HCOPY(c->d_rows, rows.data(), nbytes<int4>(p->n_row));
    DALLOC(c->d_strip_off, int, n_bl + 1);
    HCOPY(c->d_strip_off, strip_off.data(), nbytes<int>(n_bl + 1));
    DALLOC(c->d_strip_rows, int, std::max<size_t>(1, strip_rows.size()));
    if (!strip_rows.empty()) HCOPY(c->d_strip_rows, strip_rows.data(), nbytes<int>(strip_rows.size()));
    {
        // unordered antenna pairs: both orientations of a baseline share one slot of the sums
        // of a term solved from sums (qc_opts.moments)
        std::vector<int> upair((size_t)na * na, -1), up_of_bl(std::max(1, n_bl), 0);
        int n_up = 0;
        for (int a1 = 0; a1 < na; ++a1)
            for (int a2 = 0; a2 < na; ++a2) {
                const int bl = bl_of_pair[(size_t)a1 * na + a2];
                if (bl < 0) continue;
                const int lo = std::min(a1, a2), hi = std::max(a1, a2);
                int &slot = upair[(size_t)lo * na + hi];
                if (slot < 0) { slot = n_up++; upair[(size_t)hi * na + lo] = slot; }
                up_of_bl[bl] = slot;
            }
        c->n_up = n_up;
        c->pair_strips.assign(n_up, make_int2(-1, -1));
        for (int bl = 0; bl < n_bl; ++bl) {
            int2 &g = c->pair_strips[up_of_bl[bl]];
            (g.x < 0 ? g.x : g.y) = bl;
        }
        c->full_grid = c->full_grid && n_up == n_bl;
        // the last pair that had a row at each time; a pair's rows are in two strips at most
        c->pair_time_once = true;
        std::vector<int> last(p->n_time, -1);
        for (int u = 0; u < n_up; ++u)
            for (int b : { c->pair_strips[u].x, c->pair_strips[u].y })
                for (int k = b < 0 ? 0 : strip_off[b]; b >= 0 && k < strip_off[b + 1]; ++k) {
                    int &l = last[rows[strip_rows[k]].z];
                    if (l == u) c->pair_time_once = false;
                    l = u;
                }
        DALLOC(c->d_upair, int, std::max<size_t>(1, upair.size()));
        if (!upair.empty()) HCOPY(c->d_upair, upair.data(), nbytes<int>(upair.size()));
        DALLOC(c->d_up_of_bl, int, up_of_bl.size());
        HCOPY(c->d_up_of_bl, up_of_bl.data(), nbytes<int>(up_of_bl.size()));
    }

    const size_t n_vis = (size_t)p->n_row * p->n_chan;
    const float4 *model32 = nullptr;
    if (p->memory == QC_MEM_DEVICE) {
        c->d_vis = (const float4 *)p->data;
        model32 = (const float4 *)p->model;
        c->d_weight = (const float4 *)p->weight;
        c->d_flag = p->flag;
    } else {
        float4 *v, *w;
        DALLOC(v, float4, 2 * n_vis);
        HCOPY(v, p->data, nbytes<float4>(2 * n_vis));
        DALLOC(w, float4, n_vis);
        HCOPY(w, p->weight, nbytes<float4>(n_vis));
        c->d_vis = v;
        c->d_weight = w;
        float4 *m;
        DALLOC(m, float4, 2 * n_vis * p->n_dir);
        HCOPY(m, p->model, nbytes<float4>(2 * n_vis * p->n_dir));
        model32 = m;
        if (p->flag) {
            uint8_t *f;
            DALLOC(f, uint8_t, n_vis);
            HCOPY(f, p->flag, n_vis);
            c->d_flag = f;
        }
    }
    if (c->m16) {
        unsigned *bits;
        uint4 *m16;
        DALLOC(bits, unsigned, std::max(1, n_bl));
        DALLOC(m16, uint4, n_vis);
        e = cudaMemsetAsync(bits, 0, nbytes<unsigned>(std::max(1, n_bl)), c->own_stream);
        if (e == cudaSuccess && n_vis) {
            bl_scale_kernel<<<grid_for((long)n_vis, 256, c->sm_count), 256, 0, c->own_stream>>>(
                model32, c->d_rows, p->n_row, p->n_chan, bits);
            fix_scale_kernel<<<(n_bl + 255) / 256 + 1, 256, 0, c->own_stream>>>(bits, n_bl);
            pack16_kernel<<<grid_for((long)n_vis, 256, c->sm_count), 256, 0, c->own_stream>>>(
                model32, c->d_rows, p->n_row, p->n_chan, (const float *)bits, m16);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->own_stream);
        if (e != cudaSuccess) { g_create_error = std::string("fp16 model packing: ") + cudaGetErrorString(e); return QC_ECUDA; }
        c->d_model16 = m16;
        c->d_bl_scale = (const float *)bits;
        if (p->memory == QC_MEM_HOST) c->release((void *)model32);
        model32 = nullptr;
    }
    c->d_model = model32;
    {
        // weights with flags and autocorrelations folded in (w = 0), read by the streaming
        // kernel instead of the flags; the owned host-mode copy is folded in place
        float4 *wf = nullptr;
        if (p->memory == QC_MEM_HOST) wf = const_cast<float4 *>(c->d_weight);
        else DALLOC(wf, float4, std::max<size_t>(1, n_vis));
        if (n_vis) {
            fold_flags_kernel<<<grid_for((long)n_vis, 256, c->sm_count), 256, 0, c->own_stream>>>(
                c->d_weight, c->d_flag, c->d_rows, p->n_row, p->n_chan, wf);
            e = cudaGetLastError();
            if (e == cudaSuccess) e = cudaStreamSynchronize(c->own_stream);
            if (e != cudaSuccess) { g_create_error = std::string("weights: ") + cudaGetErrorString(e); return QC_ECUDA; }
        }
        c->d_wf = wf;
    }
    DALLOC(c->d_row_live, uint8_t, std::max(1, p->n_row));
    DALLOC(c->d_err, int, 1);
    e = cudaMemsetAsync(c->d_err, 0, sizeof(int), c->own_stream);
    if (e == cudaSuccess && p->n_row) {
        row_live_kernel<<<grid_for((long)p->n_row * 32, 256, c->sm_count), 256, 0, c->own_stream>>>(c->data_desc(),
                                                                                                     c->d_row_live);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->own_stream);
    if (e != cudaSuccess) { g_create_error = std::string("row flags: ") + cudaGetErrorString(e); return QC_ECUDA; }
#undef DALLOC
#undef HCOPY
    *out = c.release();
    return QC_OK;
}

extern "C" void qc_destroy(qc_ctx *c) { delete c; }

// lets the allocation-free entry point report through qc_last_error(NULL)
void qc_internal_set_error(const char *msg) { g_create_error = msg; }

extern "C" const char *qc_last_error(const qc_ctx *c)
{
    if (!c) return g_create_error.c_str();
    return c->err.c_str();
}

extern "C" const char *qc_version(void) { return "qc-gb300 1.0 (sm_103a)"; }

// ---------------------------------------------------------------------------
// term staging
// ---------------------------------------------------------------------------

static size_t term_nbins(const qc_term &t) { return (size_t)t.n_tint * t.n_fint; }

int qc_ctx::validate_terms(const qc_term *terms, int n_terms, bool need_solve_fields)
{
    if (!terms) return fail(QC_EINVAL, "terms is NULL");
    if (n_terms < 1 || n_terms > QC_MAX_TERMS) return fail(QC_EINVAL, "n_terms must be in [1, QC_MAX_TERMS]");
    for (int j = 0; j < n_terms; ++j) {
        const qc_term &t = terms[j];
        if (t.type < 0 || t.type > 3) return fail(QC_EINVAL, "unknown term type");
        if (t.type == QC_TERM_DELAY) {
            if (!t.chan_freq) return fail(QC_EINVAL, "a delay term needs chan_freq");
            for (int i = 0; i < n_chan; ++i)
                if (!std::isfinite(t.chan_freq[i])) return fail(QC_EINVAL, "chan_freq must be finite");
            if ((long long)t.n_tint * n_chan * n_ant > (1LL << 31)) return fail(QC_EINVAL, "delay term too large");
        }
        if (t.n_tint < 1 || t.n_fint < 1) return fail(QC_EINVAL, "n_tint and n_fint must be >= 1");
        if ((long long)t.n_tint * t.n_fint * n_ant > (1LL << 31)) return fail(QC_EINVAL, "term too large");
        if (!t.t_map || !t.f_map || !t.gains) return fail(QC_EINVAL, "t_map, f_map and gains are required");
        if (t.memory != QC_MEM_HOST && t.memory != QC_MEM_DEVICE) return fail(QC_EINVAL, "term memory invalid");
        for (int i = 0; i < n_time; ++i)
            if (t.t_map[i] < 0 || t.t_map[i] >= t.n_tint) return fail(QC_EINVAL, "t_map value out of range");
        for (int i = 0; i < n_chan; ++i) {
            if (t.f_map[i] < 0 || t.f_map[i] >= t.n_fint) return fail(QC_EINVAL, "f_map value out of range");
            if (i && t.f_map[i] < t.f_map[i - 1]) return fail(QC_EINVAL, "f_map must be non-decreasing");
        }
        if (need_solve_fields && t.solve) {
            if (t.max_iter < 1) return fail(QC_EINVAL, "max_iter must be >= 1 for a solved term");
            if (!(t.tol >= 0)) return fail(QC_EINVAL, "tol must be >= 0");
        }
        if (n_dir > 1) {
            if (t.type == QC_TERM_PHASE)
                return fail(QC_EUNSUPPORTED, "chains with directions take diagonal, full and delay terms");
            if (t.type == QC_TERM_DELAY && t.dd)
                return fail(QC_EUNSUPPORTED, "a delay term is direction-independent");
            if (need_solve_fields && t.solve && !t.dd)
                for (int i = 0; i < j; ++i)
                    if (terms[i].dd)
                        return fail(QC_EUNSUPPORTED, "a solved direction-independent term must not have a "
                                                     "direction-dependent term to its left");
        }
    }
    return QC_OK;
}

// The kernels' view of the chain: a delay term becomes a diagonal term with one bin per
// (time interval, channel) and the identity channel map, its table evaluated at every
// channel from the interval's parameters (the channel ranges, maps and frequencies of its
// intervals are uploaded here).  Other terms are unchanged.
int qc_ctx::expand_terms(const qc_term *terms, int n_terms, std::vector<qc_term> &xt, cudaStream_t st)
{
    qc_ctx *c = this;
    xt.assign(terms, terms + n_terms);
    if ((int)fid.size() != n_chan) {
        fid.resize(n_chan);
        for (int i = 0; i < n_chan; ++i) fid[i] = i;
    }
    for (int j = 0; j < n_terms; ++j) {
        delay[j] = terms[j].type == QC_TERM_DELAY;
        if (!delay[j]) continue;
        const qc_term &t = terms[j];
        TermBufs &B = tb[j];
        B.hfr.assign(t.n_fint, make_int2(-1, -2));
        for (int ch = 0; ch < n_chan; ++ch) {
            int2 &r = B.hfr[t.f_map[ch]];
            if (r.x < 0) r.x = ch;
            r.y = ch;
        }
        int rc;
        if ((rc = ensure(B.dfmap, nbytes<int>(std::max(1, n_chan))))) return rc;
        if ((rc = ensure(B.dfr, nbytes<int2>(t.n_fint)))) return rc;
        if ((rc = ensure(B.dnu, nbytes<double>(std::max(1, n_chan))))) return rc;
        if ((rc = ensure(B.domega, nbytes<float>(2 * (size_t)std::max(1, n_chan))))) return rc;
        B.hufmap.assign(t.f_map, t.f_map + n_chan);
        double mean_nu = 0;
        for (int ch = 0; ch < n_chan; ++ch) mean_nu += t.chan_freq[ch];
        B.omega_ref = n_chan ? DELAY_TWO_PI * (mean_nu / n_chan) : 0.0;
        std::vector<float> om(2 * (size_t)n_chan);      // heads, then tails
        B.hom_sums.assign(t.n_fint, make_double2(0.0, 0.0));
        B.om_max = 0.0;
        for (int ch = 0; ch < n_chan; ++ch) {
            const double w = DELAY_TWO_PI * t.chan_freq[ch] - B.omega_ref;
            om[ch] = (float)w;
            om[n_chan + ch] = (float)(w - (double)om[ch]);
            B.om_max = std::max(B.om_max, std::fabs(w));
            double2 &m = B.hom_sums[t.f_map[ch]];
            m.x += w;
            m.y += w * w;
        }
        if ((rc = ensure(B.dom_sums, nbytes<double2>(t.n_fint)))) return rc;
        CK(to_device(B.dom_sums.ptr, B.hom_sums.data(), nbytes<double2>(t.n_fint), st));
        if (n_chan) {
            CK(to_device(B.dfmap.ptr, t.f_map, nbytes<int>(n_chan), st));
            CK(to_device(B.dnu.ptr, t.chan_freq, nbytes<double>(n_chan), st));
            CK(to_device(B.domega.ptr, om.data(), nbytes<float>(om.size()), st));
        }
        CK(to_device(B.dfr.ptr, B.hfr.data(), nbytes<int2>(t.n_fint), st));
        xt[j].type = QC_TERM_DIAG;
        xt[j].n_fint = n_chan;
        xt[j].f_map = fid.data();
    }
    return QC_OK;
}

DelayArgs qc_ctx::delay_args(int j, const qc_term &xt_j)
{
    TermBufs &B = tb[j];
    DelayArgs d;
    d.n_tint = xt_j.n_tint;
    d.n_fint = (int)B.hfr.size();
    d.n_ant = n_ant;
    d.n_chan = n_chan;
    d.fmap = (const int *)B.dfmap.ptr;
    d.frange = (const int2 *)B.dfr.ptr;
    d.nu = (const double *)B.dnu.ptr;
    d.params = (double *)B.params.ptr;
    d.tab = (float4 *)B.tab.ptr;
    d.omega_ref = B.omega_ref;
    return d;
}

// Upload maps and gains of every term; fills chain (device descriptors).
int qc_ctx::stage_terms(const qc_term *terms, int n_terms, cudaStream_t st, Chain &chain)
{
    qc_ctx *c = this;
    chain.n_terms = n_terms;
    chain.n = -1;
    chain.n_ant = n_ant;
    for (int j = 0; j < n_terms; ++j) {
        const qc_term &t = terms[j];
        TermBufs &B = tb[j];
        cur_nd[j] = term_nd(t);
        const size_t nb = term_nbins(t);
        const size_t nent = nb * term_nat(t);
        const size_t tab_f4 = nent * (t.type == 1 ? 2 : 1);
        int rc;
        if ((rc = ensure(B.maps, nbytes<int>(n_time + n_chan)))) return rc;
        if ((rc = ensure(B.tab, nbytes<float4>(tab_f4)))) return rc;
        if ((rc = ensure(B.params, nbytes<double>(nent * (t.type == 2 ? 2 : 8))))) return rc;
        if ((rc = ensure(B.stage, nent * (t.type == 2 ? 8 : 32)))) return rc;
        B.hmaps.assign(t.t_map, t.t_map + n_time);
        B.hmaps.insert(B.hmaps.end(), t.f_map, t.f_map + n_chan);
        CK(to_device(B.maps.ptr, B.hmaps.data(), nbytes<int>(n_time + n_chan), st));
        if (delay[j]) {
            // parameters [n_tint][n_fint][n_ant][4] (float32) -> FP64 master; table per channel
            const DelayArgs da = delay_args(j, t);
            const size_t nvals = (size_t)da.n_tint * da.n_fint * n_ant * 4;
            const void *src = t.gains;
            if (t.memory == QC_MEM_HOST) {
                CK(to_device(B.stage.ptr, t.gains, nbytes<float>(nvals), st));
                src = B.stage.ptr;
            }
            delay_params_in_kernel<<<grid_for((long)nvals, 256, sm_count), 256, 0, st>>>((long)nvals, (const float *)src,
                                                                                        da.params);
            CK(cudaGetLastError());
            delay_tab_kernel<<<grid_for((long)nent, 256, sm_count), 256, 0, st>>>(da);
            CK(cudaGetLastError());
            launches += 2;
        } else {
            const void *src = t.gains;
            if (t.memory == QC_MEM_HOST) {
                CK(to_device(B.stage.ptr, t.gains, nent * (t.type == 2 ? 8 : 32), st));
                src = B.stage.ptr;
            }
            gains_in_kernel<<<grid_for((long)nent, 256, sm_count), 256, 0, st>>>(t.type, t.n_tint, t.n_fint, term_nat(t), src,
                                                                                (double *)B.params.ptr,
                                                                                (float4 *)B.tab.ptr);
            CK(cudaGetLastError());
            ++launches;
        }
        DevTerm &d = chain.t[j];
        d.type = t.type;
        d.n_tint = t.n_tint;
        d.n_fint = t.n_fint;
        d.t_map = (const int *)B.maps.ptr;
        d.f_map = (const int *)B.maps.ptr + n_time;
        d.tab = (const float4 *)B.tab.ptr;
    }
    return QC_OK;
}

Data qc_ctx::data_desc() const
{
    Data D;
    D.n_row = n_row;
    D.n_chan = n_chan;
    D.vis = d_vis;
    D.model = d_model;
    D.weight = d_weight_use ? d_weight_use : d_weight;
    D.model16 = d_model16;
    D.bl_scale = d_bl_scale;
    D.flag = d_flag;
    D.rows = d_rows;
    D.strip_rows = d_strip_rows;
    D.strip_off = d_strip_off;
    D.n_strips = n_strips;
    return D;
}

// ---------------------------------------------------------------------------
// residual / chi^2
// ---------------------------------------------------------------------------

extern "C" int qc_residual(qc_ctx *c, const qc_term *terms, int32_t n_terms, void *resid, int32_t resid_memory,
                           double *chi2)
{
    if (!c) return QC_EINVAL;
    c->err.clear();
    if (!chi2) return c->fail(QC_EINVAL, "chi2 is NULL");
    int rc = c->validate_terms(terms, n_terms, false);
    if (rc) return rc;
    cudaStream_t st = c->own_stream;
    PinScope pins(c, st);
    std::vector<qc_term> xt;
    if ((rc = c->expand_terms(terms, n_terms, xt, st))) return rc;
    Chain chain;
    if ((rc = c->stage_terms(xt.data(), n_terms, st, chain))) return rc;
    if ((rc = c->ensure(c->scalars, 64))) return rc;
    double *d_chi2 = (double *)c->scalars.ptr;
    const size_t n_vis = (size_t)c->n_row * c->n_chan;
    float4 *dres = nullptr;
    if (resid) {
        if (resid_memory == QC_MEM_DEVICE) dres = (float4 *)resid;
        else {
            if ((rc = c->ensure(c->resid_stage, nbytes<float4>(2 * n_vis)))) return rc;
            dres = (float4 *)c->resid_stage.ptr;
        }
    }
    if ((rc = c->run_residual(chain, dres, d_chi2, st))) return rc;
    if (++c->pin_calls >= c->PIN_CALLS) c->pin_reserve(64);
    CK(c->to_host(chi2, d_chi2, sizeof(double), st));
    if (resid && resid_memory != QC_MEM_DEVICE)
        CK(cudaMemcpyAsync(resid, dres, nbytes<float4>(2 * n_vis), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    c->pin_end();
    return QC_OK;
}

extern "C" int qc_delay_init(qc_ctx *c, qc_term *term, int32_t ref_ant, int32_t oversample)
{
    if (!c) return QC_EINVAL;
    c->err.clear();
    if (!term) return c->fail(QC_EINVAL, "term is NULL");
    if (term->type != QC_TERM_DELAY) return c->fail(QC_EINVAL, "qc_delay_init needs a QC_TERM_DELAY term");
    if (c->n_dir > 1) return c->fail(QC_EUNSUPPORTED, "qc_delay_init takes problems with one direction");
    int rc = c->validate_terms(term, 1, false);
    if (rc) return rc;
    if (ref_ant < 0 || ref_ant >= c->n_ant) return c->fail(QC_EINVAL, "ref_ant out of range");
    if (oversample < 0) return c->fail(QC_EINVAL, "oversample must be >= 0");
    if (oversample == 0) oversample = 4;
    const qc_term &t = *term;
    // per frequency interval: first channel, channels, transform length, spacing, first frequency
    std::vector<int4> info(t.n_fint, make_int4(0, 0, 1, 0));
    std::vector<double> dnu(t.n_fint, 0.0), nu0(t.n_fint, 0.0);
    int max_n = 1;
    for (int ch = 0; ch < c->n_chan; ++ch) {
        int4 &f = info[t.f_map[ch]];
        if (f.y == 0) f.x = ch;
        ++f.y;
    }
    for (int fi = 0; fi < t.n_fint; ++fi) {
        int4 &f = info[fi];
        if (f.y == 0) continue;
        nu0[fi] = t.chan_freq[f.x];
        if (f.y > 1) {
            const double d = (t.chan_freq[f.x + f.y - 1] - t.chan_freq[f.x]) / (f.y - 1);
            if (!(d != 0.0)) return c->fail(QC_EUNSUPPORTED, "an interval's channels have no frequency spread");
            for (int k = 0; k < f.y; ++k)
                if (std::fabs(t.chan_freq[f.x + k] - nu0[fi] - k * d) > 1e-6 * std::fabs(d))
                    return c->fail(QC_EUNSUPPORTED, "the delay estimate needs uniformly spaced channels");
            dnu[fi] = d;
        }
        long long N = 1;
        int lg = 0;
        while (N < (long long)oversample * f.y) { N *= 2; ++lg; }
        if (N > 16384) return c->fail(QC_EUNSUPPORTED, "transform longer than 16384 (reduce oversample)");
        f.z = (int)N;
        f.w = lg;
        max_n = std::max(max_n, (int)N);
    }
    cudaStream_t st = c->own_stream;
    // scratch of chain position 0: every qc_solve and qc_residual stages its buffers anew
    // (maps, accumulators, staging), and its graph is re-captured on every qc_solve
    TermBufs &B = c->tb[0];
    const size_t nx = (size_t)t.n_tint * c->n_ant * 2 * c->n_chan;
    const size_t npar = (size_t)t.n_tint * t.n_fint * c->n_ant * 4;
    if ((rc = c->ensure(B.maps, nbytes<int>(c->n_time + c->n_chan)))) return rc;
    if ((rc = c->ensure(B.acc, std::max(nbytes<float2>(nx), nbytes<float>(npar) + 64)))) return rc;
    if ((rc = c->ensure(B.stage, nbytes<float>(npar)))) return rc;
    if ((rc = c->ensure(B.dfr, nbytes<int4>(t.n_fint)))) return rc;
    if ((rc = c->ensure(B.dnu, nbytes<double>(2 * (size_t)t.n_fint)))) return rc;
    CK(cudaMemcpyAsync(B.maps.ptr, t.t_map, nbytes<int>(c->n_time), cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(B.dfr.ptr, info.data(), nbytes<int4>(t.n_fint), cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(B.dnu.ptr, dnu.data(), nbytes<double>(t.n_fint), cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync((double *)B.dnu.ptr + t.n_fint, nu0.data(), nbytes<double>(t.n_fint), cudaMemcpyHostToDevice, st));
    CK(cudaMemsetAsync(B.acc.ptr, 0, nbytes<float2>(nx), st));
    DelayInitArgs a;
    a.n_row = c->n_row;
    a.n_chan = c->n_chan;
    a.n_ant = c->n_ant;
    a.ref = ref_ant;
    a.n_tint = t.n_tint;
    a.n_fint = t.n_fint;
    a.rows = c->d_rows;
    a.vis = c->d_vis;
    a.model = c->m16 ? nullptr : c->d_model;
    a.model16 = c->d_model16;
    a.bl_scale = c->d_bl_scale;
    a.wf = c->d_wf;
    a.t_map = (const int *)B.maps.ptr;
    a.x = (float2 *)B.acc.ptr;
    a.fint_info = (const int4 *)B.dfr.ptr;
    a.fint_dnu = (const double *)B.dnu.ptr;
    a.fint_nu0 = (const double *)B.dnu.ptr + t.n_fint;
    float *dpar = t.memory == QC_MEM_DEVICE ? (float *)t.gains : (float *)B.stage.ptr;
    a.params = dpar;
    if (c->n_row) {
        delay_gather_kernel<<<grid_for((long)c->n_row * 32, 256, c->sm_count), 256, 0, st>>>(a);
        CK(cudaGetLastError());
    }
    const int smem = max_n * (int)sizeof(float2);
    if (smem > 48 * 1024) {
        if (smem > c->smem_optin) return c->fail(QC_EUNSUPPORTED, "transform does not fit in shared memory");
        CK(cudaFuncSetAttribute((const void *)delay_peak_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    }
    const long blocks = (long)t.n_tint * t.n_fint * c->n_ant * 2;
    if (blocks > 0) {
        delay_peak_kernel<<<(unsigned)blocks, 256, smem, st>>>(a);
        CK(cudaGetLastError());
    }
    if (t.memory == QC_MEM_HOST)
        CK(cudaMemcpyAsync(t.gains, dpar, nbytes<float>(npar), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    return QC_OK;
}

int qc_ctx::run_residual(const Chain &chain, float4 *dres, double *d_chi2, cudaStream_t st)
{
    qc_ctx *c = this;
    CK(cudaMemsetAsync(d_chi2, 0, sizeof(double), st));
    if (n_dir > 1) {
        DDArgs da;
        memset(&da, 0, sizeof da);
        da.D = data_desc();
        da.wf = d_wf;
        da.row_live = d_row_live;
        da.n_dir = n_dir;
        da.C = chain;
        da.C.n = -1;
        for (int j = 0; j < chain.n_terms; ++j) da.nd[j] = cur_nd[j];
        da.resid = dres;
        da.chi2 = d_chi2;
        CK(dd_launch_residual(da, grid_for((long)n_row * n_chan, 256, sm_count), st));
        ++launches;
        return QC_OK;
    }
    ResArgs ra;
    ra.D = data_desc();
    ra.C = chain;
    ra.resid = dres;
    ra.chi2 = d_chi2;
    CK(residual_launch(ra, m16, sm_count, st));
    ++launches;
    return QC_OK;
}

// ---------------------------------------------------------------------------
// solve
// ---------------------------------------------------------------------------

static int kind_of_range(const qc_term *terms, int lo, int hi)
{
    int k = KIND_NONE;
    for (int j = lo; j < hi; ++j) k = std::max(k, terms[j].type == 1 ? KIND_FULL : KIND_DIAG);
    return k;
}

int qc_ctx::pick_order(const qc_term &t, const qc_opts *o) const
{
    if (o && (o->order == 0 || o->order == 1)) return o->order;
    // mean interval extent along channels and along time (rows of one baseline)
    const double wf = (double)n_chan / t.n_fint;
    const double ht = (double)n_time / t.n_tint;
    return (wf >= 32.0 || wf >= ht) ? 0 : 1;
}

extern "C" int qc_solve(qc_ctx *c, qc_term *terms, int32_t n_terms, const qc_opts *o, qc_stats *stats)
{
    if (!c) return QC_EINVAL;
    c->err.clear();
    int rc = c->validate_terms(terms, n_terms, true);
    if (rc) return rc;
    qc_opts defaults;
    memset(&defaults, 0, sizeof defaults);
    defaults.n_epochs = 1;
    defaults.damping_mode = QC_DAMP_ALTERNATE;
    defaults.use_graph = 1;
    defaults.order = -1;
    if (!o) o = &defaults;
    if (o->n_epochs < 1) return c->fail(QC_EINVAL, "n_epochs must be >= 1");
    if (o->damping_mode != QC_DAMP_CONST && o->damping_mode != QC_DAMP_ALTERNATE)
        return c->fail(QC_EINVAL, "unknown damping_mode");
    for (int j = 0; j < n_terms; ++j)
        if (terms[j].solve && terms[j].reduce && !o->allreduce)
            return c->fail(QC_EINVAL, "a term with reduce = 1 needs opts.allreduce");
    cudaStream_t st = o->stream ? (cudaStream_t)o->stream : c->own_stream;
    c->launches = 0;
    qc_stats S;
    memset(&S, 0, sizeof S);

    cudaEvent_t ev0, ev1;
    if ((rc = c->get_event(0, ev0)) || (rc = c->get_event(1, ev1))) return rc;
    CK(cudaEventRecord(ev0, st));
    PinScope pins(c, st);
    std::vector<qc_term> xt;     // the kernels' view of the terms (delay terms per channel)
    if ((rc = c->expand_terms(terms, n_terms, xt, st))) return rc;
    Chain chain;
    if ((rc = c->stage_terms(xt.data(), n_terms, st, chain))) return rc;
    if ((rc = c->ensure(c->scalars, 64))) return rc;
    unsigned long long *d_counters = (unsigned long long *)c->scalars.ptr;   // [0] vis_iters, [1] bytes
    double *d_chi2 = (double *)c->scalars.ptr + 4;
    CK(cudaMemsetAsync(d_counters, 0, 2 * sizeof(unsigned long long), st));
    if (o->want_chi2) {
        if ((rc = c->run_residual(chain, nullptr, d_chi2, st))) return rc;
        CK(c->to_host(&S.chi2_before, d_chi2, sizeof(double), st));
    }

    // per solved term: its route, bin counts and byte weights
    c->pending.clear();
    const long long b_flag = c->has_flag ? 1 : 0;
    const long long b_unflag = 32 + (c->m16 ? 16 : 32 * c->n_dir) + 16;
    for (int j = 0; j < n_terms; ++j)
        if (terms[j].solve && (rc = c->plan_sums(xt.data(), n_terms, j, o))) return rc;
    if ((rc = c->plan_counters(xt.data(), n_terms, o->n_epochs))) return rc;
    for (int j = 0; j < n_terms; ++j) {
        if (!terms[j].solve) continue;
        const qc_term &t = xt[j];
        TermBufs &B = c->tb[j];
        const size_t nb = term_nbins(t);
        const size_t KG = t.type == 1 ? KG_FULL : KG_DIAG;
        const size_t nat = c->term_nat(t);
        const bool one_launch = B.sums.one_launch;
        if (!one_launch) {
            if ((rc = c->ensure(B.acc, nbytes<double>(nb * nat * KG)))) return rc;
            if ((rc = c->ensure(B.active, nb))) return rc;
            if ((rc = c->ensure(B.cnt, nbytes<int>(t.max_iter + 1)))) return rc;
        }
        if ((rc = c->ensure(B.nvis, nbytes<long long>(3 * nb)))) return rc;
        if ((rc = c->ensure(B.iters, nbytes<int>(nb)))) return rc;
        if ((rc = c->ensure(B.flags, nb * nat))) return rc;
        if (!one_launch) {       // the one-launch iterations write every interval's count and flags
            CK(cudaMemsetAsync(B.acc.ptr, 0, nbytes<double>(nb * nat * KG), st));
            CK(cudaMemsetAsync(B.iters.ptr, 0, nbytes<int>(nb), st));
            CK(cudaMemsetAsync(B.flags.ptr, 0, nb * nat, st));
        }
        // the counts of the previous call stand while the term's maps are the same (FNV-1a
        // over the kernels' view of them)
        uint64_t sig = 1469598103934665603ull;
        auto mix = [&](uint64_t v) { sig = (sig ^ v) * 1099511628211ull; };
        mix((uint64_t)t.type);
        mix((uint64_t)t.n_tint);
        mix((uint64_t)t.n_fint);
        mix((uint64_t)nat);
        for (int i = 0; i < c->n_time; ++i) mix((uint64_t)(uint32_t)t.t_map[i]);
        for (int i = 0; i < c->n_chan; ++i) mix((uint64_t)(uint32_t)t.f_map[i]);
        B.graph_valid = false;
        if (sig == B.count_sig && B.count_buf == B.nvis.ptr) continue;
        B.count_sig = 0;
        CK(cudaMemsetAsync(B.nvis.ptr, 0, nbytes<long long>(3 * nb), st));
        long long *nvis = (long long *)B.nvis.ptr;
        CountArgs ca;
        ca.D = c->data_desc();
        ca.t_map = chain.t[j].t_map;
        ca.f_map = chain.t[j].f_map;
        ca.n_fint = t.n_fint;
        ca.nvis = nvis;
        ca.nunflag = nvis + nb;
        if (c->n_row) {
            // about 64 warps an SM, up to 128 rows each (small data: one row a warp)
            const long cells = (long)c->n_row * ((c->n_chan + 31) / 32);
            ca.rb = (int)std::min(128L, std::max(1L, cells / (64L * c->sm_count)));
            const long units = ((c->n_row + ca.rb - 1) / ca.rb) * (long)((c->n_chan + 31) / 32);
            count_kernel<<<grid_for(units * 32, 256, c->sm_count), 256, 0, st>>>(ca);
            CK(cudaGetLastError());
            ++c->launches;
        }
        bin_bytes_kernel<<<((int)nb + 255) / 256, 256, 0, st>>>((int)nb, nvis, nvis + nb, b_flag, b_unflag, nvis + 2 * nb);
        CK(cudaGetLastError());
        ++c->launches;
        B.count_sig = sig;
        B.count_buf = B.nvis.ptr;
    }

    // robust reweighting between epochs: every kernel reads the context's folded weight copy,
    // reweighted in place; the weights before reweighting are kept and put back on return
    const bool robust = o->robust && o->n_epochs > 1;
    const double nu = o->robust_nu > 0 ? o->robust_nu : 5.0;
    const size_t n_vis = (size_t)c->n_row * c->n_chan;
    struct RobustGuard {
        qc_ctx *c = nullptr;
        cudaStream_t st = nullptr;
        size_t bytes = 0;
        ~RobustGuard()
        {
            if (!c) return;
            cudaMemcpyAsync(const_cast<float4 *>(c->d_wf), c->rob_w0.ptr, bytes, cudaMemcpyDeviceToDevice, st);
            c->d_weight_use = nullptr;
        }
    } guard;
    if (robust && n_vis) {
        if (!std::isfinite(nu)) return c->fail(QC_EINVAL, "robust_nu must be finite");
        if ((rc = c->ensure(c->rob_w0, nbytes<float4>(n_vis)))) return rc;
        if ((rc = c->ensure(c->rob_lam, nbytes<float>(n_vis)))) return rc;
        if ((rc = c->ensure(c->rob_res, nbytes<float4>(2 * n_vis)))) return rc;
        if ((rc = c->ensure(c->rob_sums, nbytes<double>(4)))) return rc;
        CK(cudaMemcpyAsync(c->rob_w0.ptr, c->d_wf, nbytes<float4>(n_vis), cudaMemcpyDeviceToDevice, st));
        robust_fill_kernel<<<grid_for((long)n_vis, 256, c->sm_count), 256, 0, st>>>((long)n_vis, (float *)c->rob_lam.ptr,
                                                                                     1.f);
        CK(cudaGetLastError());
        guard.c = c;
        guard.st = st;
        guard.bytes = nbytes<float4>(n_vis);
        c->d_weight_use = c->d_wf;
    }
    int n_iter_max = 0;
    for (int epoch = 0; epoch < o->n_epochs; ++epoch) {
        for (int n = 0; n < n_terms; ++n) {
            if (!terms[n].solve) continue;
            int it_max = 0;
            double acc_ms = 0, pass_ms = 0;
            long long acc_launches = 0;
            if (c->tb[n].sums.one_launch) {
                if ((rc = c->solve_term_sums(xt.data(), n_terms, n, chain, o, st, epoch == o->n_epochs - 1))) return rc;
                if ((int)c->pending.size() == qc_ctx::MAX_PENDING) {
                    if ((rc = c->copy_pending(st))) return rc;
                    CK(cudaStreamSynchronize(st));
                    c->pin_end();
                    c->pin_begin();
                    if ((rc = c->collect_sums(S, n_iter_max))) return rc;
                }
                continue;
            }
            if ((rc = c->solve_term(xt.data(), n_terms, n, chain, o, st, &it_max, &acc_ms, &acc_launches, &pass_ms)))
                return rc;
            S.acc_ms += acc_ms;
            S.pass_ms += pass_ms;
            S.acc_launches += acc_launches;
            if (epoch == o->n_epochs - 1) n_iter_max = std::max(n_iter_max, it_max);
        }
        if (guard.c && epoch < o->n_epochs - 1) {
            // one EM step on the residual of the current chain (whitened by the original weights)
            double *sums = (double *)c->rob_sums.ptr;
            if ((rc = c->run_residual(chain, (float4 *)c->rob_res.ptr, sums + 2, st))) return rc;
            CK(cudaMemsetAsync(sums, 0, 2 * sizeof(double), st));
            const int g = grid_for((long)n_vis, 256, c->sm_count);
            robust_sum_kernel<<<g, 256, 0, st>>>((long)n_vis, (const float4 *)c->rob_res.ptr,
                                                 (const float4 *)c->rob_w0.ptr, (const float *)c->rob_lam.ptr, sums);
            robust_apply_kernel<<<g, 256, 0, st>>>((long)n_vis, (const float4 *)c->rob_res.ptr,
                                                   (const float4 *)c->rob_w0.ptr, (float *)c->rob_lam.ptr,
                                                   const_cast<float4 *>(c->d_wf), sums, nu);
            CK(cudaGetLastError());
            c->launches += 3;
        }
    }
    if (guard.c) {
        // the caller's weights again for chi2_after and for later calls
        CK(cudaMemcpyAsync(const_cast<float4 *>(c->d_wf), c->rob_w0.ptr, nbytes<float4>(n_vis),
                           cudaMemcpyDeviceToDevice, st));
        c->d_weight_use = nullptr;
        guard.c = nullptr;
    }
    if (o->want_chi2) {
        if ((rc = c->run_residual(chain, nullptr, d_chi2, st))) return rc;
        CK(c->to_host(&S.chi2_after, d_chi2, sizeof(double), st));
    }
    // write back solved gains, flags, iteration counts
    size_t out_bytes = 64;
    for (const auto &P : c->pending) out_bytes += nbytes<int>(P.max_iter + 1) + 64;
    for (int j = 0; j < n_terms; ++j)
        if (terms[j].solve && terms[j].memory == QC_MEM_HOST) {
            const size_t nb = term_nbins(terms[j]);
            out_bytes += nb * c->term_nat(terms[j]) * 33 + nbytes<int>(nb) + 3 * 64;
        }
    c->pin_reserve(out_bytes);
    for (int j = 0; j < n_terms; ++j) {
        if (!terms[j].solve) continue;
        qc_term &t = terms[j];
        TermBufs &B = c->tb[j];
        const size_t nb = term_nbins(t), nent = nb * c->term_nat(t);
        const size_t gbytes = nent * (t.type == 2 ? 8 : (t.type == QC_TERM_DELAY ? 16 : 32));
        void *dst = t.memory == QC_MEM_DEVICE ? t.gains : B.stage.ptr;
        if (t.type == QC_TERM_DELAY)
            delay_params_out_kernel<<<grid_for((long)nent * 4, 256, c->sm_count), 256, 0, st>>>(
                (long)nent * 4, (const double *)B.params.ptr, (float *)dst);
        else
            gains_out_kernel<<<grid_for((long)nent, 256, c->sm_count), 256, 0, st>>>(t.type, (long)nent,
                                                                                   (const double *)B.params.ptr, dst);
        CK(cudaGetLastError());
        ++c->launches;
        if (t.memory == QC_MEM_HOST) {
            CK(c->to_host(t.gains, B.stage.ptr, gbytes, st));
            if (t.gain_flags) CK(c->to_host(t.gain_flags, B.flags.ptr, nent, st));
            if (t.iters) CK(c->to_host(t.iters, B.iters.ptr, nbytes<int>(nb), st));
        } else {
            if (t.gain_flags) CK(cudaMemcpyAsync(t.gain_flags, B.flags.ptr, nent, cudaMemcpyDeviceToDevice, st));
            if (t.iters) CK(cudaMemcpyAsync(t.iters, B.iters.ptr, nbytes<int>(nb), cudaMemcpyDeviceToDevice, st));
        }
    }
    unsigned long long hc[2];
    CK(c->to_host(hc, d_counters, sizeof hc, st));
    if ((rc = c->copy_pending(st))) return rc;
    CK(cudaEventRecord(ev1, st));
    CK(cudaStreamSynchronize(st));
    c->pin_end();
    if ((rc = c->collect_sums(S, n_iter_max))) return rc;
    float ms = 0;
    CK(cudaEventElapsedTime(&ms, ev0, ev1));
    S.ms = ms;
    S.vis_iters = (int64_t)hc[0];
    S.acc_bytes = (int64_t)hc[1];
    S.n_iter_max = n_iter_max;
    S.launches = c->launches;
    if (stats) *stats = S;
    return QC_OK;
}

bool qc_ctx::configured(const void *fn) const
{
    return std::find(configured_fns.begin(), configured_fns.end(), fn) != configured_fns.end();
}

int qc_ctx::get_event(int i, cudaEvent_t &ev)
{
    while ((int)events.size() <= i) {
        cudaEvent_t e;
        cudaError_t err_ = cudaEventCreate(&e);
        if (err_ != cudaSuccess) return cuda_fail(err_, "cudaEventCreate");
        events.push_back(e);
    }
    ev = events[i];
    return QC_OK;
}

// ---------------------------------------------------------------------------
// solving a term from per-(interval, antenna pair) sums
// ---------------------------------------------------------------------------

// Antennas up to which one CTA keeps an interval's gains and normal equations in shared memory
// (256 x (32 + 128 + 64) B = 56 KB) and walks all of its pairs itself.
static constexpr int SUMS_ONE_LAUNCH_ANT = 256;
// Antennas from which the full and left-full forms' slots are rounded to their heads: a slot's rounding
// averages out over the pairs.  Error of three chains and single terms against FP64 (rounding the result
// alone 2.4e-8): 20 antennas 3.6e-8 heads only, 3.2e-8 with tails, 3.6e-8 on the samples; 40 antennas 2.7,
// 2.5 and 2.5e-8; 64 antennas 2.6, 2.5 and 2.5e-8, where G and B with the FP16 model end at 3.0e-8 with and
// without tails and the tails' bytes take 13.0 instead of 10.3 ms.  The plain diagonal form's tails, 48 B a
// slot, cost 2% and are always kept.
static constexpr int SUMS_TAILS_ANT = 64;

// Whether all iterations of a term go in one launch, a CTA an interval, or in a launch an iteration, a warp
// an antenna and interval.  Time of an iteration (us, measured, nb intervals of 20 samples a pair):
//   one launch    a + c pairs ceil(nb / CTAs)     a = 5, 10, 8 and c = 0.0057, 0.0197, 0.0070 (plain diagonal, full,
//                                                 left-full form), two CTAs an SM
//   one each      f + m pairs nb                  f = 46, 78, 46 and m = 0.000065, 0.00021, 0.00009
// and the one launch has about 0.65 of m pairs nb to read as well; c with 8 warps a CTA (16, where every
// interval has an SM, take 0.85 of it).  20 iterations in ms, one launch and one each: 64 antennas, 1 interval: 0.34
// and 0.90, 0.99 and 1.58, 0.43 and 0.91; 128 antennas, 1 interval, 8 warps: 1.14 and 1.02, 3.56 and 1.90, 1.39 and
// 1.05; 152 intervals: 2.0 and 2.8, 6.7 and 7.4, 2.7 and 3.4; 256 antennas, 1 interval, 8 warps: 3.9 and 1.3, 13.2
// and 3.0, 4.8 and 1.3 (on the samples 2.0, 4.1 and 2.4); 152 intervals: 9.2 and 7.7, 27 and 24, 12.1 and 10.2.
bool qc_ctx::sums_one_launch(int form, size_t nb) const
{
    if (n_ant > SUMS_ONE_LAUNCH_ANT) return false;
    static const double a[3] = { 10, 8, 5 }, c[3] = { 0.0197, 0.0070, 0.0057 };        // FORM_FULL, FORM_E, FORM_D
    static const double f[3] = { 78, 46, 46 }, m[3] = { 0.00021, 0.00009, 0.000065 };
    const double pairs = n_up, ctas = 2.0 * sm_count;
    return a[form] + c[form] * pairs * std::ceil((double)nb / ctas) < f[form] + 0.35 * m[form] * pairs * (double)nb;
}

// The route of a solved term: from sums when the caller asks for it (qc_opts.moments), or by itself
// where that is the cheaper way to the same steps; sets B.sums and sizes its workspace.
//
// An iteration on the samples reads 80 B a sample (64 with the FP16 model) and is limited by
// instruction issue at about 0.64 of the HBM rate; the sums cost one pass, about 1.3 such
// iterations, and then 2 x 4 x words B per (interval, pair) and iteration, mostly out of L2.  The
// rule takes the sums when an iteration on them moves at most half the bytes of one on the
// samples, i.e. from 2.4 (plain diagonal form), 5.6 (E form) or 20 (full form) samples per slot
// on, and a term may take three iterations or more.  There and beyond the sums were never the slower
// ones (32 to 256 antennas, 1 to 320 intervals, 4 to 256 samples a slot; 20 iterations on 64 antennas and
// two intervals of 4 samples a pair: 0.41 against 0.98 ms).  It also bounds the heads to a quarter of
// the samples' bytes, the whole workspace to as many; it has to leave as much free memory (qc_dev_spare).  The options that name an accumulate kernel, its tiles or launch shape,
// divergence flagging and an allreduce (whose buffers are documented per iteration) keep the
// iterations on the samples.
int qc_ctx::plan_sums(const qc_term *terms, int n_terms, int n, const qc_opts *o)
{
    const qc_term &t = terms[n];
    TermBufs &B = tb[n];
    B.sums = SumsPlan();
    if (n_terms > 2 || delay[n] || n_dir > 1 || n_up == 0) return QC_OK;
    const size_t nb = term_nbins(t), slots = nb * (size_t)n_up;
    if (slots >= (size_t)INT32_MAX) return QC_OK;
    const int lk = kind_of_range(terms, 0, n), rk = kind_of_range(terms, n + 1, n_terms);
    int form, ok;
    if (t.type != QC_TERM_FULL && lk != KIND_FULL) { form = FORM_D; ok = lk != KIND_NONE ? lk : rk; }
    else if (t.type != QC_TERM_FULL) { form = FORM_E; ok = lk; }
    else if (lk == KIND_NONE) { form = FORM_FULL; ok = rk; }
    else return QC_OK;
    const bool asked = o->moments && d_model != nullptr;
    const bool one_launch = sums_one_launch(form, nb) && !t.reduce && !(o->div_flag && t.max_iter >= 4);
    if (!asked) {
        const bool plain = o->kernel == 0 && o->order == -1 && o->block_threads == 0 && o->ctas_per_sm == 0;
        if (!plain || n_ant > SUMS_ONE_LAUNCH_ANT || t.reduce || o->div_flag || t.max_iter < 3) return QC_OK;
        const double sample_bytes = (m16 ? 64.0 : 80.0) * (double)n_strip_rows * n_chan;
        if (2.0 * 4.0 * mom_words(form) * (double)slots > 0.5 * sample_bytes) return QC_OK;
    }
    // an interval several times long: the rows inside each chunk keep a lane's key (units of a strip
    // x one chunk); else a row's chunks inside each row (units of whole rows), so that an interval
    // one time long flushes once per row.  The rows are cut into blocks until there are about four
    // units per resident warp, down to 8 rows inside a chunk (a block's end is a flush)
    SumsPlan P;
    P.chunk_major = t.n_tint < n_time ? 1 : 0;
    const long max_strip = std::max(1, max_strip_rows), n_chunks = (n_chan + 31) / 32;
    const long strips = std::max(1L, (long)n_strips * (P.chunk_major ? n_chunks : 1));
    const long blocks = std::max(1L, (4L * sm_count * 12 + strips - 1) / strips);
    P.rb = (int)std::min(max_strip, std::max(P.chunk_major ? 8L : 1L, (max_strip + blocks - 1) / blocks));
    P.n_rb = (int)((max_strip + P.rb - 1) / P.rb);
    P.tails = form == FORM_D || n_ant < SUMS_TAILS_ANT;
    P.wide = !slots_once(t, form, P);
    const size_t words = slots * mom_words(form);
    P.cnt_off = nbytes<float>((P.tails ? 2 : 1) * words);
    P.mom64_off = P.cnt_off + ((nbytes<long long>(nb) + 15) / 16) * 16;
    const size_t bytes = P.mom64_off + (P.wide ? nbytes<double>(words) : 0);
    const bool grows = B.mom.bytes < bytes || mom_end.ptr == nullptr;
    if (!asked && grows && !qc_dev_spare(bytes - std::min(bytes, B.mom.bytes))) return QC_OK;
    int rc = ensure(B.mom, bytes);
    if (!rc) rc = size_mom_rows();
    if (rc) {
        if (asked || rc != QC_ENOMEM) return rc;
        cudaGetLastError();                    // no room for the sums: iterate on the samples
        err.clear();
        drop(B.mom);
        return QC_OK;
    }
    P.form = form;
    P.ok = ok;
    P.asked = asked;
    P.one_launch = one_launch;
    B.sums = P;
    return QC_OK;
}

// Whether the pass adds to each slot of a term at most once: then the additions are exact in FP32.  What
// follows is the order of mom_pass_kernel's steps and the rule by which it flushes.
bool qc_ctx::slots_once(const qc_term &t, int form, const SumsPlan &P) const
{
    if (!pair_time_once) return false;
    const int every = form == FORM_FULL ? mom_flush_every(m16) : INT32_MAX;
    std::vector<int> n_of(t.n_tint, 0);
    for (int i = 0; i < n_time; ++i) ++n_of[t.t_map[i]];
    const int deepest = n_time ? *std::max_element(n_of.begin(), n_of.end()) : 0;
    // a chunk's lanes in one interval, or each in its own: else the parts of an interval are added one by one
    for (int c0 = 0; c0 < n_chan; c0 += 32) {
        const int n = std::min(32, n_chan - c0), k = t.f_map[c0 + n - 1] - t.f_map[c0];
        if (k == 0) continue;
        for (int l = 1; l < n; ++l)
            if (t.f_map[c0 + l] == t.f_map[c0 + l - 1]) return false;
    }
    if (P.chunk_major) {
        // a strip's rows inside one chunk: the pair in one strip, the strip in one unit, the interval's times
        // in a row and no more of them than the lanes keep, the interval's channels in one chunk
        if (n_up != n_strips || P.n_rb != 1 || deepest > every) return false;
        for (int i = 1; i < n_time; ++i)
            if (t.t_map[i] < t.t_map[i - 1]) return false;
        for (int ch = 32; ch < n_chan; ch += 32)
            if (t.f_map[ch] == t.f_map[ch - 1]) return false;
        return true;
    }
    // a row's chunks: one row an interval, and no flush between an interval's chunks
    if (deepest > 1) return false;
    int run = 0;
    std::vector<int> cur(32, -1);
    for (int c0 = 0; c0 < n_chan; c0 += 32) {
        const int n = std::min(32, n_chan - c0);
        bool flush = c0 == 0;
        for (int l = 0; l < n; ++l) flush = flush || t.f_map[c0 + l] != cur[l];
        if (!flush && ++run < every) continue;
        if (c0 && t.f_map[c0] == t.f_map[c0 - 1]) return false;
        run = 0;
        for (int l = 0; l < 32; ++l) cur[l] = l < n ? t.f_map[c0 + l] : -1;
    }
    return true;
}

// Counters of the term solves pending together from the call's `first`-th one on: max_iter + 1 each.
size_t qc_ctx::sums_window(long long first) const
{
    size_t n = 0;
    const long long end = std::min(sums_total, first + MAX_PENDING);
    for (long long i = first; i < end; ++i) n += (size_t)sums_iters[i % sums_iters.size()] + 1;
    return n;
}

// Room for the counters of the call's one-launch term solves (`terms` in the order of an epoch), before
// the first of them: the buffer stays where it is while solves are pending.  A term that took the
// sums by itself goes back to the samples where there is no room.
int qc_ctx::plan_counters(const qc_term *terms, int n_terms, int n_epochs)
{
    sums_done = 0;
    for (;;) {
        sums_iters.clear();
        for (int j = 0; j < n_terms; ++j)
            if (terms[j].solve && tb[j].sums.one_launch) sums_iters.push_back(terms[j].max_iter);
        sums_total = (long long)n_epochs * (long long)sums_iters.size();
        size_t most = 0;
        for (size_t i = 0; i < sums_iters.size(); ++i) most = std::max(most, sums_window((long long)i));
        if (most == 0) return QC_OK;
        const int rc = ensure(sums_cnt, nbytes<int>(most));
        if (rc != QC_ENOMEM) return rc;
        bool left = false;
        for (int j = 0; j < n_terms; ++j)
            if (terms[j].solve && tb[j].sums.one_launch && !tb[j].sums.asked) {
                tb[j].sums = SumsPlan();
                drop(tb[j].mom);
                left = true;
            }
        if (!left) return rc;
        cudaGetLastError();
        err.clear();
    }
}

int qc_ctx::size_mom_rows()
{
    const size_t bytes = nbytes<int4>(std::max(1L, n_strip_rows)) + (m16 ? nbytes<float>(std::max(1L, n_strip_rows)) : 0);
    int rc = ensure(mom_rows, bytes);
    if (!rc) rc = ensure(mom_live, bytes);
    if (!rc) rc = ensure(mom_end, nbytes<int>(std::max(1, n_strips)));
    return rc;
}

// The context's table of strip rows as the passes read them, built the first time (a function of the
// rows and flags staged at create).
int qc_ctx::ensure_mom_rows(cudaStream_t st)
{
    qc_ctx *c = this;
    if (mom_rows_ready) return QC_OK;
    const size_t scale_off = nbytes<int4>(std::max(1L, n_strip_rows));
    const int rc = size_mom_rows();
    if (rc) return rc;
    auto scales = [&](const Buf &b) { return m16 ? (float *)((char *)b.ptr + scale_off) : nullptr; };
    CK(mom_launch_rows(n_strip_rows, d_strip_rows, d_rows, d_row_live, d_up_of_bl, d_bl_scale, (int4 *)mom_rows.ptr,
                       scales(mom_rows), n_strips, d_strip_off, (int4 *)mom_live.ptr, scales(mom_live), (int *)mom_end.ptr,
                       st));
    // built on this call's stream: finished before any later call can use it on another one
    CK(cudaStreamSynchronize(st));
    mom_rows_ready = true;
    ++launches;
    return QC_OK;
}

// A solved delay term from the products T and H of qc_delay_sums.cu (chains of one or two terms, the
// other one to the right or diagonal).  The rule: an iteration on T reads 1 KB per (time interval,
// pair, 32 channels), one on the samples 80 B (64 B with the FP16 model) a sample; T is taken when it is at most 0.6 of that, which leaves the pass that forms
// it paid for after two iterations (measured on 64 antennas, 75 x 512: pass 1.9 iterations on the
// samples, an iteration on T 0.3).  That also bounds T to 0.6 of the samples' bytes; where a slot takes
// several additions, its FP64 sums take twice T beside it.  Few intervals of many antennas leave most SMs
// without a CTA: time of an iteration in us, measured, 30 + 0.023 to 0.037 per pair and wave of CTAs on
// products, 82 + 0.024 per 1000 samples on the samples (20 iterations, products and samples: 64 antennas, 1 x
// 512: 2.1 and 2.1 ms; 75 x 512: 10.0 and 25; 128 antennas, 1 x 64: 4.7 and 2.0; 1 x 512: 6.5 and 3.5; 3 x
// 512: 6.8 and 7.3; 200 antennas, 2 x 512: 14.4 and 10.2; 3 x 512: 14.8 and 16.0).
// Times of an interval of a delay term on a full grid whose intervals are all of one length (the last
// one may be shorter) up to what a lane adds up in FP32: its blocks of rows then end where intervals do.
// Else 0.
int qc_ctx::products_depth(const qc_term &t) const
{
    int d = 1;
    while (d < n_time && t.t_map[d] == t.t_map[0]) ++d;
    bool even = full_grid && n_time > 0 && d <= 32 && t.n_tint == (n_time + d - 1) / d;
    for (int i = 0; i < n_time && even; ++i) even = t.t_map[i] == i / d;
    return even ? d : 0;
}

// Whether every product of a delay term takes one addition: such a grid, or a time an interval and a row
// a pair and time.
bool qc_ctx::products_once(const qc_term &t) const
{
    if (products_depth(t)) return true;
    std::vector<char> seen(t.n_tint, 0);
    for (int i = 0; i < n_time; ++i)
        if (seen[t.t_map[i]]++) return false;
    return pair_time_once;
}

int qc_ctx::plan_delay_sums(const qc_term *terms, int n_terms, int n, const qc_opts *o, bool &use)
{
    use = false;
    const qc_term &t = terms[n];
    TermBufs &B = tb[n];
    if (!delay[n] || n_terms > 2 || n_dir > 1 || n_up == 0 || n_ant > DSUM_MAX_ANT || t.reduce || t.max_iter < 3)
        return QC_OK;
    if (o->kernel != 0 || o->order != -1 || o->block_threads != 0 || o->ctas_per_sm != 0) return QC_OK;
    if (n == 1 && kind_of_range(terms, 0, 1) == KIND_FULL) return QC_OK;
    const size_t n_chunks = (n_chan + 31) / 32;
    const size_t iter_bytes = (size_t)t.n_tint * n_chunks * n_up * 1024;
    // the products, and the FP64 ones where a slot takes several additions
    const size_t t_bytes = iter_bytes * (products_once(t) ? 1 : 3);
    const double sample = m16 ? 64.0 : 80.0;
    const double samples = (double)n_strip_rows * n_chan;
    if ((double)iter_bytes > 0.6 * sample * samples) return QC_OK;
    // an iteration on T is a CTA per (time interval, chunk), which walks all pairs
    const double waves = std::ceil((double)t.n_tint * (double)n_chunks / (2.0 * sm_count));
    if (30 + 0.04 * n_up * waves > 82 + 3e-7 * sample * samples) return QC_OK;
    if (B.dsum_t.bytes < t_bytes && !qc_dev_spare(t_bytes - B.dsum_t.bytes)) return QC_OK;
    int rc = ensure(B.dsum_t, t_bytes);
    if (!rc) rc = ensure(B.dsum_h, nbytes<double>((size_t)t.n_tint * B.hfr.size() * n_ant * KG_HSUM));
    if (!rc) rc = size_mom_rows();
    if (rc == QC_ENOMEM) {
        cudaGetLastError();                    // no room for the products: iterate on the samples
        err.clear();
        drop(B.dsum_t);
        drop(B.dsum_h);
        return QC_OK;
    }
    use = rc == QC_OK;
    return rc;
}

DelaySumsArgs qc_ctx::delay_sums_args(const qc_term *terms, int n_terms, int n, const Chain &chain)
{
    const qc_term &t = terms[n];
    TermBufs &B = tb[n];
    DelaySumsArgs a;
    memset(&a, 0, sizeof a);
    a.n_chan = n_chan;
    a.n_ant = n_ant;
    a.n_up = n_up;
    a.n_fint = (int)B.hfr.size();
    a.n_chunks = (n_chan + 31) / 32;
    a.vis = d_vis;
    a.model = d_model;
    a.wf = d_wf;
    a.model16 = m16 ? d_model16 : nullptr;
    a.mrows = (const int4 *)mom_rows.ptr;
    a.mscale = m16 ? (const float *)((const char *)mom_rows.ptr + nbytes<int4>(std::max(1L, n_strip_rows))) : nullptr;
    a.strip_off = d_strip_off;
    a.n_strips = n_strips;
    // an interval several times long keeps its slot while the rows run inside a chunk; the blocks of
    // rows give about four units per resident warp, down to 8 rows inside a chunk
    a.chunk_major = t.n_tint < n_time ? 1 : 0;
    const long max_strip = std::max(1, max_strip_rows), want = 4L * sm_count * 16;
    const long strips = std::max(1L, (long)n_strips * (a.chunk_major ? a.n_chunks : 1));
    const long blocks = std::max(1L, (want + strips - 1) / strips);
    a.rb = (int)std::min(max_strip, std::max(a.chunk_major ? 8L : 1L, (max_strip + blocks - 1) / blocks));
    // a block ends where an interval does: every slot is written once
    const int depth = products_depth(t);
    if (depth) a.rb = (a.rb + depth - 1) / depth * depth;
    a.n_rb = (int)((max_strip + a.rb - 1) / a.rb);
    a.t_map = chain.t[n].t_map;
    a.to = n_terms == 2 ? chain.t[1 - n] : chain.t[n];
    a.store = depth > 0;
    a.active = (const uint8_t *)B.active.ptr;
    a.fmap = (const int *)B.dfmap.ptr;
    a.omega = (const float *)B.domega.ptr;
    a.T = (float4 *)B.dsum_t.ptr;
    a.T64 = products_once(t) ? nullptr : (double *)((char *)B.dsum_t.ptr + (size_t)t.n_tint * a.n_chunks * n_up * 1024);
    a.hsum = (double *)B.dsum_h.ptr;
    a.n_tint = t.n_tint;
    a.upair = d_upair;
    a.nu = (const double *)B.dnu.ptr;
    a.params = (const double *)B.params.ptr;
    a.acc = (double *)B.acc.ptr;
    return a;
}

// Arguments of the pass and of the normal equations of a term solved from sums.
int qc_ctx::sums_args(const qc_term *terms, int n_terms, int n, const Chain &chain, cudaStream_t st, MomArgs &ma,
                      MomNormArgs &mn)
{
    qc_ctx *c = this;
    const qc_term &t = terms[n];
    TermBufs &B = tb[n];
    memset(&ma, 0, sizeof ma);
    memset(&mn, 0, sizeof mn);
    const int rc = ensure_mom_rows(st);
    if (rc) return rc;
    const size_t scale_off = nbytes<int4>(std::max(1L, n_strip_rows));
    ma.n_chan = n_chan;
    ma.n_ant = n_ant;
    ma.n_up = n_up;
    ma.vis = d_vis;
    ma.model = d_model;
    ma.model16 = d_model16;
    ma.wf = d_wf;
    ma.mrows = (const int4 *)mom_live.ptr;
    ma.mscale = m16 ? (const float *)((const char *)mom_live.ptr + scale_off) : nullptr;
    ma.strip_off = d_strip_off;
    ma.strip_end = (const int *)mom_end.ptr;
    auto map_kind = [&](const qc_term &x) {
        if (x.n_fint == 1) return (int)MAP_ONE;
        bool id = true, chunk = true;
        for (int ch = 0; ch < n_chan; ++ch) {
            id = id && x.f_map[ch] == ch;
            chunk = chunk && x.f_map[ch] == x.f_map[ch / 32 * 32];
        }
        return (int)(id ? MAP_IDENTITY : (chunk ? MAP_CHUNK : MAP_ANY));
    };
    ma.tn_map = map_kind(t);
    ma.to_map = n_terms == 2 ? map_kind(terms[1 - n]) : (int)MAP_ONE;
    ma.n_strips = n_strips;
    ma.n_time = n_time;
    ma.n_chunks = (n_chan + 31) / 32;
    ma.chunk_major = B.sums.chunk_major;
    ma.group = ma.chunk_major ? 1 : ma.n_chunks;
    ma.rb = B.sums.rb;
    ma.n_rb = B.sums.n_rb;
    ma.tn = chain.t[n];
    ma.to = n_terms == 2 ? chain.t[1 - n] : chain.t[n];
    ma.mom = (float *)B.mom.ptr;
    ma.tail = B.sums.tails ? ma.mom + term_nbins(t) * n_up * mom_words(B.sums.form) : nullptr;
    ma.mom64 = B.sums.wide ? (double *)((char *)B.mom.ptr + B.sums.mom64_off) : nullptr;
    mn.n_bins = (int)term_nbins(t);
    mn.n_ant = n_ant;
    mn.n_up = n_up;
    mn.type = t.type;
    mn.form = B.sums.form;
    mn.upair = d_upair;
    mn.mom = ma.mom;
    mn.tail = ma.tail;
    mn.params = (const double *)B.params.ptr;
    mn.tab = (const float4 *)B.tab.ptr;
    mn.n_fint = t.n_fint;
    return QC_OK;
}

// One term solve from sums with its iterations in one launch; its statistics are collected when the
// stream is next synchronised (collect_sums).
int qc_ctx::solve_term_sums(const qc_term *terms, int n_terms, int n, const Chain &chain, const qc_opts *o,
                            cudaStream_t st, bool last_epoch)
{
    qc_ctx *c = this;
    const qc_term &t = terms[n];
    TermBufs &B = tb[n];
    MomArgs ma;
    MomIterArgs mi;
    memset(&mi, 0, sizeof mi);
    int rc;
    if ((rc = sums_args(terms, n_terms, n, chain, st, ma, mi.n))) return rc;
    Pending P;
    P.max_iter = t.max_iter;
    P.n_bins = mi.n.n_bins;
    P.last_epoch = last_epoch;
    P.asked = B.sums.asked;
    P.off = pending.empty() ? 0 : pending.back().off + pending.back().max_iter + 1;
    P.ev = 3 * (int)pending.size();
    while ((int)sums_events.size() < P.ev + 3) {
        cudaEvent_t e;
        CK(cudaEventCreate(&e));
        sums_events.push_back(e);
    }
    const cudaEvent_t *ev = sums_events.data() + P.ev;
    // a counter region per pending term solve, all of those up to the next collection cleared together
    int *cnt = (int *)sums_cnt.ptr + P.off;
    if (pending.empty()) CK(cudaMemsetAsync(cnt, 0, nbytes<int>(sums_window(sums_done)), st));
    ++sums_done;
    const size_t words = (size_t)P.n_bins * n_up * mom_words(B.sums.form);
    if (ma.mom64) CK(cudaMemsetAsync(ma.mom64, 0, nbytes<double>(words), st));
    else CK(cudaMemsetAsync(ma.mom, 0, nbytes<float>((ma.tail ? 2 : 1) * words), st));
    CK(cudaEventRecord(ev[0], st));
    CK(mom_launch_pass(ma, B.sums.form, B.sums.ok, sm_count, st));
    if (ma.mom64) CK(mom_launch_split(words, ma.mom64, ma.mom, ma.tail, sm_count, st));
    CK(cudaEventRecord(ev[1], st));
    mi.params = (double *)B.params.ptr;
    mi.tab = (float4 *)B.tab.ptr;
    mi.gain_flags = (int8_t *)B.flags.ptr;
    mi.iters = (int *)B.iters.ptr;
    mi.cnt = cnt;
    mi.bin_nvis = (const long long *)B.nvis.ptr;
    mi.bin_nbytes = (const long long *)B.nvis.ptr + 2 * (size_t)P.n_bins;
    mi.iter_bytes = 2LL * n_up * mom_words(B.sums.form) * 4 + 8LL * term_nat(t) * (t.type == 1 ? KG_FULL : KG_DIAG);
    mi.vis_iters = (unsigned long long *)scalars.ptr;
    mi.acc_bytes = (unsigned long long *)scalars.ptr + 1;
    mi.max_iter = t.max_iter;
    mi.alternate = o->damping_mode == QC_DAMP_ALTERNATE;
    mi.damping = o->damping > 0 ? o->damping : 1.0;
    mi.tol = t.tol;
    CK(mom_launch_iterate(mi, sm_count, st));
    CK(cudaEventRecord(ev[2], st));
    launches += ma.mom64 ? 3 : 2;
    pending.push_back(P);
    return QC_OK;
}

// Host copies of the pending term solves' counters, ordered on the stream.
int qc_ctx::copy_pending(cudaStream_t st)
{
    qc_ctx *c = this;
    if (pending.empty()) return QC_OK;
    const size_t n = (size_t)pending.back().off + pending.back().max_iter + 1;
    pending_cnt.resize(n);
    CK(to_host(pending_cnt.data(), sums_cnt.ptr, nbytes<int>(n), st));
    return QC_OK;
}

// After a synchronisation that followed copy_pending: iteration counts and device times.
int qc_ctx::collect_sums(qc_stats &S, int &n_iter_max)
{
    qc_ctx *c = this;
    for (const Pending &P : pending) {
        int its = P.n_bins > 0 ? 1 : 0;
        while (its > 0 && its < P.max_iter && pending_cnt[P.off + its] > 0) ++its;
        float ms = 0, pass = 0;
        CK(cudaEventElapsedTime(&ms, sums_events[P.ev], sums_events[P.ev + 2]));
        CK(cudaEventElapsedTime(&pass, sums_events[P.ev], sums_events[P.ev + 1]));
        S.acc_ms += ms;
        if (P.asked) S.pass_ms += pass;
        S.acc_launches += its;
        if (P.last_epoch) n_iter_max = std::max(n_iter_max, its);
    }
    pending.clear();
    return QC_OK;
}

int qc_ctx::solve_term(const qc_term *terms, int n_terms, int n, Chain chain, const qc_opts *o, cudaStream_t st,
                       int *it_max, double *acc_ms, long long *acc_launches, double *pass_ms)
{
    *pass_ms = 0;
    qc_ctx *c = this;
    const qc_term &t = terms[n];
    TermBufs &B = tb[n];
    const int nb = (int)term_nbins(t);
    chain.n = n;
    const int ts = t.type == 1 ? TS_FULL : TS_DIAG;
    const int lk = kind_of_range(terms, 0, n);
    const int rk = kind_of_range(terms, n + 1, n_terms);
    // chains with directions: chains of one or two terms with at most DDS_MAX_DIR directions
    // take the streaming direction-dependent kernel (row tiles, qc_dd_stream.cuh), longer
    // chains the general one (qc_dd.cu)
    const bool ddp = n_dir > 1;
    DDSLaunch DS;
    if (ddp && n_terms <= 2 && n_dir <= DDS_MAX_DIR && (o->kernel == 0 || o->kernel == 3) &&
        (long long)n_ant * n_dir < 32768) {
        const int ok_ = n_terms == 2 ? (terms[1 - n].type == 1 ? KIND_FULL : KIND_DIAG) : KIND_NONE;
        DS = dds_launcher(t.type == 1 ? KIND_FULL : KIND_DIAG, ok_, n == 1, delay[n], cur_nd[n] > 1);
    }
    const bool dds = DS.fn != nullptr;
    const int order = dds ? 0 : pick_order(t, o);
    // the prefetching and streaming kernels are compiled for at most 256 threads per CTA
    // (the streaming kernel for two such CTAs per SM)
    const bool bt_ok = o->block_threads >= 32 && o->block_threads % 32 == 0;
    int block = (bt_ok && o->block_threads <= 256) ? o->block_threads : 256;
    const int block_stream = block;
    AccArgs aa;
    aa.D = data_desc();
    aa.C = chain;
    aa.tn = chain.t[n];
    aa.row_live = d_row_live;
    aa.to = n_terms == 2 ? chain.t[1 - n] : chain.t[n];
    aa.acc = (double *)B.acc.ptr;
    aa.active = (const uint8_t *)B.active.ptr;
    aa.order = order;
    aa.n_chunks = (n_chan + 31) / 32;
    const long units = order == 0 ? (long)n_row : (long)n_strips * aa.n_chunks;
    int per_sm = o->ctas_per_sm > 0 ? o->ctas_per_sm : 0;
    const bool simple = n_terms <= 2;
    AccLaunch L = acc_launcher(ts, simple, lk, rk, m16);
    const int nat = term_nat(t);
    if (!L.fn && !ddp) return fail(QC_EUNSUPPORTED, "no accumulate kernel for this chain");
    // the term from per-(interval, pair) sums (qc_moments.cu), iteration by iteration (plan_sums)
    const bool mom = B.sums.form >= 0;
    // pipelined kernel: shared-memory layout of the per-warp rings for this chain
    PipeArgs pa;
    memset(&pa, 0, sizeof pa);
    int pipe_smem = 0;
    // auto and kernel 3: the streaming kernel (chains of one or two terms; antenna pairs are
    // packed as p | q << 16); kernels 1 and 2 on request, and for longer chains
    // kernel 4: the warp-specialised kernel (chains of one or two terms; a solved delay term
    // keeps its own streaming kernel)
    // kernel 5: the self-feeding variant (every warp issues its own bulk copies)
    bool ws = !mom && !ddp && L.ws_fn != nullptr && !delay[n] && n_ant < 32768 && (o->kernel == 4 || o->kernel == 5);
    const bool self_feed = o->kernel == 5;
    const void *ws_fn = self_feed ? (order == 0 ? L.wss_fn : L.wss_fn1) : L.ws_fn;
    const int ws_warps = self_feed ? L.wss_nw : L.ws_nc;     // warps that own a ring
    const bool streaming = !mom && !ddp && L.stream_fn != nullptr && n_ant < 32768 &&
                           (o->kernel == 3 || o->kernel == 0 || ((o->kernel == 4 || o->kernel == 5) && delay[n]));
    // a solved delay term under the streaming kernel: its own kernel, which applies the chain
    // rule per sample and keeps sums per parameter interval (else: the per-channel bins)
    DelayLaunch DL;
    if (delay[n] && streaming) DL = delay_launcher(lk, rk, m16);
    const bool ded = DL.fn != nullptr;
    // a solved delay term with sums per parameter interval (the streaming kernels), else
    // the per-channel bins
    // or, where that is cheaper, products of every (time interval, pair, channel) formed once
    bool dsum = false;
    {
        int rc_;
        if ((rc_ = plan_delay_sums(terms, n_terms, n, o, dsum))) return rc_;
        if (dsum && (rc_ = ensure_mom_rows(st))) return rc_;
    }
    const bool psums = dsum || ded || (dds && delay[n]);
    DevTerm tnu = chain.t[n];
    const int nbu = delay[n] ? t.n_tint * (int)B.hfr.size() : nb;
    if (psums) {
        tnu.n_fint = (int)B.hfr.size();
        tnu.f_map = (const int *)B.dfmap.ptr;
        aa.tn = tnu;
        int rc_;
        if ((rc_ = ensure(B.acc, nbytes<double>((size_t)nbu * n_ant * KG_SUMS)))) return rc_;
        CK(cudaMemsetAsync(B.acc.ptr, 0, nbytes<double>((size_t)nbu * n_ant * KG_SUMS), st));
        aa.acc = (double *)B.acc.ptr;
    }
    const void *stream_fn = dds ? DS.fn : (ded ? DL.fn : L.stream_fn);
    const int stream_smem_per_warp = dds ? dds_smem_per_warp(n_dir) : (ded ? DL.smem_per_warp : L.stream_smem_per_warp);
    bool pipelined = !mom && !ddp && !streaming && L.pipe_fn != nullptr && (o->kernel == 1 || (o->kernel == 0 && order == 1));
    const bool has_o = n_terms == 2;
    if (pipelined) {
        const int NW = L.pipe_nw;
        const int n_chunks = (n_chan + 31) / 32;
        std::vector<int4> ci(n_chunks);
        int capn = 1, capo = has_o ? 1 : 0;
        for (int ch = 0; ch < n_chunks; ++ch) {
            const int c0 = ch * 32, c1 = std::min(n_chan, c0 + 32) - 1;
            ci[ch].x = t.f_map[c0];
            ci[ch].y = t.f_map[c1] - t.f_map[c0] + 1;
            ci[ch].z = has_o ? terms[1 - n].f_map[c0] : 0;
            ci[ch].w = has_o ? terms[1 - n].f_map[c1] - terms[1 - n].f_map[c0] + 1 : 0;
            capn = std::max(capn, ci[ch].y);
            capo = std::max(capo, ci[ch].w);
        }
        const int esn = t.type == 1 ? 32 : 16;
        const int eso = has_o ? (terms[1 - n].type == 1 ? 32 : 16) : 16;
        pa.jn_cap = capn;
        pa.jo_cap = capo;
        const int mb = m16 ? 16 : 32;
        pa.off_m = 32 * 32;
        pa.off_w = pa.off_m + 32 * mb;
        pa.off_jn = pa.off_w + 32 * 16;
        pa.off_jo = pa.off_jn + 2 * pa.jn_cap * esn;
        pa.slot_bytes = pa.off_jo + 2 * pa.jo_cap * eso;
        pa.stage_fmap = n_chan <= 8192 ? 1 : 0;
        const int fmap_bytes = pa.stage_fmap ? ((2 * n_chan * 4 + 15) / 16) * 16 : 0;
        const int H = L.pipe_h;
        const int per_stage = H * (pa.slot_bytes + (int)sizeof(SlotDesc)) + 8;
        const int warp_budget = (smem_optin - fmap_bytes - 128) / NW;
        const int ns = std::min(8, warp_budget / per_stage);
        if (ns < 2) pipelined = false;
        else {
            pa.ns = ns;
            pa.desc_off = ns * H * pa.slot_bytes;
            pa.bar_off = pa.desc_off + ns * H * (int)sizeof(SlotDesc);
            pa.warp_bytes = ((pa.bar_off + ns * 8 + 15) / 16) * 16;
            pa.fmap_off = NW * pa.warp_bytes;
            pipe_smem = pa.fmap_off + fmap_bytes;
            if (!configured(L.pipe_fn)) {
                CK(cudaFuncSetAttribute(L.pipe_fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin));
                configured_fns.push_back(L.pipe_fn);
            }
        }
    }
    int ws_cap = 1;            // warp-specialised kernel: other-term entries per 32-channel chunk (max)
    {
        // static per-row and per-chunk information of this term solve (both kernels)
        const int n_chunks = (n_chan + 31) / 32;
        std::vector<int4> ci(n_chunks);
        for (int ch = 0; ch < n_chunks; ++ch) {
            const int c0 = ch * 32, c1 = std::min(n_chan, c0 + 32) - 1;
            ci[ch].x = t.f_map[c0];
            ci[ch].y = t.f_map[c1] - t.f_map[c0] + 1;
            ci[ch].z = has_o ? terms[1 - n].f_map[c0] : 0;
            ci[ch].w = has_o ? terms[1 - n].f_map[c1] - terms[1 - n].f_map[c0] + 1 : 0;
            ws_cap = std::max(ws_cap, ci[ch].w);
        }
        int rc_;
        if ((rc_ = ensure(B.row_info, nbytes<int4>(std::max(1, n_row))))) return rc_;
        if ((rc_ = ensure(B.chunk_info, nbytes<int4>(n_chunks)))) return rc_;
        CK(cudaMemcpyAsync(B.chunk_info.ptr, ci.data(), nbytes<int4>(n_chunks), cudaMemcpyHostToDevice, st));
        if (n_row) {
            row_info_kernel<<<(n_row + 255) / 256, 256, 0, st>>>(data_desc(), d_row_live, chain.t[n],
                                                                has_o ? chain.t[1 - n] : chain.t[n], has_o ? 1 : 0,
                                                                (int4 *)B.row_info.ptr);
            CK(cudaGetLastError());
            ++launches;
        }
        pa.row_info = (const int4 *)B.row_info.ptr;
        pa.chunk_info = (const int4 *)B.chunk_info.ptr;
        aa.row_info = pa.row_info;
    }
    // warp-specialised kernel: shared-memory layout of one consumer's ring stage (d, m, folded
    // weights, the 32 channel maps, the other term's entries for p and q, a 32-byte header)
    // and the ring depth that two CTAs per SM leave room for
    WsArgs wa;
    memset(&wa, 0, sizeof wa);
    int ws_smem = 0, ws_grid = 0;
    if (ws) {
        const int ok_ = lk != KIND_NONE ? lk : rk;
        const int eso = ok_ == KIND_FULL ? 32 : 16;
        const int jo = has_o ? ((ws_cap * eso + 15) / 16) * 16 : 0;
        wa.off_m = 1024;
        wa.off_w = wa.off_m + 32 * (m16 ? 16 : 32);
        wa.off_fm = wa.off_w + 512;
        wa.off_jp = wa.off_fm + 256;
        wa.off_jq = wa.off_jp + jo;
        wa.off_h = wa.off_jq + jo;
        wa.stage_bytes = ((wa.off_h + 32 + 127) / 128) * 128;
        const int NC = ws_warps;
        const int nbar = self_feed ? 1 : 2;        // barriers per stage: full (and empty)
        const int budget = std::min(smem_optin, smem_per_sm / 2 - 1024) - 2560;
        wa.depth = std::min(6, budget / (NC * (wa.stage_bytes + 8 * nbar)));
        if (wa.depth < 2) ws = false;
        else ws_smem = NC * wa.depth * wa.stage_bytes + nbar * NC * wa.depth * 8;
    }
    StreamArgs sa;
    memset(&sa, 0, sizeof sa);
    int stream_smem = 0;
    const long n_rt = order == 0 ? (long)n_row : n_strip_rows;
    if (streaming || ws || dds) {
        // step-major row table in the tile order, and the channel maps of both terms (padded
        // to whole 32-channel chunks: the warp-specialised kernel copies them 32 at a time)
        const int n_chunks = (n_chan + 31) / 32;
        int rc_;
        if ((rc_ = ensure(B.rt, nbytes<int4>(std::max(1L, n_rt))))) return rc_;
        if (m16 && (rc_ = ensure(B.rt_scale, nbytes<float>(std::max(1L, n_rt))))) return rc_;
        if ((rc_ = ensure(B.fmap2, nbytes<int2>(32 * n_chunks)))) return rc_;
        std::vector<int2> fm(32 * n_chunks, make_int2(0, 0));
        for (int ch = 0; ch < n_chan; ++ch)
            fm[ch] = make_int2(psums ? B.hufmap[ch] : t.f_map[ch], has_o ? terms[1 - n].f_map[ch] : 0);
        CK(cudaMemcpyAsync(B.fmap2.ptr, fm.data(), nbytes<int2>(32 * n_chunks), cudaMemcpyHostToDevice, st));
        if (n_rt) {
            row_table_kernel<<<(int)((n_rt + 255) / 256), 256, 0, st>>>(
                (int)n_rt, order == 0 ? nullptr : d_strip_rows, (const int4 *)B.row_info.ptr, d_rows,
                m16 ? d_bl_scale : nullptr, (int4 *)B.rt.ptr, m16 ? (float *)B.rt_scale.ptr : nullptr);
            CK(cudaGetLastError());
            ++launches;
        }
    }
    if (ws) {
        const int n_chunks = (n_chan + 31) / 32;
        int rc_;
        wa.vis = d_vis;
        wa.model = d_model;
        wa.model16 = d_model16;
        wa.wf = d_wf;
        wa.n_chan = n_chan;
        wa.n_ant = n_ant;
        wa.order = order;
        wa.n_chunks = n_chunks;
        wa.nwr = (n_chunks + 31) / 32;
        wa.nwk = (int)((n_strip_rows + 31) / 32);
        if (order == 0) {
            if ((rc_ = ensure(B.ws_rl, nbytes<int4>(std::max(1, n_row))))) return rc_;
            if (m16 && (rc_ = ensure(B.ws_rls, nbytes<float>(std::max(1, n_row))))) return rc_;
            if ((rc_ = ensure(B.ws_rlb, nbytes<unsigned>((size_t)std::max(1, n_row) * wa.nwr)))) return rc_;
            if ((rc_ = ensure(B.ws_n, sizeof(int)))) return rc_;
            wa.rl = (const int4 *)B.ws_rl.ptr;
            wa.rl_scale = m16 ? (const float *)B.ws_rls.ptr : nullptr;
            wa.rl_bits = (const unsigned *)B.ws_rlb.ptr;
            wa.n_rl = (const int *)B.ws_n.ptr;
        } else {
            if ((rc_ = ensure(B.ws_sb, nbytes<unsigned>((size_t)n_chunks * std::max(1, wa.nwk))))) return rc_;
            if ((rc_ = ensure(B.units, sizeof(int)))) return rc_;
            wa.sbits = (const unsigned *)B.ws_sb.ptr;
            wa.unit_counter = (int *)B.units.ptr;
        }
        wa.rt = (const int4 *)B.rt.ptr;
        wa.rt_scale = m16 ? (const float *)B.rt_scale.ptr : nullptr;
        wa.unit_off = d_strip_off;
        wa.n_strips = n_strips;
        wa.tn = chain.t[n];
        wa.to = has_o ? chain.t[1 - n] : chain.t[n];
        wa.fmap2 = (const int2 *)B.fmap2.ptr;
        wa.chunk_info = (const int4 *)B.chunk_info.ptr;
        wa.active = (const uint8_t *)B.active.ptr;
        wa.acc = (double *)B.acc.ptr;
        wa.err = d_err;
        wa.wait_ns = qc_wait_limit_ns();
        wa.stall_fill = qc_wait_stall_stage();
        if (!configured(ws_fn)) {
            // the kernel's static shared memory (chunk table, abort flag) counts against the limit too
            cudaFuncAttributes fa;
            CK(cudaFuncGetAttributes(&fa, ws_fn));
            CK(cudaFuncSetAttribute(ws_fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    smem_optin - (int)fa.sharedSizeBytes));
            configured_fns.push_back(ws_fn);
        }
        int occ = 0;
        const int ws_block = self_feed ? ws_warps * 32 : (ws_warps + 1) * 32;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, ws_fn, ws_block, ws_smem);
        if (e != cudaSuccess || occ < 1) return fail(QC_EUNSUPPORTED, "warp-specialised kernel does not fit on an SM");
        per_sm = per_sm > 0 ? std::min(per_sm, occ) : occ;
        ws_grid = sm_count * per_sm;
    }
    if (streaming || dds) {
        int rc_;
        block = block_stream;
        sa.vis = d_vis;
        sa.model = d_model;
        sa.model16 = d_model16;
        sa.wf = d_wf;
        sa.n_chan = n_chan;
        sa.n_ant = n_ant;
        sa.rt = (const int4 *)B.rt.ptr;
        sa.rt_scale = m16 ? (const float *)B.rt_scale.ptr : nullptr;
        sa.unit_off = d_strip_off;
        sa.order = order;
        sa.n_chunks = (n_chan + 31) / 32;
        sa.n_units = order == 0 ? n_row : n_strips * sa.n_chunks;
        sa.tn = psums ? tnu : chain.t[n];
        sa.to = has_o ? chain.t[1 - n] : chain.t[n];
        sa.fmap2 = (const int2 *)B.fmap2.ptr;
        sa.acc = (double *)B.acc.ptr;
        sa.active = (const uint8_t *)B.active.ptr;
        if (order == 1) {
            if ((rc_ = ensure(B.units, sizeof(int)))) return rc_;
            sa.unit_counter = (int *)B.units.ptr;
        }
        stream_smem = (block / 32) * stream_smem_per_warp;
        if (stream_smem > smem_optin) return fail(QC_EUNSUPPORTED, "streaming kernel ring exceeds shared memory");
        if (!configured(stream_fn)) {
            CK(cudaFuncSetAttribute(stream_fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin));
            configured_fns.push_back(stream_fn);
        }
    }
    int grid;
    DDArgs dda;
    memset(&dda, 0, sizeof dda);
    if (dds) {
        if (per_sm == 0) {
            int occ = 0;
            cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, stream_fn, block, stream_smem);
            per_sm = (e == cudaSuccess && occ > 0) ? occ : 1;
        }
        const long warps_needed = std::max(1L, (long)n_row);
        grid = (int)std::max(1L, std::min((long)sm_count * per_sm, (warps_needed * 32 + block - 1) / block));
    } else if (ddp) {
        dda.D = data_desc();
        dda.wf = d_wf;
        dda.row_live = d_row_live;
        dda.n_dir = n_dir;
        dda.C = chain;
        for (int j = 0; j < n_terms; ++j) dda.nd[j] = cur_nd[j];
        dda.dd_solved = cur_nd[n] > 1;
        dda.acc = (double *)B.acc.ptr;
        dda.active = (const uint8_t *)B.active.ptr;
        grid = sm_count * 8;
    } else if (mom) {
        grid = 0;
    } else if (ws) {
        grid = ws_grid;
    } else if (streaming) {
        if (per_sm == 0) {
            int occ = 0;
            cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, stream_fn, block, stream_smem);
            per_sm = (e == cudaSuccess && occ > 0) ? occ : 1;
        }
        const long warps_needed = std::max(1L, (long)sa.n_units);
        grid = (int)std::max(1L, std::min((long)sm_count * per_sm, (warps_needed * 32 + block - 1) / block));
    } else if (pipelined) {
        const int NW = L.pipe_nw;
        const long groups = (units + NW - 1) / NW;
        grid = (int)std::max(1L, std::min((long)sm_count, groups));
    } else {
        const int smem = (block / 32) * L.acc_smem_per_warp;
        if (!configured(L.fn)) {
            CK(cudaFuncSetAttribute(L.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin));
            configured_fns.push_back(L.fn);
        }
        if (per_sm == 0) {
            int occ = 0;
            cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, L.fn, block, smem);
            per_sm = (e == cudaSuccess && occ > 0) ? occ : 2;
        }
        const long warps_needed = std::max(1L, units);
        grid = (int)std::max(1L, std::min((long)sm_count * per_sm, (warps_needed * 32 + block - 1) / block));
    }
    int rc;
    if ((rc = ensure(B.chunk_act, (size_t)t.n_tint * aa.n_chunks))) return rc;
    aa.chunk_active = (const uint8_t *)B.chunk_act.ptr;
    sa.chunk_active = aa.chunk_active;
    pa.a = aa;
    pa.chunk_active = (const uint8_t *)B.chunk_act.ptr;
    pa.err = d_err;
    pa.wait_ns = qc_wait_limit_ns();
    pa.stall_issue = qc_wait_stall_stage();
    const int ca_threads = t.n_tint * aa.n_chunks;

    UpdArgs ua;
    ua.type = t.type;
    ua.n_bins = nb;
    ua.n_fint = t.n_fint;
    ua.n_ant = nat;
    ua.acc = (double *)B.acc.ptr;
    ua.params = (double *)B.params.ptr;
    ua.tab = (float4 *)B.tab.ptr;
    ua.gain_flags = (int8_t *)B.flags.ptr;
    ua.iters = (int *)B.iters.ptr;
    ua.active = (uint8_t *)B.active.ptr;
    ua.bin_nvis = (const long long *)B.nvis.ptr;
    ua.bin_nbytes = (const long long *)B.nvis.ptr + 2 * (size_t)nb;
    ua.vis_iters = (unsigned long long *)scalars.ptr;
    ua.acc_bytes = (unsigned long long *)scalars.ptr + 1;
    ua.tol = t.tol;
    // gain flagging on divergence: first / last relative updates and the parameters before the solve
    ua.div = (o->div_flag && !delay[n] && t.max_iter >= 4) ? 1 : 0;
    ua.max_iter = t.max_iter;
    ua.div_stats = nullptr;
    ua.params0 = nullptr;
    // the streaming kernel sums J^H W d in place of J^H W r (the update subtracts JHJ g)
    ua.b_form = (streaming && !dds && !delay[n]) ? 1 : 0;
    const size_t pbytes = nbytes<double>((size_t)nb * nat * (t.type == 2 ? 2 : 8));
    if (ua.div) {
        int rc_;
        if ((rc_ = ensure(B.div, nbytes<double>((size_t)nb * nat * 2)))) return rc_;
        if ((rc_ = ensure(B.params0, pbytes))) return rc_;
        ua.div_stats = (double *)B.div.ptr;
        ua.params0 = (const double *)B.params0.ptr;
    }
    int *cnt = (int *)B.cnt.ptr;
    const int upd_block = nat >= 128 ? 128 : (nat > 32 ? 64 : 32);
    // delay terms: the update reduces the channel bins of each parameter interval
    DelayUpdArgs dua;
    memset(&dua, 0, sizeof dua);
    if (delay[n]) {
        dua.d = delay_args(n, t);
        dua.acc = ua.acc;
        dua.gain_flags = ua.gain_flags;
        dua.iters = ua.iters;
        dua.active = ua.active;
        dua.bin_nvis = ua.bin_nvis;
        dua.bin_nbytes = ua.bin_nbytes;
        dua.vis_iters = ua.vis_iters;
        dua.acc_bytes = ua.acc_bytes;
        dua.tol = ua.tol;
        if (dsum) {
            dua.hsum = (const double *)B.dsum_h.ptr;
            dua.omega = (const float *)B.domega.ptr;
            dua.omega_lo = dua.omega + n_chan;
            dua.om_sums = (const double2 *)B.dom_sums.ptr;
            dua.om_max = B.om_max;
            dua.prod_bytes = 32 * n_up;
        }
    }
    DelaySumsArgs dsa_;
    if (dsum) dsa_ = delay_sums_args(terms, n_terms, n, chain);

    MomArgs ma;
    MomNormArgs mn;
    const int mom_n = mom ? mom_words(B.sums.form) : 0;
    const size_t mom_words_all = (size_t)nb * n_up * mom_n;
    const size_t mom_cnt_off = B.sums.cnt_off;
    if (mom) {
        int rc_ = sums_args(terms, n_terms, n, chain, st, ma, mn);
        if (rc_) return rc_;
        mn.active = (const uint8_t *)B.active.ptr;
        mn.acc = (double *)B.acc.ptr;
        ua.bin_nbytes = (const long long *)((char *)B.mom.ptr + mom_cnt_off);
    }
    const long long mom_iter_bytes = 2LL * n_up * mom_n * 4 + 8LL * n_ant * (t.type == 1 ? KG_FULL : KG_DIAG);

    const int max_iter = t.max_iter;
    for (int k = 0; k < 2 * max_iter + 2; ++k) { cudaEvent_t ev; if ((rc = get_event(2 + k, ev))) return rc; }
    const int ev_pass = 2 + 2 * max_iter;     // the sums pass (its own bracket inside iteration 1's)
    // (no graph while a test stalls a stage: a captured graph would keep the stall)
    // (a delay term from products has two short kernels an iteration: launching them costs less than
    // capturing and instantiating a graph for the one replay of a solve)
    const bool use_graph = o->use_graph && !t.reduce && qc_wait_stall_stage() < 0 && !dsum;
    const unsigned rec_flags = use_graph ? cudaEventRecordExternal : cudaEventRecordDefault;

    auto enqueue = [&]() -> int {
        init_term_kernel<<<(std::max(nb, max_iter + 1) + 255) / 256, 256, 0, st>>>(nb, (uint8_t *)B.active.ptr, cnt,
                                                                                   max_iter + 1);
        CK(cudaGetLastError());
        if (ua.div) {
            CK(cudaMemsetAsync(B.div.ptr, 0, nbytes<double>((size_t)nb * nat * 2), st));
            CK(cudaMemcpyAsync(B.params0.ptr, B.params.ptr, pbytes, cudaMemcpyDeviceToDevice, st));
        }
        for (int k = 1; k <= max_iter; ++k) {
            aa.n_active = cnt + (k - 1);
            // inside a capture the record must be an external event node to be timed on replay
            if (!dsum) {
                chunk_active_kernel<<<(ca_threads + 255) / 256, 256, 0, st>>>(aa.tn, n_chan, aa.n_chunks,
                                                                            (const uint8_t *)B.active.ptr, cnt + (k - 1),
                                                                            (uint8_t *)B.chunk_act.ptr);
                CK(cudaGetLastError());
            }
            CK(cudaEventRecordWithFlags(events[2 + 2 * (k - 1)], st, rec_flags));
            if (dsum) {
                dsa_.n_active = cnt + (k - 1);
                if (k == 1) {
                    CK(cudaMemsetAsync(B.dsum_h.ptr, 0, nbytes<double>((size_t)nbu * n_ant * KG_HSUM), st));
                    const size_t words = (size_t)t.n_tint * dsa_.n_chunks * n_up * 256;
                    if (dsa_.T64) CK(cudaMemsetAsync(dsa_.T64, 0, nbytes<double>(words), st));
                    else if (!dsa_.store) CK(cudaMemsetAsync(dsa_.T, 0, nbytes<float>(words), st));
                    CK(dsum_launch_pass(dsa_, lk != KIND_NONE ? lk : rk, sm_count, st));
                    if (dsa_.T64) CK(dsum_launch_round(words, dsa_.T64, dsa_.T, sm_count, st));
                }
                CK(dsum_launch_iter(dsa_, st));
            } else if (dds) {
                DDStreamArgs x;
                x.s = sa;
                x.s.n_active = cnt + (k - 1);
                x.n_dir = n_dir;
                x.nd_n = cur_nd[n];
                x.nd_o = n_terms == 2 ? cur_nd[1 - n] : 1;
                x.omega = delay[n] ? (const float *)B.domega.ptr : nullptr;
                const int gy = DS.dirs_per_cta > 0 ? (n_dir + DS.dirs_per_cta - 1) / DS.dirs_per_cta : 1;
                CK(DS.launch(dim3(grid, gy), block, stream_smem, st, x));
            } else if (ddp) {
                dda.n_active = cnt + (k - 1);
                CK(dd_launch_acc(dda, ts, grid, st));
            } else if (mom) {
                if (k == 1) {
                    if (ma.mom64) CK(cudaMemsetAsync(ma.mom64, 0, nbytes<double>(mom_words_all), st));
                    else CK(cudaMemsetAsync(ma.mom, 0, nbytes<float>((ma.tail ? 2 : 1) * mom_words_all), st));
                    CK(mom_launch_bytes(nb, (const long long *)B.nvis.ptr + 2 * (size_t)nb, mom_iter_bytes,
                                        (long long *)((char *)B.mom.ptr + mom_cnt_off), ua.acc_bytes, st));
                    CK(cudaEventRecordWithFlags(events[ev_pass], st, rec_flags));
                    ma.n_active = cnt;
                    CK(mom_launch_pass(ma, B.sums.form, B.sums.ok, sm_count, st));
                    if (ma.mom64) CK(mom_launch_split(mom_words_all, ma.mom64, ma.mom, ma.tail, sm_count, st));
                    CK(cudaEventRecordWithFlags(events[ev_pass + 1], st, rec_flags));
                }
                mn.n_active = cnt + (k - 1);
                CK(mom_launch_normal(mn, st));
            } else if (ws) {
                wa.n_active = cnt + (k - 1);
                const uint8_t *ca = (const uint8_t *)B.chunk_act.ptr;
                if (order == 0) {
                    CK(cudaMemsetAsync(B.ws_n.ptr, 0, sizeof(int), st));
                    if (n_row)
                        ws_rows_kernel<<<(n_row + 255) / 256, 256, 0, st>>>(
                            n_row, wa.rt, wa.rt_scale, ca, wa.n_chunks, wa.nwr, wa.n_active, (int4 *)B.ws_rl.ptr,
                            m16 ? (float *)B.ws_rls.ptr : nullptr, (unsigned *)B.ws_rlb.ptr, (int *)B.ws_n.ptr);
                } else {
                    if (wa.nwk)
                        ws_strip_bits_kernel<<<(wa.nwk + 7) / 8, 256, 0, st>>>(
                            n_strip_rows, wa.rt, ca, wa.n_chunks, wa.nwk, wa.n_active, (unsigned *)B.ws_sb.ptr);
                    CK(cudaMemsetAsync(B.units.ptr, 0, sizeof(int), st));
                }
                CK(cudaGetLastError());
                if (self_feed) CK(L.wss_launch(ws_grid, ws_smem, st, wa));
                else CK(L.ws_launch(ws_grid, ws_smem, st, wa));
            } else if (streaming) {
                sa.n_active = cnt + (k - 1);
                if (sa.unit_counter) CK(cudaMemsetAsync(sa.unit_counter, 0, sizeof(int), st));
                if (ded) {
                    DelayStreamArgs dsa;
                    dsa.s = sa;
                    dsa.omega = (const float *)B.domega.ptr;
                    CK(DL.launch(grid, block, stream_smem, st, dsa));
                } else {
                    CK(L.stream_launch(grid, block, stream_smem, st, sa));
                }
            } else if (pipelined) {
                pa.a.n_active = cnt + (k - 1);
                CK(L.pipe_launch(grid, pipe_smem, st, pa));
            } else {
                CK(L.launch(grid, block, st, aa));
            }
            CK(cudaEventRecordWithFlags(events[2 + 2 * (k - 1) + 1], st, rec_flags));
            if (t.reduce) {
                const size_t KG = psums ? KG_SUMS : (t.type == 1 ? KG_FULL : KG_DIAG);
                if (o->allreduce((double *)B.acc.ptr, (int64_t)(psums ? nbu : nb) * nat * KG, st, o->allreduce_user))
                    return fail(QC_ECUDA, "allreduce callback failed");
            }
            ua.k = k;
            ua.alpha = (o->damping_mode == QC_DAMP_ALTERNATE) ? ((k % 2 == 0) ? 0.5 : 1.0)
                                                               : (o->damping > 0 ? o->damping : 1.0);
            ua.n_active_prev = cnt + (k - 1);
            ua.n_active_next = cnt + k;
            if (delay[n]) {
                dua.k = k;
                dua.alpha = ua.alpha;
                dua.n_active_prev = ua.n_active_prev;
                dua.n_active_next = ua.n_active_next;
                if (psums) {
                    delay_update_kernel<true><<<dua.d.n_tint * dua.d.n_fint, 128, 0, st>>>(dua);
                    if (!dsum) {
                        // about four CTAs an SM, none below 512 (antenna, channel) pairs
                        CK(cudaGetLastError());
                        const long n_int = (long)dua.d.n_tint * dua.d.n_fint;
                        const long by_size = ((long)n_ant * n_chan / dua.d.n_fint + 511) / 512;
                        const unsigned split = (unsigned)std::max(1L, std::min(by_size, 4L * sm_count / n_int));
                        delay_chan_kernel<<<dim3((unsigned)n_int, split), 128, 0, st>>>(dua);
                    }
                }
                else delay_update_kernel<false><<<dua.d.n_tint * dua.d.n_fint, upd_block, 0, st>>>(dua);
            } else {
                update_kernel<<<nb, upd_block, 0, st>>>(ua);
            }
            CK(cudaGetLastError());
        }
        if (dsum) {
            delay_tab_kernel<<<grid_for((long)nb * n_ant, 256, sm_count), 256, 0, st>>>(dua.d);
            CK(cudaGetLastError());
        }
        return QC_OK;
    };
    if (use_graph) {
        if (!B.graph_valid) {
            if (B.exec) { cudaGraphExecDestroy(B.exec); B.exec = nullptr; }
            cudaGraph_t g = nullptr;
            CK(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
            rc = enqueue();
            // always end the capture, so that a failure leaves the stream usable
            cudaError_t e = cudaStreamEndCapture(st, &g);
            if (rc || e != cudaSuccess) {
                if (g) cudaGraphDestroy(g);
                cudaGetLastError();
                if (rc) return rc;
                return cuda_fail(e, "cudaStreamEndCapture");
            }
            e = cudaGraphInstantiate(&B.exec, g, 0);
            cudaGraphDestroy(g);
            if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
            B.graph_valid = true;
        }
        CK(cudaGraphLaunch(B.exec, st));
    } else {
        if ((rc = enqueue())) return rc;
    }
    launches += 1 + (delay[n] && psums && !dsum ? 4 : 3) * (long long)max_iter + (mom ? 3 + (ma.mom64 ? 1 : 0) : 0);
    // iteration bookkeeping: which accumulate launches did work, and their device time
    std::vector<int> hcnt(max_iter + 1);
    int herr = 0;
    CK(cudaMemcpyAsync(hcnt.data(), cnt, nbytes<int>(max_iter + 1), cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(&herr, d_err, sizeof(int), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (herr) {
        CK(cudaMemsetAsync(d_err, 0, sizeof(int), st));
        return fail(QC_ETIMEOUT, "a bounded wait in a bulk-copy accumulate kernel gave up");
    }
    double ms_sum = 0;
    long long worked = 0;
    int last = 0;
    for (int k = 1; k <= max_iter; ++k) {
        if (hcnt[k - 1] == 0) break;
        float ms = 0;
        CK(cudaEventElapsedTime(&ms, events[2 + 2 * (k - 1)], events[2 + 2 * (k - 1) + 1]));
        ms_sum += ms;
        ++worked;
        last = k;
    }
    if (mom && B.sums.asked && hcnt[0] != 0) {
        float ms = 0;
        CK(cudaEventElapsedTime(&ms, events[ev_pass], events[ev_pass + 1]));
        *pass_ms = ms;
    }
    *it_max = last;
    *acc_ms = ms_sum;
    *acc_launches = worked;
    return QC_OK;
}

// ---------------------------------------------------------------------------
// MAD residual flagging (Section 4, "Additional features"; global mode)
// ---------------------------------------------------------------------------
//
// The statistic of an unflagged cross-correlation sample is its whitened residual norm
// z = sqrt(sum_c w_c |r_c|^2), computed in float32 with every operation rounded (no fused
// multiply-add) in a fixed order.  Median and MAD are exact order statistics (the
// floor((n - 1) / 2)-th smallest value), found by a radix select over the float bit
// patterns, which order like the values for non-negative floats.  A sample is flagged when
// |z - median| > fl32(threshold * 1.4826) * MAD in float32.  The whole sequence runs on the
// stream (qc_residual.cu): the digits are picked on the device, so that nothing waits for the host.

extern "C" int qc_mad_flag(qc_ctx *c, const qc_term *terms, int32_t n_terms, double threshold, int32_t per_baseline,
                           uint8_t *flags_out, int32_t out_memory, int64_t *n_flagged)
{
    if (!c) return QC_EINVAL;
    c->err.clear();
    if (!flags_out) return c->fail(QC_EINVAL, "flags_out is NULL");
    if (c->n_dir > 1) return c->fail(QC_EUNSUPPORTED, "qc_mad_flag takes problems with one direction");
    if (!(threshold > 0) || !std::isfinite(threshold)) return c->fail(QC_EINVAL, "threshold must be positive and finite");
    if (out_memory != QC_MEM_HOST && out_memory != QC_MEM_DEVICE) return c->fail(QC_EINVAL, "out_memory invalid");
    int rc = c->validate_terms(terms, n_terms, false);
    if (rc) return rc;
    cudaStream_t st = c->own_stream;
    PinScope pins(c, st);
    std::vector<qc_term> xt;
    if ((rc = c->expand_terms(terms, n_terms, xt, st))) return rc;
    Chain chain;
    if ((rc = c->stage_terms(xt.data(), n_terms, st, chain))) return rc;
    const long n_vis = (long)c->n_row * c->n_chan;
    if ((rc = c->ensure(c->mad_keys, nbytes<unsigned>((size_t)std::max(1L, n_vis))))) return rc;
    if ((rc = c->ensure(c->mad_state, sizeof(MadState)))) return rc;
    unsigned *keys = (unsigned *)c->mad_keys.ptr;
    MadState *state = (MadState *)c->mad_state.ptr;
    uint8_t *dout = (uint8_t *)flags_out;
    if (out_memory == QC_MEM_HOST) {
        if ((rc = c->ensure(c->mad_out, (size_t)std::max(1L, n_vis)))) return rc;
        dout = (uint8_t *)c->mad_out.ptr;
    }
    if (n_vis == 0) {
        if (n_flagged) *n_flagged = 0;
        return QC_OK;
    }
    const float factor = (float)(threshold * 1.4826);
    CK(cudaMemsetAsync(state, 0, sizeof(MadState), st));
    ResArgs ra;
    ra.D = c->data_desc();
    ra.C = chain;
    ra.resid = nullptr;
    ra.chi2 = nullptr;
    CK(mad_keys_launch(ra, c->m16, keys, state, c->sm_count, st));
    if (per_baseline) {
        if (!c->mad_groups.ptr && !c->pair_strips.empty()) {
            // the strips of each unordered antenna pair, staged by the first call
            if ((rc = c->ensure(c->mad_groups, nbytes<int2>(c->pair_strips.size())))) return rc;
            CK(cudaMemcpyAsync(c->mad_groups.ptr, c->pair_strips.data(), nbytes<int2>(c->pair_strips.size()),
                               cudaMemcpyHostToDevice, st));
        }
        CK(cudaMemsetAsync(dout, 0, (size_t)n_vis, st));
        CK(mad_group_launch((int)c->pair_strips.size(), (const int2 *)c->mad_groups.ptr, c->d_strip_off, c->d_strip_rows,
                            c->n_chan, keys, factor, state, dout, st));
    } else {
        CK(mad_global_launch(n_vis, keys, factor, state, dout, c->sm_count, st));
    }
    unsigned long long hc = 0;
    if (++c->pin_calls >= c->PIN_CALLS) c->pin_reserve(64);
    if (out_memory == QC_MEM_HOST) CK(cudaMemcpyAsync(flags_out, dout, (size_t)n_vis, cudaMemcpyDeviceToHost, st));
    CK(c->to_host(&hc, &state->n_flagged, sizeof hc, st));
    CK(cudaStreamSynchronize(st));
    c->pin_end();
    if (n_flagged) *n_flagged = (int64_t)hc;
    return QC_OK;
}
