// qc_delay_sums.cuh -- a solved delay term from per-(time interval, pair, channel) products
// (kernels in qc_delay_sums.cu).
#pragma once

#include "qc_delay.cuh"

namespace qc {

// antennas whose gains and right-hand sides of 32 channels fit a CTA's shared memory (1 KB each)
constexpr int DSUM_MAX_ANT = 220;
constexpr int KG_HSUM = 6;           // FP64 words of the constant sums per (interval, antenna)

struct DelaySumsArgs {
    int n_chan, n_ant, n_up, n_fint, n_chunks;
    // pass
    const float4 *vis, *model, *wf;
    const uint4 *model16;            // FP16 model, or null
    const int4 *mrows;               // strip rows {row or -1, time, pair | conj << 31, p | q << 16}, p < q
    const float *mscale;             // their FP16 model scales, or null
    const int *strip_off;
    int n_strips, rb, n_rb;          // units of work: strip x block of rb rows (x chunk with chunk_major)
    int chunk_major;
    const int *t_map;                // [n_time] time interval of the delay term
    DevTerm to;                      // the other term (a copy of anything when there is none)
    int store;                       // every slot is written exactly once: plain stores, no zeroing
    const uint8_t *active;           // [bins], all set when the pass runs
    // both
    const int *fmap;                 // [n_chan] parameter interval of each channel
    const float *omega;              // [n_chan] 2 pi nu - omega_ref
    float4 *T;                       // [n_tint][n_chunks][n_up][2][32]
    double *T64;                     // the same in FP64, added to instead, or null (one addition a slot)
    double *hsum;                    // [bins][n_ant][KG_HSUM]
    // iterations
    int n_tint;
    const int *upair;                // [n_ant][n_ant] unordered pair or -1
    const double *nu;                // [n_chan]
    const double *params;            // FP64 master [bins][n_ant][4]
    const int *n_active;
    double *acc;                     // [bins][n_ant][KG_SUMS]
};

} // namespace qc

cudaError_t dsum_launch_pass(const qc::DelaySumsArgs &a, int ok, int sm_count, cudaStream_t st);
cudaError_t dsum_launch_round(size_t words, const double *src, float4 *dst, int sm_count, cudaStream_t st);
cudaError_t dsum_launch_iter(const qc::DelaySumsArgs &a, cudaStream_t st);
