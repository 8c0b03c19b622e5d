// qc_residual.cuh -- chi^2, the residual and MAD flagging of it (kernels in qc_residual.cu).
#pragma once
#include "qc_kernels.cuh"

namespace qc {

struct ResArgs {
    Data D;
    Chain C;              // n = -1: product of all terms
    float4 *resid;        // [n_row][n_chan] x 2, or nullptr
    double *chi2;         // one double
};

// Device state of one MAD selection: two exact order statistics found by radix select over the bits
// of non-negative floats (which order like the values), most significant digits first.
struct MadState {
    unsigned long long n_used, n_flagged;
    unsigned long long k;                  // rank looked for among the keys that match the prefix
    unsigned prefix;                       // digits found so far
    float med, thr;
    unsigned hist[2048];
};

constexpr int MAD_LEVELS = 3;              // digits of 11, 10 and 10 bits (the sign bit is never set)

} // namespace qc

cudaError_t residual_launch(const qc::ResArgs &a, bool m16, int sm_count, cudaStream_t st);
// z keys of every sample (a sentinel for unused ones) and the number of used ones (state zeroed
// before); no residual is written
cudaError_t mad_keys_launch(const qc::ResArgs &a, bool m16, unsigned *keys, qc::MadState *state, int sm_count, cudaStream_t st);
// median, MAD and flags over all keys
cudaError_t mad_global_launch(long n, const unsigned *keys, float factor, qc::MadState *state, uint8_t *out, int sm_count,
                              cudaStream_t st);
// the same per group: the rows of the group's one or two baseline strips (y < 0: one)
cudaError_t mad_group_launch(int n_groups, const int2 *groups, const int *strip_off, const int *strip_rows, int n_chan,
                             const unsigned *keys, float factor, qc::MadState *state, uint8_t *out, cudaStream_t st);
