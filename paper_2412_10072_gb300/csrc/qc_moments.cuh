// qc_moments.cuh -- argument blocks of the sums pass and the per-iteration normal equations of
// a single-term chain (kernels in qc_moments.cu).
#pragma once

#include "qc_kernels.cuh"
#include "qc_sums.cuh"

namespace qc {

constexpr int MOM_N = 100;          // FP32 words per (interval, pair), full form: S 64, T 32, four of padding
constexpr int MOM_T = 64;
// left-full form (a diagonal or phase-only solved term with a full term to its left): S' 16 (4x4
// Hermitian packed as S), T' 8, four words of padding (slots of whole 16-byte vectors)
constexpr int MOM_E = 28;
constexpr int MOM_ET = 16;
// plain diagonal form (a diagonal or phase-only solved term, the other term diagonal or to its
// right): S 4, T 8
constexpr int MOM_D = 12;
constexpr int FORM_FULL = 0, FORM_E = 1, FORM_D = 2;
__host__ __device__ constexpr int mom_words(int form)
{
    return form == FORM_FULL ? MOM_N : (form == FORM_E ? MOM_E : MOM_D);
}

// steps after which the full form's lanes go to the slots
__host__ __device__ constexpr int mom_flush_every(bool m16) { return m16 ? 16 : 32; }

// Hermitian pairs (u, v), u < v, of the 4x4 S blocks: packed as 4 diagonal reals then 6 (re, im)
__host__ __device__ constexpr int mom_pair(int u, int v)
{
    return u == 0 ? (v == 1 ? 0 : v == 2 ? 1 : 2) : u == 1 ? (v == 2 ? 3 : 4) : 5;
}

// what is known of a channel map: nothing, one interval, one interval per channel, or each 32-channel
// chunk in one interval
enum { MAP_ANY = 0, MAP_ONE = 1, MAP_IDENTITY = 2, MAP_CHUNK = 3 };

struct MomArgs {
    int n_chan, n_ant, n_up;             // n_up: unordered antenna pairs with data
    const float4 *vis, *model, *wf;      // wf: weights with flags and autocorrelations folded in (w = 0)
    const uint4 *model16;                // FP16 model, or null
    const float *mscale;                 // [strip rows] its scale, or null
    // [strip rows] {row, time, pair | conj << 31, p | q << 16}, rows with usable samples: p, q the
    // antennas of the baseline as oriented in the sums (p < q); conj: the row is (q, p)
    const int4 *mrows;
    const int *strip_off, *strip_end;    // first and past-the-last row of each ordered baseline in mrows
    int tn_map, to_map;                  // MAP_* of the channel maps of the solved and the fixed term
    int n_strips, n_chunks;              // n_chunks: 32-channel chunks of a row
    int group;                           // chunks per unit of work
    int rb, n_rb;                        // rows of a strip per unit of work, blocks per strip
    int n_time, stage_maps;              // data times; time maps read from shared memory (set at the launch)
    int chunk_major;                     // 1: a unit's rows inside each chunk; 0: a row's chunks inside it
    DevTerm tn;                          // the solved term (maps)
    DevTerm to;                          // the fixed other term of a two-term chain (tables)
    float *mom, *tail;                   // [bins][n_up][mom_words(form)], heads and tails (or null) of the sums
    double *mom64;                       // the same in FP64, added to instead, or null: one store a slot
    const int *n_active;                 // or null: always
};

struct MomNormArgs {
    int n_bins, n_ant, n_up, type;       // type: QC_TERM_* (diag, full, phase)
    int form;                            // FORM_*
    const int *upair;                    // [n_ant][n_ant] unordered pair index or -1
    const float *mom;                    // [bins][n_up][mom_words(form)]
    const float *tail;                   // their tails, or null
    const double *params;                // FP64 gains of the solved term
    const float4 *tab;                   // their FP32 table [n_tint][n_ant][n_fint] x (1 | 2)
    int n_fint;
    const uint8_t *active;               // [bins]
    const int *n_active;
    double *acc;                         // [bins][n_ant][KG] (written by the per-iteration form)
};

// Every iteration in one launch (mom_iterate_kernel).
struct MomIterArgs {
    MomNormArgs n;
    double *params;                      // FP64 master (read and updated)
    float4 *tab;                         // FP32 table (read at the start, written at the end)
    int8_t *gain_flags;                  // [bins][n_ant]
    int *iters;                          // [bins]
    int *cnt;                            // [max_iter + 1], zeroed: intervals still active after iteration k
    const long long *bin_nvis, *bin_nbytes;
    long long iter_bytes;                // algorithmic bytes of an interval's iteration
    unsigned long long *vis_iters, *acc_bytes;
    int max_iter, alternate;             // alternate: step 1, 1/2, 1, ...; else `damping`
    double damping, tol;
};

} // namespace qc
