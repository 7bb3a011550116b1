// The small-batch search path (small.cu): the stages before and after the scan
// in one kernel each.
#pragma once

#include "lut.cuh"
#include "scan.cuh"

namespace ksc {

constexpr int SP_MAX_P = 1024;    // probes per query of the small-batch kernels
constexpr int SP_RANK_L = 8192;   // lists, and
constexpr int SP_RANK_P = 512;    // probes, up to which they rank the lists as well
constexpr int SP_REG_KEYS = 8192; // keys of a query up to which the selection holds them in registers

struct SmallPrep {
    LutArgs T;  // tables of (query, rank); T.probes as below
    ScanArgs A;
    // ranking (c_rank != NULL): the P_q best lists of every query by exact FP32
    // score into probes_out (= T.probes); otherwise the probes are given
    const float* c_rank;
    int spherical;
    int32_t* probes_out;
    uint8_t* lut;
    int32_t* bias;
    float* scale;
    int32_t* cnt;   // [nq] keys of the unfiltered part
    int32_t* noff;  // [nq Pmax] place of a pair's first key in it
    int4 *recsA, *recsB;  // scan items of the unfiltered part and of the rest
    int32_t* nrec;  // [2] their numbers (cleared by the caller)
    int TBa, TB, Rmax, cap;
    int all_near;   // the store holds every key: all lists are in the unfiltered part
    int near_keys_per_r, near_share_div;
};

// One cluster per query: ranking (optional), tables, biases and scan items.
int launch_small_prep(const SmallPrep& S, cudaStream_t st);

// One CTA per query: the R best keys of its store (redone exactly if it
// overflowed) and their exact re-rank.
int launch_select_rerank(const ScanArgs& A, int Rmax, const int32_t* cnt, uint64_t* cand, int cap, int sel_cap,
                         const float* Q, const float* X, int d, int ip, int k, int64_t* ids, float* dists,
                         int32_t* status, unsigned long long* stats, cudaStream_t st);

}  // namespace ksc
