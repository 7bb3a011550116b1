// Query path of KScaNN (Alg. 2 with the leaf scan of Alg. 3) on sm_103a.
//
//   a1 rank     : scores of every (query, list) + per-query top-P select
//   a2 LUT      : FP32 residual tables (Eq. 1), per-query scale, u8 tables
//                 and per-(query, probe) integer bias (8-bit LUT, Sec. 2.5)
//   threshold   : per-query upper bound of the R-th key from its nearest lists
//   a3 scan     : cluster-major work list of (list, query group, block tile);
//                 16-entry sub-LUTs held in registers, looked up with PRMT,
//                 u16x2 lane sums, cross-lane reduce-scatter
//   a5 select   : R smallest (D, id) keys per query (radix select + bitonic)
//   a6 rerank   : exact FP32 distances of the R candidates, top-k
#include <atomic>
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "index.cuh"
#include "lut.cuh"
#include "mlp.cuh"
#include "rerank.cuh"
#include "rerank_low.cuh"
#include "scan.cuh"
#include "scan_ops.cuh"
#include "small.cuh"

namespace ksc {

constexpr int SEL_CAP = 4096;   // bitonic buffer of the select kernels (>= KSC_MAX_RERANK)

// Shared buffer of the exact select of overflowed queries: 8 R keys (a power
// of two, at least 1024, at most SEL_CAP; it sorts the R best).
static int sel_keys(int Rmax) { return std::min(SEL_CAP, std::max(1024, pow2_ceil(8 * Rmax))); }

// Per-query kernels come in two shapes: a warp per query (many queries: the
// GPU is full of warps) or a CTA per query (few queries: eight warps share
// each one).  The warp shape pays off once the batch fills every SM's warps.
static bool warp_per_query(int64_t nq) { return nq >= 8 * (int64_t)num_sms(); }
constexpr int MAX_NPROBE = 4096;
constexpr int NEAR_KEYS_PER_R = 4;  // keys of the unfiltered first scan: at least 4 R ...
constexpr int NEAR_SHARE_DIV = 16;  // ... and at least 1/16 of the keys the query probes

// ------------------------------------------------------------------ a1: list scores
// score[q][c] = ||c||^2 - 2<q,c> (L2, ||q||^2 dropped) or -<q,c> (spherical).
constexpr int SC_T = 64, SC_K = 32;
__global__ void __launch_bounds__(256) k_list_scores(const float* __restrict__ Q, int64_t nq, int d,
                                                     const float* __restrict__ Cc, const float* __restrict__ cn,
                                                     int L, int spherical, float* __restrict__ scores) {
    __shared__ float qs[SC_K][SC_T + 4];
    __shared__ float cs[SC_K][SC_T + 4];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t q0 = (int64_t)blockIdx.y * SC_T;
    const int c0 = blockIdx.x * SC_T;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int k0 = 0; k0 < d; k0 += SC_K) {
        for (int e = threadIdx.x; e < SC_T * SC_K; e += 256) {
            int r = e / SC_K, kk = e % SC_K;
            int gk = k0 + kk;
            int64_t gq = q0 + r;
            qs[kk][r] = (gq < nq && gk < d) ? Q[gq * d + gk] : 0.f;
            int gc = c0 + r;
            cs[kk][r] = (gc < L && gk < d) ? Cc[(int64_t)gc * d + gk] : 0.f;
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < SC_K; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = qs[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = cs[kk][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        int64_t q = q0 + ty * 4 + i;
        if (q >= nq) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            int c = c0 + tx * 4 + j;
            if (c >= L) continue;
            scores[q * L + c] = spherical ? -acc[i][j] : fmaf(-2.f, acc[i][j], cn[c]);
        }
    }
}

// P_q best lists per query.  `scores` may be approximate (each within err[q]
// of the exact score; err = NULL means exact): a float histogram finds the
// bin of the P-th smallest score, every list whose score can still be among
// the P best (score <= upper edge of that bin + 2 err) is re-scored exactly in
// FP32 (L2: sum_t (q_t - c_t)^2 in the direct form; spherical: -<q, c>), and
// the P best by (exact score, list id) are kept.  If more lists qualify than
// the re-score buffer holds (4 Pmax, at least 1024, at most RS_CAP), every
// list is re-scored when all fit, else those with the lowest given scores.
constexpr int RS_CAP = 4096;     // largest re-score buffer
constexpr int FEAT_K = 32;       // list distances of the predictor's features
constexpr int RS_SMEM_L = 8192;  // score rows up to this length are staged in shared memory
template <int NT>
__global__ void __launch_bounds__(NT) k_rank_select(const float* __restrict__ scores, const float* __restrict__ err,
                                                     const float* __restrict__ Q, const float* __restrict__ Cc,
                                                     int64_t nq, int d, int L, int spherical,
                                                     const int32_t* __restrict__ nprobe_q, int Pfix, int Pmax,
                                                     int rs_cap, int32_t* __restrict__ probes,
                                                     float* __restrict__ score_out, const int32_t* __restrict__ list) {
    extern __shared__ uint64_t cand[];  // rs_cap keys, then the row's scores when L <= RS_SMEM_L
    __shared__ uint32_t hist[HIST_BINS];
    __shared__ uint32_t warp_tot[32];
    __shared__ __align__(16) float qs[KSC_MAX_DIM];
    __shared__ uint32_t s_mn, s_mx;
    __shared__ int s_cnt, s_B;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    // every query, or (list != NULL) the list[0] queries list[1..]
    const int64_t count = list ? list[0] : nq;
    for (int64_t e = blockIdx.x; e < count; e += gridDim.x) {
    const int64_t q = list ? list[1 + e] : e;
    __syncthreads();  // the previous query's shared state is no longer read
    int P = nprobe_q ? nprobe_q[q] : Pfix;
    P = P < 1 ? 1 : (P > Pmax ? Pmax : P);
    const float* s = scores + q * L;
    if (L <= RS_SMEM_L) {
        // the row is read from global memory once
        float* ss = reinterpret_cast<float*>(cand + rs_cap);
        for (int c = threadIdx.x; c < L; c += blockDim.x) ss[c] = s[c];
        s = ss;
    }
    const float e2 = err ? 2.f * err[q] : 0.f;
    for (int t = threadIdx.x; t < d; t += blockDim.x) qs[t] = Q[q * d + t];
    if (threadIdx.x == 0) { s_mn = 0xffffffffu; s_mx = 0u; s_cnt = 0; s_B = -1; }
    for (int b = threadIdx.x; b < HIST_BINS; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    uint32_t mn = 0xffffffffu, mx = 0u;
    for (int c = threadIdx.x; c < L; c += blockDim.x) {
        uint32_t u = ordered_f32(s[c]);
        mn = min(mn, u);
        mx = max(mx, u);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) { atomicMin(&s_mn, mn); atomicMax(&s_mx, mx); }
    __syncthreads();
    const float fmn = unordered_f32(s_mn), fmx = unordered_f32(s_mx);
    const float width = (fmx - fmn) / (float)(HIST_BINS - 1);
    const float inv = width > 0.f ? 1.f / width : 0.f;
    auto bin_of = [&](float v) -> int {
        float f = (v - fmn) * inv;
        return f < (float)(HIST_BINS - 1) ? (int)f : HIST_BINS - 1;
    };
    for (int c = threadIdx.x; c < L; c += blockDim.x) atomicAdd(&hist[bin_of(s[c])], 1u);
    __syncthreads();
    {
        const int per = HIST_BINS / blockDim.x;
        const int b0 = threadIdx.x * per;
        uint32_t local = 0;
        for (int b = b0; b < b0 + per; ++b) local += hist[b];
        const uint32_t excl = block_exclusive_scan(local, warp_tot);
        if (excl < (uint32_t)P && excl + local >= (uint32_t)P) {
            uint32_t acc = excl;
            for (int b = b0; b < b0 + per; ++b) {
                if (acc + hist[b] >= (uint32_t)P) { s_B = b; break; }
                acc += hist[b];
            }
        }
    }
    __syncthreads();
    // every list that can still be among the P best
    const float tau = (s_B >= HIST_BINS - 1) ? INFINITY : fmn + (float)(s_B + 1) * width + e2;
    for (int c = threadIdx.x; c < L; c += blockDim.x) {
        if (s[c] <= tau) {
            int slot = atomicAdd(&s_cnt, 1);
            if (slot < rs_cap) cand[slot] = (uint64_t)(uint32_t)c;
        }
    }
    __syncthreads();
    int n = s_cnt;
    if (n > rs_cap) {
        // degenerate score distribution: re-score every list if they fit,
        // else the rs_cap lists with the lowest given scores
        if (L <= rs_cap) {
            n = L;
            for (int c = threadIdx.x; c < L; c += blockDim.x) cand[c] = (uint64_t)(uint32_t)c;
            __syncthreads();
        } else {
            n = rs_cap;
            auto load = [&](int c) -> uint64_t { return ((uint64_t)ordered_f32(s[c]) << 32) | (uint32_t)c; };
            block_select_smallest(load, L, rs_cap, cand, cand, rs_cap, hist);
            for (int i = threadIdx.x; i < rs_cap; i += blockDim.x) cand[i] &= 0xffffffffull;
            __syncthreads();
        }
    }
    for (int i = w; i < n; i += nw) {
        const int c = (int)(uint32_t)cand[i];
        const float v = exact_list_score(qs, Cc + (int64_t)c * d, d, spherical, lane);
        if (lane == 0) cand[i] = ((uint64_t)ordered_f32(v) << 32) | (uint32_t)c;
    }
    __syncthreads();
    if (n <= 32) {
        if (w == 0) {
            const uint64_t v = warp_sort_key(lane < n ? cand[lane] : KEY_NONE, lane);
            cand[lane] = v;
        }
    } else {
        const int S = pow2_ceil(n);
        for (int i = n + threadIdx.x; i < S; i += blockDim.x) cand[i] = KEY_NONE;
        __syncthreads();
        block_bitonic_sort(cand, S);
    }
    __syncthreads();
    for (int r = threadIdx.x; r < Pmax; r += blockDim.x) {
        if (r < P && r < n) {
            probes[q * Pmax + r] = (int32_t)(cand[r] & 0xffffffffu);
            if (score_out) score_out[q * Pmax + r] = unordered_f32((uint32_t)(cand[r] >> 32));
        } else {
            probes[q * Pmax + r] = -1;
            if (score_out) score_out[q * Pmax + r] = INFINITY;
        }
    }
    }
}

// Warp bitonic sort, ascending, of S (a power of two) keys in shared memory.
__device__ __forceinline__ void warp_bitonic_smem(uint64_t* s, int S, int lane) {
    for (int k = 2; k <= S; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = lane; i < S; i += 32) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const uint64_t a = s[i], b = s[ixj];
                    if ((a > b) == ((i & k) == 0)) {
                        s[i] = b;
                        s[ixj] = a;
                    }
                }
            }
            __syncwarp();
        }
    }
}

__device__ __forceinline__ uint32_t warp_sort_u32(uint32_t v, int lane) {  // ascending, one value per lane
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const uint32_t o = __shfl_xor_sync(0xffffffffu, v, j);
            v = (((lane & k) == 0) == ((lane & j) == 0)) ? min(o, v) : max(o, v);
        }
    }
    return v;
}

// Ascending sort of a bitonic sequence of one value per lane.
__device__ __forceinline__ uint32_t warp_merge_u32(uint32_t v, int lane) {
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const uint32_t o = __shfl_xor_sync(0xffffffffu, v, j);
        v = (lane & j) == 0 ? min(o, v) : max(o, v);
    }
    return v;
}

// The K smallest of N values load(i) (order-preserving u32 images of the
// scores, counted with multiplicity; 0 < K <= 48, K < N), ascending into
// vals[0..K), by one warp.  Each lane keeps the two smallest values it reads
// (i = lane, lane + 32, ...).  The K-th smallest t of those (at most) 64 is
// at least the K-th smallest of all values (they are K of them; with N < 64
// they are all of them), so the values at or below t hold the K smallest:
// they are gathered and sorted.  Two passes over the values and a few warp
// sorts, against the radix refinement's histogram passes.  Returns the number
// gathered (>= K), or -1 if more than 64 (the caller then selects by radix
// refinement; at K 48 of 1024 random scores about 65 values fall at or below
// t).  vals: 64 words of the warp's own shared memory.  All 32 lanes call.
template <class Load>
__device__ int warp_small_kvals(Load load, int N, int K, uint32_t* vals) {
    const int lane = threadIdx.x & 31;
    uint32_t a = 0xffffffffu, b = 0xffffffffu;  // a <= b: the two smallest values of this lane
    for (int i0 = 0; i0 < N; i0 += 32 * TOPK_U) {
        uint32_t x[TOPK_U];
#pragma unroll
        for (int u = 0; u < TOPK_U; ++u) {
            const int i = i0 + 32 * u + lane;
            x[u] = i < N ? load(i) : 0xffffffffu;
        }
#pragma unroll
        for (int u = 0; u < TOPK_U; ++u) {
            b = min(b, max(a, x[u]));
            a = min(a, x[u]);
        }
    }
    // both sets sorted across the warp; against the reversed second, the
    // element-wise minima are the 32 smallest of the 64 and the maxima the
    // 32 largest, each a bitonic sequence
    const uint32_t A = warp_sort_u32(a, lane), B = warp_sort_u32(b, lane);
    const uint32_t Br = __shfl_sync(0xffffffffu, B, 31 - lane);
    const uint32_t v = warp_merge_u32(K <= 32 ? min(A, Br) : max(A, Br), lane);
    const uint32_t t = __shfl_sync(0xffffffffu, v, (K - 1) & 31);
    const uint32_t below = (1u << lane) - 1u;
    int n = 0;
    for (int i0 = 0; i0 < N; i0 += 32) {
        const int i = i0 + lane;
        const uint32_t x = i < N ? load(i) : 0xffffffffu;
        const bool in = i < N && x <= t;
        const uint32_t m = __ballot_sync(0xffffffffu, in);
        const int at = n + __popc(m & below);
        if (in && at < 64) vals[at] = x;
        n += __popc(m);
    }
    if (n > 64) return -1;
    __syncwarp();
    const uint32_t c0 = lane < n ? vals[lane] : 0xffffffffu, c1 = lane + 32 < n ? vals[lane + 32] : 0xffffffffu;
    const uint32_t S0 = warp_sort_u32(c0, lane);
    if (n <= 32) {
        __syncwarp();
        vals[lane] = S0;
    } else {
        const uint32_t S1r = __shfl_sync(0xffffffffu, warp_sort_u32(c1, lane), 31 - lane);
        const uint32_t lo = warp_merge_u32(min(S0, S1r), lane), hi = warp_merge_u32(max(S0, S1r), lane);
        __syncwarp();
        vals[lane] = lo;
        vals[lane + 32] = hi;
    }
    __syncwarp();
    return n;
}

// One warp per query (RSW_WARPS per CTA) for L <= RSW_MAX_L: the row of given
// scores is staged in the warp's shared memory and the P-th smallest given
// score s_P found by radix refinement over (score, list) keys.  Every list of
// the exact top P has a given score <= s_P + 2 err (P lists have given scores
// <= s_P, so the exact P-th score is at most s_P + err).  Those lists are
// re-scored exactly in FP32 (8 at a time, as in the re-rank) and the P best by
// (score, id) are sorted.  A query with more than RSW_CAND such lists is put on
// `redo` for k_rank_select.
constexpr int RSW_WARPS = 4;
constexpr int RSW_MAX_L = 2048;
constexpr int RSW_CAND = 128;

// A row of L scores into the warp's shared memory ss, with up to 8 16-byte
// loads per lane in flight (ss 16-byte aligned).
__device__ __forceinline__ void stage_row(const float* __restrict__ row, float* ss, int L, int lane) {
    if ((L & 3) == 0 && (reinterpret_cast<uintptr_t>(row) & 15) == 0) {
        const float4* r4 = reinterpret_cast<const float4*>(row);
        float4* s4 = reinterpret_cast<float4*>(ss);
        const int L4 = L >> 2;
        for (int c0 = 0; c0 < L4; c0 += 32 * 8) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int c = c0 + 32 * u + lane;
                v[u] = c < L4 ? __ldg(r4 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int c = c0 + 32 * u + lane;
                if (c < L4) s4[c] = v[u];
            }
        }
    } else {
        for (int c = lane; c < L; c += 32) ss[c] = row[c];
    }
    __syncwarp();
}

// The lists of given score <= tau (staged in ss) into ck, ascending; returns
// their number (only the first RSW_CAND are stored).  One warp.
__device__ __forceinline__ int collect_lists(const float* ss, int L, float tau, uint64_t* ck, int lane) {
    const uint32_t below = (1u << lane) - 1u;
    int n = 0;
    for (int c0 = 0; c0 < L; c0 += 32) {
        const int c = c0 + lane;
        const bool in = c < L && ss[c] <= tau;
        const uint32_t m = __ballot_sync(0xffffffffu, in);
        const int at = n + __popc(m & below);
        if (in && at < RSW_CAND) ck[at] = (uint64_t)(uint32_t)c;
        n += __popc(m);
    }
    return n;
}

// The n (<= RSW_CAND) lists in ck re-scored exactly in FP32 (8 at a time, as
// in the re-rank), sorted by (score, id); the P best into row q of probes
// (and score_out), -1 (+inf) past them up to Pmax.  One warp.
__device__ void exact_top_p(int64_t q, int n, int P, int Pmax, uint64_t* ck, const float* __restrict__ Q,
                            const float* __restrict__ Cc, int d, int spherical, int32_t* __restrict__ probes,
                            float* __restrict__ score_out, int lane) {
    __syncwarp();
    // exact FP32 scores, 8 lists at a time
    const float* qv = Q + q * d;
    const bool vec = (d & 3) == 0 && d <= 128;
    const int myrow = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
    for (int i0 = 0; i0 < n; i0 += 8) {
        float a[8];
        if (vec) {
            const bool inl = lane * 4 < d;
            float4 q4 = make_float4(0.f, 0.f, 0.f, 0.f);
            if (inl) q4 = make_float4(qv[lane * 4], qv[lane * 4 + 1], qv[lane * 4 + 2], qv[lane * 4 + 3]);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int c = i0 + u < n ? (int)(uint32_t)ck[i0 + u] : -1;
                const float4 cv = (c >= 0 && inl) ? __ldg(reinterpret_cast<const float4*>(Cc + (int64_t)c * d) + lane)
                                                  : make_float4(0.f, 0.f, 0.f, 0.f);
                if (spherical) {
                    a[u] = fmaf(q4.w, cv.w, fmaf(q4.z, cv.z, fmaf(q4.y, cv.y, q4.x * cv.x)));
                } else {
                    const float e0 = q4.x - cv.x, e1 = q4.y - cv.y, e2 = q4.z - cv.z, e3 = q4.w - cv.w;
                    a[u] = fmaf(e3, e3, fmaf(e2, e2, fmaf(e1, e1, e0 * e0)));
                }
            }
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int c = i0 + u < n ? (int)(uint32_t)ck[i0 + u] : -1;
                float acc = 0.f;
                if (c >= 0) {
                    for (int t = lane; t < d; t += 32) {
                        const float x = __ldg(Cc + (int64_t)c * d + t);
                        if (spherical) acc = fmaf(qv[t], x, acc);
                        else { const float e = qv[t] - x; acc = fmaf(e, e, acc); }
                    }
                }
                a[u] = acc;
            }
        }
        // halving exchange: lane ends with the sum of row myrow
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool up = lane & 16;
            const float send = up ? a[i] : a[i + 4], keep = up ? a[i + 4] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const bool up = lane & 8;
            const float send = up ? a[i] : a[i + 2], keep = up ? a[i + 2] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
        }
        {
            const bool up = lane & 4;
            const float send = up ? a[0] : a[1], keep = up ? a[1] : a[0];
            a[0] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
        }
        a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
        a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
        __syncwarp();
        const int i = i0 + myrow;
        if ((lane & 3) == 0 && i < n) {
            const uint32_t c = (uint32_t)ck[i];
            ck[i] = ((uint64_t)ordered_f32(spherical ? -a[0] : a[0]) << 32) | c;
        }
        __syncwarp();
    }
    // the P best in order
    if (n <= 32) {
        const uint64_t v = warp_sort_key(lane < n ? ck[lane] : KEY_NONE, lane);
        ck[lane] = v;
    } else {
        const int S = pow2_ceil(n);
        for (int i = n + lane; i < S; i += 32) ck[i] = KEY_NONE;
        __syncwarp();
        warp_bitonic_smem(ck, S, lane);
    }
    __syncwarp();
    for (int r = lane; r < Pmax; r += 32) {
        if (r < P && r < n) {
            probes[q * Pmax + r] = (int32_t)(ck[r] & 0xffffffffu);
            if (score_out) score_out[q * Pmax + r] = unordered_f32((uint32_t)(ck[r] >> 32));
        } else {
            probes[q * Pmax + r] = -1;
            if (score_out) score_out[q * Pmax + r] = INFINITY;
        }
    }
}


__global__ void __launch_bounds__(RSW_WARPS * 32) k_rank_select_w(const float* __restrict__ scores,
                                                                  const float* __restrict__ err,
                                                                  const float* __restrict__ Q,
                                                                  const float* __restrict__ Cc, int64_t nq, int d,
                                                                  int L, int spherical,
                                                                  const int32_t* __restrict__ nprobe_q, int Pfix,
                                                                  int Pmax, int32_t* __restrict__ probes,
                                                                  float* __restrict__ score_out,
                                                                  int32_t* __restrict__ redo,
                                                                  float* __restrict__ feat) {
    extern __shared__ uint64_t rsm[];  // RSW_WARPS x RSW_CAND keys, then RSW_WARPS x L scores
    __shared__ uint32_t hist[RSW_WARPS][256];
    __shared__ uint64_t bb[RSW_WARPS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t q = (int64_t)blockIdx.x * RSW_WARPS + w;
    if (q >= nq) return;
    uint64_t* ck = rsm + w * RSW_CAND;
    float* ss = reinterpret_cast<float*>(rsm + RSW_WARPS * RSW_CAND) + (size_t)w * L;
    int P = nprobe_q ? nprobe_q[q] : Pfix;
    P = P < 1 ? 1 : (P > Pmax ? Pmax : P);
    stage_row(scores + q * L, ss, L, lane);
    float tau = INFINITY;
    auto load = [&](int c) -> uint64_t { return ((uint64_t)ordered_f32(ss[c]) << 32) | (uint32_t)c; };
    auto load32 = [&](int c) -> uint32_t { return ordered_f32(ss[c]); };
    uint32_t* kv = reinterpret_cast<uint32_t*>(ck);  // the small selection's values (ck's first 64 words)
    if (feat) {
        // the K = max(P, FEAT_K) smallest given scores, sorted: the predictor's
        // distances (+ ||q||^2 for L2, which the score leaves out) and s_P
        const int K = min(max(P, FEAT_K), L);
        uint32_t fv, sP = 0u;  // this lane's distance, the P-th smallest (ordered images)
        if (K < L && K <= 48 && warp_small_kvals(load32, L, K, kv) >= 0) {
            fv = kv[lane];
            if (P < L) sP = kv[P - 1];
        } else {
            auto emit = [&](int i, uint64_t k) { ck[i] = k; };
            if (K < L) warp_topk(load, L, K, emit, hist[w], bb[w]);
            else for (int c = lane; c < L; c += 32) ck[c] = load(c);
            const int S = pow2_ceil(K);
            for (int i = K + lane; i < S; i += 32) ck[i] = KEY_NONE;
            __syncwarp();
            warp_bitonic_smem(ck, S, lane);
            fv = (uint32_t)(ck[lane] >> 32);
            if (P < L) sP = (uint32_t)(ck[P - 1] >> 32);
        }
        float qq = 0.f;
        if (!spherical) {
            for (int t = lane; t < d; t += 32) qq = fmaf(Q[q * d + t], Q[q * d + t], qq);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) qq += __shfl_xor_sync(0xffffffffu, qq, o);
        }
        feat[q * FEAT_K + lane] = unordered_f32(fv) + qq;
        if (P < L) tau = unordered_f32(sP) + (err ? 2.f * err[q] : 0.f);
        __syncwarp();
    } else if (P < L) {
        uint32_t sP;
        if (P <= 48 && warp_small_kvals(load32, L, P, kv) >= 0) {
            sP = kv[P - 1];
            __syncwarp();  // ck is reused for the lists below
        } else {
            auto none = [](int, uint64_t) {};
            sP = (uint32_t)(warp_topk(load, L, P, none, hist[w], bb[w]) >> 32);
        }
        tau = unordered_f32(sP) + (err ? 2.f * err[q] : 0.f);
    }
    // the lists that can still be among the P best
    const int n = collect_lists(ss, L, tau, ck, lane);
    if (n > RSW_CAND) {
        if (lane == 0) redo[1 + atomicAdd(&redo[0], 1)] = (int32_t)q;
        return;
    }
    exact_top_p(q, n, P, Pmax, ck, Q, Cc, d, spherical, probes, score_out, lane);
}

// The adaptive search's ranking in one kernel (Sec. 4.2.1-4.2.2, Eq. 2), a
// warp per query, persistent CTAs of RH_WARPS warps: the FEAT_K smallest
// given scores (the predictor's distances, as k_feat_scores), the features,
// network and settings (as k_features and k_mlp_infer, the same operations
// in the same order: bit for bit their settings), then the exact ranking of
// the predicted nprobe lists (as k_rank_select_w).  The BF16-rounded hidden
// weights are staged once per CTA as BF16 pairs [input f][units 2l, 2l + 1]
// (rows of 33 words: the transposing stores fall in distinct banks; BF16
// keeps the CTA small enough for three per SM), so that lane l accumulates
// units 2l and 2l + 1 from one 4-byte load and one packed FMA per input
// (each half the scalar FMA's result); the inputs are broadcast by shuffles.
// Writes nprobe_out / rerank_out; a query with more than RSW_CAND lists
// inside its bound goes on `redo`.
constexpr int RH_WARPS = 8;
constexpr int RH_WLD = 33;  // words per input row of the staged weight pairs
constexpr size_t rh_head_bytes() { return sizeof(uint32_t) * 2 * MLP_F * RH_WLD + sizeof(float) * (4 * MLP_H + 4); }

// The two BF16 values of a staged pair as FP32 (exact).
__device__ __forceinline__ float2 bf16_pair(uint32_t pk) {
    return make_float2(__uint_as_float(pk << 16), __uint_as_float(pk & 0xffff0000u));
}
constexpr size_t rh_warp_bytes(int L) {
    return sizeof(uint64_t) * (RSW_CAND + 32) + sizeof(uint32_t) * 256 + sizeof(float) * (size_t)((L + 3) & ~3);
}

__global__ void __launch_bounds__(RH_WARPS * 32) k_rank_head_w(const float* __restrict__ scores,
                                                               const float* __restrict__ err,
                                                               const float* __restrict__ Q,
                                                               const float* __restrict__ Cc, int64_t nq, int d, int L,
                                                               int spherical, const float* __restrict__ wm,
                                                               ksc_adaptive_params prm, int Pmax,
                                                               int32_t* __restrict__ probes,
                                                               int32_t* __restrict__ redo,
                                                               int32_t* __restrict__ nprobe_out,
                                                               int32_t* __restrict__ rerank_out) {
    extern __shared__ uint64_t hsm[];
    uint32_t* WB1 = reinterpret_cast<uint32_t*>(hsm);
    uint32_t* WB2 = WB1 + MLP_F * RH_WLD;
    float* hb1 = reinterpret_cast<float*>(WB2 + MLP_H * RH_WLD);
    float* hb2 = hb1 + MLP_H;
    float* hW3 = hb2 + MLP_H;  // [f][o]
    float* hb3 = hW3 + MLP_O * MLP_H;
    unsigned char* wbase = reinterpret_cast<unsigned char*>(hsm) + rh_head_bytes();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned char* mine = wbase + (size_t)w * rh_warp_bytes(L);
    uint64_t* ck = reinterpret_cast<uint64_t*>(mine);
    uint64_t* bb = ck + RSW_CAND;
    uint32_t* hist = reinterpret_cast<uint32_t*>(bb + 32);
    float* ss = reinterpret_cast<float*>(hist + 256);
    uint32_t* kv = reinterpret_cast<uint32_t*>(ck);
    {
        // hidden weights: coalesced 16-byte loads of rows a, stored transposed
        // as BF16 (units 2l, 2l + 1 of input f in word f * RH_WLD + l)
        const MlpW G = mlp_views(wm);
        constexpr int V = MLP_H * MLP_F / 4 / (RH_WARPS * 32);
        float4 v1[V], v2[V];
#pragma unroll
        for (int u = 0; u < V; ++u) {
            v1[u] = __ldg(reinterpret_cast<const float4*>(G.W1) + threadIdx.x + RH_WARPS * 32 * u);
            v2[u] = __ldg(reinterpret_cast<const float4*>(G.W2) + threadIdx.x + RH_WARPS * 32 * u);  // (MLP_F == MLP_H)
        }
#pragma unroll
        for (int u = 0; u < V; ++u) {
            const int e4 = threadIdx.x + RH_WARPS * 32 * u, a = e4 >> 4, f = 4 * (e4 & 15);
            const float x1[4] = {v1[u].x, v1[u].y, v1[u].z, v1[u].w}, x2[4] = {v2[u].x, v2[u].y, v2[u].z, v2[u].w};
            __nv_bfloat16* B1 = reinterpret_cast<__nv_bfloat16*>(WB1);
            __nv_bfloat16* B2 = reinterpret_cast<__nv_bfloat16*>(WB2);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                B1[2 * (f + k) * RH_WLD + a] = __float2bfloat16_rn(x1[k]);
                B2[2 * (f + k) * RH_WLD + a] = __float2bfloat16_rn(x2[k]);
            }
        }
        for (int e = threadIdx.x; e < MLP_H; e += blockDim.x) {
            hb1[e] = bf(G.b1[e]);
            hb2[e] = bf(G.b2[e]);
        }
        for (int e = threadIdx.x; e < MLP_O * MLP_H; e += blockDim.x) {  // interleaved: [f][o]
            const int o = e / MLP_H, f = e - o * MLP_H;
            hW3[2 * f + o] = bf(G.W3[e]);
        }
        if (threadIdx.x < MLP_O) hb3[threadIdx.x] = bf(G.b3[threadIdx.x]);
    }
    __syncthreads();
    auto load = [&](int c) -> uint64_t { return ((uint64_t)ordered_f32(ss[c]) << 32) | (uint32_t)c; };
    auto load32 = [&](int c) -> uint32_t { return ordered_f32(ss[c]); };
    for (int64_t q = (int64_t)blockIdx.x * RH_WARPS + w; q < nq; q += (int64_t)gridDim.x * RH_WARPS) {
        stage_row(scores + q * L, ss, L, lane);
        // the FEAT_K smallest scores, ascending (order-preserving images)
        uint32_t fv;
        if (L > FEAT_K && warp_small_kvals(load32, L, FEAT_K, kv) >= 0) {
            fv = kv[lane];
        } else {
            auto emit = [&](int i, uint64_t k) { ck[i] = k; };
            if (L > FEAT_K) warp_topk(load, L, FEAT_K, emit, hist, bb);
            else ck[lane] = load(lane);
            __syncwarp();
            fv = (uint32_t)(warp_sort_key(ck[lane], lane) >> 32);
        }
        __syncwarp();
        float qq = 0.f;
        if (!spherical) {
            for (int t = lane; t < d; t += 32) qq = fmaf(Q[q * d + t], Q[q * d + t], qq);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) qq += __shfl_xor_sync(0xffffffffu, qq, o);
        }
        // features: lane i holds d_i / mean and d_1 / d_i (BF16)
        const float u = fmaxf(feat_dist(unordered_f32(fv) + qq, spherical), 0.f);
        float mean = 0.f;
#pragma unroll
        for (int i = 0; i < MLP_FEAT_K; ++i) mean += __shfl_sync(0xffffffffu, u, i);
        mean = mean / MLP_FEAT_K + 1e-12f;
        const float d1 = __shfl_sync(0xffffffffu, u, 0) + 1e-12f, di = u + 1e-12f;
        const float xa = bf(di / mean), xb = bf(d1 / di);
        // hidden layers: lane l computes units 2l and 2l + 1
        float2 acc = *reinterpret_cast<const float2*>(hb1 + 2 * lane);
#pragma unroll 8
        for (int f = 0; f < MLP_F; ++f) {
            const float x = __shfl_sync(0xffffffffu, f < MLP_FEAT_K ? xa : xb, f & 31);
            acc = f2_fma(make_float2(x, x), bf16_pair(WB1[f * RH_WLD + lane]), acc);
        }
        const float h0 = bf(acc.x > 0.f ? acc.x : 0.f), h1 = bf(acc.y > 0.f ? acc.y : 0.f);
        acc = *reinterpret_cast<const float2*>(hb2 + 2 * lane);
#pragma unroll 8
        for (int f = 0; f < MLP_H; ++f) {
            const float x = __shfl_sync(0xffffffffu, (f & 1) ? h1 : h0, f >> 1);
            acc = f2_fma(make_float2(x, x), bf16_pair(WB2[f * RH_WLD + lane]), acc);
        }
        const float g0 = bf(acc.x > 0.f ? acc.x : 0.f), g1 = bf(acc.y > 0.f ? acc.y : 0.f);
        float2 z = make_float2(hb3[0], hb3[1]);
#pragma unroll 8
        for (int f = 0; f < MLP_H; ++f) {
            const float x = __shfl_sync(0xffffffffu, (f & 1) ? g1 : g0, f >> 1);
            z = f2_fma(make_float2(x, x), *reinterpret_cast<const float2*>(hW3 + 2 * f), z);
        }
        const float p0 = 1.f / (1.f + expf(-z.x)), p1 = 1.f / (1.f + expf(-z.y));
        const int np = prm.regression ? regmap(p0, prm.pmin, prm.pmax, prm.p0, prm.p1)
                                      : eq2(p0, prm.pmin, prm.pmax, prm.p0, prm.p1);
        const int rr = prm.regression ? regmap(p1, prm.rmin, prm.rmax, prm.r0, prm.r1)
                                      : eq2(p1, prm.rmin, prm.rmax, prm.r0, prm.r1);
        if (lane == 0) {
            nprobe_out[q] = np;
            rerank_out[q] = rr;
        }
        // the exact ranking of the predicted lists
        const int P = np < 1 ? 1 : (np > Pmax ? Pmax : np);
        float tau = INFINITY;
        if (P < L) {
            uint32_t sP;
            if (P <= FEAT_K) {
                sP = __shfl_sync(0xffffffffu, fv, P - 1);
            } else if (P <= 48 && warp_small_kvals(load32, L, P, kv) >= 0) {
                sP = kv[P - 1];
                __syncwarp();
            } else {
                auto none = [](int, uint64_t) {};
                sP = (uint32_t)(warp_topk(load, L, P, none, hist, bb) >> 32);
            }
            tau = unordered_f32(sP) + (err ? 2.f * err[q] : 0.f);
        }
        const int n = collect_lists(ss, L, tau, ck, lane);
        if (n > RSW_CAND) {
            if (lane == 0) redo[1 + atomicAdd(&redo[0], 1)] = (int32_t)q;
        } else {
            exact_top_p(q, n, P, Pmax, ck, Q, Cc, d, spherical, probes, nullptr, lane);
        }
        __syncwarp();  // ss and ck are reused by the warp's next query
    }
}

// The predictor's distances (Sec. 4.2.1): per query the FEAT_K smallest list
// scores, ascending, from the given score matrix (the tensor-core scores,
// within their bound of the exact ones); for L2 the query's squared norm,
// which the ranking score leaves out, is added back.  One warp per query.
__global__ void __launch_bounds__(256) k_feat_scores(const float* __restrict__ scores, const float* __restrict__ Q,
                                                     int d, int spherical, int64_t nq, int L,
                                                     float* __restrict__ out) {
    __shared__ uint32_t hist[8][256];
    __shared__ uint64_t bb[8][32];
    __shared__ uint64_t kk[8][FEAT_K];
    __shared__ uint32_t kv[8][64];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t q = (int64_t)blockIdx.x * 8 + w;
    if (q >= nq) return;
    const float* row = scores + q * L;
    auto load = [&](int c) -> uint64_t { return ((uint64_t)ordered_f32(row[c]) << 32) | (uint32_t)c; };
    auto load32 = [&](int c) -> uint32_t { return ordered_f32(row[c]); };
    auto emit = [&](int i, uint64_t k) { kk[w][i] = k; };
    uint32_t v;  // this lane's distance (ordered image) in ascending order
    if (L > FEAT_K && warp_small_kvals(load32, L, FEAT_K, kv[w]) >= 0) {
        v = kv[w][lane];
    } else {
        if (L > FEAT_K) warp_topk(load, L, FEAT_K, emit, hist[w], bb[w]);
        else kk[w][lane] = load(lane);  // L == FEAT_K (the predictor needs 32 lists)
        __syncwarp();
        v = (uint32_t)(warp_sort_key(kk[w][lane], lane) >> 32);
    }
    float qq = 0.f;
    if (!spherical) {
        for (int t = lane; t < d; t += 32) qq = fmaf(Q[q * d + t], Q[q * d + t], qq);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) qq += __shfl_xor_sync(0xffffffffu, qq, o);
    }
    out[q * FEAT_K + lane] = unordered_f32(v) + qq;
}

// ------------------------------------------------------------------ a2: quantised LUTs (rule: lut.cuh)

// Two-pass tables when a query's tables do not fit one CTA's shared memory
// (many probes): a warp per item (query, probe rank), lane l computing the
// rows j = l, l + 32, ... (M <= KSC_MAX_M), no block barrier.  Pass 1: the
// largest row range of each query, R_q (a warp maximum per item, then one
// global atomic maximum; R >= 0, so the bit order is the value order).
constexpr int LUT_WARPS = 8;

template <int DS>
__global__ void __launch_bounds__(LUT_WARPS * 32) k_lut_range(LutArgs A, uint32_t* __restrict__ range_bits) {
    extern __shared__ __align__(16) float cbs[];
    stage_codebook(A, cbs);
    const int ld = cb_ld(A.dsub);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t n0;
    const int64_t items = lut_items(A, &n0);
    for (int64_t i = (int64_t)blockIdx.x * LUT_WARPS + warp; i < items; i += (int64_t)gridDim.x * LUT_WARPS) {
        const int64_t item = lut_item(A, i, n0);
        const int64_t q = item / A.Pmax;
        const int r = (int)(item - q * A.Pmax);
        const int p = A.probes[item];
        if (r >= probes_of(A, q) || p < 0 || p >= A.L) continue;  // invalid probe ids are skipped (warp-uniform)
        float R = 0.f;
        for (int j = lane; j < A.M; j += 32) {
            float T[PQ_K];
            row_table<DS>(A.dsub, A.ip, A.Q + q * A.d + j * A.dsub, A.c_mean + (int64_t)p * A.d + j * A.dsub,
                          cbs + j * ld, T);
            float mn = T[0], mx = T[0];
#pragma unroll
            for (int e = 1; e < PQ_K; ++e) { mn = fminf(mn, T[e]); mx = fmaxf(mx, T[e]); }
            R = fmaxf(R, __fsub_rn(mx, mn));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) R = fmaxf(R, __shfl_xor_sync(0xffffffffu, R, o));
        if (lane == 0 && R > 0.f) atomicMax(&range_bits[q], __float_as_uint(R));
    }
}

// Pass 2: u8 tables Q = min(255, floor((T - m_j) a + 1/2)), a = 255 / R_q,
// then the item's bias from its row minima (summed in ascending j by lane 0,
// the FP32 rule's order).
template <int DS>
__global__ void __launch_bounds__(LUT_WARPS * 32) k_lut_quant(LutArgs A, const uint32_t* __restrict__ range_bits,
                                                              uint8_t* __restrict__ lut, int32_t* __restrict__ bias,
                                                              float* __restrict__ scale) {
    extern __shared__ __align__(16) float cbs[];
    __shared__ float s_min[LUT_WARPS][KSC_MAX_M];
    stage_codebook(A, cbs);
    const int ld = cb_ld(A.dsub);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t n0;
    const int64_t items = lut_items(A, &n0);
    for (int64_t i = (int64_t)blockIdx.x * LUT_WARPS + warp; i < items; i += (int64_t)gridDim.x * LUT_WARPS) {
        const int64_t item = lut_item(A, i, n0);
        const int64_t q = item / A.Pmax;
        const int r = (int)(item - q * A.Pmax);
        const int p = A.probes[item];
        if (r >= probes_of(A, q) || p < 0 || p >= A.L) continue;  // warp-uniform
        const float Rq = __uint_as_float(range_bits[q]);
        const float a = (Rq == 0.f) ? 1.f : __fdiv_rn(255.f, Rq);
        for (int j = lane; j < A.M; j += 32) {
            float T[PQ_K];
            row_table<DS>(A.dsub, A.ip, A.Q + q * A.d + j * A.dsub, A.c_mean + (int64_t)p * A.d + j * A.dsub,
                          cbs + j * ld, T);
            float mn = T[0];
#pragma unroll
            for (int e = 1; e < PQ_K; ++e) mn = fminf(mn, T[e]);
            reinterpret_cast<uint4*>(lut + item * (int64_t)A.M * PQ_K)[j] =
                make_uint4(quant4(T, mn, a), quant4(T + 4, mn, a), quant4(T + 8, mn, a), quant4(T + 12, mn, a));
            s_min[warp][j] = mn;
        }
        __syncwarp();
        if (lane == 0) {
            bias[item] = lut_bias(A, A.Q + q * A.d, A.c_mean + (int64_t)p * A.d, s_min[warp], a);
            if (r == 0) scale[q] = a;
        }
        __syncwarp();  // s_min is read before the warp's next item overwrites it
    }
}

// Persistent CTAs, one query at a time, when all of a query's tables fit in
// shared memory: the codebook is staged once per CTA; the FP32 tables of the
// query's P_q probes are computed once, their largest range gives the scale,
// and they are quantised from shared memory (same FP32 rule, same results as
// the two-pass kernels above).  Rows of 16 entries sit 20 floats apart (16-byte
// aligned; 8 consecutive rows of a 128-bit access fall in distinct banks).  A
// thread walks rows (r, j) = (probe rank, subspace) by a fixed step, no
// division.  Two barriers per query: the next query's vector is loaded into
// the other of two buffers while this one is quantised.
constexpr int LUT_TROW = 20;

template <int DS>
__global__ void __launch_bounds__(512) k_lut_fused(LutArgs A, int Pb, int Pm, uint8_t* __restrict__ lut,
                                                   int32_t* __restrict__ bias, float* __restrict__ scale) {
    extern __shared__ __align__(16) float fsm[];
    const int M = A.M;
    const int ld = cb_ld(A.dsub);
    const int dpad = (A.d + 3) & ~3;
    float* cbs = fsm;                                                  // M x ld
    float* T = cbs + (((size_t)M * ld + 3) & ~(size_t)3);              // Pb x M rows, LUT_TROW apart
    float* mins = T + (size_t)Pb * M * LUT_TROW;                       // Pm x M
    float* qsb = mins + (((size_t)Pm * M + 3) & ~(size_t)3);           // 2 x dpad
    int32_t* prb = reinterpret_cast<int32_t*>(qsb + 2 * dpad);         // 2 x Pm probe ids
    __shared__ uint32_t s_rbits[2];
    const int r0 = threadIdx.x / M, j0 = threadIdx.x - r0 * M;         // first row of this thread
    const int dr = blockDim.x / M, dj = blockDim.x - dr * M;           // step of blockDim.x rows
    int64_t q = blockIdx.x;
    if (q < A.nq) {
        for (int t = threadIdx.x; t < A.d; t += blockDim.x) qsb[t] = A.Q[q * A.d + t];
        for (int r = threadIdx.x; r < Pm; r += blockDim.x) prb[r] = A.probes[q * A.Pmax + r];
    }
    if (threadIdx.x == 0) s_rbits[0] = 0u;
    stage_codebook(A, cbs);  // ends with __syncthreads
    for (int buf = 0; q < A.nq; q += gridDim.x, buf ^= 1) {
        const float* qs = qsb + buf * dpad;
        // the tables of the first Pb probes are kept for the quantisation
        // pass; those of later probes (a query with more) are computed again
        const int P = min(probes_of(A, q), Pm);
        const int nstored = Pb * M;
        const int32_t* pr = prb + buf * Pm;  // the query's probes, staged in shared memory
        float R = 0.f;
        {
            int r = r0, j = j0;
            for (int row = threadIdx.x; row < P * M; row += blockDim.x) {
                const int p = pr[r];
                float* Tr = T + (size_t)row * LUT_TROW;
                const bool stored = row < nstored;
                if (p < 0 || p >= A.L) {
                    if (stored)
#pragma unroll
                        for (int i = 0; i < PQ_K; i += 4) *reinterpret_cast<float4*>(Tr + i) = make_float4(0.f, 0.f, 0.f, 0.f);
                    mins[row] = 0.f;
                } else {
                    float Tv[PQ_K];
                    row_table<DS>(A.dsub, A.ip, qs + j * A.dsub, A.c_mean + (int64_t)p * A.d + j * A.dsub,
                                  cbs + j * ld, Tv);
                    float mn = Tv[0], mx = Tv[0];
#pragma unroll
                    for (int i = 1; i < PQ_K; ++i) {
                        mn = fminf(mn, Tv[i]);
                        mx = fmaxf(mx, Tv[i]);
                    }
                    if (stored)
#pragma unroll
                        for (int i = 0; i < PQ_K; i += 4)
                            *reinterpret_cast<float4*>(Tr + i) = make_float4(Tv[i], Tv[i + 1], Tv[i + 2], Tv[i + 3]);
                    mins[row] = mn;
                    R = fmaxf(R, __fsub_rn(mx, mn));
                }
                j += dj;
                r += dr;
                if (j >= M) {
                    j -= M;
                    ++r;
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) R = fmaxf(R, __shfl_xor_sync(0xffffffffu, R, o));
        if ((threadIdx.x & 31) == 0) atomicMax(&s_rbits[buf], __float_as_uint(R));
        __syncthreads();
        const float Rq = __uint_as_float(s_rbits[buf]);
        const float a = (Rq == 0.f) ? 1.f : __fdiv_rn(255.f, Rq);
        // the next query's vector into the other buffer (its last readers
        // passed the barrier above)
        const int64_t qn = q + gridDim.x;
        float* qs_next = qsb + (buf ^ 1) * dpad;
        const bool pre = qn < A.nq && threadIdx.x < A.d;
        const float nx = pre ? A.Q[qn * A.d + threadIdx.x] : 0.f;
        if (threadIdx.x == 0) s_rbits[buf ^ 1] = 0u;
        {
            int r = r0, j = j0;
            for (int row = threadIdx.x; row < P * M; row += blockDim.x) {
                const float mn = mins[row];
                float Tv[PQ_K];
                bool ok = true;
                if (row < nstored) {
                    const float* Tr = T + (size_t)row * LUT_TROW;
#pragma unroll
                    for (int i = 0; i < PQ_K; i += 4) {
                        const float4 v = *reinterpret_cast<const float4*>(Tr + i);
                        Tv[i] = v.x;
                        Tv[i + 1] = v.y;
                        Tv[i + 2] = v.z;
                        Tv[i + 3] = v.w;
                    }
                } else {
                    const int p = pr[r];
                    ok = p >= 0 && p < A.L;
                    if (ok)
                        row_table<DS>(A.dsub, A.ip, qs + j * A.dsub, A.c_mean + (int64_t)p * A.d + j * A.dsub,
                                      cbs + j * ld, Tv);
                }
                if (ok)
                    reinterpret_cast<uint4*>(lut + (q * A.Pmax + r) * (int64_t)M * PQ_K)[j] = make_uint4(
                        quant4(Tv, mn, a), quant4(Tv + 4, mn, a), quant4(Tv + 8, mn, a), quant4(Tv + 12, mn, a));
                j += dj;
                r += dr;
                if (j >= M) {
                    j -= M;
                    ++r;
                }
            }
        }
        // biases by the last threads (those with the fewest rows above)
        for (int r = blockDim.x - 1 - threadIdx.x; r < P; r += blockDim.x) {
            const int p = pr[r];
            if (p < 0 || p >= A.L) continue;
            bias[q * A.Pmax + r] = lut_bias(A, qs, A.c_mean + (int64_t)p * A.d, mins + r * M, a);
        }
        if (threadIdx.x == 0) scale[q] = a;
        if (pre) qs_next[threadIdx.x] = nx;
        if (qn < A.nq) {
            for (int t = threadIdx.x + blockDim.x; t < A.d; t += blockDim.x) qs_next[t] = A.Q[qn * A.d + t];
            for (int r = threadIdx.x; r < Pm; r += blockDim.x) prb[(buf ^ 1) * Pm + r] = A.probes[qn * A.Pmax + r];
        }
        __syncthreads();  // the next query reuses the shared tables
    }
}

static size_t lut_fused_smem(int M, int dsub, int d, int Pb, int Pm) {
    return sizeof(float) * ((((size_t)M * cb_ld(dsub) + 3) & ~(size_t)3) + (size_t)Pb * M * LUT_TROW +
                            (((size_t)Pm * M + 3) & ~(size_t)3) + 2 * (((size_t)d + 3) & ~(size_t)3)) +
           sizeof(int32_t) * 2 * (size_t)Pm;
}

// The fixed row width of the tables (0: any): vector loads of the rows need
// the query matrix aligned to them (d is a multiple of dsub; the fused kernel
// reads the query from shared memory).
static int lut_width(const LutArgs& A, bool from_shared) {
    const uintptr_t q = from_shared ? 0 : reinterpret_cast<uintptr_t>(A.Q);
    if (A.dsub == 2 && (q & 7) == 0) return 2;
    if (A.dsub == 4 && (q & 15) == 0) return 4;
    return 0;
}

static int launch_luts(const LutArgs& A, uint32_t* rb, uint8_t* lut, int32_t* bias, float* scale, cudaStream_t st);

// ------------------------------------------------------------------ candidate-key selection
// The need smallest keys of distance word h among keys[0..N) (the others
// mapped above every key, uniquely by index), into out[0..need) unless out
// is null; returns the need-th.  The tie case of warp_topk_hi.
__device__ __forceinline__ uint64_t warp_topk_tied(const uint64_t* __restrict__ keys, int N, int need, uint32_t h,
                                                uint64_t* out, uint32_t* hist, uint64_t* bb) {
    auto load_t = [&](int i) -> uint64_t {
        const uint64_t k = keys[i];
        return (uint32_t)(k >> 32) == h ? k : ((0xffffffffull << 32) | (uint32_t)i);
    };
    auto emit_t = [&](int i, uint64_t k) {
        if (out) out[i] = k;
    };
    return warp_topk(load_t, N, need, emit_t, hist, bb);
}

// The K smallest (0 < K < N) of N unique candidate keys keys[0..N) (high word:
// the integer distance + 2^31, below 2^32 - 1; low word: the vector id), by
// one warp, as warp_topk but with the range, histogram and emission decided
// on the keys' high words alone (32-bit loads and compares: the distance
// range always spans more than the id bits matter for) until the K-th key's
// bin holds at most 32 keys, which are sorted on their full 64 bits.  A bin
// narrowed to a single distance with more than 32 keys in it (ties) hands the
// rest to warp_topk over those keys.  Writes the K smallest to dst[0..K) in
// no particular order (nothing if dst is null) and returns the K-th.
__device__ uint64_t warp_topk_hi(const uint64_t* __restrict__ keys, int N, int K, uint64_t* dst, uint32_t* hist,
                                 uint64_t* bb) {
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    const uint32_t* hw = reinterpret_cast<const uint32_t*>(keys) + 1;  // key i's high word at hw[2 i]
    uint32_t lo = 0xffffffffu, hi = 0u;
    for (int i0 = 0; i0 < N; i0 += 32 * TOPK_U) {
        uint32_t h[TOPK_U];
#pragma unroll
        for (int u = 0; u < TOPK_U; ++u) {
            const int i = i0 + 32 * u + lane;
            h[u] = i < N ? hw[2 * i] : 0u;
        }
#pragma unroll
        for (int u = 0; u < TOPK_U; ++u)
            if (i0 + 32 * u + lane < N) {
                lo = min(lo, h[u]);
                hi = max(hi, h[u]);
            }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    int out = 0, need = K;
    while (lo < hi) {
        const int shift = bin_shift(hi - lo);
        for (int b = lane; b < 256; b += 32) hist[b] = 0u;
        __syncwarp();
        for (int i0 = 0; i0 < N; i0 += 32 * TOPK_U) {
            uint32_t h[TOPK_U];
#pragma unroll
            for (int u = 0; u < TOPK_U; ++u) {
                const int i = i0 + 32 * u + lane;
                h[u] = i < N ? hw[2 * i] : 0xffffffffu;
            }
#pragma unroll
            for (int u = 0; u < TOPK_U; ++u)
                if (i0 + 32 * u + lane < N && h[u] >= lo && h[u] <= hi) atomicAdd(&hist[(h[u] - lo) >> shift], 1u);
        }
        __syncwarp();
        uint32_t c[8], local = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            c[j] = hist[8 * lane + j];
            local += c[j];
        }
        uint32_t incl = local;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t excl = incl - local;
        int B = -1, lt = 0, inB = 0;
        if (excl < (uint32_t)need && (uint32_t)need <= incl) {
            uint32_t acc = excl;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (B < 0 && acc + c[j] >= (uint32_t)need) {
                    B = 8 * lane + j;
                    lt = (int)acc;
                    inB = (int)c[j];
                }
                acc += c[j];
            }
        }
        const int owner = __ffs(__ballot_sync(0xffffffffu, B >= 0)) - 1;
        B = __shfl_sync(0xffffffffu, B, owner);
        lt = __shfl_sync(0xffffffffu, lt, owner);  // keys of the range below bin B
        inB = __shfl_sync(0xffffffffu, inB, owner);
        const uint32_t blo = lo + ((uint32_t)B << shift);
        const uint32_t bhi = (hi - blo < (1u << shift)) ? hi : blo + ((1u << shift) - 1u);
        const bool last = inB <= 32;
        int nb = 0;
        for (int i0 = 0; i0 < N; i0 += 32 * TOPK_U) {
            uint32_t h[TOPK_U];
#pragma unroll
            for (int u = 0; u < TOPK_U; ++u) {
                const int i = i0 + 32 * u + lane;
                h[u] = i < N ? hw[2 * i] : 0xffffffffu;
            }
#pragma unroll
            for (int u = 0; u < TOPK_U; ++u) {
                const int i = i0 + 32 * u + lane;
                const bool e = i < N && h[u] >= lo && h[u] < blo;
                const bool g = last && i < N && h[u] >= blo && h[u] <= bhi;
                const uint32_t me = __ballot_sync(0xffffffffu, e), mg = __ballot_sync(0xffffffffu, g);
                if (e && dst) dst[out + __popc(me & below)] = keys[i];
                if (g) bb[nb + __popc(mg & below)] = keys[i];
                out += __popc(me);
                nb += __popc(mg);
            }
        }
        need -= lt;
        if (last) {
            __syncwarp();
            const uint64_t v = warp_sort_key(lane < inB ? bb[lane] : KEY_NONE, lane);
            if (lane < need && dst) dst[out + lane] = v;
            const uint64_t kth = __shfl_sync(0xffffffffu, v, need - 1);
            __syncwarp();
            return kth;
        }
        lo = blo;
        hi = bhi;
        __syncwarp();
    }
    // one distance left with more keys than the sort takes: the need smallest
    // of its keys by their ids
    return warp_topk_tied(keys, N, need, lo, dst ? dst + out : nullptr, hist, bb);
}

// The K smallest (0 < K < n) of n unique keys (block_topk's rules), by a CTA of NT
// threads: up to NT U keys are held in registers, read once, and emit may then
// overwrite them; more (or U = 0) are read again in each pass.
template <int NT, int U, class Emit>
__device__ __forceinline__ uint64_t cta_topk(const uint64_t* keys, int n, int K, Emit emit, uint32_t* hist,
                                             uint64_t* bb) {
    if constexpr (U > 0) {
        if (n <= NT * U) {
            uint64_t kk[U];
#pragma unroll
            for (int u = 0; u < U; ++u) kk[u] = (int)threadIdx.x + u * NT < n ? keys[threadIdx.x + u * NT] : KEY_NONE;
            auto each = [&](auto f) {
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (u * NT < n) f((int)threadIdx.x + u * NT < n, kk[u]);
            };
            return block_topk_each(each, K, emit, hist, bb);
        }
    }
    return block_topk([&](int i) -> uint64_t { return keys[i]; }, n, K, emit, hist, bb);
}

// ------------------------------------------------------------------ threshold
// Per query, after the scan of its nearest list(s) with no filter: the R-th
// smallest of the keys found so far bounds the R-th smallest key of the whole
// search from above (any subset with at least R members gives such a bound);
// the scan of the remaining lists keeps only keys at or below it.  Fewer than
// R keys: no bound (all ones).  One warp per query.  Nothing above the R-th
// key can enter the final R, so the store keeps only the R keys at or below it
// (gathered in `scratch`, a row of Rmax keys per query, then copied back),
// unless it overflowed (the final select then redoes the query).
constexpr int SW_WARPS = 8;        // queries per CTA of the warp selection kernels
constexpr int SW_MAX_KEYS = 2048;  // expected keys per query up to which a warp selects ...
// ... in batches that fill the GPU; above SW_CTA_KEYS a CTA of 128 threads with its
// keys in registers, in batches that do not give every SM SW_CTA_NQ warps.  A warp
// reads its keys from L2 in each of three passes and more, a CTA once, at the cost
// of some nine barriers: the search by warps / CTAs in us at R 400 (3001 queries)
// 547 / 498, the hybrid search with 1560 near keys 732 / 705, at R 200 (10,000
// queries) 904 / 951; at R 300 to 512 and nprobe 2 to 48 on three index shapes 3 to 12%
// faster by CTAs with 1216 queries, 0 to 6% with 3000, 0 to 4% slower with 8000 (500k
// x 64, R 400, nprobe 8: 678 / 707).
constexpr int SW_CTA_KEYS = 1024, SW_CTA_NQ = 32;
static bool select_by_warp(int64_t nq, double keys) {
    return warp_per_query(nq) && keys <= SW_MAX_KEYS && (keys <= SW_CTA_KEYS || nq >= SW_CTA_NQ * (int64_t)num_sms());
}

__global__ void __launch_bounds__(SW_WARPS * 32) k_threshold(ScanArgs A, int Rmax, int32_t* __restrict__ cnt,
                                                             uint64_t* __restrict__ cand, int cap,
                                                             uint64_t* __restrict__ scratch,
                                                             uint64_t* __restrict__ thr) {
    __shared__ uint32_t hist[SW_WARPS][256];
    __shared__ uint64_t bb[SW_WARPS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t q = (int64_t)blockIdx.x * SW_WARPS + w;
    if (q >= A.nq) return;
    const int R = rerank_of(A.rerank_q, A.Rfix, A.Rmin, Rmax, q);
    const int n0 = cnt[q];
    const int n = min(n0, cap);  // an overflowed store still bounds the R-th key
    const bool ovf = n0 > cap;
    uint64_t* cq = cand + q * cap;
    uint64_t t = KEY_NONE;
    if (n == R) {
        uint64_t m = 0ull;
        for (int i = lane; i < n; i += 32) m = cq[i] > m ? cq[i] : m;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const uint64_t y = __shfl_xor_sync(0xffffffffu, m, o);
            m = y > m ? y : m;
        }
        t = m;
    } else if (n > R) {
        uint64_t* sq = scratch + q * Rmax;
        t = warp_topk_hi(cq, n, R, ovf ? nullptr : sq, hist[w], bb[w]);
        if (!ovf) {
            __syncwarp();
            for (int i = lane; i < R; i += 32) cq[i] = sq[i];
            if (lane == 0) cnt[q] = R;
        }
    }
    if (lane == 0) thr[q] = t;
}

// The same with one CTA per query, for queries with many keys (NT threads:
// 1024 when the batch is too small to fill the GPU with 256-thread CTAs; U keys
// per thread in registers).
template <int NT, int U>
__global__ void __launch_bounds__(NT) k_threshold_cta(ScanArgs A, int Rmax, int32_t* __restrict__ cnt,
                                                       uint64_t* __restrict__ cand, int cap,
                                                       uint64_t* __restrict__ scratch,
                                                       uint64_t* __restrict__ thr) {
    __shared__ __align__(16) uint32_t hist[256];
    __shared__ uint64_t bb[32];
    __shared__ unsigned long long s_m;
    const int64_t q = blockIdx.x;
    const int R = rerank_of(A.rerank_q, A.Rfix, A.Rmin, Rmax, q);
    const int n0 = cnt[q];
    const int n = min(n0, cap);
    const bool ovf = n0 > cap;
    uint64_t* cq = cand + q * cap;
    uint64_t t = KEY_NONE;
    if (n == R) {
        if (threadIdx.x == 0) s_m = 0ull;
        __syncthreads();
        unsigned long long m = 0ull;
        for (int i = threadIdx.x; i < n; i += blockDim.x) m = cq[i] > m ? cq[i] : m;
        atomicMax(&s_m, m);
        __syncthreads();
        t = s_m;
    } else if (n > R) {
        uint64_t* sq = n <= NT * U ? cq : scratch + q * Rmax;
        auto emit = [&](int i, uint64_t k) {
            if (!ovf) sq[i] = k;
        };
        t = cta_topk<NT, U>(cq, n, R, emit, hist, bb);
        if (!ovf) {
            if (sq != cq)
                for (int i = threadIdx.x; i < R; i += blockDim.x) cq[i] = sq[i];
            if (threadIdx.x == 0) cnt[q] = R;
        }
    }
    if (threadIdx.x == 0) thr[q] = t;
}

// ------------------------------------------------------------------ work list (cluster-major)
// pairs of (query, probe rank) grouped by list; items = (list, query group,
// block tile).
// Work lists of both parts of every query's probe ranks, in one pass: a warp
// per query finds the end of the unfiltered first part and counts the pairs
// of each part per list.  First part (plain search): the fewest nearest lists
// holding S = max(NEAR_KEYS_PER_R * R, N / NEAR_SHARE_DIV) keys, N = the keys
// the query probes.  The R-th key of a first set of S keys sits near the R/S
// quantile of the nearest keys and the remaining lists are farther, so at most
// about N R / S of their keys pass it: a few R.  S is at most half the
// candidate store, and the first part never holds more keys than the store
// (at least one list).  Hybrid search: the first `rs` ranks.  split[q] (plain
// only) records the boundary for k_fill_parts.

__global__ void k_count_parts(ScanArgs A, int Rmax, int cap, int rs, int32_t* __restrict__ split,
                              int32_t* __restrict__ cntA, int32_t* __restrict__ cntB,
                              int32_t* __restrict__ near_cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t q = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (q >= A.nq) return;
    const int P = nprobe_of(A, q);
    const int32_t* pr = A.probes + q * A.Pmax;
    int b = rs;
    if (split) {
        long long total = 0;
        for (int r = lane; r < P; r += 32) total += list_size(A, pr[r]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
        long long target = (long long)NEAR_KEYS_PER_R * rerank_of(A.rerank_q, A.Rfix, A.Rmin, Rmax, q);
        target = max(target, total / NEAR_SHARE_DIV);
        target = min(target, (long long)cap / 2);
        // first rank r whose keys-before reach the target, or (r > 0) whose list
        // would overflow the store
        long long acc = 0;
        int bnd = P;
        for (int r0 = 0; r0 < P; r0 += 32) {
            const int r = r0 + lane;
            const long long n = r < P ? list_size(A, pr[r]) : 0;
            long long incl = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const long long before = acc + incl - n;
            const bool stop = r < P && (before >= target || (r > 0 && before + n > cap));
            const uint32_t m = __ballot_sync(0xffffffffu, stop);
            if (m) {
                bnd = r0 + __ffs(m) - 1;
                break;
            }
            acc += __shfl_sync(0xffffffffu, incl, 31);
        }
        b = bnd < 1 ? 1 : bnd;
        if (lane == 0) split[q] = b;
    }
    long long nn = 0;
    for (int r = lane; r < P; r += 32) {
        const int p = pr[r];
        if (p >= 0 && p < A.L) atomicAdd(r < b ? &cntA[p] : &cntB[p], 1);
        if (r < b) nn += list_size(A, p);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
    // the unfiltered scan writes every key of the first part at a fixed place
    if (lane == 0) near_cnt[q] = (int32_t)(nn < 0x7fffffffll ? nn : 0x7fffffffll);
}


// exclusive scans: pair_off = scan(cnt); item_off = scan(ceil(cnt/QG) * ntiles)
// Several work lists at once: CTA i scans cnt + i L into pair_off / item_off +
// i (L + 1) and clears fill + i L; the first list's items hold QG0 queries and
// tiles of TB0 blocks, the others' QG1 and TB1.
__global__ void __launch_bounds__(1024) k_scan_lists(const int32_t* __restrict__ cnt0, const int32_t* __restrict__ list_n,
                                                     int L, int QG0, int QG1, int TB0, int TB1,
                                                     int64_t* __restrict__ pair_off0, int64_t* __restrict__ item_off0,
                                                     int32_t* __restrict__ fill0) {
    const int TB = blockIdx.x == 0 ? TB0 : TB1;  // tile length of this CTA's work list
    const int QG = blockIdx.x == 0 ? QG0 : QG1;  // queries per item
    const int32_t* cnt = cnt0 + (size_t)blockIdx.x * L;
    int64_t* pair_off = pair_off0 + (size_t)blockIdx.x * (L + 1);
    int64_t* item_off = item_off0 + (size_t)blockIdx.x * (L + 1);
    int32_t* fill = fill0 + (size_t)blockIdx.x * L;
    __shared__ int64_t s_p[1024], s_i[1024];
    const int per = (L + 1023) / 1024;
    const int c0 = threadIdx.x * per;
    int64_t sp = 0, si = 0;
    for (int c = c0; c < c0 + per && c < L; ++c) {
        sp += cnt[c];
        int nb = (list_n[c] + 31) >> 5;
        int nt = (nb + TB - 1) / TB;
        si += (int64_t)((cnt[c] + QG - 1) / QG) * nt;
    }
    s_p[threadIdx.x] = sp;
    s_i[threadIdx.x] = si;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        int64_t vp = threadIdx.x >= o ? s_p[threadIdx.x - o] : 0;
        int64_t vi = threadIdx.x >= o ? s_i[threadIdx.x - o] : 0;
        __syncthreads();
        s_p[threadIdx.x] += vp;
        s_i[threadIdx.x] += vi;
        __syncthreads();
    }
    int64_t bp = s_p[threadIdx.x] - sp, bi = s_i[threadIdx.x] - si;
    for (int c = c0; c < c0 + per && c < L; ++c) {
        pair_off[c] = bp;
        item_off[c] = bi;
        fill[c] = 0;
        bp += cnt[c];
        int nb = (list_n[c] + 31) >> 5;
        int nt = (nb + TB - 1) / TB;
        bi += (int64_t)((cnt[c] + QG - 1) / QG) * nt;
    }
    if (threadIdx.x == 1023) {
        pair_off[L] = s_p[1023];
        item_off[L] = s_i[1023];
    }
}

__global__ void k_fill_parts(ScanArgs A, int rs, const int32_t* __restrict__ split,
                             const int64_t* __restrict__ offA, int32_t* __restrict__ fillA, uint32_t* __restrict__ pairsA,
                             const int64_t* __restrict__ offB, int32_t* __restrict__ fillB,
                             uint32_t* __restrict__ pairsB) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= A.nq * A.Pmax) return;
    int64_t q = e / A.Pmax;
    int r = (int)(e - q * A.Pmax);
    if (r >= nprobe_of(A, q)) return;
    const int p = A.probes[e];
    if (p < 0 || p >= A.L) return;
    const bool first = r < (split ? split[q] : rs);
    const int slot = atomicAdd(first ? &fillA[p] : &fillB[p], 1);
    (first ? pairsA : pairsB)[(first ? offA : offB)[p] + slot] = (uint32_t)e;  // e = q * Pmax + r
}

// ------------------------------------------------------------------ a3: LUT16 scan

// Persistent, cluster-major scan with shared-memory staging of the codes.
// A warp takes one item = (list p, group of QG = 32/G queries that probe p,
// tile of at most TB blocks of p) and walks the tile in chunks of
// SCAN_CHUNK blocks.  Lane 0 bulk-copies each chunk's codes (contiguous in
// global memory) into the warp's own shared-memory buffer with cp.async.bulk,
// completing the warp's mbarrier; two buffers alternate so that the next
// chunk -- of this item or of the warp's next item -- is in flight while the
// current one is scanned.  Group lane g of query slot s holds the sub-LUTs of
// subspaces j = g + G*u (u < SMAX) in registers.  A key is formed only for a
// vector whose distance reaches its query's threshold, so ids are read from
// global memory only for those.  With no threshold (the first part of every
// query, O.thr null) every key is kept and written straight to its fixed place
// in the store (near_offset of its probe rank + its index in the list; the
// count is preset by k_count_parts), its id loaded before the block's lookups.
// No CTA-wide barrier: warps run independently.
constexpr int SCAN_WARPS = 8;
constexpr int SCAN_CHUNK_BYTES = 4096;           // per buffer, per warp
constexpr int SCAN_CHUNK_BYTES_SEL = 3072;       // the same with shared selectors (room for their buffer)
constexpr int SCAN_BUF_KEYS = 64;                // kept keys buffered per (warp, query slot)

// With 8 lanes per query the four query slots of a warp read the same code
// words: their selectors are computed once per block into a shared buffer of
// M x 64 bytes per warp.
template <int G>
__host__ __device__ constexpr bool scan_shared_sel() { return G == 8; }
template <int G>
__host__ __device__ constexpr int scan_chunk_bytes() { return scan_shared_sel<G>() ? SCAN_CHUNK_BYTES_SEL : SCAN_CHUNK_BYTES; }
// The chunk stream of one warp: items it0, it0 + stride, ...; each item's
// blocks [b0, b1) in chunks of cb blocks.
struct ChunkCursor {
    int64_t it;
    int c;  // chunk index within the item
};

template <int G, int SMAX, bool DIRECT, bool FULL, bool REC>
__global__ void __launch_bounds__(SCAN_WARPS * 32, (SMAX <= 2 ? 3 : (SMAX <= 8 ? 2 : 1))) k_scan(ScanArgs A, ScanOut O, const int64_t* __restrict__ pair_off,
                                                          const int64_t* __restrict__ item_off,
                                                          const uint32_t* __restrict__ pairs, int L, int TB,
                                                          int32_t* __restrict__ status) {
    constexpr int QG = 32 / G;
    constexpr int V = 32 / G;
    constexpr bool SEL = scan_shared_sel<G>();
    constexpr int CHUNK = scan_chunk_bytes<G>();
    // SCAN_WARPS x 2 x CHUNK code buffers, then (SEL) SCAN_WARPS x M x 64 selector bytes
    extern __shared__ __align__(128) uint8_t bufs[];
    __shared__ __align__(8) uint64_t full[SCAN_WARPS][2];
    // kept keys of the warp's current item, per query slot, flushed to the
    // candidate store with one atomic per slot when a slot fills and when the
    // item ends (so a block's atomic latency is not on the scan's path)
    __shared__ uint64_t kbuf[SCAN_WARPS][QG][SCAN_BUF_KEYS];
    __shared__ int kcnt[SCAN_WARPS][QG];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int slot = lane / G, g = lane % G;
    constexpr bool direct = DIRECT;  // no threshold (O.thr null): keys to fixed places
    if (lane < QG) kcnt[warp][lane] = 0;
    const int M = A.M;
    const int S = (M + G - 1) / G;
    const int blk_bytes = M * 16;
    const int cb = CHUNK / blk_bytes;  // blocks per chunk (>= 1)
    // REC: items given one by one (a small batch: one pair each), else located
    // in the cluster-major work list
    const int64_t total = REC ? (int64_t)*O.nrec : item_off[L];
    auto locate = [&](int64_t i) -> ScanItem {
        if constexpr (REC) {
            const int4 r = __ldg(O.recs + i);
            return ScanItem{r.w, r.y, r.z, (int64_t)r.x, 1};
        } else {
            return locate_item(A, pair_off, item_off, L, TB, QG, i);
        }
    };
    const int64_t stride = (int64_t)gridDim.x * SCAN_WARPS;
    uint8_t* mybuf = bufs + (size_t)warp * 2 * CHUNK;
    uint4* sel = reinterpret_cast<uint4*>(bufs + (size_t)SCAN_WARPS * 2 * CHUNK) + (size_t)warp * 4 * M;
    const uint32_t bar0 = smem_addr(&full[warp][0]), bar1 = smem_addr(&full[warp][1]);
    if (lane == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    // lane 0: bulk copy of chunk (x, c) into buffer b
    auto issue = [&](const ScanItem& x, int c, int b) {
        const int c0 = x.b0 + c * cb, c1 = min(x.b1, c0 + cb);
        const uint32_t bytes = (uint32_t)(c1 - c0) * blk_bytes;
        const uint32_t bar = b ? bar1 : bar0;
        const uint8_t* src = A.codes + (A.boff[x.p] + c0) * (int64_t)blk_bytes;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         smem_addr(mybuf + b * CHUNK)),
                     "l"(src), "r"(bytes), "r"(bar)
                     : "memory");
    };
    int64_t it = (int64_t)blockIdx.x * SCAN_WARPS + warp;
    if (it >= total) return;
    ScanItem x = locate(it), nx = x;
    if (lane == 0) issue(x, 0, 0);
    uint32_t phase[2] = {0u, 0u};
    int b = 0;
    bool failed = false;
    while (true) {
        // item set-up: LUTs, bias and threshold of this lane group's query.
        // An item with fewer pairs than query slots (few queries probe the
        // list) gives every pair rep = QG / npw slots (npw: the pair count
        // rounded up to a power of two), which take interleaved blocks of each
        // chunk: slot = ph * npw + pi scans blocks ph, ph + rep, ...
        const int np_eff = (int)(x.npairs < QG ? x.npairs : QG);
        int npw = 1;
        while (npw < np_eff) npw <<= 1;
        const int rep = QG / npw;
        const int64_t pi = slot % npw;
        const int ph = slot / npw;
        const bool active = pi < np_eff;
        int64_t q = 0;
        uint4 t[SMAX];
        int32_t bias = 0, lim = -1;
        uint32_t thI = 0;
        int64_t noff = 0;
        if (active) {
            const uint32_t e = REC ? (uint32_t)x.g0 : pairs[x.g0 + pi];
            q = e / A.Pmax;
            if (direct) noff = REC ? (int64_t)O.noff[e] : near_offset(A, q, (int)(e - q * A.Pmax));
            const uint4* lp = reinterpret_cast<const uint4*>(A.lut + (int64_t)e * M * PQ_K);
#pragma unroll
            for (int u = 0; u < SMAX; ++u) {
                const int j = g + G * u;
                t[u] = (FULL || (u < S && j < M)) ? __ldg(lp + j) : make_uint4(0, 0, 0, 0);
            }
            bias = A.bias[e];
            const uint64_t th = O.thr ? O.thr[q] : KEY_NONE;
            thI = (uint32_t)th;
            // key high word (bias + sum) + 2^31 vs the threshold's: sum < lim
            // passes, sum == lim is decided by the id (sums are below 2^24)
            const int64_t l = (int64_t)(th >> 32) - 2147483648ll - bias;
            lim = (int32_t)(l < -1 ? -1 : (l > (1 << 24) ? (1 << 24) : l));
        } else {
#pragma unroll
            for (int u = 0; u < SMAX; ++u) t[u] = make_uint4(0, 0, 0, 0);
        }
        // all lanes: each lane group writes its slot's buffered keys; a buffered
        // entry holds (distance word, vector slot in blk_ids), the id is
        // looked up here, many at once
        auto flush = [&]() {
            const int n = kcnt[warp][slot];
            int base = 0;
            if (g == 0 && n > 0) base = atomicAdd(&O.cnt[q], n);
            base = __shfl_sync(0xffffffffu, base, 0, G);
            for (int i0 = g; i0 < n; i0 += 4 * G) {  // four id loads in flight per lane
                uint64_t e[4];
                uint32_t id[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) e[u] = i0 + u * G < n ? kbuf[warp][slot][i0 + u * G] : 0ull;
#pragma unroll
                for (int u = 0; u < 4; ++u) id[u] = i0 + u * G < n ? (uint32_t)A.ids[(uint32_t)e[u]] : 0u;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = i0 + u * G;
                    if (i < n && base + i < O.cap) O.cand[q * O.cap + base + i] = (e[u] & 0xffffffff00000000ull) | id[u];
                }
            }
            __syncwarp();
            if (g == 0) kcnt[warp][slot] = 0;
            __syncwarp();
        };
        const int listn = A.list_n[x.p];
        const int nch = (x.b1 - x.b0 + cb - 1) / cb;
        const int64_t next_it = it + stride;
        for (int c = 0; c < nch; ++c) {
            // prefetch the chunk after this one into the other buffer
            if (c + 1 == nch && next_it < total) nx = locate(next_it);
            if (lane == 0) {
                if (c + 1 < nch) issue(x, c + 1, b ^ 1);
                else if (next_it < total) issue(nx, 0, b ^ 1);
            }
            const bool ready = !failed && scan_wait(b ? bar1 : bar0, phase[b]);
            phase[b] ^= 1u;
            if (!ready) {
                if (lane == 0 && !failed) atomicOr(status, 4);  // a chunk never arrived: the warp stops
                failed = true;
            } else {
                const uint8_t* chunk = mybuf + b * CHUNK;
                const int c0 = x.b0 + c * cb, nblk = min(x.b1, c0 + cb) - c0;
                const int64_t gb0 = A.boff[x.p] + c0;
                // the same number of steps on every lane (the reduction is a
                // warp-wide shuffle); a slot past the chunk's last block reads
                // the last block again and keeps nothing
                for (int blk0 = 0; blk0 < nblk; blk0 += rep) {
                    const int blk = blk0 + ph;
                    const bool vb = active && blk < nblk;
                    const uint4* cp = reinterpret_cast<const uint4*>(chunk + min(blk, nblk - 1) * blk_bytes);
                    const uint32_t vslot = (uint32_t)((gb0 + blk) * 32 + V * g);
                    uint32_t idv[V];
                    if (direct && vb) {
#pragma unroll
                        for (int v = 0; v < V; ++v) idv[v] = (uint32_t)A.ids[vslot + v];
                    }
                    uint32_t a32[32];
#pragma unroll
                    for (int m = 0; m < 32; ++m) a32[m] = 0;
                    if (SEL && rep == 1) {
                        // every slot scans this block: its selectors once, into
                        // the warp's buffer (word k of subspace j at k M + j),
                        // then the lookups from there
                        for (int jj = lane; jj < M; jj += 32) {
                            const uint4 cw = cp[jj];
                            sel[0 * M + jj] = lut16_selectors(cw.x);
                            sel[1 * M + jj] = lut16_selectors(cw.y);
                            sel[2 * M + jj] = lut16_selectors(cw.z);
                            sel[3 * M + jj] = lut16_selectors(cw.w);
                        }
                        __syncwarp();
#pragma unroll
                        for (int u = 0; u + 1 < SMAX; u += 2) {
                            const int j = g + G * u;
                            if (FULL || (u + 1 < S && j + G < M)) accum_pair_sel(sel, M, j, j + G, t[u], t[u + 1], a32);
                            else if (u < S && j < M) accum_chunk_sel(sel, M, j, t[u], a32);
                        }
                        if (SMAX & 1) {
                            const int u = SMAX - 1, j = g + G * u;
                            if (FULL || (u < S && j < M)) accum_chunk_sel(sel, M, j, t[u], a32);
                        }
                        __syncwarp();  // all reads done before the next block's selectors
                    } else {
#pragma unroll
                        for (int u = 0; u + 1 < SMAX; u += 2) {
                            const int j = g + G * u;
                            if (FULL || (u + 1 < S && j + G < M)) accum_pair32(cp[j], t[u], cp[j + G], t[u + 1], a32);
                            else if (u < S && j < M) accum_chunk32(cp[j], t[u], a32);
                        }
                        if (SMAX & 1) {
                            const int u = SMAX - 1, j = g + G * u;
                            if (FULL || (u < S && j < M)) accum_chunk32(cp[j], t[u], a32);
                        }
                    }
                    // partial sums < 2^16: pack vector pairs for the reduction
                    uint32_t acc[16];
#pragma unroll
                    for (int m = 0; m < 16; ++m) acc[m] = prmt(a32[2 * m], a32[2 * m + 1], 0x5410u);
                    uint32_t sums[V];
                    reduce_scatter<G>(acc, lane, sums);
                    if (direct) {
                        if (vb) {
                            const int nv = listn - (c0 + blk) * 32;
                            const int64_t pos = noff + (int64_t)(c0 + blk) * 32 + V * g;
                            uint64_t* out = O.cand + q * O.cap;
#pragma unroll
                            for (int v = 0; v < V; ++v) {
                                const uint32_t Dk = (uint32_t)(bias + (int32_t)sums[v]) ^ 0x80000000u;
                                if (V * g + v < nv && pos + v < O.cap) out[pos + v] = ((uint64_t)Dk << 32) | idv[v];
                            }
                        }
                        continue;
                    }
                    // keys at or below the threshold (padding, only at a list's
                    // tail, excluded by the list length); an id is read only
                    // on a tie with the threshold's distance
                    uint32_t kmask = 0;
                    if (vb) {
                        const int nv = listn - (c0 + blk) * 32 - V * g;  // valid vectors of this lane
                        const uint32_t vm = nv >= V ? (1u << V) - 1u : (nv > 0 ? (1u << nv) - 1u : 0u);
                        uint32_t eq = 0;
#pragma unroll
                        for (int v = 0; v < V; ++v) {
                            kmask |= (uint32_t)((int)sums[v] < lim) << v;
                            eq |= (uint32_t)((int)sums[v] == lim) << v;
                        }
                        kmask &= vm;
                        eq &= vm;
                        while (eq) {
                            const int v = __ffs(eq) - 1;
                            eq &= eq - 1u;
                            if ((uint32_t)A.ids[vslot + v] <= thI) kmask |= 1u << v;
                        }
                    }
                    // into the slot's buffer, which always has room for a whole
                    // block (32 keys): each lane reserves its keys with a shared
                    // atomic; a slot left with less room is flushed.  Entry:
                    // high word (D + 2^31) as an unsigned integer, low word the
                    // vector's slot (the id is looked up at the flush)
                    if (__any_sync(0xffffffffu, kmask != 0u)) {
                        if (kmask) {
                            const int pos = atomicAdd(&kcnt[warp][slot], __popc(kmask));
#pragma unroll
                            for (int v = 0; v < V; ++v)
                                if ((kmask >> v) & 1u) {
                                    const uint32_t Dk = (uint32_t)(bias + (int32_t)sums[v]) ^ 0x80000000u;
                                    kbuf[warp][slot][pos + __popc(kmask & ((1u << v) - 1u))] =
                                        ((uint64_t)Dk << 32) | (vslot + v);
                                }
                        }
                        __syncwarp();
                        if (__any_sync(0xffffffffu, kcnt[warp][slot] > SCAN_BUF_KEYS - 32)) flush();
                    }
                }
            }
            __syncwarp();  // the whole warp is done with buffer b before lane 0 refills it
            b ^= 1;
        }
        if (__any_sync(0xffffffffu, kcnt[warp][slot] > 0)) flush();
        if (next_it >= total || failed) break;
        it = next_it;
        x = nx;
    }
}

// ------------------------------------------------------------------ a3: LUT16 scan, one lane per block
// Same warp items as k_scan with 4 lanes per query (list p, 8 queries that
// probe p, tile [b0, b1) of p's blocks), but the 4 lanes of a query take 4
// different blocks of each step and each sums all M subspaces of its block's
// 32 vectors, so no cross-lane reduction is needed.  Lane = (slot s = lane & 7,
// block bo = lane >> 3).  The item's 8 tables of subspace j sit side by side in
// shared memory (T[j][s], 16 B each): the 8 lanes of a quarter-warp (same bo,
// s = 0..7) read 128 contiguous bytes, and they share one block, so its code
// chunk is a broadcast.  Codes arrive in steps of 4 blocks by cp.async.bulk
// into two alternating buffers, as in k_scan.
constexpr int S4_WARPS = 4;
constexpr int S4_Q = 8;  // queries per item
constexpr int S4_B = 4;  // blocks per step

template <int MAXM>
__host__ __device__ constexpr int s4_warp_bytes() { return MAXM * S4_Q * 16 + 2 * S4_B * MAXM * 16; }

template <int MAXM>
__global__ void __launch_bounds__(S4_WARPS * 32, MAXM <= 64 ? 3 : 1)
    k_scan4(ScanArgs A, ScanOut O, const int64_t* __restrict__ pair_off, const int64_t* __restrict__ item_off,
            const uint32_t* __restrict__ pairs, int L, int TB, int32_t* __restrict__ status) {
    constexpr int TAB_BYTES = MAXM * S4_Q * 16;
    constexpr int BUF_BYTES = S4_B * MAXM * 16;
    extern __shared__ __align__(128) uint8_t sm4[];
    __shared__ __align__(8) uint64_t full[S4_WARPS][2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int s = lane & 7, bo = lane >> 3;
    const int M = A.M, blk_bytes = M * 16;
    const bool direct = O.thr == nullptr;
    uint8_t* wb = sm4 + (size_t)warp * s4_warp_bytes<MAXM>();
    uint4* tab = reinterpret_cast<uint4*>(wb);
    uint8_t* cbuf = wb + TAB_BYTES;
    const uint32_t bar0 = smem_addr(&full[warp][0]), bar1 = smem_addr(&full[warp][1]);
    if (lane == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    auto issue = [&](const ScanItem& x, int c, int b) {
        const int c0 = x.b0 + c * S4_B, c1 = min(x.b1, c0 + S4_B);
        const uint32_t bytes = (uint32_t)(c1 - c0) * blk_bytes;
        const uint32_t bar = b ? bar1 : bar0;
        const uint8_t* src = A.codes + (A.boff[x.p] + c0) * (int64_t)blk_bytes;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         smem_addr(cbuf + b * BUF_BYTES)),
                     "l"(src), "r"(bytes), "r"(bar)
                     : "memory");
    };
    const int64_t total = item_off[L];
    const int64_t stride = (int64_t)gridDim.x * S4_WARPS;
    int64_t it = (int64_t)blockIdx.x * S4_WARPS + warp;
    if (it >= total) return;
    ScanItem x = locate_item(A, pair_off, item_off, L, TB, S4_Q, it, S4_B), nx = x;
    if (lane == 0) issue(x, 0, 0);
    uint32_t phase[2] = {0u, 0u};
    int b = 0;
    bool failed = false;
    while (true) {
        // the item's tables, transposed to T[j][s] (zeros for empty slots)
        const int nslots = x.npairs < S4_Q ? (int)x.npairs : S4_Q;
        for (int e = lane; e < S4_Q * M; e += 32) {
            const int qs = e / M, j = e - qs * M;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (qs < nslots) v = __ldg(reinterpret_cast<const uint4*>(A.lut + (int64_t)pairs[x.g0 + qs] * M * PQ_K) + j);
            tab[j * S4_Q + qs] = v;
        }
        const bool active = s < nslots;
        int64_t q = 0, noff = 0;
        int32_t bias = 0, lim = -1;
        uint32_t thI = 0;
        if (active) {
            const uint32_t e = pairs[x.g0 + s];
            q = e / A.Pmax;
            if (direct) noff = near_offset(A, q, (int)(e - q * A.Pmax));
            bias = A.bias[e];
            const uint64_t th = O.thr ? O.thr[q] : KEY_NONE;
            thI = (uint32_t)th;
            // key high word (bias + sum) + 2^31 <= thD  <=>  sum <= thD - 2^31 - bias
            const int64_t l = (int64_t)(th >> 32) - 2147483648ll - bias;
            lim = (int32_t)(l < -1 ? -1 : (l > 65536 ? 65536 : l));
        }
        const int listn = A.list_n[x.p];
        const int64_t gb_list = A.boff[x.p];
        __syncwarp();
        const int nch = (x.b1 - x.b0 + S4_B - 1) / S4_B;
        const int64_t next_it = it + stride;
        for (int c = 0; c < nch; ++c) {
            if (c + 1 == nch && next_it < total) nx = locate_item(A, pair_off, item_off, L, TB, S4_Q, next_it, S4_B);
            if (lane == 0) {
                if (c + 1 < nch) issue(x, c + 1, b ^ 1);
                else if (next_it < total) issue(nx, 0, b ^ 1);
            }
            const bool ready = !failed && scan_wait(b ? bar1 : bar0, phase[b]);
            phase[b] ^= 1u;
            if (!ready) {
                if (lane == 0 && !failed) atomicOr(status, 4);  // a chunk never arrived: the warp stops
                failed = true;
            } else {
                const int c0 = x.b0 + c * S4_B, nblk = min(x.b1, c0 + S4_B) - c0;
                const int blk = c0 + bo;
                uint32_t acc[32];  // sum of vector v of the block
#pragma unroll
                for (int m = 0; m < 32; ++m) acc[m] = 0u;
                uint32_t kmask = 0;
                if (bo < nblk) {
                    const uint4* cp = reinterpret_cast<const uint4*>(cbuf + b * BUF_BYTES + bo * blk_bytes);
                    const uint4* tp = tab + s;
                    int j = 0;
                    for (; j + 1 < M; j += 2) accum_pair32(cp[j], tp[j * S4_Q], cp[j + 1], tp[(j + 1) * S4_Q], acc);
                    if (j < M) accum_chunk32(cp[j], tp[j * S4_Q], acc);
                    if (direct && active) {
                        // no threshold: every key of the block to its fixed place
                        const int nv = listn - blk * 32;
                        const int64_t pos = noff + (int64_t)blk * 32;
                        const int32_t* idp = A.ids + (gb_list + blk) * 32;
                        uint64_t* out = O.cand + q * O.cap;
#pragma unroll
                        for (int v = 0; v < 32; ++v) {
                            const uint32_t Dk = (uint32_t)(bias + (int32_t)acc[v]) ^ 0x80000000u;
                            if (v < nv && pos + v < O.cap) out[pos + v] = ((uint64_t)Dk << 32) | (uint32_t)idp[v];
                        }
                    } else if (active) {
                        const int nv = listn - blk * 32;
                        const uint32_t vmask = nv >= 32 ? 0xffffffffu : ((1u << nv) - 1u);
                        uint32_t lt = 0, eq = 0;
#pragma unroll
                        for (int v = 0; v < 32; ++v) {
                            lt |= (uint32_t)((int)acc[v] < lim) << v;
                            eq |= (uint32_t)((int)acc[v] == lim) << v;
                        }
                        lt &= vmask;
                        eq &= vmask;
                        while (eq) {  // a key equal to the threshold's distance: its id decides
                            const int v = __ffs(eq) - 1;
                            eq &= eq - 1u;
                            if ((uint32_t)A.ids[(gb_list + blk) * 32 + v] <= thI) lt |= 1u << v;
                        }
                        kmask = lt;
                    }
                }
                // one atomic per query and step: counts of its 4 lanes (kmask
                // stays empty with no threshold: those keys are already placed)
                const int n = __popc(kmask);
                const int n0 = __shfl_sync(0xffffffffu, n, s), n1 = __shfl_sync(0xffffffffu, n, s + 8);
                const int n2 = __shfl_sync(0xffffffffu, n, s + 16), n3 = __shfl_sync(0xffffffffu, n, s + 24);
                const int tot = n0 + n1 + n2 + n3;
                int base = (bo == 0 && tot > 0) ? atomicAdd(&O.cnt[q], tot) : 0;
                base = __shfl_sync(0xffffffffu, base, s) + (bo > 0 ? n0 : 0) + (bo > 1 ? n1 : 0) + (bo > 2 ? n2 : 0);
                if (kmask) {
                    const int32_t* idp = A.ids + (gb_list + blk) * 32;
                    uint64_t* out = O.cand + q * O.cap;
#pragma unroll
                    for (int v = 0; v < 32; ++v) {
                        if ((kmask >> v) & 1u) {
                            const int at = base + __popc(kmask & ((1u << v) - 1u));
                            const uint32_t Dk = (uint32_t)(bias + (int32_t)acc[v]) ^ 0x80000000u;
                            if (at < O.cap) out[at] = ((uint64_t)Dk << 32) | (uint32_t)idp[v];
                        }
                    }
                }
            }
            __syncwarp();  // the whole warp is done with buffer b (and the tables) before they are refilled
            b ^= 1;
        }
        if (next_it >= total || failed) break;
        it = next_it;
        x = nx;
    }
}

// ------------------------------------------------------------------ a4: hybrid graph search
// Work lists from an explicit pair array (the lists marked for a full scan).
__global__ void k_count_from(const uint32_t* __restrict__ src, const int64_t* __restrict__ nsrc,
                             const int32_t* __restrict__ probes, int32_t* __restrict__ cnt) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= *nsrc) return;
    atomicAdd(&cnt[probes[src[i]]], 1);
}

__global__ void k_fill_from(const uint32_t* __restrict__ src, const int64_t* __restrict__ nsrc,
                            const int32_t* __restrict__ probes, const int64_t* __restrict__ pair_off,
                            int32_t* __restrict__ fill, uint32_t* __restrict__ dst) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= *nsrc) return;
    const uint32_t e = src[i];
    const int p = probes[e];
    dst[pair_off[p] + atomicAdd(&fill[p], 1)] = e;
}

struct GraphArgs {
    const int32_t* nbr_pos;    // [nslots x 32] neighbour list positions, -1 padding
    const uint8_t* nbr_codes;  // [nslots x M x 16] neighbour codes as one block per node
    const int32_t* entry_pos;  // [L]
    int efs, tau, vwords;
    uint32_t* full_pairs;      // out: (query, rank) pairs whose list is scanned fully
    int64_t* nfull;            // out: their count
};

constexpr int GS_WARPS = 4;
constexpr int GS_MAX_EFS = 96;    // result-set capacity: three keys per lane
constexpr int GS_INSERT_MAX = 8;  // new keys of an expansion inserted one by one (more: sorted and merged)
// Shared bytes per CTA that bound the list length this search accepts (a
// visited bit per member and a fixed allowance per warp).
static size_t gs_smem_bound(int vwords) { return (size_t)GS_WARPS * (2048 + (size_t)vwords * 4); }

// 32 distances of one block for the lane group of the whole warp (G = 32):
// lane l receives vector l's sum.
template <int SMAX>
__device__ __forceinline__ uint32_t block_sums32(const uint4* __restrict__ cp, const uint4 (&t)[SMAX], int M,
                                                 int lane) {
    uint32_t acc[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) acc[m] = 0;
#pragma unroll
    for (int u = 0; u < SMAX; ++u) {
        const int j = lane + 32 * u;
        if (j < M) accum_chunk(__ldg(cp + j), t[u], acc);
    }
    uint32_t out[1];
    reduce_scatter<32>(acc, lane, out);
    return out[0];
}

// Ascending sort of a bitonic sequence of one key per lane.
__device__ __forceinline__ uint64_t warp_merge_key(uint64_t v, int lane) {
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const uint64_t o = __shfl_xor_sync(0xffffffffu, v, j);
        v = ((lane & j) == 0) == (o < v) ? o : v;
    }
    return v;
}

// One warp per (query, distant list): best-first search of the list's graph
// with result set W of capacity efs (Sec. 4.4).  An expansion takes W's
// smallest unexpanded entry, computes its 32 neighbours' keys with one LUT16
// block, marks them visited, and keeps the efs smallest of W and the unvisited
// neighbours.  The search ends when every entry of W is expanded
// (equivalently: the best candidate is worse than W's worst once W is full).
// Then, with theta the query's threshold: at least tau keys of W below theta
// -> the list is scanned fully later; otherwise W's keys at or below theta
// join the candidates.
//
// W lives in registers, sorted: entry 32 i + lane in W[i].  An entry is one
// word, distance word << 32 | list position << 1 | expanded: a list's members
// stand in ascending id, so positions order ties as ids do, and the expanded
// bit of unique positions changes no order (an empty entry, all ones, reads as
// expanded).  Ids are looked up once, for the final W.  Only new keys below
// W's worst can enter: a few of them are inserted one by one (a compare and a
// shift by one lane), more are sorted across the warp and merged.
// The kernel is bound by instruction issue: about 450 issue slots per
// expansion, a third of them the block's lookups.  Sorting W and the new keys
// together in shared memory took about 4500 (100k x 64, M 32, 2000 queries, 10
// distant lists each, efs 64: 6.2 ms against 0.51 ms now).
template <int SMAX, int NR>
__global__ void __launch_bounds__(GS_WARPS * 32) k_graph_search(ScanArgs A, ScanOut O, GraphArgs Gr,
                                                                const uint32_t* __restrict__ pairs,
                                                                const int64_t* __restrict__ npairs) {
    extern __shared__ uint32_t gvis[];  // a visited bit per member, vwords per warp
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* vis = gvis + (size_t)warp * Gr.vwords;
    const int M = A.M;
    const int64_t n_items = *npairs;
    for (int64_t it = (int64_t)blockIdx.x * GS_WARPS + warp; it < n_items; it += (int64_t)gridDim.x * GS_WARPS) {
        const uint32_t e = pairs[it];
        const int64_t q = e / A.Pmax;
        const int p = A.probes[e];
        const int np_ = A.list_n[p];
        const int ep = Gr.entry_pos[p];
        if (ep < 0) continue;
        uint4 t[SMAX];
        const uint4* lp = reinterpret_cast<const uint4*>(A.lut + (int64_t)e * M * PQ_K);
#pragma unroll
        for (int u = 0; u < SMAX; ++u) {
            const int j = lane + 32 * u;
            t[u] = j < M ? __ldg(lp + j) : make_uint4(0, 0, 0, 0);
        }
        const int32_t bias = A.bias[e];
        const uint64_t th = O.thr[q];
        const int64_t slot0 = A.boff[p] * 32;
        auto entry_of = [&](uint32_t sum, int pos) -> uint64_t {
            return ((uint64_t)((uint32_t)(bias + (int32_t)sum) ^ 0x80000000u) << 32) | ((uint32_t)pos << 1);
        };
        for (int w = lane; w < (np_ + 31) / 32; w += 32) vis[w] = 0u;
        __syncwarp();
        uint64_t W[NR];
#pragma unroll
        for (int i = 0; i < NR; ++i) W[i] = KEY_NONE;
        // entry: its block's 32 sums, keep the entry's
        {
            const int64_t gb = A.boff[p] + (ep >> 5);
            const uint32_t sum = block_sums32<SMAX>(reinterpret_cast<const uint4*>(A.codes + gb * M * 16), t, M, lane);
            const uint64_t k = __shfl_sync(0xffffffffu, entry_of(sum, ep), ep & 31);
            if (lane == 0) {
                W[0] = k;
                vis[ep >> 5] = 1u << (ep & 31);
            }
            __syncwarp();
        }
        for (int guard = 0; guard <= np_; ++guard) {
            // smallest unexpanded entry of W
            int src = -1;
            uint32_t up = 0;
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                const uint32_t m = __ballot_sync(0xffffffffu, (W[i] & 1ull) == 0ull);
                if (src < 0 && m) {
                    src = __ffs(m) - 1;
                    up = __shfl_sync(0xffffffffu, (uint32_t)W[i], src) >> 1;
                    if (lane == src) W[i] |= 1ull;
                }
            }
            if (src < 0) break;
            // expand: the 32 neighbours' keys in one block
            const int64_t su = slot0 + up;
            const int pe = Gr.nbr_pos[su * 32 + lane];
            const uint32_t sum =
                block_sums32<SMAX>(reinterpret_cast<const uint4*>(Gr.nbr_codes + su * M * 16), t, M, lane);
            uint64_t kn = KEY_NONE;
            if (pe >= 0) {
                const uint32_t bit = 1u << (pe & 31);
                const uint32_t old = atomicOr(&vis[pe >> 5], bit);
                if (!(old & bit)) kn = entry_of(sum, pe);
            }
            // only keys below W's last entry (all ones until W is full) can enter
            uint64_t worst = KEY_NONE;
#pragma unroll
            for (int i = 0; i < NR; ++i)
                if ((Gr.efs - 1) >> 5 == i) worst = __shfl_sync(0xffffffffu, W[i], (Gr.efs - 1) & 31);
            if (kn >= worst) kn = KEY_NONE;
            uint32_t m = __ballot_sync(0xffffffffu, kn != KEY_NONE);
            if (!m) continue;
            if (__popc(m) <= GS_INSERT_MAX) {
                while (m) {
                    const uint64_t k = __shfl_sync(0xffffffffu, kn, __ffs(m) - 1);
                    m &= m - 1u;
                    // entries above k move up by one place, k takes the first of theirs
#pragma unroll
                    for (int i = NR - 1; i >= 0; --i) {
                        uint64_t prev = __shfl_up_sync(0xffffffffu, W[i], 1);
                        const uint64_t below = i > 0 ? __shfl_sync(0xffffffffu, W[i > 0 ? i - 1 : 0], 31) : 0ull;
                        if (lane == 0) prev = below;
                        if (W[i] > k) W[i] = prev > k ? prev : k;
                    }
                }
            } else {
                // from the top 32 entries down: of W[i] and the new keys, the 32
                // largest are final (those past the last register drop out), the
                // 32 smallest go on against W[i - 1]
                uint64_t N = warp_sort_key(kn, lane);
#pragma unroll
                for (int i = NR - 1; i >= 0; --i) {
                    const uint64_t r = __shfl_sync(0xffffffffu, N, 31 - lane);
                    const uint64_t lo = r < W[i] ? r : W[i], hi = r < W[i] ? W[i] : r;
                    if (i + 1 < NR) W[i + 1 < NR ? i + 1 : 0] = warp_merge_key(hi, lane);
                    N = warp_merge_key(lo, lane);
                }
                W[0] = N;
            }
#pragma unroll
            for (int i = 0; i < NR; ++i)
                if (32 * i + lane >= Gr.efs) W[i] = KEY_NONE;
        }
        // decide: full scan later, or W's keys join the candidates
        int good = 0;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            // the entry as a candidate key: its id in place of its position
            if (W[i] != KEY_NONE)
                W[i] = (W[i] & 0xffffffff00000000ull) | (uint32_t)A.ids[slot0 + ((uint32_t)W[i] >> 1)];
            good += __popc(__ballot_sync(0xffffffffu, W[i] < th && W[i] != KEY_NONE));
        }
        if (good >= Gr.tau) {
            if (lane == 0) Gr.full_pairs[atomicAdd(reinterpret_cast<unsigned long long*>(Gr.nfull), 1ull)] = e;
        } else {
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                const bool keep = W[i] != KEY_NONE && W[i] <= th;
                const unsigned b = __ballot_sync(0xffffffffu, keep);
                if (!b) continue;
                int base = 0;
                if (lane == 0) base = atomicAdd(&O.cnt[q], __popc(b));
                base = __shfl_sync(0xffffffffu, base, 0) + __popc(b & ((1u << lane) - 1u));
                if (keep && base < O.cap) O.cand[q * O.cap + base] = W[i];
            }
        }
        __syncwarp();
    }
}

// The scan's lookup sequence with shared selectors (8 lanes per query): the
// selectors of a subspace pair from the warp's shared buffer (at indices that
// depend on a per-iteration random number, so that nothing can be hoisted
// out of the loop), the lookups and the interleaved widening of two
// subspaces -- the lookup rate of the scan's inner loop with no code or
// table traffic beyond shared memory.
__global__ void __launch_bounds__(256) k_lut16_peak_sel(int iters, uint32_t seed, uint32_t* __restrict__ sink) {
    __shared__ uint4 sel[4 * 64];
    for (int i = threadIdx.x; i < 4 * 64; i += blockDim.x) {
        uint32_t h = (uint32_t)i * 2654435761u + seed;
        h ^= h >> 15;
        h *= 0x2c1b3c6du;
        sel[i] = lut16_selectors(h ^ (h >> 12));
    }
    __syncthreads();
    const int g = threadIdx.x & 7;
    const uint4 t0 = make_uint4(seed, seed * 3u + 1u, seed * 5u + 7u, seed * 9u + 3u);
    const uint4 t1 = make_uint4(t0.y, t0.z, t0.w, t0.x);
    uint32_t acc[32];
#pragma unroll
    for (int m = 0; m < 32; ++m) acc[m] = 0;
    uint32_t w = seed ^ (blockIdx.x * blockDim.x + threadIdx.x);
    for (int i = 0; i < iters; i += 2) {  // 64 lookups per pair of iterations
        const int j = (g + 8 * (int)(w >> 29)) & 63;
        accum_pair_sel(sel, 64, j, (j + 32) & 63, t0, t1, acc);
        w = w * 1664525u + 1013904223u;
    }
    uint32_t s_ = 0;
#pragma unroll
    for (int m = 0; m < 32; ++m) s_ ^= acc[m];
    if (s_ == 0x12345678u) sink[0] = s_;  // keeps the loop alive
}

// Register-only copy of the scan's earlier lookup/accumulate sequence (each
// query slot computing its own selectors, one byte dot product per lookup;
// no memory traffic): still the sequence of the scan's sparse items.
__global__ void __launch_bounds__(128) k_lut16_peak(int iters, uint32_t seed, uint32_t* __restrict__ sink) {
    uint4 t = make_uint4(seed, seed * 3u + 1u, seed * 5u + 7u, seed * 9u + 3u);
    uint32_t acc[32];
#pragma unroll
    for (int m = 0; m < 32; ++m) acc[m] = 0;
    uint32_t w = seed ^ (blockIdx.x * blockDim.x + threadIdx.x);
    const uint4 t2 = make_uint4(t.y, t.z, t.w, t.x);
    for (int i = 0; i < iters; i += 2) {
        uint4 c = make_uint4(w, w ^ 0x5a5a5a5au, w + 0x01234567u, w ^ 0xf0f0f0f0u);
        uint4 c2 = make_uint4(w ^ 0x0f0f0f0fu, w + 0x89abcdefu, w ^ 0x33333333u, w + 0x13579bdfu);
        accum_pair32(c, t, c2, t2, acc);
        w = w * 1664525u + 1013904223u;
    }
    uint32_t s = 0;
#pragma unroll
    for (int m = 0; m < 32; ++m) s ^= acc[m];
    if (s == 0x12345678u) sink[0] = s;  // keeps the loop alive
}

// ------------------------------------------------------------------ a5: select
// R smallest candidate keys per query, in no particular order (the re-rank
// does not need one); one warp per query.  A query whose store overflowed is
// put on the redo list for k_select_redo.
__global__ void __launch_bounds__(SW_WARPS * 32) k_select(ScanArgs A, int Rmax, const int32_t* __restrict__ cnt,
                                                          const uint64_t* __restrict__ cand, int cap,
                                                          uint64_t* __restrict__ topr, int32_t* __restrict__ ncand,
                                                          int32_t* __restrict__ status,
                                                          unsigned long long* __restrict__ stats,
                                                          int32_t* __restrict__ redo) {
    __shared__ uint32_t hist[SW_WARPS][256];
    __shared__ uint64_t bb[SW_WARPS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t q = (int64_t)blockIdx.x * SW_WARPS + w;
    if (q >= A.nq) return;
    const int R = rerank_of(A.rerank_q, A.Rfix, A.Rmin, Rmax, q);
    const int n = cnt[q];
    if (lane == 0) {
        atomicAdd(&stats[1], (unsigned long long)n);
        atomicMax(&stats[2], (unsigned long long)n);
    }
    if (n > cap) {
        if (lane == 0) {
            atomicAdd(&stats[0], 1ull);
            atomicOr(status, KSC_STATUS_CAND_OVERFLOW);
            redo[1 + atomicAdd(&redo[0], 1)] = (int32_t)q;
        }
        return;
    }
    const uint64_t* cq = cand + q * cap;
    uint64_t* out = topr + q * Rmax;
    const int K = min(R, n);
    if (n <= K) {
        for (int i = lane; i < n; i += 32) out[i] = cq[i];
    } else {
        warp_topk_hi(cq, n, K, out, hist[w], bb[w]);
    }
    for (int i = K + lane; i < Rmax; i += 32) out[i] = KEY_NONE;
    if (lane == 0 && ncand) ncand[q] = K;
}

// The same with one CTA per query, for queries with many candidates.
template <int NT, int U>
__global__ void __launch_bounds__(NT) k_select_cta(ScanArgs A, int Rmax, const int32_t* __restrict__ cnt,
                                                    const uint64_t* __restrict__ cand, int cap,
                                                    uint64_t* __restrict__ topr, int32_t* __restrict__ ncand,
                                                    int32_t* __restrict__ status,
                                                    unsigned long long* __restrict__ stats,
                                                    int32_t* __restrict__ redo) {
    __shared__ __align__(16) uint32_t hist[256];
    __shared__ uint64_t bb[32];
    const int64_t q = blockIdx.x;
    const int R = rerank_of(A.rerank_q, A.Rfix, A.Rmin, Rmax, q);
    const int n = cnt[q];
    if (threadIdx.x == 0) {
        atomicAdd(&stats[1], (unsigned long long)n);
        atomicMax(&stats[2], (unsigned long long)n);
    }
    if (n > cap) {
        if (threadIdx.x == 0) {
            atomicAdd(&stats[0], 1ull);
            atomicOr(status, KSC_STATUS_CAND_OVERFLOW);
            redo[1 + atomicAdd(&redo[0], 1)] = (int32_t)q;
        }
        return;
    }
    const uint64_t* cq = cand + q * cap;
    uint64_t* out = topr + q * Rmax;
    const int K = min(R, n);
    if (n <= K) {
        for (int i = threadIdx.x; i < n; i += blockDim.x) out[i] = cq[i];
    } else {
        auto emit = [&](int i, uint64_t k) { out[i] = k; };
        cta_topk<NT, U>(cq, n, K, emit, hist, bb);
    }
    for (int i = K + threadIdx.x; i < Rmax; i += blockDim.x) out[i] = KEY_NONE;
    if (threadIdx.x == 0 && ncand) ncand[q] = K;
}

// The queries on the redo list.  A persistent grid walks it (usually empty).
__global__ void __launch_bounds__(1024) k_select_redo(ScanArgs A, int Rmax, int sel_cap, uint64_t* cand, int cap,
                                                      uint64_t* __restrict__ topr, int32_t* __restrict__ ncand,
                                                      const int32_t* __restrict__ redo) {
    extern __shared__ uint64_t sbuf[];  // sel_cap keys
    __shared__ __align__(16) uint32_t hist[256];
    __shared__ uint64_t bb[32];
    __shared__ int32_t s_pref[MAX_NPROBE + 1];
    const int nredo = redo[0];
    for (int r0 = blockIdx.x; r0 < nredo; r0 += gridDim.x) {
        const int64_t q = redo[1 + r0];
        const int R = rerank_of(A.rerank_q, A.Rfix, A.Rmin, Rmax, q);
        uint64_t* out = topr + q * Rmax;
        const int K = redo_select(A, q, R, cand + q * cap, cap, out, sbuf, sel_cap, hist, bb, s_pref);
        for (int i = K + threadIdx.x; i < Rmax; i += blockDim.x) out[i] = KEY_NONE;
        if (threadIdx.x == 0 && ncand) ncand[q] = K;
    }
}

// ------------------------------------------------------------------ a6: rerank
// A CTA per query (rerank.cuh): the candidates' exact distances, the k best.
template <int NT>
__global__ void __launch_bounds__(NT) k_rerank(const float* __restrict__ Q, const float* __restrict__ X, int d,
                                                int ip, const uint64_t* __restrict__ topr, int Rmax,
                                                const int32_t* __restrict__ rerank_q, int Rfix, int k,
                                                int64_t* __restrict__ out_ids, float* __restrict__ out_d) {
    extern __shared__ uint64_t keys[];  // Rmax keys, then rerank_kbuf(k) for the selection of more than RR_RANK_R
    __shared__ __align__(16) float qs[KSC_MAX_DIM];
    const int64_t q = blockIdx.x;
    const int R = rerank_of(rerank_q, Rfix, k, Rmax, q);
    for (int t = threadIdx.x; t < d; t += blockDim.x) qs[t] = Q[q * d + t];
    // the candidate keys staged in shared memory (each row load then waits
    // for a shared load)
    for (int c = threadIdx.x; c < R; c += blockDim.x) keys[c] = topr[q * Rmax + c];
    __syncthreads();
    cta_rerank<NT>(keys, R, keys + Rmax, qs, X, d, ip, k, out_ids + q * k, out_d + q * k);
}

// One warp per query (8 per CTA) when k <= 32, R <= RW_MAXR, d <= 128 and
// d % 4 == 0: lane l holds query coordinates 4l..4l+3; each step gathers 8
// candidate rows (one 16-byte load per lane and row) and sums the 8 partial
// dot products across the warp in a halving exchange (9 shuffles for 8 rows);
// the k best keys are then taken by k rounds of a warp minimum.  Same
// distance rule as k_rerank (L2 direct difference squares, IP -<q, x>), FP32.
//
// With xb (BF16 copies of the rows; or xu, U8 copies, when every coordinate
// is an integer in [0, 255] and a byte holds it exactly) and xe (per row:
// n >= |x| and r >= |x~ - x|, the norm of its rounding error, both from FP64
// sums rounded up), a first pass reads the low-precision rows (half or a
// quarter of the bytes) and bounds
// each candidate's FP32 distance: |d~ - d| <= e, from the rounding of the row
// (|<v, x~ - x>| <= |v| r) and the FP32 evaluation of both sums (relative
// g = 2^-20, above the at most 14 rounding steps of 2^-24 on a term's path in
// either pass):
//   L2: e = 2 r s + r^2 + g (s^2 + (s + r)^2), s >= sqrt of the exact
//       BF16-row distance (so s + r >= |q - x|);
//   IP: e = |q| (r + 2.01 g (n + r)),
// all evaluated with a factor (1 + 2^-10) and directed rounding of d~ -/+ e.
// r is the row's own rounding error, not the format's worst case
// (2^-8 |x|): a row that BF16 holds exactly (integer coordinates up to 256,
// say) has r = 0 and a band of the evaluation term alone.  U is the k-th
// smallest d~ + e; a candidate with d~ - e > U has an FP32 distance above k
// FP32 distances, so it cannot be among the k best.  The others get the FP32
// distance by the very code of the plain pass (a row's sum does not depend on
// the rows beside it in the exchange), so the result is bit for bit the
// plain pass's.
constexpr int RW_WARPS = 8;
constexpr int RW_MAXR = 512;

// The distance terms of 16 low-precision rows at once, 8 lanes per row:
// lane l = 8 h + j takes rows 4 h .. 4 h + 3 of the step (idv[], -1: none)
// and, of each, the 4-coordinate chunks j, j + 8, j + 16, j + 24 below d (one
// load each: 8 bytes of BF16, or 4 bytes of U8 rows; qv[] holds the query's
// coordinates of those chunks), summed in FP32 pairs; a halving exchange over
// lane bits 2, 1 and a sum over bit 0 leave row (lane >> 1) & 15 in both
// lanes of a pair.  The row's id, address and exchange cost one lane in
// eight, not every lane.  Only bounded, not compared bit for bit, so the
// summation order is free (its depth, at most 8 + 1 + 3 additions after the
// square, stays inside the bound's g).  A U8 byte b becomes the float
// (2^23 + b) - 2^23, exact.
template <bool U8>
__device__ __forceinline__ float rerank_rows16_band(const float4 (&qv)[4], const void* __restrict__ rows, int d,
                                                    int ip, int nch, const int32_t (&idv)[4], int lane) {
    const int j = lane & 7;
    uint2 r[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool ok = k < nch && idv[i] >= 0 && 4 * (j + 8 * k) < d;
            if (U8)
                r[i][k] = make_uint2(ok ? __ldg(reinterpret_cast<const uint32_t*>(
                                              static_cast<const uint8_t*>(rows) + (int64_t)idv[i] * d) + j + 8 * k)
                                        : 0u, 0u);
            else
                r[i][k] = ok ? __ldg(reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(rows) +
                                                                    (int64_t)idv[i] * d) + j + 8 * k)
                             : make_uint2(0u, 0u);
        }
    float a[4];
    const float2 m23 = make_float2(8388608.f, 8388608.f);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k >= nch) break;  // warp-uniform
            float2 x01, x23;
            if (U8) {
                const uint32_t w = r[i][k].x;
                x01 = f2_sub(make_float2(__uint_as_float(prmt(w, 0x4B000000u, 0x7540u)),
                                         __uint_as_float(prmt(w, 0x4B000000u, 0x7541u))), m23);
                x23 = f2_sub(make_float2(__uint_as_float(prmt(w, 0x4B000000u, 0x7542u)),
                                         __uint_as_float(prmt(w, 0x4B000000u, 0x7543u))), m23);
            } else {
                x01 = make_float2(__uint_as_float(r[i][k].x << 16), __uint_as_float(r[i][k].x & 0xffff0000u));
                x23 = make_float2(__uint_as_float(r[i][k].y << 16), __uint_as_float(r[i][k].y & 0xffff0000u));
            }
            const float2 q01 = make_float2(qv[k].x, qv[k].y), q23 = make_float2(qv[k].z, qv[k].w);
            if (ip) {
                acc = f2_fma(q01, x01, acc);
                acc = f2_fma(q23, x23, acc);
            } else {
                const float2 e01 = f2_sub(q01, x01), e23 = f2_sub(q23, x23);
                acc = f2_fma(e01, e01, acc);
                acc = f2_fma(e23, e23, acc);
            }
        }
        a[i] = acc.x + acc.y;
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const bool up = lane & 4;
        const float send = up ? a[i] : a[i + 2], keep = up ? a[i + 2] : a[i];
        a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    {
        const bool up = lane & 2;
        const float send = up ? a[0] : a[1], keep = up ? a[1] : a[0];
        a[0] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    return a[0];
}

// U8: the band's rows are U8 (xu), else BF16 (xb).
template <bool U8>
__global__ void __launch_bounds__(RW_WARPS * 32) k_rerank_w(const float* __restrict__ Q, const float* __restrict__ X,
                                                            int d, int ip, const uint64_t* __restrict__ topr,
                                                            int Rmax, const int32_t* __restrict__ rerank_q, int Rfix,
                                                            int k, int64_t nq, int64_t* __restrict__ out_ids,
                                                            float* __restrict__ out_d,
                                                            const uint16_t* __restrict__ xb,
                                                            const uint8_t* __restrict__ xu,
                                                            const float2* __restrict__ xe) {
    // RW_WARPS x Rmax keys; with xb also RW_WARPS x Rmax bound pairs and RW_WARPS x (Rmax + 64) words
    extern __shared__ uint64_t wkeys[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t q = (int64_t)blockIdx.x * RW_WARPS + w;
    if (q >= nq) return;
    uint64_t* keys = wkeys + (size_t)w * Rmax;  // the candidates' keys, staged; then their FP32 keys
    const int R = rerank_of(rerank_q, Rfix, k, Rmax, q);
    const bool inl = lane * 4 < d;
    float4 qv = make_float4(0.f, 0.f, 0.f, 0.f);
    if (inl) {  // the query matrix may be only 4-byte aligned
        const float* qp = Q + q * d + lane * 4;
        qv = make_float4(qp[0], qp[1], qp[2], qp[3]);
    }
    // the candidate keys in shared memory (one coalesced pass), so that a
    // step's row loads wait for a shared load, not for a global one
    {
        const uint64_t* cq = topr + q * Rmax;
        for (int c = lane; c < R; c += 32) keys[c] = cq[c];
        __syncwarp();
    }
    // row of the sum this lane holds after the exchange
    const int myrow = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
    auto id_of = [&](int c) -> int32_t {
        const uint64_t kk = c < R ? keys[c] : KEY_NONE;
        return kk != KEY_NONE ? (int32_t)(kk & 0xffffffffu) : -1;
    };
    auto fp32_key = [&](uint64_t kk, float a0) -> uint64_t {
        return kk != KEY_NONE ? (((uint64_t)ordered_f32(ip ? -a0 : a0) << 32) | (kk & 0xffffffffull)) : KEY_NONE;
    };
    // the k smallest of arr[0..cnt) to the outputs: one warp sort when they
    // fit a warp, else k rounds of a warp minimum
    auto emit_best = [&](uint64_t* arr, int cnt) {
        uint64_t mine = KEY_NONE;  // lane r keeps the r-th smallest
        if (cnt <= 32) {
            mine = warp_sort_key(lane < cnt ? arr[lane] : KEY_NONE, lane);
        } else {
            for (int r = 0; r < k; ++r) {
                uint64_t m = KEY_NONE;
                int at = -1;
                for (int i = lane; i < cnt; i += 32) {
                    if (arr[i] < m) { m = arr[i]; at = i; }
                }
                uint64_t gk = m;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const uint64_t y = __shfl_xor_sync(0xffffffffu, gk, o);
                    gk = y < gk ? y : gk;
                }
                if (gk != KEY_NONE && m == gk) arr[at] = KEY_NONE;  // keys are unique: one lane matches
                __syncwarp();
                if (lane == r) mine = gk;
            }
        }
        if (lane < k) {
            if (mine == KEY_NONE) {
                out_ids[q * k + lane] = -1;
                out_d[q * k + lane] = ip ? -INFINITY : INFINITY;
            } else {
                out_ids[q * k + lane] = (int64_t)(mine & 0xffffffffu);
                const float dist = unordered_f32((uint32_t)(mine >> 32));
                out_d[q * k + lane] = ip ? -dist : dist;
            }
        }
    };
    if ((xb || xu) && R > k) {
        float2* band = reinterpret_cast<float2*>(wkeys + (size_t)RW_WARPS * Rmax) + (size_t)w * Rmax;
        uint32_t* sv = reinterpret_cast<uint32_t*>(wkeys + (size_t)2 * RW_WARPS * Rmax) + (size_t)w * (Rmax + 64);
        uint32_t* kv = sv + Rmax;  // the small selection's values
        const float g = 0x1p-20f, safe = 1.f + 0x1p-10f;
        float qn = 0.f;  // IP: an upper bound of |q|
        if (ip) {
            float t = fmaf(qv.x, qv.x, fmaf(qv.y, qv.y, fmaf(qv.z, qv.z, qv.w * qv.w)));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            qn = sqrtf(t) * (1.f + 0x1p-18f);
        }
        // this lane's query chunks for the 8-lanes-per-row BF16 pass
        const int nch = (d + 31) >> 5;
        float4 qc[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int t0 = 4 * ((lane & 7) + 8 * h);
            qc[h] = t0 < d ? make_float4(Q[q * d + t0], Q[q * d + t0 + 1], Q[q * d + t0 + 2], Q[q * d + t0 + 3])
                           : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const int myrow16 = (lane >> 1) & 15;
        // the candidates' ids (-1: none) to 16 past R, in sv until the
        // survivors replace them: one shared load per row and step
        const int R16 = (R + 15) & ~15;
        for (int c = lane; c < R16; c += 32) sv[c] = (uint32_t)id_of(c);
        __syncwarp();
        for (int c0 = 0; c0 < R; c0 += 16) {
            int32_t idv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) idv[i] = (int32_t)sv[c0 + 4 * (lane >> 3) + i];
            // this lane's row bounds, loaded beside the rows
            const int c = c0 + myrow16;
            const int32_t id = (int32_t)sv[c];
            const float2 nr = id >= 0 ? __ldg(xe + id) : make_float2(0.f, 0.f);
            const float a0 = U8 ? rerank_rows16_band<true>(qc, xu, d, ip, nch, idv, lane)
                                : rerank_rows16_band<false>(qc, xb, d, ip, nch, idv, lane);
            if ((lane & 1) == 0 && c < R) {
                float lo = INFINITY, hi = INFINITY;
                if (id >= 0) {
                    const float n = nr.x, r = nr.y;
                    float e, dt;
                    if (ip) {
                        dt = -a0;
                        e = qn * (r + 2.01f * g * (n + r)) * safe;
                    } else {
                        dt = a0;
                        const float sq = sqrtf(fmaxf(dt, 0.f) * (1.f + 2.f * g)) * (1.f + 0x1p-20f);
                        e = (2.f * r * sq + r * r + g * (sq * sq + (sq + r) * (sq + r))) * safe;
                    }
                    lo = __fsub_rd(dt, e);
                    hi = __fadd_ru(dt, e);
                    if (!(lo <= hi)) {  // a NaN: no bound, the candidate is read in FP32
                        lo = -INFINITY;
                        hi = INFINITY;
                    }
                }
                band[c] = make_float2(lo, hi);
            }
        }
        __syncwarp();
        // U: the k-th smallest upper bound (+inf when the small selection
        // cannot tell: then every candidate is re-scored)
        float U = INFINITY;
        auto load_hi = [&](int c) -> uint32_t { return ordered_f32(band[c].y); };
        if (k <= 48 && warp_small_kvals(load_hi, R, k, kv) >= 0) U = unordered_f32(kv[k - 1]);
        // survivors: lower bound <= U
        const uint32_t below = (1u << lane) - 1u;
        int ns = 0;
        for (int c0 = 0; c0 < R; c0 += 32) {
            const int c = c0 + lane;
            const bool in = c < R && band[c].x <= U;
            const uint32_t m = __ballot_sync(0xffffffffu, in);
            if (in) sv[ns + __popc(m & below)] = (uint32_t)c;
            ns += __popc(m);
        }
        __syncwarp();
        // their FP32 keys, by survivor index, where the bounds were
        uint64_t* fk = reinterpret_cast<uint64_t*>(band);
        for (int s0 = 0; s0 < ns; s0 += 8) {
            int32_t idv[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) idv[u] = s0 + u < ns ? id_of((int)sv[s0 + u]) : -1;
            const float a0 = rerank_rows8(qv, X, d, ip, inl, idv, lane);
            const int si = s0 + myrow;
            if ((lane & 3) == 0 && si < ns) fk[si] = fp32_key(keys[sv[si]], a0);
        }
        __syncwarp();
        emit_best(fk, ns);
    } else {
        for (int c0 = 0; c0 < R; c0 += 8) {
            int32_t idv[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) idv[u] = id_of(c0 + u);
            const float a0 = rerank_rows8(qv, X, d, ip, inl, idv, lane);
            const int c = c0 + myrow;
            const uint64_t kk = c < R ? keys[c] : KEY_NONE;
            __syncwarp();  // this step's keys are read before they are replaced
            if ((lane & 3) == 0 && c < R) keys[c] = fp32_key(kk, a0);
        }
        __syncwarp();
        emit_best(keys, R);
    }
}

// Per row of X and of its low-precision copy (BF16 xb, or U8 xu): (an upper
// bound of |x|, an upper bound of |x~ - x|), each the sqrt of an FP64 sum of
// squares rounded up to FP32 (x~ - x is exact in FP64).  A row the copy holds
// exactly gets r = 0; a row with a non-finite coordinate gets r = +inf (every
// bound infinite).  A warp per row.
__global__ void k_band_rows(const float* __restrict__ X, const uint16_t* __restrict__ xb,
                            const uint8_t* __restrict__ xu, int64_t n, int d, float2* __restrict__ out) {
    const int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (r >= n) return;
    double s = 0.0, e = 0.0;
    for (int t = lane; t < d; t += 32) {
        const double v = X[r * d + t];
        const double w = xu ? (double)xu[r * d + t] : (double)__uint_as_float((uint32_t)xb[r * d + t] << 16);
        s += v * v;
        e += (v - w) * (v - w);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        e += __shfl_xor_sync(0xffffffffu, e, o);
    }
    if (lane == 0) {
        float nb = __double2float_ru(sqrt(s) * (1.0 + 0x1p-40));
        float rb = e == 0.0 ? 0.f : __double2float_ru(sqrt(e) * (1.0 + 0x1p-40));
        if (!(nb < INFINITY) || !(rb < INFINITY)) nb = rb = INFINITY;
        out[r] = make_float2(nb, rb);
    }
}

// Clears *ok unless every element of X [m] is an integer in [0, 255] (a
// byte holds it exactly; -0 counts as 0).
__global__ void k_bytes_exact(const float* __restrict__ X, int64_t m, int32_t* __restrict__ ok) {
    bool all = true;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int round = 0; i < m && all; i += (int64_t)gridDim.x * blockDim.x, ++round) {
        // (real-valued rows end the check at once, in every CTA)
        if ((round & 15) == 15 && *reinterpret_cast<const volatile int32_t*>(ok) == 0) break;
        const float v = X[i];
        all &= v >= 0.f && v <= 255.f && v == rintf(v);
    }
    __syncwarp();
    if (!__all_sync(0xffffffffu, all) && (threadIdx.x & 31) == 0) atomicAnd(ok, 0);
}

__global__ void k_x_u8(const float* __restrict__ X, int64_t m, uint8_t* __restrict__ xu) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        xu[i] = (uint8_t)X[i];
}

// ------------------------------------------------------------------ precision variant
// Low-precision copies of X for the widened first re-rank: BF16 rows, or FP8
// e4m3 rows with one FP32 scale per row (x ~ fp8(x / s) * s, s = max|x| / 448).
__global__ void k_x_lowp(const float* __restrict__ X, int64_t n, int d, int prec, uint16_t* __restrict__ xb,
                         uint8_t* __restrict__ x8, float* __restrict__ sc) {
    const int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (r >= n) return;
    const float* x = X + r * d;
    if (prec == 1) {
        for (int t = lane; t < d; t += 32) xb[r * d + t] = __bfloat16_as_ushort(__float2bfloat16_rn(x[t]));
        return;
    }
    float mx = 0.f;
    for (int t = lane; t < d; t += 32) mx = fmaxf(mx, fabsf(x[t]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const float s = mx > 0.f ? mx / 448.f : 1.f;
    if (lane == 0) sc[r] = s;
    for (int t = lane; t < d; t += 32)
        x8[r * d + t] = (uint8_t)__nv_cvt_float_to_fp8(x[t] / s, __NV_SATFINITE, __NV_E4M3);
}

// Diagnostic: distances of given (query, id) pairs in a precision.
__global__ void k_pair_dist(const float* __restrict__ Q, int64_t nq, int d, int ip, int prec,
                            const float* __restrict__ X, const uint16_t* __restrict__ xb,
                            const uint8_t* __restrict__ x8, const float* __restrict__ sc,
                            const int64_t* __restrict__ ids, int c, float* __restrict__ out) {
    __shared__ __align__(16) float qs[KSC_MAX_DIM];
    const int64_t q = blockIdx.x;
    for (int t = threadIdx.x; t < d; t += blockDim.x) qs[t] = Q[q * d + t];
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = w; i < c; i += nw) {
        const int64_t id = ids[q * c + i];
        const float v = id >= 0 ? lowp_dist(prec, qs, X, xb, x8, sc, (int32_t)id, d, ip, lane) : NAN;
        if (lane == 0) out[q * c + i] = ip ? -v : v;
    }
}

// Candidate export: each query's R selected keys, ascending (the select
// leaves them unordered).  One CTA per query.
__global__ void __launch_bounds__(256) k_copy_cands(const uint64_t* __restrict__ topr, int Rmax,
                                                    uint64_t* __restrict__ out) {
    extern __shared__ uint64_t cs[];
    const int64_t q = blockIdx.x;
    const int S = pow2_ceil(Rmax < 2 ? 2 : Rmax);
    for (int i = threadIdx.x; i < S; i += blockDim.x) cs[i] = i < Rmax ? topr[q * Rmax + i] : KEY_NONE;
    __syncthreads();
    block_bitonic_sort(cs, S);
    for (int i = threadIdx.x; i < Rmax; i += blockDim.x) out[q * Rmax + i] = cs[i];
}

// ------------------------------------------------------------------ host pipeline
// Stage boundary i (0 = start of stage 0, KSC_NUM_STAGES = end of the last).
static void mark(ksc_index* ix, int i, cudaStream_t st) {
    if (!ix->prof) return;
    cudaEventRecord(ix->ev[i], st);
    ix->ev_used[i] = true;
}

// Status word, item counts and counters of a search, cleared in one go (they
// share an allocation: index.cuh).
static int reset_counters(ksc_index* ix, cudaStream_t st) {
    KSC_CUDA(cudaMemsetAsync(ix->status, 0, STATUS_BYTES, st));
    return KSC_OK;
}
// The item counts alone (searches inside a training call keep the rest).
static int reset_items(ksc_index* ix, cudaStream_t st) {
    KSC_CUDA(cudaMemsetAsync(ix->status + STATUS_NREC, 0, 2 * sizeof(int32_t), st));
    return KSC_OK;
}

static unsigned blocks_for(int64_t work, int threads) { return (unsigned)((work + threads - 1) / threads); }

struct Plan {
    int64_t nq;
    int k, Pmax, Rmax, Pfix, Rfix;
    const int32_t* nprobe_q;
    const int32_t* rerank_q;
    int G, TB, TBa, cap;  // TB: tile blocks of the filtered scan, TBa: of the unfiltered first part
    int rank_mode;  // RankMode of the list scores
    bool hybrid;
    int n_near, efs, tau;
    int prec, Rf;  // precision variant: first re-rank of R (= Rmax) in prec, then FP32 of the best Rf
    bool band;     // exact re-rank with the band of U8 / BF16 rows (k_rerank_w, k_rerank_u8)
    bool band_now; // asked for by the caller: its copies are made at once
    int Pq_max;    // bound on the per-query nprobe (<= Pmax)
    double Pexp;   // expected nprobe
    bool tc;       // filtered scan on the tensor cores (k_scan_tc)
    bool tc_opt;   // asked for by the caller
    int nt;        // its queries per item
    bool small;    // the small-batch kernels (small.cu) around the scan,
    bool rank;     // which also rank the lists (no ranking has run)
    bool all_near; // no filtered part: the store holds every key a query can probe
    int64_t nrec;  // bound on the scan items of either part
};

static int choose_G(const ksc_index* ix, int64_t nq, int Pmax, int want) {
    if (want == 4 && ix->M <= 128) return 4;
    if (want == 8 || want == 16 || want == 32) {
        int S = (ix->M + want - 1) / want;
        if (S <= 16) return want;
    }
    // 8 lanes per query (4 query slots per warp) up to 128 subspaces: when
    // fewer queries than slots probe a list, the item's slots split its
    // blocks instead, so every lane stays busy at any batch size, and the
    // per-block reduction runs over 8 lanes only
    (void)nq;
    (void)Pmax;
    if (ix->M <= 128) return 8;
    if (ix->M <= 256) return 16;
    return 32;
}

template <int G, int SMAX>
static int launch_scan(const ScanArgs& A, const ScanOut& O, const int64_t* pair_off, const int64_t* item_off,
                       const uint32_t* pairs, int L, int TB, int32_t* status, cudaStream_t st) {
    const size_t smem = (size_t)SCAN_WARPS * 2 * scan_chunk_bytes<G>() +
                        (scan_shared_sel<G>() ? (size_t)SCAN_WARPS * A.M * 64 : 0);
    // M = G SMAX: every lane has SMAX subspaces, no per-subspace guards
    const bool full = A.M == G * SMAX;
    auto kern = O.thr ? (full ? k_scan<G, SMAX, false, true, false> : k_scan<G, SMAX, false, false, false>)
                      : (full ? k_scan<G, SMAX, true, true, false> : k_scan<G, SMAX, true, false, false>);
    if constexpr (G <= 16)
        if (O.recs) kern = O.thr ? k_scan<G, SMAX, false, false, true> : k_scan<G, SMAX, true, false, true>;
    KSC_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    KSC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, SCAN_WARPS * 32, smem));
    const int grid = num_sms() * (per_sm > 0 ? per_sm : 1);
    kern<<<grid, SCAN_WARPS * 32, smem, st>>>(A, O, pair_off, item_off, pairs, L, TB, status);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

template <int MAXM>
static int launch_scan4(const ScanArgs& A, const ScanOut& O, const int64_t* pair_off, const int64_t* item_off,
                        const uint32_t* pairs, int L, int TB, int32_t* status, cudaStream_t st) {
    const size_t smem = (size_t)S4_WARPS * s4_warp_bytes<MAXM>();
    KSC_CUDA(cudaFuncSetAttribute(k_scan4<MAXM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    KSC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_scan4<MAXM>, S4_WARPS * 32, smem));
    const int grid = num_sms() * (per_sm > 0 ? per_sm : 1);
    k_scan4<MAXM><<<grid, S4_WARPS * 32, smem, st>>>(A, O, pair_off, item_off, pairs, L, TB, status);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

template <int G>
static int dispatch_scan(int S, const ScanArgs& A, const ScanOut& O, const int64_t* pair_off,
                         const int64_t* item_off, const uint32_t* pairs, int L, int TB, int32_t* status,
                         cudaStream_t st) {
    if (S <= 2) return launch_scan<G, 2>(A, O, pair_off, item_off, pairs, L, TB, status, st);
    if (S <= 4) return launch_scan<G, 4>(A, O, pair_off, item_off, pairs, L, TB, status, st);
    if constexpr (G == 8)
        if (S == 6) return launch_scan<G, 6>(A, O, pair_off, item_off, pairs, L, TB, status, st);  // M 48
    if (S <= 8) return launch_scan<G, 8>(A, O, pair_off, item_off, pairs, L, TB, status, st);
    if (S <= 16) return launch_scan<G, 16>(A, O, pair_off, item_off, pairs, L, TB, status, st);
    set_error("M too large for %d lanes per query", G);
    return KSC_EINVAL;
}

// Operand type of the list scores (a1): 16-bit tensor cores, FP32 CUDA
// cores, or FP8 tensor cores.
enum RankMode { RANK_TC16 = 0, RANK_FP32 = 1, RANK_FP8 = 2 };
// Widest rows whose given scores come from the tensor cores everywhere; wider
// ones only where the scores just preselect lists for the exact ranking.
constexpr int TC_SCORES_D = 256;

// List scores [nq x L] on the 16-bit or FP8 tensor cores or the FP32 CUDA
// cores, with the per-query bound err [nq] on their distance from the exact
// scores.
static int list_scores(ksc_index* ix, const float* Q, int64_t nq, int mode, float* scores, float** err,
                       cudaStream_t st, bool preselect = false) {
    KSC_TRY(ensure(ix->ws_err, sizeof(float) * nq, st));
    *err = (float*)ix->ws_err.p;
    // rows past TC_SCORES_D: the scores themselves stay FP32 (ksc_list_scores,
    // the predictor's features); a ranking re-scores exactly whatever the
    // scores' bound cannot exclude, so it takes the 16-bit tensor cores there
    // too where that bound excludes most lists and the rest always fit the
    // re-score buffer (10,000 x 784 against 256 lists: 365 us of FP32 scores and
    // bounds before, 32 us now)
    bool wide_tc = false;
    if (preselect && mode == RANK_TC16 && ix->d > TC_SCORES_D) KSC_TRY(rank_tc_narrow(ix, &wide_tc, st));
    if (mode != RANK_FP32 && (ix->d <= TC_SCORES_D || wide_tc))
        return mode == RANK_FP8 ? rank_scores_tc8(ix, Q, nq, scores, *err, st)
                                : rank_scores_tc(ix, Q, nq, scores, *err, st);
    dim3 grid(blocks_for(ix->L, SC_T), blocks_for(nq, SC_T));
    k_list_scores<<<grid, 256, 0, st>>>(Q, nq, ix->d, ix->c_rank, ix->c_rank_sq, ix->L, ix->spherical, scores);
    ix->launches++;
    KSC_LAUNCH_CHECK();
    return score_err(ix, Q, nq, false, *err, st);
}

// The Pmax best lists of every query (exact ranking); feat (optional, L >=
// FEAT_K) receives each query's FEAT_K smallest given list distances.
// The warp kernel ranks a batch when its lists fit a warp's share of shared
// memory and the batch fills the GPU.
static bool rank_by_warp(const ksc_index* ix, int64_t nq, int Pmax) {
    return ix->L <= RSW_MAX_L && Pmax <= 4 * RSW_CAND / 8 && warp_per_query(nq);
}

// The P best lists of every query from the given approximate scores (an
// error bound per query in err), exactly re-scored; feat: the predictor's
// distances as well.
static int select_lists(ksc_index* ix, const float* scores, const float* err, const float* Q, int64_t nq,
                        const int32_t* nprobe_q, int Pfix, int Pmax, int32_t* probes, float* score_out,
                        cudaStream_t st, float* feat);

static int rank_lists(ksc_index* ix, const float* Q, int64_t nq, const int32_t* nprobe_q, int Pfix, int Pmax,
                      int32_t* probes, float* score_out, int mode, cudaStream_t st, float* feat = nullptr) {
    KSC_TRY(ensure(ix->ws_scores, sizeof(float) * nq * ix->L, st));
    float* scores = (float*)ix->ws_scores.p;
    float* err = nullptr;
    KSC_TRY(list_scores(ix, Q, nq, mode, scores, &err, st, !feat));
    return select_lists(ix, scores, err, Q, nq, nprobe_q, Pfix, Pmax, probes, score_out, st, feat);
}

static int select_lists(ksc_index* ix, const float* scores, const float* err, const float* Q, int64_t nq,
                        const int32_t* nprobe_q, int Pfix, int Pmax, int32_t* probes, float* score_out,
                        cudaStream_t st, float* feat) {
    // re-score buffer of the CTA kernel: 4 Pmax lists (a power of two, at least 1024, at most RS_CAP)
    static_assert(RANK_TC_LISTS <= 1024, "wide rows' 16-bit scores rely on a buffer of every list");
    const int rs_cap = std::min(RS_CAP, std::max(1024, pow2_ceil(4 * Pmax)));
    const size_t smem = rs_cap * sizeof(uint64_t) + (ix->L <= RS_SMEM_L ? sizeof(float) * ix->L : 0);
    KSC_CUDA(cudaFuncSetAttribute(k_rank_select<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    KSC_CUDA(cudaFuncSetAttribute(k_rank_select<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (rank_by_warp(ix, nq, Pmax)) {
        // a warp per query; queries with too many lists inside the bound go to the CTA kernel
        KSC_TRY(ensure(ix->ws_redo, sizeof(int32_t) * (nq + 1), st));
        int32_t* redo = (int32_t*)ix->ws_redo.p;
        KSC_CUDA(cudaMemsetAsync(redo, 0, sizeof(int32_t), st));
        const size_t wsm = sizeof(uint64_t) * RSW_WARPS * RSW_CAND + sizeof(float) * RSW_WARPS * ix->L;
        KSC_CUDA(cudaFuncSetAttribute(k_rank_select_w, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wsm));
        k_rank_select_w<<<(unsigned)((nq + RSW_WARPS - 1) / RSW_WARPS), RSW_WARPS * 32, wsm, st>>>(
            scores, err, Q, ix->c_rank, nq, ix->d, ix->L, ix->spherical, nprobe_q, Pfix, Pmax, probes, score_out,
            redo, feat);
        feat = nullptr;  // written
        KSC_LAUNCH_CHECK();
        k_rank_select<256><<<num_sms() * 2, 256, smem, st>>>(scores, err, Q, ix->c_rank, nq, ix->d, ix->L, ix->spherical,
                                                        nprobe_q, Pfix, Pmax, rs_cap, probes, score_out, redo);
        ix->launches += 2;
    } else {
        // a CTA per query; 1024 threads when the batch is too small to fill the GPU
        if (nq < 2 * (int64_t)num_sms())
            k_rank_select<1024><<<(unsigned)nq, 1024, smem, st>>>(scores, err, Q, ix->c_rank, nq, ix->d, ix->L,
                                                                  ix->spherical, nprobe_q, Pfix, Pmax, rs_cap, probes,
                                                                  score_out, nullptr);
        else
            k_rank_select<256><<<(unsigned)nq, 256, smem, st>>>(scores, err, Q, ix->c_rank, nq, ix->d, ix->L,
                                                                ix->spherical, nprobe_q, Pfix, Pmax, rs_cap, probes,
                                                                score_out, nullptr);
        ix->launches++;
    }
    KSC_LAUNCH_CHECK();
    if (feat) {
        k_feat_scores<<<(unsigned)((nq + 7) / 8), 256, 0, st>>>(scores, Q, ix->d, ix->spherical, nq, ix->L, feat);
        KSC_LAUNCH_CHECK();
        ix->launches++;
    }
    return KSC_OK;
}

static int launch_luts(const LutArgs& A, uint32_t* rb, uint8_t* lut, int32_t* bias, float* scale, cudaStream_t st) {
    const size_t smem = sizeof(float) * (size_t)A.M * cb_ld(A.dsub);
    const int64_t warps = (A.nq * A.Pmax + LUT_WARPS - 1) / LUT_WARPS;  // a warp per item
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(warps, (int64_t)num_sms() * 8));
    const int w = lut_width(A, false);
    auto kr = w == 2 ? k_lut_range<2> : (w == 4 ? k_lut_range<4> : k_lut_range<0>);
    auto kq = w == 2 ? k_lut_quant<2> : (w == 4 ? k_lut_quant<4> : k_lut_quant<0>);
    KSC_CUDA(cudaFuncSetAttribute(kr, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    KSC_CUDA(cudaFuncSetAttribute(kq, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kr<<<grid, LUT_WARPS * 32, smem, st>>>(A, rb);
    KSC_LAUNCH_CHECK();
    kq<<<grid, LUT_WARPS * 32, smem, st>>>(A, rb, lut, bias, scale);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

static int compute_luts(ksc_index* ix, const float* Q, int64_t nq, const int32_t* probes, const int32_t* nprobe_q,
                        int Pfix, int Pmax, uint8_t* lut, int32_t* bias, float* scale, cudaStream_t st) {
    KSC_TRY(ensure(ix->ws_range, sizeof(uint32_t) * nq, st));
    uint32_t* rb = (uint32_t*)ix->ws_range.p;
    KSC_CUDA(cudaMemsetAsync(rb, 0, sizeof(uint32_t) * nq, st));
    LutArgs A{Q, nq, ix->d, ix->M, ix->dsub, ix->metric == KSC_IP, Pmax, probes, nprobe_q, Pfix, ix->c_mean,
              ix->codebook, ix->L};
    KSC_TRY(launch_luts(A, rb, lut, bias, scale, st));
    ix->launches += 2;
    return KSC_OK;
}

// BF16 / FP8 copies of the re-rank vectors, made on first use.
static int ensure_lowp(ksc_index* ix, int prec, cudaStream_t st) {
    const int dr = rr_d(ix);
    if (prec == 1 && !ix->X_bf16) {
        KSC_CUDA(cudaMalloc(&ix->X_bf16, sizeof(uint16_t) * ix->n * dr));
        k_x_lowp<<<(unsigned)((ix->n + 7) / 8), 256, 0, st>>>(rr_X(ix), ix->n, dr, 1, (uint16_t*)ix->X_bf16, nullptr,
                                                              nullptr);
        KSC_LAUNCH_CHECK();
    }
    if (prec == 2 && !ix->X_fp8) {
        KSC_CUDA(cudaMalloc(&ix->X_fp8, (size_t)ix->n * dr));
        KSC_CUDA(cudaMalloc(&ix->X_scale, sizeof(float) * ix->n));
        k_x_lowp<<<(unsigned)((ix->n + 7) / 8), 256, 0, st>>>(rr_X(ix), ix->n, dr, 2, nullptr, (uint8_t*)ix->X_fp8,
                                                              ix->X_scale);
        KSC_LAUNCH_CHECK();
    }
    return KSC_OK;
}

// U8 copies of the re-rank rows when every coordinate is an integer in [0,
// 255] (checked once, x_u8_state).  Synchronises the stream on first use.
static int ensure_u8(ksc_index* ix, cudaStream_t st) {
    const int64_t m = ix->n * (int64_t)rr_d(ix);
    if (ix->x_u8_state == 0) {
        KSC_TRY(ensure(ix->ws_flag, sizeof(int32_t), st));
        int32_t* ok = (int32_t*)ix->ws_flag.p;
        const int32_t one = 1;
        KSC_CUDA(cudaMemcpyAsync(ok, &one, sizeof(int32_t), cudaMemcpyHostToDevice, st));
        k_bytes_exact<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>((m + 255) / 256, 8 * (int64_t)num_sms())),
                        256, 0, st>>>(rr_X(ix), m, ok);
        KSC_LAUNCH_CHECK();
        int32_t h = 0;
        KSC_CUDA(cudaMemcpyAsync(&h, ok, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        KSC_CUDA(cudaStreamSynchronize(st));
        ix->x_u8_state = (h && m > 0) ? 2 : -1;
    }
    if (ix->x_u8_state == 2) {
        if (!ix->X_u8) KSC_CUDA(cudaMalloc(&ix->X_u8, (size_t)m));
        k_x_u8<<<(unsigned)std::min<int64_t>((m + 255) / 256, 8 * (int64_t)num_sms()), 256, 0, st>>>(
            rr_X(ix), m, (uint8_t*)ix->X_u8);
        KSC_LAUNCH_CHECK();
        ix->x_u8_state = 1;  // only once the copy exists
    }
    return KSC_OK;
}

// Whether U8 copies of the re-rank rows are there for a re-rank of `rows`
// candidates.  Making them (a pass over the rows, their check and copy, n d bytes
// of memory, a synchronisation) costs about what re-ranking 19 candidates per
// row of the index in bytes saves (60k x 784: 450 us; 10,000 queries of 200
// candidates 848 -> 477 us), so they are made once the handle has re-ranked
// U8_AFTER per row, at once (`now`) for a plan and for a caller who asks for the
// band: a program that searches an index a few times does not pay for them.  Not while the stream is captured; where the
// device has no room, tried again after as many candidates more.
constexpr int64_t U8_AFTER = 16;
static bool u8_rows(ksc_index* ix, int64_t rows, bool now, cudaStream_t st) {
    if (ix->x_u8_state == 0 || ix->x_u8_state == 2) {
        ix->u8_wanted += rows;
        if (!now && !ix->u8_now && ix->u8_wanted < U8_AFTER * ix->n) return false;
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) return false;
        if (ensure_u8(ix, st) != KSC_OK) {
            cudaGetLastError();
            ix->u8_wanted = 0;
        }
    }
    return ix->x_u8_state == 1;
}

// The band of the exact re-rank, made on first use: U8 copies of the rows
// when every coordinate is an integer in [0, 255] (checked once; exact, a
// quarter of the FP32 bytes), else BF16 copies; and the rows' bounds (norm,
// rounding error).
static int ensure_band(ksc_index* ix, cudaStream_t st) {
    KSC_TRY(ensure_u8(ix, st));
    const bool u8 = ix->x_u8_state == 1;
    if (!u8) KSC_TRY(ensure_lowp(ix, 1, st));
    if (!ix->X_band) {
        KSC_CUDA(cudaMalloc(&ix->X_band, sizeof(float2) * ix->n));
        k_band_rows<<<(unsigned)((ix->n + 7) / 8), 256, 0, st>>>(
            rr_X(ix), u8 ? nullptr : (const uint16_t*)ix->X_bf16, u8 ? (const uint8_t*)ix->X_u8 : nullptr, ix->n,
            rr_d(ix), ix->X_band);
        KSC_LAUNCH_CHECK();
    }
    return KSC_OK;
}

template <int SMAX, int NR>
static int launch_graph_search_t(const ScanArgs& A, const ScanOut& O, const GraphArgs& Gr, const uint32_t* pairs,
                                 const int64_t* npairs, cudaStream_t st) {
    const size_t smem = sizeof(uint32_t) * GS_WARPS * (size_t)Gr.vwords;
    auto kern = k_graph_search<SMAX, NR>;
    KSC_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    KSC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, GS_WARPS * 32, smem));
    kern<<<num_sms() * (per_sm > 0 ? per_sm : 1), GS_WARPS * 32, smem, st>>>(A, O, Gr, pairs, npairs);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

// The graph search with as many subspaces and result entries per lane as M
// and efs need.
static int launch_graph_search(const ScanArgs& A, const ScanOut& O, const GraphArgs& Gr, const uint32_t* pairs,
                               const int64_t* npairs, cudaStream_t st) {
    const int sg = (A.M + 31) / 32, nr = (Gr.efs + 31) / 32;
#define KSC_GS(SM)                                                                            \
    (nr <= 1 ? launch_graph_search_t<SM, 1>(A, O, Gr, pairs, npairs, st)                      \
             : (nr == 2 ? launch_graph_search_t<SM, 2>(A, O, Gr, pairs, npairs, st)           \
                        : launch_graph_search_t<SM, 3>(A, O, Gr, pairs, npairs, st)))
    if (sg <= 1) return KSC_GS(1);
    if (sg <= 2) return KSC_GS(2);
    if (sg <= 4) return KSC_GS(4);
    return KSC_GS(8);
#undef KSC_GS
}

// Cluster-major work list of the (query, rank) pairs of one part of the probe
// ranks (the unfiltered first part or the rest).
struct WorkList {
    int64_t* pair_off;  // [L + 1]
    int64_t* item_off;  // [L + 1]
    int32_t* cnt;       // [L]
    int32_t* fill;      // [L]
    uint32_t* pairs;    // [<= nq * Pmax]
    int TB;             // blocks per item tile
};

static int run_scan(const Plan& pl, int M, const ScanArgs& A, const ScanOut& O, const WorkList& w, int L,
                    int32_t* status, cudaStream_t st, unsigned long long* next_item, bool tc) {
    if (tc) return launch_scan_tc(A, O, w.pair_off, w.item_off, w.pairs, L, w.TB, pl.nt, next_item, status, st);
    const int S = (M + pl.G - 1) / pl.G;
    if (pl.G == 4) {
        if (M <= 64) return launch_scan4<64>(A, O, w.pair_off, w.item_off, w.pairs, L, w.TB, status, st);
        if (M <= 128) return launch_scan4<128>(A, O, w.pair_off, w.item_off, w.pairs, L, w.TB, status, st);
        set_error("M too large for 4 lanes per query");
        return KSC_EINVAL;
    }
    if (pl.G == 8) return dispatch_scan<8>(S, A, O, w.pair_off, w.item_off, w.pairs, L, w.TB, status, st);
    if (pl.G == 16) return dispatch_scan<16>(S, A, O, w.pair_off, w.item_off, w.pairs, L, w.TB, status, st);
    return dispatch_scan<32>(S, A, O, w.pair_off, w.item_off, w.pairs, L, w.TB, status, st);
}

// a2 .. a6 for given probe lists.  Stages: 1 work lists, 2 LUTs, 3 scan of
// the nearest list(s) + threshold, 4 scan of the other lists, 5 select,
// 6 rerank.
// Queries in the index's working dimensions: with component filtration
// (Sec. 4.3, Alg. 2 FilterComponents) the kept dimensions of Q, gathered into
// a workspace buffer (zeros in the padding); otherwise Q itself.
static int work_queries(ksc_index* ix, const float* Q, int64_t nq, cudaStream_t st, const float** Qw) {
    *Qw = Q;
    if (!ix->dims || nq == 0) return KSC_OK;
    KSC_TRY(ensure(ix->ws_qf, sizeof(float) * nq * ix->d, st));
    KSC_TRY(gather_dims(Q, nq, ix->d_rr, ix->dims, ix->d, (float*)ix->ws_qf.p, st));
    ix->launches++;
    *Qw = (const float*)ix->ws_qf.p;
    return KSC_OK;
}

// 6. exact rerank of the selected keys topr (precision variant: a BF16 / FP8
//    re-rank of the widened shortlist first, then FP32 of its best Rf), with
//    the full queries and vectors (Alg. 2: q_init)
static int rerank_stage(ksc_index* ix, const float* Qr, const Plan& pl, const uint64_t* topr, int64_t* ids,
                        float* dists, cudaStream_t st) {
    const int64_t nq = pl.nq;
    mark(ix, 6, st);
    const float* Xr = rr_X(ix);
    const int dr = rr_d(ix);
    const uint64_t* rr_keys = topr;
    int rr_R = pl.Rmax;
    const int32_t* rr_q = pl.rerank_q;
    if (pl.prec > 0) {
        KSC_TRY(ensure_lowp(ix, pl.prec, st));
        KSC_TRY(ensure(ix->ws_topr2, sizeof(uint64_t) * nq * pl.Rf, st));
        uint64_t* topr2 = (uint64_t*)ix->ws_topr2.p;
        KSC_TRY(launch_rerank_lowp(Qr, nq, dr, ix->metric == KSC_IP, pl.prec, (const uint16_t*)ix->X_bf16,
                                   (const uint8_t*)ix->X_fp8, ix->X_scale, topr, pl.Rmax, pl.rerank_q, pl.Rfix, pl.k,
                                   pl.Rf, topr2, st));
        ix->launches++;
        rr_keys = topr2;
        rr_R = pl.Rf;
        rr_q = nullptr;
    }
    if (pl.k <= 32 && rr_R <= RW_MAXR && dr <= 128 && (dr & 3) == 0 && warp_per_query(nq)) {
        const bool band = pl.band && pl.prec == 0 && rr_R > pl.k;
        if (band) KSC_TRY(ensure_band(ix, st));
        const size_t smem = sizeof(uint64_t) * RW_WARPS * rr_R * (band ? 2 : 1) +
                            (band ? sizeof(uint32_t) * RW_WARPS * (rr_R + 64) : 0);
        auto kr = band && ix->x_u8_state == 1 ? k_rerank_w<true> : k_rerank_w<false>;
        KSC_CUDA(cudaFuncSetAttribute(kr, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kr<<<(unsigned)((nq + RW_WARPS - 1) / RW_WARPS), RW_WARPS * 32, smem, st>>>(
            Qr, Xr, dr, ix->metric == KSC_IP, rr_keys, rr_R, rr_q, rr_R, pl.k, nq, ids, dists,
            band && ix->x_u8_state != 1 ? (const uint16_t*)ix->X_bf16 : nullptr,
            band && ix->x_u8_state == 1 ? (const uint8_t*)ix->X_u8 : nullptr, band ? ix->X_band : nullptr);
        ix->launches++;
        KSC_LAUNCH_CHECK();
    } else if (pl.band && pl.prec == 0 && rr_R > pl.k && ix->metric != KSC_IP && nq >= 2 * (int64_t)num_sms() &&
               rerank_u8_supported(dr) && u8_rows(ix, nq * rr_R, pl.band_now, st)) {
        KSC_TRY(launch_rerank_u8(Qr, nq, Xr, (const uint8_t*)ix->X_u8, dr, rr_keys, rr_R, rr_q, rr_R, pl.k, ids, dists,
                                 st));
        ix->launches++;
    } else {
        const size_t smem = rerank_smem(rr_R, pl.k);
        // a CTA per query; 1024 threads (more rows in flight) when the batch is
        // too small to fill the GPU with 256-thread CTAs
        if (nq < 2 * (int64_t)num_sms()) {
            KSC_CUDA(cudaFuncSetAttribute(k_rerank<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k_rerank<1024><<<(unsigned)nq, 1024, smem, st>>>(Qr, Xr, dr, ix->metric == KSC_IP, rr_keys, rr_R, rr_q,
                                                             rr_R, pl.k, ids, dists);
        } else {
            KSC_CUDA(cudaFuncSetAttribute(k_rerank<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k_rerank<256><<<(unsigned)nq, 256, smem, st>>>(Qr, Xr, dr, ix->metric == KSC_IP, rr_keys, rr_R, rr_q,
                                                           rr_R, pl.k, ids, dists);
        }
        ix->launches++;
        KSC_LAUNCH_CHECK();
    }
    mark(ix, KSC_NUM_STAGES, st);
    return KSC_OK;
}

// 5. the R best keys per query into topr (and, sorted, cand_out)
static int select_stage(ksc_index* ix, const Plan& pl, const ScanArgs& A, const int32_t* cnt, uint64_t* cand,
                        uint64_t* topr, uint64_t* cand_out, int32_t* ncand_out, cudaStream_t st) {
    const int64_t nq = pl.nq;
    {
        KSC_TRY(ensure(ix->ws_redo, sizeof(int32_t) * (nq + 1), st));
        int32_t* redo = (int32_t*)ix->ws_redo.p;
        KSC_CUDA(cudaMemsetAsync(redo, 0, sizeof(int32_t), st));
        // candidates per query: the R kept by the threshold plus a few R more
        if (select_by_warp(nq, 4.0 * pl.Rmax)) {
            k_select<<<(unsigned)((nq + SW_WARPS - 1) / SW_WARPS), SW_WARPS * 32, 0, st>>>(
                A, pl.Rmax, cnt, cand, pl.cap, topr, ncand_out, ix->status, ix->stats, redo);
        } else {
            const bool few = nq < 2 * (int64_t)num_sms(), narrow = 4 * pl.Rmax <= SW_MAX_KEYS && warp_per_query(nq);
            auto kf = few ? k_select_cta<1024, 0> : narrow ? k_select_cta<128, 16> : k_select_cta<256, 0>;
            kf<<<(unsigned)nq, few ? 1024 : narrow ? 128 : 256, 0, st>>>(A, pl.Rmax, cnt, cand, pl.cap, topr, ncand_out,
                                                                        ix->status, ix->stats, redo);
        }
        KSC_LAUNCH_CHECK();
        // overflowed queries (usually none): their keys recomputed
        const int sel_cap = sel_keys(pl.Rmax);
        const size_t smem = sel_cap * sizeof(uint64_t);
        KSC_CUDA(cudaFuncSetAttribute(k_select_redo, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        k_select_redo<<<num_sms(), 1024, smem, st>>>(A, pl.Rmax, sel_cap, cand, pl.cap, topr, ncand_out, redo);
        KSC_LAUNCH_CHECK();
        ix->launches += 2;
    }
    if (cand_out) {
        const size_t csm = sizeof(uint64_t) * pow2_ceil(pl.Rmax < 2 ? 2 : pl.Rmax);
        KSC_CUDA(cudaFuncSetAttribute(k_copy_cands, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)csm));
        k_copy_cands<<<(unsigned)nq, 256, csm, st>>>(topr, pl.Rmax, cand_out);
        ix->launches++;
        KSC_LAUNCH_CHECK();
    }
    return KSC_OK;
}

// The search of a few queries (small.cu).
static int search_small(ksc_index* ix, const float* Q, const Plan& pl, const int32_t* probes, int64_t* ids,
                        float* dists, uint64_t* cand_out, int32_t* ncand_out, cudaStream_t st, const float* Qr) {
    const int64_t nq = pl.nq;
    const int M = ix->M;
    KSC_TRY(ensure(ix->ws_lut, (size_t)nq * pl.Pmax * M * PQ_K, st));
    KSC_TRY(ensure(ix->ws_bias, sizeof(int32_t) * nq * pl.Pmax, st));
    KSC_TRY(ensure(ix->ws_scale, sizeof(float) * nq, st));
    KSC_TRY(ensure(ix->ws_thr, sizeof(uint64_t) * nq, st));
    KSC_TRY(ensure(ix->ws_cnt, sizeof(int32_t) * nq, st));
    KSC_TRY(ensure(ix->ws_cand, sizeof(uint64_t) * nq * pl.cap, st));
    KSC_TRY(ensure(ix->ws_topr, sizeof(uint64_t) * nq * pl.Rmax, st));
    KSC_TRY(ensure(ix->ws_items, sizeof(int4) * 2 * pl.nrec + sizeof(int32_t) * nq * pl.Pmax, st));
    int32_t* bias = (int32_t*)ix->ws_bias.p;
    uint8_t* lut = (uint8_t*)ix->ws_lut.p;
    int32_t* cnt = (int32_t*)ix->ws_cnt.p;
    uint64_t* thr = (uint64_t*)ix->ws_thr.p;
    uint64_t* cand = (uint64_t*)ix->ws_cand.p;
    uint64_t* topr = (uint64_t*)ix->ws_topr.p;
    int4* recs = (int4*)ix->ws_items.p;
    int32_t* nrec = ix->status + STATUS_NREC;
    ScanArgs A{M, pl.Pmax, nq, probes, pl.nprobe_q, pl.Pfix, pl.rerank_q, pl.Rfix, pl.k, lut, bias,
               ix->list_boff, ix->list_n, ix->blk_codes, ix->blk_ids, ix->L};
    SmallPrep S{};
    S.T = LutArgs{Q, nq, ix->d, M, ix->dsub, ix->metric == KSC_IP, pl.Pmax, probes, pl.nprobe_q, pl.Pfix, ix->c_mean,
                  ix->codebook, ix->L};
    S.A = A;
    S.c_rank = pl.rank ? ix->c_rank : nullptr;
    S.spherical = ix->spherical;
    S.probes_out = const_cast<int32_t*>(probes);  // written only when pl.rank: then the handle's own buffer
    S.lut = lut;
    S.bias = bias;
    S.scale = (float*)ix->ws_scale.p;
    S.cnt = cnt;
    S.noff = (int32_t*)(recs + 2 * pl.nrec);
    S.recsA = recs;
    S.recsB = recs + pl.nrec;
    S.nrec = nrec;
    S.TBa = pl.TBa;
    S.TB = pl.TB;
    S.Rmax = pl.Rmax;
    S.cap = pl.cap;
    S.all_near = pl.all_near;
    S.near_keys_per_r = NEAR_KEYS_PER_R;
    S.near_share_div = NEAR_SHARE_DIV;
    KSC_TRY(launch_small_prep(S, st));
    ix->launches++;
    for (int i = 1; i <= 3; ++i) mark(ix, i, st);
    const WorkList none{};
    KSC_TRY(run_scan(pl, M, A, ScanOut{nullptr, cnt, cand, pl.cap, S.recsA, nrec, S.noff}, none, ix->L, ix->status, st,
                     nullptr, false));
    ix->launches++;
    if (!pl.all_near) {
        k_threshold_cta<1024, 0><<<(unsigned)nq, 1024, 0, st>>>(A, pl.Rmax, cnt, cand, pl.cap, topr, thr);
        KSC_LAUNCH_CHECK();
        ix->launches++;
    }
    mark(ix, 4, st);
    if (!pl.all_near) {
        KSC_TRY(run_scan(pl, M, A, ScanOut{thr, cnt, cand, pl.cap, S.recsB, nrec + 1, S.noff}, none, ix->L, ix->status,
                         st, nullptr, false));
        ix->launches++;
    }
    mark(ix, 5, st);
    if (cand_out || pl.prec > 0 || !ids) {
        KSC_TRY(select_stage(ix, pl, A, cnt, cand, topr, cand_out, ncand_out, st));
        if (!ids && !dists) {  // candidates only
            mark(ix, 6, st);
            mark(ix, KSC_NUM_STAGES, st);
            return KSC_OK;
        }
        return rerank_stage(ix, Qr, pl, topr, ids, dists, st);
    }
    KSC_TRY(launch_select_rerank(A, pl.Rmax, cnt, cand, pl.cap, pl.all_near ? 0 : sel_keys(pl.Rmax), Qr, rr_X(ix),
                                 rr_d(ix), ix->metric == KSC_IP, pl.k, ids, dists, ix->status, ix->stats, st));
    ix->launches++;
    mark(ix, 6, st);
    mark(ix, KSC_NUM_STAGES, st);
    return KSC_OK;
}

// Whether the small-batch kernels serve this search (small.cu).  They give a
// query a cluster and a CTA of its own, so they pay off while those fill the
// GPU at most about twice (2 SMs' worth of queries: the general kernels then
// share lists and tables between queries); the rest are limits of their
// buffers.  distinct: no list occurs twice in a query's probes (a ranking);
// can_rank: the lists are not ranked yet.
//  - ranking: every list is scored exactly by the query's own cluster, L d
//    floats from L2 per query: up to SMALL_RANK_BYTES over the batch (1024 x
//    128, one query: 5 us of k_small_prep against 20 us of the three ranking
//    kernels; at 128 queries those 64 MB take about as long as the tensor
//    cores' path).
// One query of 1M x 128 at nprobe 7 from a plan: 97.6 us before, 49 now; 100
// queries of 10k x 128 by direct calls 112.9 and 58; 16 queries at nprobe up to
// 256 and R up to 1000 of 1M x 96 158 and 72.
//  - all_near: if no query can probe more than SMALL_NEAR_KEYS keys, the store
//    holds all of them and the threshold, the second scan and its items go.
//  - pairs of a query and a probed list: with many, the general path's shared
//    lists win (299 queries at up to 144 probes of 758k x 96, 43,000 pairs: 288 us
//    here, 265 there; 158 at up to 199, 31,000 pairs: 205 here, 234 there).
//  - sharing: the general path reads a list's codes and builds its selectors once
//    for several queries, the small one for each.  Where more than two queries
//    share a list (one, past 256 queries), it is taken only up to SMALL_SHARED_NQ
//    queries and SMALL_LOOKUPS table lookups, fewer the more queries there are
//    (SMALL_NQ_LOOKUPS over their number).  Here / there in us, 1M x 64 subspaces in 1024
//    lists: 303 queries at nprobe 16 259 / 212, at 4 162 / 169; 200 at 16 206 /
//    188, at 8 158 / 170; 150 at 32 213 / 191, at 16 163 / 170; 64 at 256 382 /
//    331, at 64 164 / 194; 303 on 10k x 64 in 64 lists at 16 174 / 144; 250 on 1M x
//    48 in 4096 lists at 64 201 / 204, at 16 136 / 154; 303 there at 64 226 / 212.
constexpr int64_t SMALL_MAX_PAIRS = 40000;
constexpr int64_t SMALL_RANK_BYTES = 64 << 20;
constexpr int64_t SMALL_NEAR_KEYS = 32768;
constexpr int64_t SMALL_MAX_RECS = 1 << 22;
constexpr int64_t SMALL_SHARED_NQ = 200;
constexpr double SMALL_LOOKUPS = 450e6, SMALL_NQ_LOOKUPS = 36e9;
static void plan_small(const ksc_index* ix, Plan& pl, const ksc_search_opts* opts, bool distinct, bool can_rank) {
    const int64_t nq = pl.nq, P = pl.Pmax;
    if (nq == 0 || nq >= 2 * (int64_t)num_sms() || pl.hybrid || pl.tc_opt || (pl.G != 8 && pl.G != 16) || P > SP_MAX_P ||
        nq * P > SMALL_MAX_PAIRS || P * ix->max_list >= (1ll << 31))
        return;
    const double share = (double)nq * pl.Pexp / ix->L, lookups = share * (double)ix->n * ix->M;
    if (share > (nq > 256 ? 1.0 : 2.0) &&
        (nq > SMALL_SHARED_NQ || lookups > SMALL_LOOKUPS || nq * lookups > SMALL_NQ_LOOKUPS))
        return;
    const int64_t maxb = (ix->max_list + 31) / 32;
    const int64_t blocks = distinct ? ix->h_top_blocks[P] : P * maxb;
    const int64_t keys = std::min(32 * blocks, P * (int64_t)ix->max_list);
    const bool own_cap = opts && opts->cand_cap > 0;
    const bool near = keys <= (own_cap ? std::min<int64_t>(pl.cap, SMALL_NEAR_KEYS) : SMALL_NEAR_KEYS);
    int TB = pl.TB, TBa = pl.TBa;
    if (!(opts && opts->tile_blocks > 0)) {
        // a pair per item: about 8 items per warp of the scan, 4 to 32 blocks each
        const double per = (double)nq * P * ix->nblocks / ix->L / (60.0 * num_sms());
        TB = TBa = per < 4 ? 4 : (per > 32 ? 32 : (int)per);
    }
    const int64_t nrec = nq * (P + blocks / std::min(TB, TBa) + 1);
    if (nrec > SMALL_MAX_RECS) return;
    pl.small = true;
    pl.tc = false;
    pl.all_near = near;
    if (near && !own_cap) pl.cap = (int)std::max<int64_t>(pl.cap, keys);
    pl.TB = TB;
    pl.TBa = TBa;
    pl.nrec = nrec;
    pl.rank = can_rank && pl.rank_mode == RANK_TC16 && ix->L <= SP_RANK_L && P <= SP_RANK_P &&
              nq * (int64_t)ix->L * ix->d * 4 <= SMALL_RANK_BYTES;
}

// Q: the queries in the index's (working) dimensions; Qr: the same queries
// with all their dimensions for the re-rank (null: Q; they differ only under
// component filtration).
static int search_from_probes(ksc_index* ix, const float* Q, const Plan& pl, const int32_t* probes,
                              int64_t* ids, float* dists, uint64_t* cand_out, int32_t* ncand_out, cudaStream_t st,
                              const float* Qr = nullptr) {
    const int64_t nq = pl.nq;
    const int M = ix->M, L = ix->L;
    if (!Qr) Qr = Q;
    if (pl.small) return search_small(ix, Q, pl, probes, ids, dists, cand_out, ncand_out, st, Qr);
    // queries per work item: the unfiltered first part always runs the
    // byte-permute scan (the tensor-core scan keeps only filtered keys; with the
    // part's one or two lists a query, few queries share a list there unless the
    // index has few lists), the rest the chosen scan
    const int QGa = 32 / pl.G;
    const int QG = pl.tc ? pl.nt : QGa;
    // hybrid: the n_near nearest lists are the fully scanned ones (Sec. 4.4);
    // plain: a per-query split (k_count_parts)
    const int rA = std::min(pl.hybrid ? pl.n_near : 1, pl.Pmax);
    KSC_TRY(ensure(ix->ws_lut, (size_t)nq * pl.Pmax * M * PQ_K, st));
    KSC_TRY(ensure(ix->ws_bias, sizeof(int32_t) * nq * pl.Pmax, st));
    KSC_TRY(ensure(ix->ws_scale, sizeof(float) * nq, st));
    KSC_TRY(ensure(ix->ws_thr, sizeof(uint64_t) * nq, st));
    KSC_TRY(ensure(ix->ws_cnt, sizeof(int32_t) * nq, st));
    KSC_TRY(ensure(ix->ws_cand, sizeof(uint64_t) * nq * pl.cap, st));
    KSC_TRY(ensure(ix->ws_topr, sizeof(uint64_t) * nq * pl.Rmax, st));
    const size_t wl_head = sizeof(int64_t) * 2 * (L + 1) + sizeof(int32_t) * 2 * L;  // per work list
    KSC_TRY(ensure(ix->ws_items, 2 * wl_head + sizeof(uint32_t) * nq * (2 * pl.Pmax + 1) + 320, st));
    uint8_t* lut = (uint8_t*)ix->ws_lut.p;
    int32_t* bias = (int32_t*)ix->ws_bias.p;
    float* scale = (float*)ix->ws_scale.p;
    uint64_t* thr = (uint64_t*)ix->ws_thr.p;
    int32_t* cnt = (int32_t*)ix->ws_cnt.p;
    uint64_t* cand = (uint64_t*)ix->ws_cand.p;
    uint64_t* topr = (uint64_t*)ix->ws_topr.p;
    // both work lists side by side: pair_off [2][L+1], item_off [2][L+1],
    // cnt [2][L], fill [2][L], then the pairs
    WorkList wa, wb;
    {
        int64_t* po = (int64_t*)ix->ws_items.p;
        int64_t* io = po + 2 * (L + 1);
        int32_t* cn = (int32_t*)(io + 2 * (L + 1));
        int32_t* fl = cn + 2 * L;
        wa.pair_off = po;
        wb.pair_off = po + (L + 1);
        wa.item_off = io;
        wb.item_off = io + (L + 1);
        wa.cnt = cn;
        wb.cnt = cn + L;
        wa.fill = fl;
        wb.fill = fl + L;
        wa.pairs = (uint32_t*)(fl + 2 * L);
        wb.pairs = wa.pairs + nq * pl.Pmax;
    }
    int32_t* split = pl.hybrid ? nullptr : (int32_t*)(wb.pairs + nq * pl.Pmax);
    // item counters of the two tensor-core scans, after the split array
    unsigned long long* tc_next = reinterpret_cast<unsigned long long*>(
        (reinterpret_cast<uintptr_t>(wb.pairs + nq * pl.Pmax + nq) + 15) & ~uintptr_t(15));
    ScanArgs A{M, pl.Pmax, nq, probes, pl.nprobe_q, pl.Pfix, pl.rerank_q, pl.Rfix, pl.k, lut, bias,
               ix->list_boff, ix->list_n, ix->blk_codes, ix->blk_ids, ix->L};
    // 1. work lists: the nearest list of every query, and the rest
    mark(ix, 1, st);
    KSC_CUDA(cudaMemsetAsync(wa.cnt, 0, sizeof(int32_t) * 2 * L, st));
    if (pl.tc) KSC_CUDA(cudaMemsetAsync(tc_next, 0, 2 * sizeof(unsigned long long), st));
    k_count_parts<<<(unsigned)((nq + 7) / 8), 256, 0, st>>>(A, pl.Rmax, pl.cap, rA, split, wa.cnt, wb.cnt, cnt);
    wa.TB = pl.TBa;
    wb.TB = pl.TB;
    k_scan_lists<<<2, 1024, 0, st>>>(wa.cnt, ix->list_n, L, QGa, QG, wa.TB, wb.TB, wa.pair_off, wa.item_off,
                                     wa.fill);
    k_fill_parts<<<blocks_for(nq * pl.Pmax, 256), 256, 0, st>>>(A, rA, split, wa.pair_off, wa.fill, wa.pairs,
                                                                wb.pair_off, wb.fill, wb.pairs);
    KSC_LAUNCH_CHECK();
    ix->launches += 3;
    // 2. quantised LUTs of every probed (query, list)
    mark(ix, 2, st);
    {
        KSC_TRY(ensure(ix->ws_range, sizeof(uint32_t) * nq, st));
        uint32_t* rb = (uint32_t*)ix->ws_range.p;
        KSC_CUDA(cudaMemsetAsync(rb, 0, sizeof(uint32_t) * nq, st));
        LutArgs LA{Q, nq, ix->d, M, ix->dsub, ix->metric == KSC_IP, pl.Pmax, probes, pl.nprobe_q, pl.Pfix,
                   ix->c_mean, ix->codebook, ix->L, wa.pairs, wa.pair_off + L, wb.pairs, wb.pair_off + L};
        // tables stored for up to Pb probes per query (per-query nprobe: 8, the
        // rest of a larger query recomputed), so that more CTAs fit per SM
        const int Pb = pl.nprobe_q ? std::min(pl.Pq_max, 8) : pl.Pq_max;
        const size_t fsm = lut_fused_smem(M, ix->dsub, ix->d, Pb, pl.Pq_max);
        // one CTA per query at a time: worth it once every SM has queries to take
        if (fsm <= 160 * 1024 && nq >= 2 * (int64_t)num_sms()) {
            const int lw = lut_width(LA, true);
            auto kf = lw == 2 ? k_lut_fused<2> : (lw == 4 ? k_lut_fused<4> : k_lut_fused<0>);
            KSC_CUDA(cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fsm));
            // 512 threads per CTA where they cost no CTA, so the tables alone limit
            // them (60k x 784, M 196, nprobe 4: the search 1567 -> 1438 us), or a query
            // has many rows (M 48, up to 256 probes: 800 -> 745); with 4 CTAs of 256
            // against 3 (M 64, nprobe 8) they were slower (904 -> 916)
            int per_sm = 0, per_sm2 = 0, nt = 256;
            KSC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kf, 256, fsm));
            KSC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm2, kf, 512, fsm));
            if (per_sm2 >= std::max(per_sm, 1) || (per_sm2 > 0 && (int64_t)pl.Pq_max * M >= 4096)) {
                nt = 512;
                per_sm = per_sm2;
            }
            const int64_t grid = std::min<int64_t>(nq, (int64_t)num_sms() * (per_sm > 0 ? per_sm : 1));
            kf<<<(unsigned)grid, nt, fsm, st>>>(LA, Pb, pl.Pq_max, lut, bias, scale);
            KSC_LAUNCH_CHECK();
            ix->launches++;
        } else {
            KSC_TRY(launch_luts(LA, rb, lut, bias, scale, st));
            ix->launches += 2;
        }
    }
    // 3. scan of the nearest lists with no filter, then the threshold
    mark(ix, 3, st);
    KSC_TRY(run_scan(pl, M, A, ScanOut{nullptr, cnt, cand, pl.cap}, wa, L, ix->status, st, tc_next, false));
    // expected keys per query of the unfiltered scan from the mean list length:
    // max(4 R, N / 16), or the hybrid search's near lists
    const double near = pl.hybrid ? (double)rA * ix->n / L
                                  : std::max(4.0 * pl.Rmax, (double)pl.Pmax * ix->n / L / 16.0);
    if (select_by_warp(nq, near)) {
        k_threshold<<<(unsigned)((nq + SW_WARPS - 1) / SW_WARPS), SW_WARPS * 32, 0, st>>>(A, pl.Rmax, cnt, cand,
                                                                                           pl.cap, topr, thr);
    } else {
        const bool few = nq < 2 * (int64_t)num_sms(), narrow = near <= SW_MAX_KEYS && warp_per_query(nq);
        auto kf = few ? k_threshold_cta<1024, 0> : narrow ? k_threshold_cta<128, 16> : k_threshold_cta<256, 0>;
        kf<<<(unsigned)nq, few ? 1024 : narrow ? 128 : 256, 0, st>>>(A, pl.Rmax, cnt, cand, pl.cap, topr, thr);
    }
    KSC_LAUNCH_CHECK();
    ix->launches += 2;
    // 4. scan of the other lists, keeping keys at or below the threshold;
    //    hybrid: graph search of every other list first, full scans only of
    //    the lists it marks (Sec. 4.4)
    mark(ix, 4, st);
    if (pl.hybrid) {
        KSC_TRY(ensure(ix->ws_full, sizeof(uint32_t) * nq * pl.Pmax + 64, st));
        int64_t* nfull = (int64_t*)ix->ws_full.p;
        uint32_t* full = (uint32_t*)(nfull + 2);
        KSC_CUDA(cudaMemsetAsync(nfull, 0, sizeof(int64_t), st));
        const int vwords = (((ix->max_list + 31) / 32) + 1) & ~1;
        GraphArgs Gr{ix->nbr_pos, ix->nbr_codes, ix->entry_pos, pl.efs, pl.tau, vwords, full, nfull};
        KSC_CHECK_ARG(gs_smem_bound(vwords) <= 200 * 1024, "lists too large for the hybrid search (%d members)",
                      ix->max_list);
        KSC_TRY(launch_graph_search(A, ScanOut{thr, cnt, cand, pl.cap}, Gr, wb.pairs, wb.pair_off + L, st));
        KSC_LAUNCH_CHECK();
        // work list of the marked lists, then their scan
        KSC_CUDA(cudaMemsetAsync(wb.cnt, 0, sizeof(int32_t) * L, st));
        const int64_t nmax = nq * pl.Pmax;
        k_count_from<<<blocks_for(nmax, 256), 256, 0, st>>>(full, nfull, probes, wb.cnt);
        k_scan_lists<<<1, 1024, 0, st>>>(wb.cnt, ix->list_n, L, QG, QG, wb.TB, wb.TB, wb.pair_off, wb.item_off,
                                         wb.fill);
        k_fill_from<<<blocks_for(nmax, 256), 256, 0, st>>>(full, nfull, probes, wb.pair_off, wb.fill, wb.pairs);
        KSC_LAUNCH_CHECK();
        ix->launches += 4;
    }
    KSC_TRY(run_scan(pl, M, A, ScanOut{thr, cnt, cand, pl.cap}, wb, L, ix->status, st, tc_next + 1, pl.tc));
    ix->launches++;
    // 5. the R best keys per query
    mark(ix, 5, st);
    KSC_TRY(select_stage(ix, pl, A, cnt, cand, topr, cand_out, ncand_out, st));
    if (!ids && !dists) {  // candidates only (a shard's first step): no re-rank
        mark(ix, KSC_NUM_STAGES, st);
        return KSC_OK;
    }
    return rerank_stage(ix, Qr, pl, topr, ids, dists, st);
}

// The filtered scan takes the tensor cores from this many queries per list of its
// part (nq P / L times the part's share of the keys) on lists of this many
// vectors: an item's cost is mostly the expansion of its
// codes, whatever its queries, and the staging of their tables, whatever its
// vectors.  Search with byte permutes / tensor cores in us, 1M x 64 subspaces in
// 1024 lists, 7 probed: 224 / 277 at 7 queries per list, 318 / 324 at 14, 396 / 353
// at 20, 490 / 404 at 28, 976 / 718 at 68; 200k x 48 in 512 lists: 146 / 150 at 16,
// 203 / 189 at 32, 793 / 613 at 256; in 2048 lists (100 vectors each): 210 / 232 at
// 16, 531 / 521 at 64 (queries per list of the whole search; at nprobe 7 the
// filtered part has 0.8 of the keys, at nprobe 2 and R 257 of 390-vector lists none,
// and 8000 queries took 433 / 444 us).
// Above 96 subspaces an item holds 16 queries only, and takes as long as byte
// permutes do: from this many vectors of the part's pairs on (128 subspaces, 400
// queries at nprobe 4 of 100k in 64 lists, 2.0M: 185 / 202; 332 at nprobe 8 of 200k x 128 in
// 128, 3.7M: 275 / 268; 2500 at nprobe 8 of 300k in 256, 21M: 1037 / 886).
constexpr int64_t TC_MIN_SHARE = 16, TC_MIN_LIST = 256, TC_MIN_VECTORS_16 = 3'000'000;
constexpr int SCAN_TC_RULE = 2;  // ksc_search_opts.scan_tc: the rule also where lanes are given

// Tile lengths of the scan's warp items for an expected P probes per query.
// Short tiles balance the persistent warps, long ones amortise an item's
// set-up: about 220 items per SM for the filtered scan, and for the smaller
// unfiltered first part (its share from the split rule of k_count_parts:
// max(4 R, N / 16) keys, rounded up to whole lists) about 120, each within
// 4 to 32 blocks (on the 1M x 128 workload at nprobe 7: tiles of 14 and 6
// blocks; filtered tiles of 12 to 17 blocks ran within 1% of each other).
static void set_tiles(const ksc_index* ix, Plan& pl, int64_t nq, double P, const ksc_search_opts* opts) {
    pl.Pexp = P;
    const int QG = 32 / pl.G;
    const double nbar = (double)ix->n / ix->L;
    const double blocks = std::ceil((double)nq * P / ix->L / QG) * ix->nblocks;
    const double keys = std::max(P * nbar, 1.0);
    const double near =
        std::min(1.0, (std::max((double)NEAR_KEYS_PER_R * pl.Rmax, keys / NEAR_SHARE_DIV) + 0.5 * nbar) / keys);
    auto tile = [&](double b, double per_sm) {
        int t = (int)(b / (per_sm * num_sms()));
        t = t < 4 ? 4 : (t > 32 ? 32 : t);
        if (pl.G == 4) t = (t + S4_B - 1) / S4_B * S4_B;  // whole steps of 4 blocks
        return t;
    };
    pl.TB = tile(blocks * (1.0 - near), 220.0);
    pl.TBa = tile(blocks * near, 60.0);
    if (opts && opts->tile_blocks > 0) pl.TB = pl.TBa = std::min(opts->tile_blocks, 1 << 20);
    // tensor-core scan of the filtered part: asked for, or by default where
    // enough queries share a list; tiles of whole 128-vector products, 32 blocks
    // unless given
    const double tc_pairs = (double)nq * P * (1.0 - near);
    pl.tc = pl.nt > 0 && !pl.hybrid &&
            (pl.tc_opt || ((!(opts && opts->lanes_per_query) || opts->scan_tc == SCAN_TC_RULE) &&
                           tc_pairs >= (double)TC_MIN_SHARE * ix->L && ix->n >= TC_MIN_LIST * ix->L &&
                           (pl.nt >= 32 || tc_pairs * nbar >= (double)TC_MIN_VECTORS_16)));
    if (pl.tc)
        pl.TB = (opts && opts->tile_blocks > 0) ? (std::min(opts->tile_blocks, TCS_MAX_TILE) + 3) / 4 * 4 : 32;
}

static int make_plan(ksc_index* ix, int64_t nq, int k, int Pmax, int Rmax, const ksc_search_opts* opts, Plan& pl) {
    KSC_CHECK_ARG(nq >= 0, "nq < 0");
    KSC_CHECK_ARG(k >= 1 && k <= KSC_MAX_K, "k must be in [1, %d]", KSC_MAX_K);
    KSC_CHECK_ARG(Pmax >= 1 && Pmax <= ix->L && Pmax <= MAX_NPROBE, "nprobe must be in [1, min(nlist, %d)]",
                  MAX_NPROBE);
    if (Rmax < k) Rmax = k;
    KSC_CHECK_ARG(Rmax <= KSC_MAX_RERANK, "rerank must be <= %d", KSC_MAX_RERANK);
    pl.nq = nq;
    pl.k = k;
    pl.Pmax = Pmax;
    pl.Rmax = Rmax;
    pl.Pfix = Pmax;
    pl.Rfix = Rmax;
    pl.nprobe_q = nullptr;
    pl.rerank_q = nullptr;
    pl.G = choose_G(ix, nq, Pmax, opts ? opts->lanes_per_query : 0);
    pl.nt = tcs_nt(ix->M);
    pl.hybrid = opts && opts->hybrid;
    pl.tc_opt = opts && opts->scan_tc && opts->scan_tc != SCAN_TC_RULE;
    set_tiles(ix, pl, nq, Pmax, opts);
    int cap = (opts && opts->cand_cap > 0) ? opts->cand_cap : std::max(32 * Rmax, 8192);
    pl.cap = std::max(cap, Rmax);
    pl.rank_mode = (opts && opts->rank_fp32) ? RANK_FP32 : ((opts && opts->rank_fp8) ? RANK_FP8 : RANK_TC16);
    pl.Pq_max = Pmax;
    pl.small = pl.rank = pl.all_near = false;
    pl.nrec = 0;
    pl.prec = opts ? opts->precision : 0;
    // the re-rank band: on by default for L2 (for inner products of
    // real-valued rows the BF16 band is wide against the gaps between the
    // best scores)
    pl.band = opts && opts->rerank_band != 0 ? opts->rerank_band > 0 : ix->metric != KSC_IP;
    pl.band_now = opts && opts->rerank_band > 0;
    KSC_CHECK_ARG(pl.prec >= 0 && pl.prec <= 2, "precision must be 0 (FP32), 1 (BF16) or 2 (FP8)");
    pl.Rf = pl.Rmax;
    if (pl.prec > 0) {
        const int rf = (opts->rerank_final > 0) ? opts->rerank_final : std::max(k, Rmax / 2);
        pl.Rf = std::min(std::max(rf, k), Rmax);
    }
    pl.n_near = (opts && opts->n_near > 0) ? opts->n_near : 2;
    pl.efs = (opts && opts->efs > 0) ? opts->efs : 64;
    pl.tau = (opts && opts->tau >= 0 && opts->hybrid) ? opts->tau : 8;
    if (pl.hybrid) {
        KSC_CHECK_ARG(pl.efs <= GS_MAX_EFS, "efs must be <= %d", GS_MAX_EFS);
        if (!ix->nbr_codes) {
            set_error("the hybrid search needs an index built or imported with graphs");
            return KSC_ESTATE;
        }
    }
    return KSC_OK;
}

}  // namespace ksc

using namespace ksc;

extern "C" {

int ksc_rank_lists(ksc_index* ix, const float* Q_dev, int64_t nq, int32_t P, int32_t* probes_dev,
                   float* scores_dev, void* stream) {
    KSC_CHECK_ARG(ix, "null index");
    KSC_CHECK_ARG(P >= 1 && P <= ix->L && P <= MAX_NPROBE, "P must be in [1, min(nlist, %d)]", MAX_NPROBE);
    if (nq == 0) return KSC_OK;
    KSC_CHECK_ARG(Q_dev && probes_dev, "null argument");
    cudaStream_t st = as_stream(stream);
    const float* Qw;
    KSC_TRY(work_queries(ix, Q_dev, nq, st, &Qw));
    return rank_lists(ix, Qw, nq, nullptr, P, P, probes_dev, scores_dev, RANK_TC16, st);
}

int ksc_list_scores(ksc_index* ix, const float* Q_dev, int64_t nq, int32_t tensor_cores, float* scores_dev,
                    float* err_dev, void* stream) {
    KSC_CHECK_ARG(ix, "null index");
    if (nq == 0) return KSC_OK;
    KSC_CHECK_ARG(Q_dev && scores_dev, "null argument");
    cudaStream_t st = as_stream(stream);
    KSC_CHECK_ARG(tensor_cores >= 0 && tensor_cores <= 2, "tensor_cores must be 0 (FP32), 1 (16-bit) or 2 (FP8)");
    const int mode = tensor_cores == 0 ? RANK_FP32 : (tensor_cores == 2 ? RANK_FP8 : RANK_TC16);
    float* err = nullptr;
    const float* Qw;
    KSC_TRY(work_queries(ix, Q_dev, nq, st, &Qw));
    KSC_TRY(list_scores(ix, Qw, nq, mode, scores_dev, &err, st));
    if (err_dev) KSC_CUDA(cudaMemcpyAsync(err_dev, err, sizeof(float) * nq, cudaMemcpyDeviceToDevice, st));
    return KSC_OK;
}

int ksc_compute_luts(ksc_index* ix, const float* Q_dev, int64_t nq, const int32_t* probes_dev, int32_t P,
                     uint8_t* lut_dev, int32_t* bias_dev, float* scale_dev, void* stream) {
    KSC_CHECK_ARG(ix, "null index");
    KSC_CHECK_ARG(P >= 1 && P <= ix->L, "P must be in [1, nlist]");
    if (nq == 0) return KSC_OK;
    KSC_CHECK_ARG(Q_dev && probes_dev && lut_dev && bias_dev && scale_dev, "null argument");
    cudaStream_t st = as_stream(stream);
    const float* Qw;
    KSC_TRY(work_queries(ix, Q_dev, nq, st, &Qw));
    return compute_luts(ix, Qw, nq, probes_dev, nullptr, P, P, lut_dev, bias_dev, scale_dev, st);
}

int ksc_search_with_probes(ksc_index* ix, const float* Q_dev, int64_t nq, const int32_t* probes_dev, int32_t P,
                           int32_t k, int32_t rerank, int64_t* ids_dev, float* dists_dev, uint64_t* cand_dev,
                           int32_t* ncand_dev, const ksc_search_opts* opts, void* stream) {
    KSC_CHECK_ARG(ix, "null index");
    Plan pl;
    KSC_TRY(make_plan(ix, nq, k, P, rerank, opts, pl));
    if (nq == 0) return KSC_OK;  // empty batch: pointers may be NULL
    KSC_CHECK_ARG(Q_dev && probes_dev && ids_dev && dists_dev, "null argument");
    cudaStream_t st = as_stream(stream);
    KSC_TRY(reset_counters(ix, st));
    ix->launches = 0;
    mark(ix, 0, st);
    const float* Qw;
    KSC_TRY(work_queries(ix, Q_dev, nq, st, &Qw));
    plan_small(ix, pl, opts, false, false);
    return search_from_probes(ix, Qw, pl, probes_dev, ids_dev, dists_dev, cand_dev, ncand_dev, st, Q_dev);
}

}  // extern "C"

namespace ksc {
// A shard's first step (list sharding): steps a1 .. a5 with a fixed nprobe,
// the R = max(rerank, k) selected keys of every query, ascending, into
// keys [nq x R] (local ids; KEY_NONE pads a short list).
int search_keys(ksc_index* ix, const float* Q, int64_t nq, int nprobe, int rerank, const ksc_search_opts* opts,
                uint64_t* keys, cudaStream_t st) {
    Plan pl;
    KSC_TRY(make_plan(ix, nq, 1, nprobe, rerank, opts, pl));
    KSC_CHECK_ARG(!pl.hybrid && pl.prec == 0, "sharded search: plain scan and FP32 re-rank only");
    if (nq == 0) return KSC_OK;
    KSC_TRY(reset_counters(ix, st));
    KSC_TRY(ensure(ix->ws_probes, sizeof(int32_t) * nq * pl.Pmax, st));
    int32_t* probes = (int32_t*)ix->ws_probes.p;
    ix->launches = 0;
    mark(ix, 0, st);
    const float* Qw;
    KSC_TRY(work_queries(ix, Q, nq, st, &Qw));
    plan_small(ix, pl, opts, true, true);
    if (!pl.rank) KSC_TRY(rank_lists(ix, Qw, nq, nullptr, pl.Pmax, pl.Pmax, probes, nullptr, pl.rank_mode, st));
    return search_from_probes(ix, Qw, pl, probes, nullptr, nullptr, keys, nullptr, st, Q);
}

// Exact re-rank (a6) of given candidate keys [nq x R] (local ids, KEY_NONE
// skipped): the k best by (distance, id) per query.
int rerank_keys(ksc_index* ix, const float* Q, int64_t nq, int k, const uint64_t* keys, int R, int64_t* ids,
                float* dists, cudaStream_t st) {
    const float* Xr = rr_X(ix);
    const int dr = rr_d(ix);
    const int ip = ix->metric == KSC_IP;
    if (k <= 32 && R <= RW_MAXR && dr <= 128 && (dr & 3) == 0 && warp_per_query(nq)) {
        const size_t smem = sizeof(uint64_t) * RW_WARPS * R;
        KSC_CUDA(cudaFuncSetAttribute(k_rerank_w<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        k_rerank_w<false><<<(unsigned)((nq + RW_WARPS - 1) / RW_WARPS), RW_WARPS * 32, smem, st>>>(
            Q, Xr, dr, ip, keys, R, nullptr, R, k, nq, ids, dists, nullptr, nullptr, nullptr);
    } else {
        const size_t smem = rerank_smem(R, k);
        if (nq < 2 * (int64_t)num_sms()) {
            KSC_CUDA(cudaFuncSetAttribute(k_rerank<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k_rerank<1024><<<(unsigned)nq, 1024, smem, st>>>(Q, Xr, dr, ip, keys, R, nullptr, R, k, ids, dists);
        } else {
            KSC_CUDA(cudaFuncSetAttribute(k_rerank<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k_rerank<256><<<(unsigned)nq, 256, smem, st>>>(Q, Xr, dr, ip, keys, R, nullptr, R, k, ids, dists);
        }
    }
    KSC_LAUNCH_CHECK();
    ix->launches++;
    return KSC_OK;
}
}  // namespace ksc

extern "C" {

int ksc_search(ksc_index* ix, const float* Q_dev, int64_t nq, int32_t k, int32_t nprobe, int32_t rerank,
               int64_t* ids_dev, float* dists_dev, const ksc_search_opts* opts, void* stream) {
    KSC_CHECK_ARG(ix, "null index");
    Plan pl;
    KSC_TRY(make_plan(ix, nq, k, nprobe, rerank, opts, pl));
    if (nq == 0) return KSC_OK;  // empty batch: pointers may be NULL
    KSC_CHECK_ARG(Q_dev && ids_dev && dists_dev, "null argument");
    cudaStream_t st = as_stream(stream);
    KSC_TRY(reset_counters(ix, st));
    KSC_TRY(ensure(ix->ws_probes, sizeof(int32_t) * nq * pl.Pmax, st));
    int32_t* probes = (int32_t*)ix->ws_probes.p;
    ix->launches = 0;
    mark(ix, 0, st);
    const float* Qw;
    KSC_TRY(work_queries(ix, Q_dev, nq, st, &Qw));
    plan_small(ix, pl, opts, true, true);
    if (!pl.rank) KSC_TRY(rank_lists(ix, Qw, nq, nullptr, pl.Pmax, pl.Pmax, probes, nullptr, pl.rank_mode, st));
    return search_from_probes(ix, Qw, pl, probes, ids_dev, dists_dev, nullptr, nullptr, st, Q_dev);
}

int ksc_search_varprobe(ksc_index* ix, const float* Q_dev, int64_t nq, int32_t k, const int32_t* nprobe_dev,
                        int32_t nprobe_max, const int32_t* rerank_dev, int32_t rerank_max, int64_t* ids_dev,
                        float* dists_dev, const ksc_search_opts* opts, void* stream) {
    KSC_CHECK_ARG(ix, "null index");
    Plan pl;
    KSC_TRY(make_plan(ix, nq, k, nprobe_max, rerank_max, opts, pl));
    if (nq == 0) return KSC_OK;  // empty batch: pointers may be NULL
    KSC_CHECK_ARG(Q_dev && ids_dev && dists_dev && nprobe_dev && rerank_dev, "null argument");
    cudaStream_t st = as_stream(stream);
    pl.nprobe_q = nprobe_dev;
    pl.rerank_q = rerank_dev;
    set_tiles(ix, pl, nq, 0.5 * pl.Pmax, opts);  // per-query nprobe: about half the largest on average
    KSC_TRY(reset_counters(ix, st));
    KSC_TRY(ensure(ix->ws_probes, sizeof(int32_t) * nq * pl.Pmax, st));
    int32_t* probes = (int32_t*)ix->ws_probes.p;
    ix->launches = 0;
    mark(ix, 0, st);
    const float* Qw;
    KSC_TRY(work_queries(ix, Q_dev, nq, st, &Qw));
    plan_small(ix, pl, opts, true, true);
    if (!pl.rank) KSC_TRY(rank_lists(ix, Qw, nq, nprobe_dev, pl.Pmax, pl.Pmax, probes, nullptr, pl.rank_mode, st));
    return search_from_probes(ix, Qw, pl, probes, ids_dev, dists_dev, nullptr, nullptr, st, Q_dev);
}

int ksc_profile_enable(ksc_index* ix, int32_t on) {
    KSC_CHECK_ARG(ix, "null argument");
    if (on) {
        for (int i = 0; i <= KSC_NUM_STAGES; ++i)
            if (!ix->ev[i]) KSC_CUDA(cudaEventCreate(&ix->ev[i]));
    }
    ix->prof = on != 0;
    for (int i = 0; i <= KSC_NUM_STAGES; ++i) ix->ev_used[i] = false;
    return KSC_OK;
}

int ksc_profile_read(ksc_index* ix, float* ms_host, int32_t n, int32_t* launches_host) {
    KSC_CHECK_ARG(ix && ms_host && n >= 0 && n <= 8, "bad argument");
    KSC_CHECK_ARG(ix->prof, "profiling is not enabled on this index");
    if (launches_host) *launches_host = ix->launches;
    for (int i = 0; i < n; ++i) ms_host[i] = 0.f;
    int prev = -1;
    for (int i = 0; i <= KSC_NUM_STAGES; ++i) {
        if (!ix->ev_used[i]) continue;
        KSC_CUDA(cudaEventSynchronize(ix->ev[i]));
        if (prev >= 0 && prev < n) {
            float ms = 0.f;
            KSC_CUDA(cudaEventElapsedTime(&ms, ix->ev[prev], ix->ev[i]));
            ms_host[prev] = ms;
        }
        prev = i;
    }
    return KSC_OK;
}

int ksc_lut16_peak(double* glookups_host, void* stream) {
    KSC_CHECK_ARG(glookups_host, "null argument");
    cudaStream_t st = as_stream(stream);
    uint32_t* sink = nullptr;
    KSC_CUDA(cudaMalloc(&sink, 16));
    const int iters = 4096;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    // [0] the shared-selector sequence, 8 CTAs of 256 threads per SM;
    // [1] the per-slot sequence, 16 CTAs of 128 threads per SM
    double rate[2] = {0.0, 0.0};
    cudaError_t err = cudaSuccess;
    for (int v = 0; v < 2 && err == cudaSuccess; ++v) {
        const int threads = v == 0 ? 256 : 128, grid = num_sms() * (v == 0 ? 8 : 16);
        for (int rep = 0; rep < 2; ++rep) {  // the first launch warms up
            if (rep == 1) cudaEventRecord(e0, st);
            if (v == 0) k_lut16_peak_sel<<<grid, threads, 0, st>>>(iters, 12345u + rep, sink);
            else k_lut16_peak<<<grid, threads, 0, st>>>(iters, 12345u + rep, sink);
        }
        cudaEventRecord(e1, st);
        err = cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        rate[v] = (double)grid * threads * iters * 32 / (ms * 1e-3) / 1e9;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(sink);
    KSC_CUDA(err);
    glookups_host[0] = rate[0];
    glookups_host[1] = rate[1];
    return KSC_OK;
}

int ksc_pair_distances(ksc_index* ix, const float* Q_dev, int64_t nq, const int64_t* ids_dev, int32_t c,
                       int32_t precision, float* out_dev, void* stream) {
    KSC_CHECK_ARG(ix, "null index");
    KSC_CHECK_ARG(precision >= 0 && precision <= 2, "precision must be 0, 1 or 2");
    if (nq == 0 || c == 0) return KSC_OK;
    KSC_CHECK_ARG(Q_dev && ids_dev && out_dev && c > 0, "bad argument");
    cudaStream_t st = as_stream(stream);
    KSC_TRY(ensure_lowp(ix, precision, st));
    k_pair_dist<<<(unsigned)nq, 256, 0, st>>>(Q_dev, nq, rr_d(ix), ix->metric == KSC_IP, precision, rr_X(ix),
                                              (const uint16_t*)ix->X_bf16, (const uint8_t*)ix->X_fp8, ix->X_scale,
                                              ids_dev, c, out_dev);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

int ksc_search_stats(ksc_index* ix, int64_t* stats_host) {
    KSC_CHECK_ARG(ix && stats_host, "null argument");
    unsigned long long v[4];
    KSC_CUDA(cudaMemcpy(v, ix->stats, sizeof(v), cudaMemcpyDeviceToHost));
    for (int i = 0; i < 4; ++i) stats_host[i] = (int64_t)v[i];
    return KSC_OK;
}

int ksc_last_status(ksc_index* ix, int32_t* status_host) {
    KSC_CHECK_ARG(ix && status_host, "null argument");
    KSC_CUDA(cudaMemcpy(status_host, ix->status, sizeof(int32_t), cudaMemcpyDeviceToHost));
    return KSC_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ allocation-free LUT entry
// Some callers cannot let this library call cudaMalloc: a host program whose
// device memory is wholly reserved by its own allocator (a framework's caching
// pool, a serving runtime that pre-reserves the device) has no headroom for a
// foreign allocation, and a latency-critical caller cannot afford the device
// synchronisation that cudaMalloc / cudaFree may imply.  For them,
// ksc_compute_luts_noalloc keeps its only scratch -- the per-query table range
// that ksc_compute_luts otherwise keeps in a workspace buffer -- in the
// fixed-size array below.  Every GPU that loads the library holds the array
// (KSC_NOALLOC_MAX_NQ * 4 bytes = 256 KiB) until the process exits.
static __device__ __align__(256) uint32_t g_noalloc_range[KSC_NOALLOC_MAX_NQ];

namespace ksc {
// Device address of g_noalloc_range per device ordinal, looked up on the first
// call made with that device current (host code cannot use the symbol itself:
// in host code it names a host-side stand-in, not device memory).  Atomic, so
// that host threads making their first call on one device at the same time
// do not race on the cache (they store the same address).
static std::atomic<void*> g_noalloc_addr[64] = {};
}  // namespace ksc

extern "C" int ksc_compute_luts_noalloc(ksc_index* ix, const float* Q_dev, int64_t nq, const int32_t* probes_dev,
                                        int32_t P, uint8_t* lut_dev, int32_t* bias_dev, float* scale_dev,
                                        void* stream) {
    KSC_CHECK_ARG(ix, "null index");
    if (ix->dims) {
        set_error("ksc_compute_luts_noalloc needs an index without component filtration");
        return KSC_EUNSUPPORTED;
    }
    KSC_CHECK_ARG(P >= 1 && P <= ix->L, "P must be in [1, nlist]");
    KSC_CHECK_ARG(nq >= 0 && nq <= KSC_NOALLOC_MAX_NQ,
                  "nq = %lld exceeds the fixed scratch of ksc_compute_luts_noalloc (at most %d queries per call)",
                  (long long)nq, KSC_NOALLOC_MAX_NQ);
    if (nq == 0) return KSC_OK;
    KSC_CHECK_ARG(Q_dev && probes_dev && lut_dev && bias_dev && scale_dev, "null argument");
    int dev = 0;
    KSC_CUDA(cudaGetDevice(&dev));
    KSC_CHECK_ARG(dev >= 0 && dev < 64, "device ordinal %d out of range", dev);
    void* addr = g_noalloc_addr[dev].load(std::memory_order_acquire);
    if (!addr) {
        KSC_CUDA(cudaGetSymbolAddress(&addr, g_noalloc_range));
        g_noalloc_addr[dev].store(addr, std::memory_order_release);
    }
    uint32_t* rb = static_cast<uint32_t*>(addr);
    cudaStream_t st = as_stream(stream);
    // the array keeps the previous call's ranges: clear this call's slots
    KSC_CUDA(cudaMemsetAsync(rb, 0, sizeof(uint32_t) * nq, st));
    LutArgs A{Q_dev, nq, ix->d, ix->M, ix->dsub, ix->metric == KSC_IP, P, probes_dev, nullptr, P, ix->c_mean,
              ix->codebook, ix->L};
    return launch_luts(A, rb, lut_dev, bias_dev, scale_dev, st);
}

// ------------------------------------------------------------------ learned nprobe / rerank
namespace ksc {
static const int32_t DEF_GRID[] = {4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128};
static const int32_t DEF_RGRID[] = {20, 50, 100, 200, 400};

// Rank with P probes (P >= 32) and derive the predictor features.
// The P best lists of every query (exact ranking) and the predictor's
// features, from the FEAT_K smallest given list scores (L >= FEAT_K).
static int rank_and_features(ksc_index* ix, const float* Q, int64_t nq, int P, int32_t* probes, float* feats,
                             cudaStream_t st) {
    KSC_TRY(ensure(ix->ws_rscore, sizeof(float) * nq * FEAT_K, st));
    float* rs = (float*)ix->ws_rscore.p;
    KSC_TRY(rank_lists(ix, Q, nq, nullptr, P, P, probes, nullptr, RANK_TC16, st, rs));
    KSC_TRY(mlp_features(rs, nq, FEAT_K, ix->spherical, feats, st));
    ix->launches++;
    return KSC_OK;
}

// The adaptive search's ranking (Sec. 4.2.1).  The predictor's distances
// are the FEAT_K smallest approximate list scores; the network sets each
// query's nprobe and R from them; only then are the nprobe best lists of each
// query ranked exactly, the threshold of the exact pass taken from the same
// sorted scores -- all in k_rank_head_w, with the CTA kernel for the queries
// it leaves on `redo`.  The probes equal the first nprobe of an exact ranking
// of Pr lists (an exact top-P is a prefix of the exact top-Pr); rows past
// nprobe hold -1.  Batches the warp kernels do not serve: the ranking of Pr
// lists with the features, then the head kernel.
static int rank_adaptive(ksc_index* ix, const float* Q, int64_t nq, int Pr, int32_t* probes,
                         const ksc_adaptive_params& prm, int32_t* np_q, int32_t* r_q, cudaStream_t st) {
    if (!rank_by_warp(ix, nq, Pr) || ix->L < FEAT_K) {
        KSC_TRY(ensure(ix->ws_rscore, sizeof(float) * nq * FEAT_K, st));
        float* rs = (float*)ix->ws_rscore.p;
        KSC_TRY(rank_lists(ix, Q, nq, nullptr, Pr, Pr, probes, nullptr, RANK_TC16, st, rs));
        KSC_TRY(mlp_infer_scores(ix->mlp_w, rs, FEAT_K, ix->spherical, nq, prm, np_q, r_q, st));
        ix->launches++;
        return KSC_OK;
    }
    KSC_TRY(ensure(ix->ws_scores, sizeof(float) * nq * ix->L, st));
    KSC_TRY(ensure(ix->ws_redo, sizeof(int32_t) * (nq + 1), st));
    float* scores = (float*)ix->ws_scores.p;
    int32_t* redo = (int32_t*)ix->ws_redo.p;
    float* err = nullptr;
    KSC_TRY(list_scores(ix, Q, nq, RANK_TC16, scores, &err, st));
    KSC_CUDA(cudaMemsetAsync(redo, 0, sizeof(int32_t), st));
    const size_t hsm = rh_head_bytes() + RH_WARPS * rh_warp_bytes(ix->L);
    KSC_CUDA(cudaFuncSetAttribute(k_rank_head_w, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hsm));
    int per_sm = 0;
    KSC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_rank_head_w, RH_WARPS * 32, hsm));
    const int64_t grid = std::min<int64_t>((nq + RH_WARPS - 1) / RH_WARPS,
                                           (int64_t)num_sms() * (per_sm > 0 ? per_sm : 1));
    k_rank_head_w<<<(unsigned)grid, RH_WARPS * 32, hsm, st>>>(scores, err, Q, ix->c_rank, nq, ix->d, ix->L,
                                                             ix->spherical, ix->mlp_w, prm, Pr, probes, redo, np_q,
                                                             r_q);
    KSC_LAUNCH_CHECK();
    // queries with too many lists inside the bound: the CTA kernel
    const int rs_cap = std::min(RS_CAP, std::max(1024, pow2_ceil(4 * Pr)));
    const size_t smem = rs_cap * sizeof(uint64_t) + (ix->L <= RS_SMEM_L ? sizeof(float) * ix->L : 0);
    KSC_CUDA(cudaFuncSetAttribute(k_rank_select<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_rank_select<256><<<num_sms() * 2, 256, smem, st>>>(scores, err, Q, ix->c_rank, nq, ix->d, ix->L, ix->spherical,
                                                        np_q, Pr, Pr, rs_cap, probes, nullptr, redo);
    KSC_LAUNCH_CHECK();
    ix->launches += 2;
    return KSC_OK;
}

static uint64_t mix64(uint64_t& s) {  // splitmix64 (Steele, Lea, Flood 2014)
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

static float median_of(std::vector<int32_t> v) {
    if (v.empty()) return 0.f;
    std::nth_element(v.begin(), v.begin() + v.size() / 2, v.end());
    return (float)v[v.size() / 2];
}

// Columns 0 .. w of the rows idx[r] (NULL: row r) of a matrix of 4-byte words
// with ld words per row.
__global__ void k_gather_words(const uint32_t* __restrict__ src, int ld, const int32_t* __restrict__ idx, int64_t cnt,
                               int w, uint32_t* __restrict__ out) {
    const int64_t tot = cnt * w;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / w;
        out[e] = src[(idx ? idx[r] : r) * ld + (e - r * w)];
    }
}

static int gather_words(const void* src, int ld, const int32_t* idx, int64_t cnt, int w, void* out, cudaStream_t st) {
    const int64_t blocks = std::min<int64_t>((cnt * w + 255) / 256, 16 * (int64_t)num_sms());
    k_gather_words<<<(unsigned)std::max<int64_t>(1, blocks), 256, 0, st>>>((const uint32_t*)src, ld, idx, cnt, w,
                                                                          (uint32_t*)out);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

// Smallest grid value per query whose search finds >= target hits; queries
// that never reach it take the last grid value.  grid: nprobe values, or
// (np given, each query's nprobe) rerank values.
// A query's label is settled by the first value that suffices, so each value
// is searched only for the queries still without one, packed into a smaller
// batch with probe rows of that value's length: searching every query at
// nprobe 4 .. 128 takes tables and scans of 438 lists per query, most of them
// after its label is known.  16,384 queries on 100k x 128 in 256 lists: 46 ms
// of searches before, 3 ms now.
static int label_queries(ksc_index* ix, const float* Q, const float* Qr, int64_t nq, const float* kth,
                         const int32_t* probes, int Pr, const std::vector<int32_t>& grid,
                         const std::vector<int32_t>* np, int R_fixed, int k, int target, std::vector<int32_t>& label,
                         cudaStream_t st) {
    std::vector<int32_t> hits_h(nq), rem(nq), npr;
    int32_t *hits = nullptr, *idx = nullptr, *pc = nullptr, *npd = nullptr;
    int64_t* ids = nullptr;
    float *dists = nullptr, *qc = nullptr, *qrc = nullptr, *kc = nullptr;
    const int d = ix->d, dr = rr_d(ix);
    int rc = KSC_OK;
    label.assign(nq, -1);
    for (int64_t q = 0; q < nq; ++q) rem[q] = (int32_t)q;
    for (int32_t gv : grid) {  // every value is checked, also one that no query gets to
        Plan pl;
        KSC_TRY(make_plan(ix, nq, k, Pr, np ? gv : R_fixed, nullptr, pl));
    }
    do {
        if (cudaMalloc(&hits, sizeof(int32_t) * nq) != cudaSuccess || cudaMalloc(&ids, sizeof(int64_t) * nq * k) != cudaSuccess ||
            cudaMalloc(&dists, sizeof(float) * nq * k) != cudaSuccess || cudaMalloc(&idx, sizeof(int32_t) * nq) != cudaSuccess ||
            cudaMalloc(&pc, sizeof(int32_t) * nq * Pr) != cudaSuccess || cudaMalloc(&npd, sizeof(int32_t) * nq) != cudaSuccess ||
            cudaMalloc(&qc, sizeof(float) * nq * d) != cudaSuccess || cudaMalloc(&kc, sizeof(float) * nq) != cudaSuccess ||
            (Qr != Q && cudaMalloc(&qrc, sizeof(float) * nq * dr) != cudaSuccess)) {
            set_error("allocation failed while labelling");
            rc = KSC_ENOMEM;
            break;
        }
        for (int32_t gv : grid) {
            const int64_t m = (int64_t)rem.size();
            if (m == 0) break;
            const bool part = m < nq;
            int P = std::min(std::max(gv, 1), Pr);
            if (np) {
                npr.resize(m);
                P = 1;
                for (int64_t i = 0; i < m; ++i) {
                    npr[i] = std::min(std::max((*np)[rem[i]], 1), Pr);
                    P = std::max(P, npr[i]);
                }
            }
            if ((part && cudaMemcpyAsync(idx, rem.data(), sizeof(int32_t) * m, cudaMemcpyHostToDevice, st) != cudaSuccess) ||
                (np && cudaMemcpyAsync(npd, npr.data(), sizeof(int32_t) * m, cudaMemcpyHostToDevice, st) != cudaSuccess)) {
                set_error("label upload failed");
                rc = KSC_ECUDA;
                break;
            }
            const int32_t* sel = part ? idx : nullptr;
            if ((rc = gather_words(probes, Pr, sel, m, P, pc, st))) break;
            if (part) {
                if ((rc = gather_words(Q, d, sel, m, d, qc, st))) break;
                if ((rc = gather_words(kth, 1, sel, m, 1, kc, st))) break;
                if (qrc && (rc = gather_words(Qr, dr, sel, m, dr, qrc, st))) break;
            }
            const float* Qs = part ? qc : Q;
            Plan pl;
            if ((rc = make_plan(ix, m, k, P, np ? gv : R_fixed, nullptr, pl))) break;
            if (np) pl.nprobe_q = npd;
            plan_small(ix, pl, nullptr, true, false);
            if ((rc = reset_items(ix, st))) break;
            if ((rc = search_from_probes(ix, Qs, pl, pc, ids, dists, nullptr, nullptr, st,
                                         qrc ? (part ? qrc : Qr) : Qs)))
                break;
            if ((rc = mlp_hits(dists, m, k, part ? kc : kth, ix->metric == KSC_IP, hits, st))) break;
            if (cudaMemcpyAsync(hits_h.data(), hits, sizeof(int32_t) * m, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                cudaStreamSynchronize(st) != cudaSuccess) {
                set_error("label readback failed");
                rc = KSC_ECUDA;
                break;
            }
            int64_t left = 0;
            for (int64_t i = 0; i < m; ++i) {
                if (hits_h[i] >= target) label[rem[i]] = gv;
                else rem[left++] = rem[i];
            }
            rem.resize(left);
        }
    } while (0);
    for (auto& l : label)
        if (l < 0) l = grid.back();
    void* tmp[] = {hits, ids, dists, idx, pc, npd, qc, kc, qrc};
    for (void* p : tmp)
        if (p) cudaFree(p);
    return rc;
}
}  // namespace ksc

extern "C" {

int ksc_mlp_grad(const float* w_dev, const float* x_dev, const float* y_dev, int64_t B, float* grad_dev,
                 float* loss_dev, void* stream) {
    KSC_CHECK_ARG(w_dev && x_dev && y_dev && grad_dev && B > 0, "bad argument");
    return mlp_grad(w_dev, x_dev, y_dev, B, grad_dev, loss_dev, as_stream(stream));
}

int ksc_mlp_forward(const float* w_dev, const float* x_dev, int64_t B, float* prob_dev, void* stream) {
    KSC_CHECK_ARG(w_dev && x_dev && prob_dev && B > 0, "bad argument");
    ksc_adaptive_params prm = {1, 1, 1, 1, 0.f, 0.f, 0.f, 0.f};
    return mlp_infer(w_dev, x_dev, B, prm, prob_dev, nullptr, nullptr, as_stream(stream));
}

int ksc_query_features(ksc_index* ix, const float* Q_dev, int64_t nq, float* feats_dev, void* stream) {
    KSC_CHECK_ARG(ix, "null index");
    KSC_CHECK_ARG(ix->L >= 32, "the predictor needs at least 32 lists");
    if (nq == 0) return KSC_OK;
    KSC_CHECK_ARG(Q_dev && feats_dev, "null argument");
    cudaStream_t st = as_stream(stream);
    KSC_TRY(ensure(ix->ws_probes, sizeof(int32_t) * nq, st));
    const float* Qw;
    KSC_TRY(work_queries(ix, Q_dev, nq, st, &Qw));
    return rank_and_features(ix, Qw, nq, 1, (int32_t*)ix->ws_probes.p, feats_dev, st);
}

int ksc_predictor_params(ksc_index* ix, const ksc_adaptive_params* prm) {
    KSC_CHECK_ARG(ix && prm, "null argument");
    KSC_CHECK_ARG(prm->pmin >= 1 && prm->pmin <= prm->pmax && prm->pmax <= ix->L && prm->pmax <= MAX_NPROBE,
                  "nprobe range must satisfy 1 <= pmin <= pmax <= min(nlist, %d)", MAX_NPROBE);
    KSC_CHECK_ARG(prm->rmin >= 1 && prm->rmin <= prm->rmax && prm->rmax <= KSC_MAX_RERANK, "bad rerank range");
    ix->mlp_prm = *prm;
    return KSC_OK;
}

int ksc_predictor_weights(ksc_index* ix, float* w_host, const float* w_in_host) {
    KSC_CHECK_STATE(!ix || !w_in_host || !ix->parent, "models are set on the index, not on a view of it");
    KSC_CHECK_ARG(ix && (w_host || w_in_host), "null argument");
    if (w_in_host) {
        if (!ix->mlp_w) KSC_CUDA(cudaMalloc(&ix->mlp_w, sizeof(float) * KSC_MLP_NPARAMS));
        KSC_CUDA(cudaMemcpy(ix->mlp_w, w_in_host, sizeof(float) * KSC_MLP_NPARAMS, cudaMemcpyHostToDevice));
        if (ix->mlp_prm.pmax == 0) {
            ix->mlp_prm = {DEF_GRID[0], std::min(DEF_GRID[10], ix->L), DEF_RGRID[0], DEF_RGRID[4], 0.3f, 0.5f,
                           0.3f, 0.5f};
            if (ix->mlp_prm.pmin > ix->mlp_prm.pmax) ix->mlp_prm.pmin = ix->mlp_prm.pmax;
        }
    }
    if (w_host) {
        if (!ix->mlp_w) {
            set_error("no predictor has been trained or loaded");
            return KSC_ESTATE;
        }
        KSC_CUDA(cudaMemcpy(w_host, ix->mlp_w, sizeof(float) * KSC_MLP_NPARAMS, cudaMemcpyDeviceToHost));
    }
    return KSC_OK;
}

int ksc_train_predictor(ksc_index* ix, const float* Qtrain_dev, int64_t nt, const float* kth_dev,
                        const ksc_train_opts* opts, void* stream, float* loss_host) {
    KSC_CHECK_STATE(!ix || !ix->parent, "the predictor is trained on an index, not on a view of it");
    KSC_CHECK_ARG(ix && Qtrain_dev && kth_dev && nt > 0, "bad argument");
    KSC_CHECK_ARG(ix->L >= 32, "the predictor needs at least 32 lists");
    cudaStream_t st = as_stream(stream);
    const int k = (opts && opts->k > 0) ? opts->k : 10;
    const int target = (opts && opts->target_hits > 0) ? opts->target_hits : 9;
    const int R_lab = (opts && opts->rerank_label > 0) ? opts->rerank_label : 200;
    const int epochs = (opts && opts->epochs > 0) ? opts->epochs : 8;
    const int batch = (int)std::min<int64_t>((opts && opts->batch > 0) ? opts->batch : 256, nt);
    const float lr = (opts && opts->lr > 0.f) ? opts->lr : 1e-3f;
    uint64_t seed = (opts && opts->seed) ? opts->seed : 0x6d6c70ull;
    const bool regression = opts && opts->regression;
    std::vector<int32_t> grid, rgrid;
    if (opts && opts->grid_host && opts->ngrid > 0) grid.assign(opts->grid_host, opts->grid_host + opts->ngrid);
    else grid.assign(DEF_GRID, DEF_GRID + 11);
    if (opts && opts->rgrid_host && opts->nrgrid > 0) rgrid.assign(opts->rgrid_host, opts->rgrid_host + opts->nrgrid);
    else rgrid.assign(DEF_RGRID, DEF_RGRID + 5);
    while (!grid.empty() && grid.back() > ix->L) grid.pop_back();
    KSC_CHECK_ARG(!grid.empty() && !rgrid.empty(), "empty grid");
    KSC_CHECK_ARG(rgrid.back() <= KSC_MAX_RERANK && R_lab >= k, "bad rerank grid");
    const int Pr = std::min(std::max(grid.back(), 32), ix->L);
    const int64_t chunk = 8192;
    float* feats = nullptr;
    float* Y = nullptr;
    int32_t* probes = nullptr;
    float *w = nullptr, *m = nullptr, *v = nullptr, *act = nullptr, *lossd = nullptr;
    int64_t* idx = nullptr;
    std::vector<int32_t> lab_n(nt), lab_r(nt);
    int rc = KSC_OK;
    const int steps = (int)((nt + batch - 1) / batch);
#define T_CUDA(call) { cudaError_t e_ = (call); if (e_ != cudaSuccess) { set_error("%s: %s", #call, cudaGetErrorString(e_)); rc = KSC_ECUDA; break; } }
    do {
        T_CUDA(cudaMalloc(&feats, sizeof(float) * nt * KSC_MLP_FEATURES));
        T_CUDA(cudaMalloc(&Y, sizeof(float) * nt * 2));
        T_CUDA(cudaMalloc(&probes, sizeof(int32_t) * chunk * Pr));
        // 1. labels from the plain search, chunk by chunk
        for (int64_t c0 = 0; c0 < nt && rc == KSC_OK; c0 += chunk) {
            const int64_t nc = std::min(chunk, nt - c0);
            const float* Qc = Qtrain_dev + c0 * rr_d(ix);
            const float* Qcw;
            if ((rc = work_queries(ix, Qc, nc, st, &Qcw))) break;
            if ((rc = rank_and_features(ix, Qcw, nc, Pr, probes, feats + c0 * KSC_MLP_FEATURES, st))) break;
            std::vector<int32_t> ln, lr_;
            if ((rc = label_queries(ix, Qcw, Qc, nc, kth_dev + c0, probes, Pr, grid, nullptr, R_lab, k, target, ln, st)))
                break;
            if ((rc = label_queries(ix, Qcw, Qc, nc, kth_dev + c0, probes, Pr, rgrid, &ln, 0, k, target, lr_, st))) break;
            std::copy(ln.begin(), ln.end(), lab_n.begin() + c0);
            std::copy(lr_.begin(), lr_.end(), lab_r.begin() + c0);
        }
        if (rc) break;
        const float med_n = median_of(lab_n), med_r = median_of(lab_r);
        std::vector<float> yh(nt * 2);
        // regression heads: soft targets, the normalised log of the label
        auto soft = [](int32_t v, int32_t lo, int32_t hi) {
            return hi > lo ? (float)((std::log((double)v) - std::log((double)lo)) / (std::log((double)hi) - std::log((double)lo)))
                           : 0.f;
        };
        for (int64_t q = 0; q < nt; ++q) {
            if (regression) {
                yh[2 * q] = soft(lab_n[q], grid.front(), grid.back());
                yh[2 * q + 1] = soft(lab_r[q], rgrid.front(), rgrid.back());
            } else {
                yh[2 * q] = lab_n[q] > med_n ? 1.f : 0.f;
                yh[2 * q + 1] = lab_r[q] > med_r ? 1.f : 0.f;
            }
        }
        T_CUDA(cudaMemcpy(Y, yh.data(), sizeof(float) * nt * 2, cudaMemcpyHostToDevice));
        // 2. weights: He-uniform from the seed, zero biases
        std::vector<float> wh(KSC_MLP_NPARAMS, 0.f);
        const int fan[3] = {KSC_MLP_FEATURES, 64, 64}, rows[3] = {64, 64, 2};
        int off = 0;
        for (int l = 0; l < 3; ++l) {
            const float a = sqrtf(6.f / fan[l]);
            for (int e = 0; e < rows[l] * fan[l]; ++e)
                wh[off + e] = a * (2.f * (float)((mix64(seed) >> 11) * (1.0 / 9007199254740992.0)) - 1.f);
            off += rows[l] * fan[l] + rows[l];
        }
        T_CUDA(cudaMalloc(&w, sizeof(float) * KSC_MLP_NPARAMS));
        T_CUDA(cudaMalloc(&m, sizeof(float) * KSC_MLP_NPARAMS));
        T_CUDA(cudaMalloc(&v, sizeof(float) * KSC_MLP_NPARAMS));
        T_CUDA(cudaMalloc(&act, sizeof(float) * mlp_train_act(batch)));
        T_CUDA(cudaMalloc(&idx, sizeof(int64_t) * nt));
        T_CUDA(cudaMalloc(&lossd, sizeof(float) * steps));
        T_CUDA(cudaMemcpy(w, wh.data(), sizeof(float) * KSC_MLP_NPARAMS, cudaMemcpyHostToDevice));
        T_CUDA(cudaMemset(m, 0, sizeof(float) * KSC_MLP_NPARAMS));
        T_CUDA(cudaMemset(v, 0, sizeof(float) * KSC_MLP_NPARAMS));
        // 3. Adam over shuffled minibatches
        std::vector<int64_t> perm(nt);
        int t = 0;
        for (int ep = 0; ep < epochs && rc == KSC_OK; ++ep) {
            for (int64_t i = 0; i < nt; ++i) perm[i] = i;
            for (int64_t i = nt - 1; i > 0; --i) std::swap(perm[i], perm[(int64_t)(mix64(seed) % (uint64_t)(i + 1))]);
            T_CUDA(cudaMemcpyAsync(idx, perm.data(), sizeof(int64_t) * nt, cudaMemcpyHostToDevice, st));
            T_CUDA(cudaMemsetAsync(lossd, 0, sizeof(float) * steps, st));
            for (int s_ = 0; s_ < steps; ++s_) {
                const int64_t b0 = (int64_t)s_ * batch, nb = std::min<int64_t>(batch, nt - b0);
                if ((rc = mlp_train_step(w, m, v, feats, Y, idx + b0, nb, batch, act, lossd + s_, ++t, lr, st))) break;
            }
            T_CUDA(cudaStreamSynchronize(st));  // perm is reused by the next epoch
        }
        if (rc) break;
        if (loss_host) {
            std::vector<float> lh(steps);
            T_CUDA(cudaMemcpy(lh.data(), lossd, sizeof(float) * steps, cudaMemcpyDeviceToHost));
            double sum = 0.0;
            for (float x : lh) sum += x;
            *loss_host = (float)(sum / steps);
        }
        if (ix->mlp_w) cudaFree(ix->mlp_w);
        ix->mlp_w = w;
        w = nullptr;
        ix->mlp_prm = regression
                          ? ksc_adaptive_params{grid.front(), grid.back(), rgrid.front(), rgrid.back(), 0.f, 0.f, 0.f,
                                                0.f, 1}
                          : ksc_adaptive_params{grid.front(), grid.back(), rgrid.front(), rgrid.back(), 0.3f, 0.5f,
                                                0.3f, 0.5f, 0};
    } while (0);
#undef T_CUDA
    cudaFree(feats); cudaFree(Y); cudaFree(probes); cudaFree(w); cudaFree(m); cudaFree(v); cudaFree(act);
    cudaFree(idx); cudaFree(lossd);
    return rc;
}

int ksc_search_adaptive(ksc_index* ix, const float* Q_dev, int64_t nq, int32_t k, int64_t* ids_dev,
                        float* dists_dev, int32_t* nprobe_dev, int32_t* rerank_dev, const ksc_search_opts* opts,
                        void* stream) {
    KSC_CHECK_ARG(ix, "null index");
    if (!ix->mlp_w) {
        set_error("no predictor has been trained or loaded");
        return KSC_ESTATE;
    }
    const ksc_adaptive_params& prm = ix->mlp_prm;
    const int Pr = std::min(std::max(prm.pmax, 1), ix->L);  // the lists a query may probe
    Plan pl;
    KSC_TRY(make_plan(ix, nq, k, Pr, prm.rmax, opts, pl));
    if (nq == 0) return KSC_OK;
    KSC_CHECK_ARG(Q_dev && ids_dev && dists_dev, "null argument");
    cudaStream_t st = as_stream(stream);
    KSC_TRY(reset_counters(ix, st));
    KSC_TRY(ensure(ix->ws_probes, sizeof(int32_t) * nq * Pr, st));
    KSC_TRY(ensure(ix->ws_nprobe, sizeof(int32_t) * nq, st));
    KSC_TRY(ensure(ix->ws_rerank, sizeof(int32_t) * nq, st));
    int32_t* probes = (int32_t*)ix->ws_probes.p;
    int32_t* np_q = (int32_t*)ix->ws_nprobe.p;
    int32_t* r_q = (int32_t*)ix->ws_rerank.p;
    ix->launches = 0;
    mark(ix, 0, st);
    const float* Qw;
    KSC_TRY(work_queries(ix, Q_dev, nq, st, &Qw));
    KSC_TRY(rank_adaptive(ix, Qw, nq, Pr, probes, prm, np_q, r_q, st));
    pl.nprobe_q = np_q;
    pl.rerank_q = r_q;
    pl.Pq_max = std::min(prm.pmax, Pr);
    const int32_t* sprobes = probes;
    if (ix->pr_theta >= 0.f && ix->pr_model && ix->pr_have_stats) {
        // Alg. 2: predictive pruning of the predicted nprobe lists
        KSC_TRY(ensure(ix->ws_pprobes, sizeof(int32_t) * nq * Pr, st));
        KSC_TRY(ensure(ix->ws_pn, sizeof(int32_t) * nq, st));
        int32_t* kept = (int32_t*)ix->ws_pprobes.p;
        int32_t* pn = (int32_t*)ix->ws_pn.p;
        KSC_TRY(prune_rows(ix, Qw, nq, probes, Pr, np_q, Pr, ix->pr_theta, nullptr, nullptr, kept, pn, st));
        ix->launches += 2;
        sprobes = kept;
        np_q = pn;
        pl.nprobe_q = pn;
    }
    set_tiles(ix, pl, nq, 0.5 * (prm.pmin + prm.pmax), opts);
    plan_small(ix, pl, opts, true, false);
    KSC_TRY(search_from_probes(ix, Qw, pl, sprobes, ids_dev, dists_dev, nullptr, nullptr, st, Q_dev));
    if (nprobe_dev) KSC_CUDA(cudaMemcpyAsync(nprobe_dev, np_q, sizeof(int32_t) * nq, cudaMemcpyDeviceToDevice, st));
    if (rerank_dev) KSC_CUDA(cudaMemcpyAsync(rerank_dev, r_q, sizeof(int32_t) * nq, cudaMemcpyDeviceToDevice, st));
    return KSC_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ captured plans, autotuner
struct ksc_plan {
    ksc_index* ix = nullptr;
    int64_t nq = 0;
    int32_t k = 0, nprobe = 0, rerank = 0, adaptive = 0;
    ksc_search_opts opts = {};
    bool has_opts = false;
    float* Q = nullptr;
    int64_t* ids = nullptr;
    float* dists = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    unsigned long long gen = 0;
};

namespace ksc {
static int plan_search(ksc_plan* pl, cudaStream_t st) {
    const ksc_search_opts* o = pl->has_opts ? &pl->opts : nullptr;
    if (pl->adaptive)
        return ksc_search_adaptive(pl->ix, pl->Q, pl->nq, pl->k, pl->ids, pl->dists, nullptr, nullptr, o, st);
    return ksc_search(pl->ix, pl->Q, pl->nq, pl->k, pl->nprobe, pl->rerank, pl->ids, pl->dists, o, st);
}

// Warm the workspace with one search, then capture the next into a graph.
static int plan_capture(ksc_plan* pl, cudaStream_t st) {
    if (pl->exec) { cudaGraphExecDestroy(pl->exec); pl->exec = nullptr; }
    if (pl->graph) { cudaGraphDestroy(pl->graph); pl->graph = nullptr; }
    const bool prof = pl->ix->prof;
    pl->ix->prof = false;
    pl->ix->u8_now = true;
    int rc = plan_search(pl, st);
    pl->ix->u8_now = false;
    if (rc == KSC_OK) {
        cudaError_t e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { set_error("warm-up failed: %s", cudaGetErrorString(e)); rc = KSC_ECUDA; }
    }
    if (rc == KSC_OK) {
        pl->gen = workspace_generation();
        cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) {
            set_error("stream capture failed to start: %s", cudaGetErrorString(e));
            rc = KSC_ECUDA;
        } else {
            rc = plan_search(pl, st);
            cudaGraph_t g = nullptr;
            e = cudaStreamEndCapture(st, &g);
            if (rc == KSC_OK && e != cudaSuccess) {
                set_error("stream capture failed: %s", cudaGetErrorString(e));
                rc = KSC_ECUDA;
            }
            pl->graph = g;
            if (rc == KSC_OK && workspace_generation() != pl->gen) {
                set_error("workspace changed during capture");
                rc = KSC_ESTATE;
            }
            if (rc == KSC_OK) {
                e = cudaGraphInstantiate(&pl->exec, pl->graph, 0);
                if (e != cudaSuccess) {
                    set_error("graph instantiation failed: %s", cudaGetErrorString(e));
                    rc = KSC_ECUDA;
                }
            }
        }
    }
    pl->ix->prof = prof;
    return rc;
}
}  // namespace ksc

extern "C" {

void ksc_plan_free(ksc_plan* pl) {
    if (!pl) return;
    if (pl->exec) cudaGraphExecDestroy(pl->exec);
    if (pl->graph) cudaGraphDestroy(pl->graph);
    cudaFree(pl->Q);
    cudaFree(pl->ids);
    cudaFree(pl->dists);
    delete pl;
}

int ksc_plan_create(ksc_index* ix, int64_t nq, int32_t k, int32_t nprobe, int32_t rerank, int32_t adaptive,
                    const ksc_search_opts* opts, void* stream, ksc_plan** out) {
    KSC_CHECK_ARG(ix && out && nq > 0 && k >= 1, "bad argument");
    KSC_CHECK_ARG(stream != nullptr, "plans need a non-default stream (graph capture)");
    cudaStream_t st = as_stream(stream);
    ksc_plan* pl = new ksc_plan();
    pl->ix = ix;
    pl->nq = nq;
    pl->k = k;
    pl->nprobe = nprobe;
    pl->rerank = rerank;
    pl->adaptive = adaptive;
    if (opts) { pl->opts = *opts; pl->has_opts = true; }
    int rc = KSC_OK;
    if (cudaMalloc(&pl->Q, sizeof(float) * nq * rr_d(ix)) != cudaSuccess ||
        cudaMalloc(&pl->ids, sizeof(int64_t) * nq * k) != cudaSuccess ||
        cudaMalloc(&pl->dists, sizeof(float) * nq * k) != cudaSuccess) {
        set_error("plan buffer allocation failed");
        rc = KSC_ENOMEM;
    }
    if (rc == KSC_OK && cudaMemsetAsync(pl->Q, 0, sizeof(float) * nq * rr_d(ix), st) != cudaSuccess) rc = KSC_ECUDA;
    if (rc == KSC_OK) rc = plan_capture(pl, st);
    if (rc != KSC_OK) {
        ksc_plan_free(pl);
        return rc;
    }
    *out = pl;
    return KSC_OK;
}

int ksc_plan_buffers(ksc_plan* pl, float** Q_dev, int64_t** ids_dev, float** dists_dev) {
    KSC_CHECK_ARG(pl, "null plan");
    if (Q_dev) *Q_dev = pl->Q;
    if (ids_dev) *ids_dev = pl->ids;
    if (dists_dev) *dists_dev = pl->dists;
    return KSC_OK;
}

int ksc_plan_execute(ksc_plan* pl, const float* Q_dev, int64_t* ids_dev, float* dists_dev, void* stream) {
    KSC_CHECK_ARG(pl && pl->exec, "null plan");
    cudaStream_t st = as_stream(stream);
    KSC_CHECK_ARG(stream != nullptr, "plans need a non-default stream (graph capture)");
    if (Q_dev && Q_dev != pl->Q)
        KSC_CUDA(cudaMemcpyAsync(pl->Q, Q_dev, sizeof(float) * pl->nq * rr_d(pl->ix), cudaMemcpyDeviceToDevice, st));
    if (workspace_generation() != pl->gen) KSC_TRY(plan_capture(pl, st));
    KSC_CUDA(cudaGraphLaunch(pl->exec, st));
    if (ids_dev && ids_dev != pl->ids)
        KSC_CUDA(cudaMemcpyAsync(ids_dev, pl->ids, sizeof(int64_t) * pl->nq * pl->k, cudaMemcpyDeviceToDevice, st));
    if (dists_dev && dists_dev != pl->dists)
        KSC_CUDA(cudaMemcpyAsync(dists_dev, pl->dists, sizeof(float) * pl->nq * pl->k, cudaMemcpyDeviceToDevice, st));
    return KSC_OK;
}

int ksc_autotune(ksc_index* ix, const float* Q_dev, int64_t nq, int32_t k, int32_t nprobe, int32_t rerank,
                 ksc_search_opts* opts, void* stream, float* best_ms_host) {
    KSC_CHECK_ARG(ix && Q_dev && opts && nq > 0, "bad argument");
    cudaStream_t st = as_stream(stream);
    int64_t* ids = nullptr;
    float* dists = nullptr;
    KSC_CUDA(cudaMalloc(&ids, sizeof(int64_t) * nq * k));
    cudaError_t ea = cudaMalloc(&dists, sizeof(float) * nq * k);
    if (ea != cudaSuccess) { cudaFree(ids); KSC_CUDA(ea); }
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const int Gs[4] = {4, 8, 16, 32};
    const int TBs[5] = {0, 8, 16, 32, 64};
    ksc_search_opts best = *opts;
    float best_ms = INFINITY;
    // (lanes alone, whatever an earlier call left in opts: byte permutes.)
    // First what the batch takes by itself, where that is the tensor cores (lanes
    // alone ask for byte permutes): its own lanes for the first part, and
    // scan_tc 2, which leaves the scan to the rule.  (10,000 queries of 1M x 64
    // subspaces at nprobe 7: 718 us, 976 at the best lanes.)
    ksc_search_opts own = *opts;
    own.lanes_per_query = own.tile_blocks = 0;
    Plan pl;
    int rc = make_plan(ix, nq, k, nprobe, rerank, &own, pl);
    if (rc == KSC_OK) plan_small(ix, pl, &own, true, true);
    own.lanes_per_query = pl.G;
    own.scan_tc = SCAN_TC_RULE;
    for (int gi = pl.tc && !pl.tc_opt ? -1 : 0; gi < 4 && rc == KSC_OK; ++gi) {
        if (gi >= 0 && (Gs[gi] == 4 ? ix->M > 128 : (ix->M + Gs[gi] - 1) / Gs[gi] > 16)) continue;
        for (int ti = 0; ti < 5 && rc == KSC_OK; ++ti) {
            ksc_search_opts o = gi < 0 ? own : *opts;
            if (gi >= 0) {
                o.lanes_per_query = Gs[gi];
                if (o.scan_tc == SCAN_TC_RULE) o.scan_tc = 0;
            }
            o.tile_blocks = TBs[ti];
            float ms = 0.f, tot = 0.f;
            for (int rep = 0; rep < 4 && rc == KSC_OK; ++rep) {
                cudaEventRecord(e0, st);
                rc = ksc_search(ix, Q_dev, nq, k, nprobe, rerank, ids, dists, &o, st);
                cudaEventRecord(e1, st);
                if (cudaEventSynchronize(e1) != cudaSuccess) { set_error("autotune run failed"); rc = KSC_ECUDA; }
                cudaEventElapsedTime(&ms, e0, e1);
                if (rep >= 1) tot += ms;  // the first run warms the workspace
            }
            if (rc == KSC_OK && tot / 3 < best_ms) {
                best_ms = tot / 3;
                best = o;
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(ids);
    cudaFree(dists);
    if (rc != KSC_OK) return rc;
    opts->lanes_per_query = best.lanes_per_query;
    opts->tile_blocks = best.tile_blocks;
    opts->scan_tc = best.scan_tc;
    if (best_ms_host) *best_ms_host = best_ms;
    return KSC_OK;
}

}  // extern "C"


// ------------------------------------------------------------------ predictive cluster pruning
// Sec. 4.2.3, Table 4, Alg. 2 f_prune: statistics, features and the
// classifier live in prune.cu; here are the entry points that tie them to the
// ranking, the plain search (labels) and the search of the kept lists.
extern "C" {

int ksc_pruner_stats(ksc_index* ix, int32_t iters, void* stream) {
    KSC_CHECK_STATE(!ix || !ix->parent, "the pruning statistics belong to the index, not to a view of it");
    KSC_CHECK_ARG(ix, "null index");
    return prune_stats(ix, iters, as_stream(stream));
}

int ksc_pruner_export(ksc_index* ix, float* stats_host, float* vecs_host, float* model_host) {
    KSC_CHECK_ARG(ix, "null index");
    if (stats_host || vecs_host) KSC_CHECK_STATE(ix->pr_have_stats, "the pruning statistics have not been computed");
    if (model_host) KSC_CHECK_STATE(ix->pr_model, "no pruning model");
    KSC_CUDA(cudaDeviceSynchronize());
    if (stats_host)
        KSC_CUDA(cudaMemcpy(stats_host, ix->pr_stats, sizeof(float) * ix->L * KSC_PRUNE_STATS, cudaMemcpyDeviceToHost));
    if (vecs_host)
        KSC_CUDA(cudaMemcpy(vecs_host, ix->pr_vecs, sizeof(float) * ix->L * 3 * ix->d, cudaMemcpyDeviceToHost));
    if (model_host)
        KSC_CUDA(cudaMemcpy(model_host, ix->pr_model, sizeof(float) * KSC_PRUNE_MODEL, cudaMemcpyDeviceToHost));
    return KSC_OK;
}

int ksc_pruner_import_model(ksc_index* ix, const float* model_host) {
    KSC_CHECK_STATE(!ix || !ix->parent, "models are set on the index, not on a view of it");
    KSC_CHECK_ARG(ix && model_host, "null argument");
    if (!ix->pr_model) KSC_CUDA(cudaMalloc(&ix->pr_model, sizeof(float) * KSC_PRUNE_MODEL));
    KSC_CUDA(cudaMemcpy(ix->pr_model, model_host, sizeof(float) * KSC_PRUNE_MODEL, cudaMemcpyHostToDevice));
    bump_workspace_generation();
    return KSC_OK;
}

int ksc_pruner_theta(ksc_index* ix, float theta) {
    KSC_CHECK_ARG(ix, "null index");
    KSC_CHECK_STATE(theta < 0.f || (ix->pr_have_stats && ix->pr_model), "no pruning model");
    ix->pr_theta = theta;
    bump_workspace_generation();
    return KSC_OK;
}

int ksc_prune_probes(ksc_index* ix, const float* Q_dev, int64_t nq, const int32_t* probes_dev, int32_t Pmax,
                     const int32_t* nprobe_dev, int32_t P, float theta, float* feats_dev, float* prob_dev,
                     int32_t* probes_out_dev, int32_t* nprobe_out_dev, void* stream) {
    KSC_CHECK_ARG(ix && nq >= 0 && Pmax >= 1 && (nprobe_dev || (P >= 1 && P <= Pmax)), "bad argument");
    if (nq == 0) return KSC_OK;
    KSC_CHECK_ARG(Q_dev && probes_dev, "null argument");
    cudaStream_t st = as_stream(stream);
    const float* Qw;
    KSC_TRY(work_queries(ix, Q_dev, nq, st, &Qw));
    return prune_rows(ix, Qw, nq, probes_dev, Pmax, nprobe_dev, P, theta, feats_dev, prob_dev, probes_out_dev,
                      nprobe_out_dev, st);
}

int ksc_prune_labels(ksc_index* ix, const int64_t* ids_dev, const float* dists_dev, int64_t nq, int32_t k,
                     const float* kth_dev, const int32_t* probes_dev, int32_t Pmax, int32_t P, float* label_dev,
                     void* stream) {
    KSC_CHECK_ARG(ix && nq >= 0 && k >= 1 && Pmax >= 1 && P >= 0, "bad argument");
    if (nq == 0) return KSC_OK;
    KSC_CHECK_ARG(ids_dev && dists_dev && kth_dev && probes_dev && label_dev, "null argument");
    return prune_labels(ix, ids_dev, dists_dev, nq, k, kth_dev, probes_dev, Pmax, P, label_dev, as_stream(stream));
}

int ksc_prune_mlp_grad(const float* w_dev, const float* x_dev, const float* y_dev, int64_t B, float* grad_dev,
                       float* loss_dev, void* stream) {
    KSC_CHECK_ARG(w_dev && x_dev && y_dev && grad_dev && B > 0, "bad argument");
    return prune_mlp_grad(w_dev, x_dev, y_dev, B, grad_dev, loss_dev, as_stream(stream));
}

int ksc_search_pruned(ksc_index* ix, const float* Q_dev, int64_t nq, int32_t k, int32_t nprobe, int32_t rerank,
                      float theta, int64_t* ids_dev, float* dists_dev, int32_t* nprobe_out_dev,
                      const ksc_search_opts* opts, void* stream) {
    KSC_CHECK_ARG(ix, "null index");
    KSC_CHECK_STATE(ix->pr_have_stats && ix->pr_model, "no pruning model: train one with ksc_train_pruner");
    Plan pl;
    KSC_TRY(make_plan(ix, nq, k, nprobe, rerank, opts, pl));
    if (nq == 0) return KSC_OK;  // empty batch: pointers may be NULL
    KSC_CHECK_ARG(Q_dev && ids_dev && dists_dev, "null argument");
    cudaStream_t st = as_stream(stream);
    KSC_TRY(reset_counters(ix, st));
    KSC_TRY(ensure(ix->ws_probes, sizeof(int32_t) * nq * pl.Pmax, st));
    KSC_TRY(ensure(ix->ws_pprobes, sizeof(int32_t) * nq * pl.Pmax, st));
    KSC_TRY(ensure(ix->ws_pn, sizeof(int32_t) * nq, st));
    int32_t* probes = (int32_t*)ix->ws_probes.p;
    int32_t* kept = (int32_t*)ix->ws_pprobes.p;
    int32_t* pn = (int32_t*)ix->ws_pn.p;
    ix->launches = 0;
    mark(ix, 0, st);
    const float* Qw;
    KSC_TRY(work_queries(ix, Q_dev, nq, st, &Qw));
    KSC_TRY(rank_lists(ix, Qw, nq, nullptr, pl.Pmax, pl.Pmax, probes, nullptr, pl.rank_mode, st));
    // Alg. 2: keep rank 0 and the ranks with f_prune > theta, in rank order
    KSC_TRY(prune_rows(ix, Qw, nq, probes, pl.Pmax, nullptr, pl.Pmax, theta, nullptr, nullptr, kept, pn, st));
    ix->launches++;
    pl.nprobe_q = pn;
    set_tiles(ix, pl, nq, 0.75 * pl.Pmax, opts);
    if (nprobe_out_dev)
        KSC_CUDA(cudaMemcpyAsync(nprobe_out_dev, pn, sizeof(int32_t) * nq, cudaMemcpyDeviceToDevice, st));
    plan_small(ix, pl, opts, true, false);
    return search_from_probes(ix, Qw, pl, kept, ids_dev, dists_dev, nullptr, nullptr, st, Q_dev);
}

#define T_CUDA(call) { cudaError_t e_ = (call); if (e_ != cudaSuccess) { set_error("%s: %s", #call, cudaGetErrorString(e_)); rc = KSC_ECUDA; break; } }
int ksc_train_pruner(ksc_index* ix, const float* Qtrain_dev, int64_t nt, const float* kth_dev, int32_t k,
                     int32_t P, int32_t R, const ksc_train_opts* opts, void* stream, float* loss_host) {
    KSC_CHECK_STATE(!ix || !ix->parent, "the pruner is trained on an index, not on a view of it");
    KSC_CHECK_ARG(ix && Qtrain_dev && kth_dev && nt > 0, "bad argument");
    KSC_CHECK_ARG(k >= 1 && k <= KSC_MAX_K && R >= k && R <= KSC_MAX_RERANK, "bad k or rerank");
    KSC_CHECK_ARG(P >= 1 && P <= ix->L && P <= MAX_NPROBE, "bad nprobe");
    cudaStream_t st = as_stream(stream);
    if (!ix->pr_have_stats) KSC_TRY(prune_stats(ix, 30, st));
    const int epochs = (opts && opts->epochs > 0) ? opts->epochs : 4;
    const int batch = (int)std::min<int64_t>((opts && opts->batch > 0) ? opts->batch : 1024, nt * P);
    const float lr = (opts && opts->lr > 0.f) ? opts->lr : 1e-3f;
    uint64_t seed = (opts && opts->seed) ? opts->seed : 0x707275ull;
    const int64_t chunk = 8192, rows = nt * P;
    const int NF = KSC_PRUNE_FEATURES, NP = KSC_PRUNE_NPARAMS;
    float *feats = nullptr, *lab = nullptr, *Y = nullptr, *dists = nullptr, *model = nullptr;
    float *w = nullptr, *m = nullptr, *v = nullptr, *act = nullptr, *lossd = nullptr;
    int32_t* probes = nullptr;
    int64_t *ids = nullptr, *idx = nullptr;
    int rc = KSC_OK;
    const int steps = (int)((rows + batch - 1) / batch);
    do {
        T_CUDA(cudaMalloc(&feats, sizeof(float) * rows * NF));
        T_CUDA(cudaMalloc(&lab, sizeof(float) * rows));
        T_CUDA(cudaMalloc(&Y, sizeof(float) * rows * 2));
        T_CUDA(cudaMalloc(&probes, sizeof(int32_t) * chunk * P));
        T_CUDA(cudaMalloc(&ids, sizeof(int64_t) * chunk * k));
        T_CUDA(cudaMalloc(&dists, sizeof(float) * chunk * k));
        T_CUDA(cudaMalloc(&model, sizeof(float) * KSC_PRUNE_MODEL));
        // 1. rows of the P nearest lists of every training query: labels from
        //    the plain search of those lists, features
        for (int64_t c0 = 0; c0 < nt && rc == KSC_OK; c0 += chunk) {
            const int64_t nc = std::min(chunk, nt - c0);
            const float* Qc = Qtrain_dev + c0 * rr_d(ix);
            const float* Qcw;
            if ((rc = work_queries(ix, Qc, nc, st, &Qcw))) break;
            if ((rc = rank_lists(ix, Qcw, nc, nullptr, P, P, probes, nullptr, RANK_TC16, st))) break;
            Plan pl;
            if ((rc = make_plan(ix, nc, k, P, R, nullptr, pl))) break;
            if ((rc = search_from_probes(ix, Qcw, pl, probes, ids, dists, nullptr, nullptr, st, Qc))) break;
            if ((rc = prune_labels(ix, ids, dists, nc, k, kth_dev + c0, probes, P, P, lab + c0 * P, st))) break;
            if ((rc = prune_rows(ix, Qcw, nc, probes, P, nullptr, P, 0.f, feats + c0 * P * NF, nullptr, nullptr,
                                 nullptr, st)))
                break;
        }
        if (rc) break;
        // 2. standardised features, targets
        if ((rc = prune_standardise(feats, rows, model, st))) break;
        if ((rc = prune_targets(lab, rows, Y, st))) break;
        // 3. weights: He-uniform from the seed, zero biases
        std::vector<float> wh(NP, 0.f);
        const int fan[3] = {NF, 32, 32}, nrow[3] = {32, 32, 2};
        int off = 0;
        for (int l = 0; l < 3; ++l) {
            const float a = sqrtf(6.f / fan[l]);
            for (int e = 0; e < nrow[l] * fan[l]; ++e)
                wh[off + e] = a * (2.f * (float)((mix64(seed) >> 11) * (1.0 / 9007199254740992.0)) - 1.f);
            off += nrow[l] * fan[l] + nrow[l];
        }
        T_CUDA(cudaMalloc(&w, sizeof(float) * NP));
        T_CUDA(cudaMalloc(&m, sizeof(float) * NP));
        T_CUDA(cudaMalloc(&v, sizeof(float) * NP));
        T_CUDA(cudaMalloc(&act, sizeof(float) * prune_train_act(batch)));
        T_CUDA(cudaMalloc(&idx, sizeof(int64_t) * rows));
        T_CUDA(cudaMalloc(&lossd, sizeof(float) * steps));
        T_CUDA(cudaMemcpy(w, wh.data(), sizeof(float) * NP, cudaMemcpyHostToDevice));
        T_CUDA(cudaMemset(m, 0, sizeof(float) * NP));
        T_CUDA(cudaMemset(v, 0, sizeof(float) * NP));
        // 4. Adam over shuffled minibatches of rows
        std::vector<int64_t> perm(rows);
        int t = 0;
        for (int ep = 0; ep < epochs && rc == KSC_OK; ++ep) {
            for (int64_t i = 0; i < rows; ++i) perm[i] = i;
            for (int64_t i = rows - 1; i > 0; --i) std::swap(perm[i], perm[(int64_t)(mix64(seed) % (uint64_t)(i + 1))]);
            T_CUDA(cudaMemcpyAsync(idx, perm.data(), sizeof(int64_t) * rows, cudaMemcpyHostToDevice, st));
            T_CUDA(cudaMemsetAsync(lossd, 0, sizeof(float) * steps, st));
            for (int s_ = 0; s_ < steps; ++s_) {
                const int64_t b0 = (int64_t)s_ * batch, nb = std::min<int64_t>(batch, rows - b0);
                if ((rc = prune_train_step(w, m, v, feats, Y, idx + b0, nb, batch, act, lossd + s_, ++t, lr, st))) break;
            }
            T_CUDA(cudaStreamSynchronize(st));  // perm is reused by the next epoch
        }
        if (rc) break;
        if (loss_host) {
            std::vector<float> lh(steps);
            T_CUDA(cudaMemcpy(lh.data(), lossd, sizeof(float) * steps, cudaMemcpyDeviceToHost));
            double sum = 0.0;
            for (float x : lh) sum += x;
            *loss_host = (float)(sum / steps);
        }
        T_CUDA(cudaMemcpy(model, w, sizeof(float) * NP, cudaMemcpyDeviceToDevice));
        if (ix->pr_model) cudaFree(ix->pr_model);
        ix->pr_model = model;
        model = nullptr;
        bump_workspace_generation();
    } while (0);
    void* tmp[] = {feats, lab, Y, dists, model, w, m, v, act, lossd, probes, ids, idx};
    for (void* p : tmp)
        if (p) cudaFree(p);
    return rc;
}
#undef T_CUDA

}  // extern "C"
