// Centroid ranking scores (Alg. 2 TopNClusters) on the 5th-generation tensor
// cores: S = Q16 . C16^T (16-bit operands: FP16 when the centroids fit it,
// else BF16) accumulated in FP32 in tensor memory.
//
// One CTA computes a 128 x 256 tile (128 queries x 256 lists): TMA loads the
// K-major BF16 operands into shared memory as 128-byte-swizzled boxes of 64
// elements, one elected thread issues tcgen05.mma (M 128, N 256, K 16 per
// instruction) into a 256-column TMEM accumulator, tcgen05.commit signals an
// mbarrier, and the four warps read their 32 TMEM lanes back with
// tcgen05.ld and write score = ||c||^2 - 2 <q, c> (L2) or -<q, c>.  These
// scores are approximate (16-bit operands); the ranking kernel re-scores in
// FP32 every list that their error bound cannot exclude.
//
// FP8 option (kind::f8f6f4, e4m3 x e4m3, FP32 accumulate): every query and
// centroid row is scaled by a power of two s = 2^(e - 8), e the exponent of
// the row's largest magnitude (so the scaled row peaks in [128, 256), inside
// e4m3's range, and the scaling itself is exact), rounded to e4m3, and the
// accumulated dot product is multiplied back by s_q s_c (exact: a power of
// two).  A 128-element e4m3 box is 128 bytes per row, the same swizzle atom
// as a 64-element 16-bit box, and one MMA takes K = 32, so the tile loop and
// the descriptors are those of the 16-bit path.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <cstdio>
#include <vector>

#include "index.cuh"
#include "scan.cuh"
#include "tc.cuh"

namespace ksc {

// scores[q][c] for one 128 x 256 tile.  KB = number of K boxes of 128 bytes
// per row (64 16-bit or 128 8-bit elements); up to RG_STAGES boxes are in
// shared memory, a box's place is loaded again once its MMAs are done.  F8:
// e4m3 operands whose rows carry the power-of-two scales qs [nq] and cs [L].
constexpr int RG_STAGES = 4;
template <bool F8>
__global__ void __launch_bounds__(128, 1) k_rank_gemm_tc(const __grid_constant__ CUtensorMap mapA,
                                                         const __grid_constant__ CUtensorMap mapB, int KB, int64_t nq,
                                                         int L, const float* __restrict__ cn, int spherical,
                                                         int fmt, const float* __restrict__ qs,
                                                         const float* __restrict__ cs, float* __restrict__ scores,
                                                         int32_t* __restrict__ status) {
    constexpr int BOX_K = F8 ? 128 : TC_KB;  // elements per 128-byte box row
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * RG_STAGES + 1];
    __shared__ uint32_t tmem_base;
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int NS = KB < RG_STAGES ? KB : RG_STAGES;
    const uint32_t sA = smem_u32(smem), sB = sA + NS * (TC_M * 128);
    auto full = [&](int i) { return smem_u32(&bars[i]); };               // stage i's copies have landed
    auto used = [&](int i) { return smem_u32(&bars[RG_STAGES + i]); };   // stage i's MMAs are done
    const uint32_t bar_mma = smem_u32(&bars[2 * RG_STAGES]);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.y * TC_M, n0 = blockIdx.x * TC_N;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2 * RG_STAGES; ++i) mbar_init(full(i), 1);
        mbar_init(bar_mma, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(TC_N));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    bool ok = true;
    if (threadIdx.x == 0) {
        auto load = [&](int kb) {
            const int i = kb % NS;
            mbar_expect_tx(full(i), (TC_M + TC_N) * 128);
            tma_load_2d(sA + i * (TC_M * 128), &mapA, full(i), kb * BOX_K, m0);
            tma_load_2d(sB + i * (TC_N * 128), &mapB, full(i), kb * BOX_K, n0);
        };
        for (int kb = 0; kb < NS; ++kb) load(kb);
        const uint32_t idesc = idesc_f16kind(fmt, TC_M, TC_N);
        int loaded = NS, kb = 0;
        for (; kb < KB; ++kb) {
            const int i = kb % NS;
            ok = mbar_wait(full(i), (kb / NS) & 1, TC_WAIT_LIMIT);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // four MMAs per 128-byte box: K = 16 16-bit or 32 8-bit elements = 32 bytes each
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint64_t a = smem_desc(sA + i * (TC_M * 128) + k * 32);
                const uint64_t b = smem_desc(sB + i * (TC_N * 128) + k * 32);
                if (F8) tc_mma_f8(tmem, a, b, idesc, (kb | k) != 0);
                else tc_mma(tmem, a, b, idesc, (kb | k) != 0);
            }
            tc_commit(used(i));
            if (kb > 0 && loaded < KB) {  // the stage before this one again, once its MMAs have read it
                ok = mbar_wait(used((kb - 1) % NS), ((kb - 1) / NS) & 1, TC_WAIT_LIMIT);
                if (!ok) break;
                load(loaded++);
            }
        }
        if (ok) {
            tc_commit(bar_mma);
        } else {  // a copy or MMA never completed: what is in flight is waited for (bounded) once more
            atomicOr(status, 2);
            for (int l = kb; l < loaded; ++l) mbar_wait(full(l % NS), (l / NS) & 1, TC_WAIT_LIMIT);
            tc_commit(bar_mma);
            mbar_wait(bar_mma, 0, TC_WAIT_LIMIT);
        }
    }
    __syncthreads();
    const bool done = __syncthreads_and(threadIdx.x == 0 ? ok : 1);
    // warp-uniform decision (tcgen05.ld is a warp-collective instruction)
    const bool mma_ok = done && __all_sync(0xffffffffu, mbar_wait(bar_mma, 0, TC_WAIT_LIMIT));
    if (mma_ok) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // 32 x 32 sub-tiles go through the operand buffers (no longer read: the
        // MMAs have completed) so that each store writes 32 consecutive
        // columns of one row; row stride 33 keeps both sides free of bank conflicts
        float* stage = reinterpret_cast<float*>(smem) + warp * (32 * 33);
        const int64_t qb = (int64_t)m0 + warp * 32;
        for (int c0 = 0; c0 < TC_N; c0 += 32) {
            uint32_t r[32];
            tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + c0, r);  // lane = row, r[i] = column c0 + i
#pragma unroll
            for (int i = 0; i < 32; ++i) stage[lane * 33 + i] = __uint_as_float(r[i]);
            __syncwarp();
            const int c = n0 + c0 + lane;
            if (c < L) {
                const float cc = spherical ? 0.f : cn[c];
                const float sc = F8 ? cs[c] : 1.f;
                const int nr = nq - qb < 32 ? (int)(nq - qb) : 32;  // rows of this warp inside the batch
                // sixteen rows at a time: their shared loads, then their stores
#pragma unroll 1
                for (int r0 = 0; r0 < nr; r0 += 16) {
                    float v[16];
#pragma unroll
                    for (int u = 0; u < 16; ++u) {
                        const int rr = r0 + u < nr ? r0 + u : nr - 1;
                        // F8: the product of two powers of two, an exact rescaling
                        const float dot = F8 ? stage[rr * 33 + lane] * (qs[qb + rr] * sc) : stage[rr * 33 + lane];
                        v[u] = spherical ? -dot : fmaf(-2.f, dot, cc);
                    }
#pragma unroll
                    for (int u = 0; u < 16; ++u)
                        if (r0 + u < nr) scores[(qb + r0 + u) * L + c] = v[u];
                }
            }
            __syncwarp();
        }
    } else if (done && lane == 0) {
        atomicOr(status, 2);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_N));
}

// rows of X (fp32 [n x d]) to 16-bit operands [n x Kp] (FP16 when fp16 is
// set, else BF16; round to nearest), zero-padded K.
__global__ void k_to_16(const float* __restrict__ X, int64_t n, int d, int Kp, int fp16, uint16_t* __restrict__ out) {
    int64_t tot = n * Kp;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e / Kp;
        int t = (int)(e - r * Kp);
        const float v = t < d ? X[r * d + t] : 0.f;
        out[e] = fp16 ? __half_as_ushort(__float2half_rn(v)) : __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
}

// Per-query bound on |given score - exact score| for every list:
// rel * ||q|| * max||c|| (times 2 for L2, whose score carries -2 <q, c>) plus
// (d + 8) 2^-23 (||q|| + max||c||)^2 for the FP32 rounding of ||c||^2 and of
// the exact FP32 re-score.
//  16-bit tensor-core operands: |<q~, c~> - <q, c>| <= (2u + u^2) sum |q_t c_t|
//    + FP32 accumulation, u = 2^-11 (FP16) or 2^-8 (BF16), and
//    sum |q_t c_t| <= ||q|| ||c|| (Cauchy-Schwarz); for FP16 also the
//    subnormal range's absolute error, 2^-25 per element.  FP16 is used when every
//    centroid element is below 2^14 and a query element above 6e4 voids the
//    bound (err = inf: every list is re-scored).
//  FP32 CUDA cores: a dot product of d terms errs by at most about d 2^-24
//    of sum |q_t c_t|.
__global__ void k_score_err(const float* __restrict__ Q, int64_t nq, int d, float cmax, int spherical, float rel,
                            float qmax, float* __restrict__ err) {
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= nq) return;
    float s = 0.f, mx = 0.f;
    for (int t = 0; t < d; ++t) {
        s = fmaf(Q[q * d + t], Q[q * d + t], s);
        mx = fmaxf(mx, fabsf(Q[q * d + t]));
    }
    if (mx > qmax) {  // an element the 16-bit operand cannot hold: no bound
        err[q] = INFINITY;
        return;
    }
    const float qn = sqrtf(s);
    const float e = rel * qn * cmax * 1.0001f;
    // plus the FP32 rounding of ||c||^2 and of the exact re-score itself
    const float r = (float)(d + 8) * 1.2e-7f * (qn + cmax) * (qn + cmax);
    err[q] = (spherical ? e : 2.f * e) + r;
}

// Queries to 16-bit operands [nq x Kp] (zero-padded K) and, in the same pass,
// the per-query bound of k_score_err.  One warp per query (coalesced rows).
__global__ void k_q16_err(const float* __restrict__ Q, int64_t nq, int d, int Kp, int fp16, float cmax,
                          int spherical, float rel, float qmax, uint16_t* __restrict__ out,
                          float* __restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int64_t q = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (q >= nq) return;
    float s = 0.f, mx = 0.f;
    for (int t = lane; t < Kp; t += 32) {
        const float v = t < d ? Q[q * d + t] : 0.f;
        s = fmaf(v, v, s);
        mx = fmaxf(mx, fabsf(v));
        out[q * Kp + t] = fp16 ? __half_as_ushort(__float2half_rn(v)) : __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane != 0) return;
    if (mx > qmax) {  // an element the 16-bit operand cannot hold: no bound
        err[q] = INFINITY;
        return;
    }
    const float qn = sqrtf(s);
    // FP16 elements below 2^-14 are subnormal: their rounding error is up to
    // half the spacing 2^-24 rather than relative, for the query's and the
    // centroids' elements alike: eta sum(|c_t| + |q_t|) <= eta sqrt(d) (|q| +
    // max|c|) (BF16 keeps the FP32 exponent range: its 2^-134 is far below r)
    const float sub = fp16 ? 0x1p-25f * sqrtf((float)d) * (qn + cmax) * 1.01f : 0.f;
    const float e = (rel * qn * cmax + sub) * 1.0001f;
    const float r = (float)(d + 8) * 1.2e-7f * (qn + cmax) * (qn + cmax);
    err[q] = (spherical ? e : 2.f * e) + r;
}

// Power-of-two scale of a row whose largest magnitude is mx: 2^(e - 8) with
// mx = m 2^e, m in [0.5, 1), so mx / s = 256 m lies in [128, 256); 1 for a
// zero row.
__device__ __forceinline__ float f8_row_scale(float mx) {
    if (!(mx > 0.f)) return 1.f;
    int e;
    frexpf(mx, &e);
    return ldexpf(1.f, e - 8);
}

__device__ __forceinline__ uint8_t to_e4m3(float v) {
    return (uint8_t)__nv_cvt_float_to_fp8(v, __NV_SATFINITE, __NV_E4M3);
}

// Rows of X [n x d] to e4m3 [n x Kp] (zero-padded K) with their power-of-two
// scales [n].  One warp per row.
__global__ void k_rows_f8(const float* __restrict__ X, int64_t n, int d, int Kp, uint8_t* __restrict__ out,
                          float* __restrict__ scale) {
    const int lane = threadIdx.x & 31;
    const int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= n) return;
    float mx = 0.f;
    for (int t = lane; t < d; t += 32) mx = fmaxf(mx, fabsf(X[r * d + t]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const float s = f8_row_scale(mx);
    const float inv = 1.f / s;  // a power of two: exact
    for (int t = lane; t < Kp; t += 32) out[r * Kp + t] = t < d ? to_e4m3(X[r * d + t] * inv) : (uint8_t)0;
    if (lane == 0) scale[r] = s;
}

// Queries to e4m3 rows [nq x Kp] with their scales and, in the same pass, the
// per-query bound of the FP8 scores (rel from fp8_rel below).
__global__ void k_q8_err(const float* __restrict__ Q, int64_t nq, int d, int Kp, float cmax, int spherical,
                         float rel, uint8_t* __restrict__ out, float* __restrict__ qs, float* __restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int64_t q = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (q >= nq) return;
    float s = 0.f, mx = 0.f;
    for (int t = lane; t < d; t += 32) {
        const float v = Q[q * d + t];
        s = fmaf(v, v, s);
        mx = fmaxf(mx, fabsf(v));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    const float sq = f8_row_scale(mx);
    const float inv = 1.f / sq;
    for (int t = lane; t < Kp; t += 32) out[q * Kp + t] = t < d ? to_e4m3(Q[q * d + t] * inv) : (uint8_t)0;
    if (lane != 0) return;
    qs[q] = sq;
    const float qn = sqrtf(s);
    const float e = rel * qn * cmax * 1.0001f;
    const float r = (float)(d + 8) * 1.2e-7f * (qn + cmax) * (qn + cmax);
    err[q] = (spherical ? e : 2.f * e) + r;
}

// Approximate scores [nq x L] with the tensor cores plus the per-query error
// bound err [nq]; the caller re-scores exactly what the bound cannot exclude.
static int err_params(ksc_index* ix, bool tensor_cores, float* rel, float* qmax, cudaStream_t st);

int rank_scores_tc(ksc_index* ix, const float* Q, int64_t nq, float* scores, float* err, cudaStream_t st) {
    const int Kp = (ix->d + TC_KB - 1) / TC_KB * TC_KB;
    const int KB = Kp / TC_KB;
    float rel, qmax;
    if (!ix->c_rank_bf16) {
        // operand type: FP16 (11-bit significand) when the centroids fit it, which
        // the largest norm mostly shows (else from the coordinates, on the host)
        KSC_TRY(err_params(ix, true, &rel, &qmax, st));
        ix->tc_fp16 = ix->c_rank_max_norm < 16384.f;
        if (!ix->tc_fp16) {
            std::vector<float> ch((size_t)ix->L * ix->d);
            KSC_CUDA(cudaMemcpy(ch.data(), ix->c_rank, sizeof(float) * ch.size(), cudaMemcpyDeviceToHost));
            float mx = 0.f;
            for (float v : ch) mx = fmaxf(mx, fabsf(v));
            ix->tc_fp16 = mx < 16384.f;
        }
        KSC_CUDA(cudaMalloc(&ix->c_rank_bf16, sizeof(uint16_t) * (size_t)ix->L * Kp));
        k_to_16<<<(unsigned)std::min<int64_t>(((int64_t)ix->L * Kp + 255) / 256, 4096), 256, 0, st>>>(
            ix->c_rank, ix->L, ix->d, Kp, ix->tc_fp16, (uint16_t*)ix->c_rank_bf16);
        KSC_LAUNCH_CHECK();
        KSC_TRY(make_map(reinterpret_cast<CUtensorMap*>(ix->map_c), ix->c_rank_bf16, ix->L, Kp, TC_N, ix->tc_fp16));
    }
    KSC_TRY(ensure(ix->ws_qbf16, sizeof(uint16_t) * (size_t)nq * Kp, st));
    uint16_t* qb = (uint16_t*)ix->ws_qbf16.p;
    KSC_TRY(err_params(ix, true, &rel, &qmax, st));
    k_q16_err<<<(unsigned)((nq + 7) / 8), 256, 0, st>>>(Q, nq, ix->d, Kp, ix->tc_fp16, ix->c_rank_max_norm,
                                                         ix->spherical, rel, qmax, qb, err);
    KSC_LAUNCH_CHECK();
    CUtensorMap mapA;
    KSC_TRY(make_map(&mapA, qb, nq, Kp, TC_M, ix->tc_fp16));
    const size_t smem = (size_t)std::min(KB, RG_STAGES) * (TC_M + TC_N) * 128 + 1024;
    KSC_CUDA(cudaFuncSetAttribute(k_rank_gemm_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    dim3 grid((ix->L + TC_N - 1) / TC_N, (unsigned)((nq + TC_M - 1) / TC_M));
    k_rank_gemm_tc<false><<<grid, 128, smem, st>>>(mapA, *reinterpret_cast<const CUtensorMap*>(ix->map_c), KB, nq,
                                                   ix->L, ix->c_rank_sq, ix->spherical, ix->tc_fp16 ? 0 : 1, nullptr,
                                                   nullptr, scores, ix->status);
    KSC_LAUNCH_CHECK();
    ix->launches += 2;
    return KSC_OK;
}

// Relative bound of the FP8 scores' dot products, per ||q|| max||c||.
//  Rounding of a scaled element y to e4m3: |fl(y) - y| <= 2^-4 |y| + 2^-10
//  (relative 2^-4 in the normal range, half the subnormal spacing 2^-9
//  below it).  With the row scale s <= max|x_t| / 128 <= ||x|| / 128 and
//  sum |x_t| <= sqrt(d) ||x||, the error of <q~, c~> is at most
//  (2 u + u^2) ||q|| ||c|| + 2 (1 + u) 2^-10 sqrt(d) / 128 ||q|| ||c|| plus
//  a d 2^-34 term (u = 2^-4).  Products of two e4m3 values are exact in
//  FP32; the accumulation inside the MMA is taken as no worse than 13 bits
//  of precision per addition (d 2^-13 (1 + u)^2 of sum |q~_t c~_t|; a
//  reading: the accumulator's internal precision is not documented here);
//  the rescaling by s_q s_c is exact.
static float fp8_rel(int d) {
    const float u = 0.0625f;
    return (2.f * u + u * u) + 2.f * (1.f + u) * 9.765625e-4f * sqrtf((float)d) / 128.f +
           (float)d * 1.2207e-4f * (1.f + u) * (1.f + u) + 1e-6f;
}

// The same scores from e4m3 operands with per-row power-of-two scales.
int rank_scores_tc8(ksc_index* ix, const float* Q, int64_t nq, float* scores, float* err, cudaStream_t st) {
    const int Kp = (ix->d + 127) / 128 * 128;
    const int KB = Kp / 128;
    if (!ix->c_rank_f8) {
        KSC_CUDA(cudaMalloc(&ix->c_rank_f8, (size_t)ix->L * Kp));
        KSC_CUDA(cudaMalloc(&ix->c_rank_f8_scale, sizeof(float) * ix->L));
        k_rows_f8<<<(unsigned)((ix->L + 7) / 8), 256, 0, st>>>(ix->c_rank, ix->L, ix->d, Kp,
                                                               (uint8_t*)ix->c_rank_f8, ix->c_rank_f8_scale);
        KSC_LAUNCH_CHECK();
        KSC_TRY(make_map(reinterpret_cast<CUtensorMap*>(ix->map_c8), ix->c_rank_f8, ix->L, Kp, TC_N, false, 1));
    }
    float rel, qmax;
    KSC_TRY(err_params(ix, true, &rel, &qmax, st));  // max ||c||
    // e4m3 rows (a multiple of 128 bytes each), then the row scales
    const size_t rows_bytes = (size_t)nq * Kp;
    KSC_TRY(ensure(ix->ws_qbf16, rows_bytes + sizeof(float) * (size_t)nq, st));
    uint8_t* q8 = (uint8_t*)ix->ws_qbf16.p;
    float* qsc = reinterpret_cast<float*>(q8 + rows_bytes);
    k_q8_err<<<(unsigned)((nq + 7) / 8), 256, 0, st>>>(Q, nq, ix->d, Kp, ix->c_rank_max_norm, ix->spherical,
                                                        fp8_rel(ix->d), q8, qsc, err);
    KSC_LAUNCH_CHECK();
    CUtensorMap mapA;
    KSC_TRY(make_map(&mapA, q8, nq, Kp, TC_M, false, 1));
    const size_t smem = (size_t)std::min(KB, RG_STAGES) * (TC_M + TC_N) * 128 + 1024;
    KSC_CUDA(cudaFuncSetAttribute(k_rank_gemm_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    dim3 grid((ix->L + TC_N - 1) / TC_N, (unsigned)((nq + TC_M - 1) / TC_M));
    k_rank_gemm_tc<true><<<grid, 128, smem, st>>>(mapA, *reinterpret_cast<const CUtensorMap*>(ix->map_c8), KB, nq,
                                                  ix->L, ix->c_rank_sq, ix->spherical, 0, qsc, ix->c_rank_f8_scale,
                                                  scores, ix->status);
    KSC_LAUNCH_CHECK();
    ix->launches += 2;
    return KSC_OK;
}

// Constants of the score bound: max ||c|| (once per index), the relative
// rounding of the operand type and the largest representable query element.
static int err_params(ksc_index* ix, bool tensor_cores, float* rel, float* qmax, cudaStream_t st) {
    if (ix->c_rank_max_norm <= 0.f) {
        std::vector<float> cn(ix->L);
        KSC_CUDA(cudaMemcpyAsync(cn.data(), ix->c_rank_sq, sizeof(float) * ix->L, cudaMemcpyDeviceToHost, st));
        KSC_CUDA(cudaStreamSynchronize(st));
        float m = 0.f;
        for (float v : cn) m = v > m ? v : m;
        ix->c_rank_max_norm = m > 0.f ? sqrtf(m) : 1e-30f;
    }
    const float u2 = ix->tc_fp16 ? 9.77e-4f + 1e-6f : 0.0078125f + 6.2e-5f;  // 2u + u^2
    *rel = tensor_cores ? u2 + (float)ix->d * 4.8e-7f : (float)(ix->d + 8) * 1.2e-7f;
    *qmax = (tensor_cores && ix->tc_fp16) ? 6.0e4f : INFINITY;
    return KSC_OK;
}

// Lists that the 16-bit scores' bound cannot tell from the 8 best, counted over
// sampled centroids taken as queries: a CTA per sample.  rel: the relative
// bound of the dot products; *total: their number over all samples.
constexpr int RW_SAMPLES = 32, RW_BEST = 8, RW_T = 256;
__global__ void __launch_bounds__(RW_T) k_rank_width(const float* __restrict__ C, const float* __restrict__ csq, int L,
                                                     int d, int spherical, float rel, float cmax,
                                                     int32_t* __restrict__ total) {
    __shared__ __align__(16) float qs[KSC_MAX_DIM];
    __shared__ float sc[RANK_TC_LISTS];
    __shared__ float s_t;
    const int s = (int)((int64_t)blockIdx.x * L / RW_SAMPLES);
    const int lane = threadIdx.x & 31;
    for (int t = threadIdx.x; t < d; t += RW_T) qs[t] = C[(int64_t)s * d + t];
    if (threadIdx.x == 0) s_t = INFINITY;
    __syncthreads();
    for (int c = threadIdx.x >> 5; c < L; c += RW_T / 32) {
        const float v = exact_list_score(qs, C + (int64_t)c * d, d, spherical, lane);
        if (lane == 0) sc[c] = v;
    }
    __syncthreads();
    for (int c = threadIdx.x; c < L; c += RW_T) {
        int r = 0;
        for (int j = 0; j < L; ++j) r += sc[j] < sc[c] || (sc[j] == sc[c] && j < c);
        if (r == min(RW_BEST, L) - 1) s_t = sc[c];
    }
    __syncthreads();
    const float dot = rel * sqrtf(csq[s]) * cmax, lim = s_t + 2.f * (spherical ? dot : 2.f * dot);
    int n = 0;
    for (int c = threadIdx.x; c < L; c += RW_T) n += sc[c] <= lim;
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) atomicAdd(total, n);
}

// Whether the 16-bit scores of rows wider than the tensor cores' own range
// (search.cu: TC_SCORES_D) tell most lists apart, from the centroids alone
// (once per index; the bound grows with the norms, so centroids far from the
// origin and close together defeat it).  Every list inside the bound is
// re-scored exactly: 512 x 784, 10,000 queries: 583 us with FP32 scores, 353
// with 16-bit ones where they leave 12 lists, 1197 where 96, 3170 where all.
// At most RANK_TC_LISTS lists, so that the re-score buffer always holds them.
int rank_tc_narrow(ksc_index* ix, bool* narrow, cudaStream_t st) {
    if (ix->rank_tc_state == 0 && ix->L > RANK_TC_LISTS) ix->rank_tc_state = -1;
    if (ix->rank_tc_state == 0) {
        float rel, qmax;
        KSC_TRY(err_params(ix, true, &rel, &qmax, st));  // max ||c||
        const float u2 = ix->c_rank_max_norm < 16384.f ? 9.77e-4f + 1e-6f : 0.0078125f + 6.2e-5f;
        rel = u2 + (float)ix->d * 4.8e-7f;
        KSC_TRY(ensure(ix->ws_flag, sizeof(int32_t), st));
        int32_t* total = (int32_t*)ix->ws_flag.p;
        int32_t h = 0;
        KSC_CUDA(cudaMemsetAsync(total, 0, sizeof(int32_t), st));
        k_rank_width<<<RW_SAMPLES, RW_T, 0, st>>>(ix->c_rank, ix->c_rank_sq, ix->L, ix->d, ix->spherical, rel,
                                                  ix->c_rank_max_norm, total);
        KSC_LAUNCH_CHECK();
        KSC_CUDA(cudaMemcpyAsync(&h, total, sizeof(h), cudaMemcpyDeviceToHost, st));
        KSC_CUDA(cudaStreamSynchronize(st));
        ix->rank_tc_state = h <= 4 * RW_BEST * RW_SAMPLES ? 1 : -1;
    }
    *narrow = ix->rank_tc_state > 0;
    return KSC_OK;
}

int score_err(ksc_index* ix, const float* Q, int64_t nq, bool tensor_cores, float* err, cudaStream_t st) {
    float rel, qmax;
    KSC_TRY(err_params(ix, tensor_cores, &rel, &qmax, st));
    k_score_err<<<(unsigned)((nq + 255) / 256), 256, 0, st>>>(Q, nq, ix->d, ix->c_rank_max_norm, ix->spherical,
                                                              rel, qmax, err);
    KSC_LAUNCH_CHECK();
    ix->launches++;
    return KSC_OK;
}

}  // namespace ksc
