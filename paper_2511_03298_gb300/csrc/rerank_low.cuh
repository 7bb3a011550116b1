// Re-ranks that read low-precision rows first (rerank_low.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "common.cuh"

namespace ksc {

__device__ __forceinline__ float lowp_elem(int prec, const uint16_t* xb, const uint8_t* x8, int64_t off) {
    if (prec == 1) return __bfloat162float(__ushort_as_bfloat16(xb[off]));
    __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)x8[off], __NV_E4M3);
    return __half2float(__half(h));
}

// Distance of query row qs (shared) to row id in the given precision (0 FP32,
// 1 BF16, 2 FP8 with row scale); one warp, result in every lane.
__device__ __forceinline__ float lowp_dist(int prec, const float* __restrict__ qs, const float* __restrict__ X,
                                           const uint16_t* __restrict__ xb, const uint8_t* __restrict__ x8,
                                           const float* __restrict__ sc, int32_t id, int d, int ip, int lane) {
    float acc = 0.f;
    const float s = prec == 2 ? sc[id] : 1.f;
    for (int t = lane; t < d; t += 32) {
        const float xv = prec == 0 ? __ldg(X + (int64_t)id * d + t) : lowp_elem(prec, xb, x8, (int64_t)id * d + t) * s;
        if (ip) acc = fmaf(qs[t], xv, acc);
        else { const float e = qs[t] - xv; acc = fmaf(e, e, acc); }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return ip ? -acc : acc;
}

// The widened first re-rank (precision 1: BF16 rows, 2: FP8 rows): each query's
// R candidates (topr) by low-precision distance, the best Rf of them as keys in
// out [nq x Rf] (in no particular order, padded with KEY_NONE).
int launch_rerank_lowp(const float* Q, int64_t nq, int d, int ip, int prec, const uint16_t* xb, const uint8_t* x8,
                       const float* sc, const uint64_t* topr, int Rmax, const int32_t* rerank_q, int Rfix, int Rmin,
                       int Rf, uint64_t* out, cudaStream_t st);

// The exact L2 re-rank by a CTA per query with exact U8 rows first, for row
// widths the vector loads serve.
bool rerank_u8_supported(int d);
int launch_rerank_u8(const float* Q, int64_t nq, const float* X, const uint8_t* xu, int d, const uint64_t* topr,
                     int Rmax, const int32_t* rerank_q, int Rfix, int k, int64_t* ids, float* dists, cudaStream_t st);

}  // namespace ksc
