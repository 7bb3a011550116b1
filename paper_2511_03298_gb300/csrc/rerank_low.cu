// Re-ranks that read low-precision copies of the candidate rows first: the
// widened shortlist by BF16 / FP8 rows (an approximation the caller asks for)
// and the exact L2 re-rank with exact U8 rows and a proven bound.
//
// Both read a row with 8 lanes, 16 bytes (U8) or 8 / 4 bytes (BF16 / FP8) per
// lane and step, 4 rows per lane group and 16 per warp in flight, and reduce 16
// rows with 7 shuffles.
#include <algorithm>

#include "rerank.cuh"
#include "rerank_low.cuh"
#include "scan.cuh"

namespace ksc {

constexpr int RL_T = 256;  // threads per CTA

// Sums of 4 rows per 8-lane group (a[i]: this lane's part of row 4 g + i) over
// the group: afterwards row (lane >> 1) & 15 of the warp's 16 is in both lanes
// of a pair.
__device__ __forceinline__ float reduce_rows16(float (&a)[4], int lane) {
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

// ------------------------------------------------------------------ widened shortlist
// A CTA per query.  PREC 1: BF16 rows, 2: FP8 e4m3 rows with a scale per row;
// FP32 accumulation.  V: elements per load (4, or 1 for widths that are no
// multiple of 4).  The best Rf by (distance, id): radix refinement, no sort
// (the FP32 pass orders).  Bound by the rows' bytes from L2; with one row per
// warp in flight, 2-byte loads and a 512-key bitonic sort 3001 queries of 400
// rows x 100 took 353 us, 73 us now.
template <int PREC, int V>
__global__ void __launch_bounds__(RL_T) k_rerank_lowp(const float* __restrict__ Q, int d, int ip,
                                                      const uint16_t* __restrict__ xb, const uint8_t* __restrict__ x8,
                                                      const float* __restrict__ sc, const uint64_t* __restrict__ topr,
                                                      int Rmax, const int32_t* __restrict__ rerank_q, int Rfix,
                                                      int Rmin, int Rf, uint64_t* __restrict__ out) {
    extern __shared__ uint64_t keys[];  // Rmax
    __shared__ __align__(16) float qs[KSC_MAX_DIM];
    __shared__ __align__(16) uint32_t hist[256];
    __shared__ uint64_t bb[32];
    const int64_t q = blockIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, j = lane & 7;
    const int R = rerank_of(rerank_q, Rfix, Rmin, Rmax, q);
    for (int t = threadIdx.x; t < d; t += RL_T) qs[t] = Q[q * d + t];
    for (int c = threadIdx.x; c < R; c += RL_T) keys[c] = topr[q * Rmax + c];
    __syncthreads();
    const int myrow = (lane >> 1) & 15;
    for (int c0 = 16 * w; c0 < R; c0 += 16 * (RL_T / 32)) {
        int32_t id[4];
        float s[4], a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c = c0 + 4 * (lane >> 3) + i;
            const uint64_t kk = c < R ? keys[c] : KEY_NONE;
            id[i] = kk != KEY_NONE ? (int32_t)(kk & 0xffffffffu) : -1;
            s[i] = PREC == 2 && id[i] >= 0 ? __ldg(sc + id[i]) : 1.f;
            a[i] = 0.f;
        }
        for (int t = V * j; t < d; t += 8 * V) {
            float x[4][V];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if constexpr (PREC == 1 && V == 4) {
                    const uint2 r = id[i] >= 0 ? __ldg(reinterpret_cast<const uint2*>(xb + (int64_t)id[i] * d + t))
                                               : make_uint2(0u, 0u);
                    x[i][0] = __uint_as_float(r.x << 16);
                    x[i][1] = __uint_as_float(r.x & 0xffff0000u);
                    x[i][2] = __uint_as_float(r.y << 16);
                    x[i][3] = __uint_as_float(r.y & 0xffff0000u);
                } else if constexpr (PREC == 2 && V == 4) {
                    const uint32_t r =
                        id[i] >= 0 ? __ldg(reinterpret_cast<const uint32_t*>(x8 + (int64_t)id[i] * d + t)) : 0u;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const __half_raw h =
                            __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)((r >> (8 * u)) & 255u), __NV_E4M3);
                        x[i][u] = __half2float(__half(h)) * s[i];
                    }
                } else {
                    x[i][0] = id[i] >= 0 ? lowp_elem(PREC, xb, x8, (int64_t)id[i] * d + t) * s[i] : 0.f;
                }
            }
#pragma unroll
            for (int u = 0; u < V; ++u) {
                const float qv = qs[t + u];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (ip) a[i] = fmaf(qv, x[i][u], a[i]);
                    else { const float e = qv - x[i][u]; a[i] = fmaf(e, e, a[i]); }
                }
            }
        }
        const float v = reduce_rows16(a, lane);
        const int c = c0 + myrow;
        const uint64_t kk = c < R ? keys[c] : KEY_NONE;
        __syncwarp();  // the step's keys are read before they are replaced
        if ((lane & 1) == 0 && kk != KEY_NONE)
            keys[c] = ((uint64_t)ordered_f32(ip ? -v : v) << 32) | (kk & 0xffffffffull);
    }
    __syncthreads();
    uint64_t* o = out + q * Rf;
    if (R <= Rf) {
        for (int i = threadIdx.x; i < Rf; i += RL_T) o[i] = i < R ? keys[i] : KEY_NONE;
        return;
    }
    // (an empty slot i counts as KEY_NONE - i: unique keys)
    auto load = [&](int i) -> uint64_t {
        const uint64_t v = keys[i];
        return v == KEY_NONE ? KEY_NONE - (uint64_t)i : v;
    };
    auto emit = [&](int i, uint64_t v) { o[i] = v >= KEY_NONE - (uint64_t)R ? KEY_NONE : v; };
    block_topk(load, R, Rf, emit, hist, bb);
}

int launch_rerank_lowp(const float* Q, int64_t nq, int d, int ip, int prec, const uint16_t* xb, const uint8_t* x8,
                       const float* sc, const uint64_t* topr, int Rmax, const int32_t* rerank_q, int Rfix, int Rmin,
                       int Rf, uint64_t* out, cudaStream_t st) {
    const bool vec = (d & 3) == 0;
    auto kern = prec == 1 ? (vec ? k_rerank_lowp<1, 4> : k_rerank_lowp<1, 1>)
                          : (vec ? k_rerank_lowp<2, 4> : k_rerank_lowp<2, 1>);
    const size_t smem = sizeof(uint64_t) * (size_t)Rmax;
    KSC_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<(unsigned)nq, RL_T, smem, st>>>(Q, d, ip, xb, x8, sc, topr, Rmax, rerank_q, Rfix, Rmin, Rf, out);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

// ------------------------------------------------------------------ exact L2 re-rank, U8 rows first
// A CTA per query.  The U8 copies hold the rows exactly, so a first pass over
// them (a quarter of the bytes) gives every candidate's distance up to FP32
// evaluation: with s~ its value, the FP32 pass's value lies within
//   e = 2^-17 (2 s~ (1 + 2^-16)) (1 + 2^-10)
// of it, 2^-17 above the relative error of either sum (at most 70 roundings of
// 2^-24 on a term's path up to 1024 dimensions: a difference counts twice, 64
// additions of a lane, 4 across the lanes).  U = the k-th smallest s~ + e; a
// candidate with s~ - e > U has an FP32 distance above k others' and is out;
// the rest take the FP32 re-rank itself, so the result is its result bit for
// bit.  Bound by L2 reads and by the bytes' conversion: 10,000 queries of 200
// rows x 784: 848 us with every row in FP32, 477 us now.
bool rerank_u8_supported(int d) { return d % 16 == 0 && d <= KSC_MAX_DIM; }

__global__ void __launch_bounds__(RL_T) k_rerank_u8(const float* __restrict__ Q, const float* __restrict__ X,
                                                    const uint8_t* __restrict__ xu, int d,
                                                    const uint64_t* __restrict__ topr, int Rmax,
                                                    const int32_t* __restrict__ rerank_q, int Rfix, int k,
                                                    int64_t* __restrict__ out_ids, float* __restrict__ out_d) {
    // Rmax keys (later the re-rank's kbuf: rerank_kbuf(k)), Rmax survivors' keys (first: bounds)
    extern __shared__ uint64_t keys[];
    __shared__ __align__(16) float qs[KSC_MAX_DIM];
    __shared__ __align__(16) uint32_t hist[256];
    __shared__ uint64_t bb[32];
    __shared__ int s_n;
    uint64_t* live = keys + max(Rmax, rerank_kbuf(k));
    float* dist = reinterpret_cast<float*>(live);  // [Rmax] the U8 pass's distances, read before live is written
    const int64_t q = blockIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, j = lane & 7;
    const int R = rerank_of(rerank_q, Rfix, k, Rmax, q);
    for (int t = threadIdx.x; t < d; t += RL_T) qs[t] = Q[q * d + t];
    for (int c = threadIdx.x; c < R; c += RL_T) keys[c] = topr[q * Rmax + c];
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int myrow = (lane >> 1) & 15;
    const float2 m23 = make_float2(8388608.f, 8388608.f);
    for (int c0 = 16 * w; c0 < R; c0 += 16 * (RL_T / 32)) {
        const uint8_t* row[4];
        bool in[4];
        float2 a2[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c = c0 + 4 * (lane >> 3) + i;
            const uint64_t kk = c < R ? keys[c] : KEY_NONE;
            in[i] = kk != KEY_NONE;
            row[i] = xu + (in[i] ? (int64_t)(kk & 0xffffffffu) * d : 0);
            a2[i] = make_float2(0.f, 0.f);
        }
        for (int t = 16 * j; t < d; t += 128) {
            uint4 r[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                r[i] = in[i] ? __ldg(reinterpret_cast<const uint4*>(row[i] + t)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const float4 qv = *reinterpret_cast<const float4*>(qs + t + 4 * h);
                const float2 q01 = make_float2(qv.x, qv.y), q23 = make_float2(qv.z, qv.w);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t b = h == 0 ? r[i].x : (h == 1 ? r[i].y : (h == 2 ? r[i].z : r[i].w));
                    // byte b as (2^23 + b) - 2^23, exact
                    const float2 x01 = f2_sub(make_float2(__uint_as_float(prmt(b, 0x4B000000u, 0x7540u)),
                                                          __uint_as_float(prmt(b, 0x4B000000u, 0x7541u))), m23);
                    const float2 x23 = f2_sub(make_float2(__uint_as_float(prmt(b, 0x4B000000u, 0x7542u)),
                                                          __uint_as_float(prmt(b, 0x4B000000u, 0x7543u))), m23);
                    const float2 e01 = f2_sub(q01, x01), e23 = f2_sub(q23, x23);
                    a2[i] = f2_fma(e01, e01, a2[i]);
                    a2[i] = f2_fma(e23, e23, a2[i]);
                }
            }
        }
        float a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = a2[i].x + a2[i].y;
        const float v = reduce_rows16(a, lane);
        if ((lane & 1) == 0 && c0 + myrow < R) dist[c0 + myrow] = v;
    }
    __syncthreads();
    // bounds of a candidate's FP32 distance (NaN: none, it is re-read)
    constexpr float G2 = 0x1p-16f * (1.f + 0x1p-9f);
    auto lower = [&](int c) -> float {
        const float s = dist[c], v = __fsub_rd(s, G2 * s);
        return v <= INFINITY ? v : -INFINITY;
    };
    // the k-th smallest upper bound; an empty slot's is above all (and unique)
    auto load = [&](int c) -> uint64_t {
        const float s = dist[c], v = __fadd_ru(s, G2 * s);
        const uint32_t u = keys[c] == KEY_NONE ? 0xffffffffu : ordered_f32(v <= INFINITY ? v : INFINITY);
        return ((uint64_t)u << 32) | (uint32_t)c;
    };
    auto none = [](int, uint64_t) {};
    const uint32_t ub = (uint32_t)(block_topk(load, R, k, none, hist, bb) >> 32);
    const float U = ub == 0xffffffffu ? INFINITY : unordered_f32(ub);
    uint64_t kk[4];
    bool keep[4];
    // (dist shares memory with live: every bound is read before any key is written)
    for (int c0 = 0; c0 < R; c0 += 4 * RL_T) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = c0 + u * RL_T + threadIdx.x;
            kk[u] = c < R ? keys[c] : KEY_NONE;
            keep[u] = c < R && (kk[u] == KEY_NONE ? ub == 0xffffffffu : lower(c) <= U);
        }
        if (c0 == 0 && R > 4 * RL_T) {
            // more candidates than one sweep holds: mark the dropped ones in keys instead
            for (int c = threadIdx.x; c < R; c += RL_T)
                if (keys[c] != KEY_NONE && !(lower(c) <= U)) keys[c] = KEY_NONE;
            __syncthreads();
            for (int c = threadIdx.x; c < R; c += RL_T) {
                const uint64_t v = keys[c];
                if (v != KEY_NONE) live[atomicAdd(&s_n, 1)] = v;
            }
            break;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (keep[u] && kk[u] != KEY_NONE) live[atomicAdd(&s_n, 1)] = kk[u];
    }
    __syncthreads();
    cta_rerank<RL_T>(live, s_n, keys, qs, X, d, 0, k, out_ids + q * k, out_d + q * k);
}

int launch_rerank_u8(const float* Q, int64_t nq, const float* X, const uint8_t* xu, int d, const uint64_t* topr,
                     int Rmax, const int32_t* rerank_q, int Rfix, int k, int64_t* ids, float* dists, cudaStream_t st) {
    const size_t smem = sizeof(uint64_t) * ((size_t)std::max(Rmax, rerank_kbuf(k)) + Rmax);
    KSC_CUDA(cudaFuncSetAttribute(k_rerank_u8, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_rerank_u8<<<(unsigned)nq, RL_T, smem, st>>>(Q, X, xu, d, topr, Rmax, rerank_q, Rfix, k, ids, dists);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

}  // namespace ksc
