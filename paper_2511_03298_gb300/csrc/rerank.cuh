// The exact re-rank (a6) by a warp or a CTA: FP32 distances of candidate rows
// and the k best of them, shared by the re-rank kernels (search.cu) and the
// small-batch kernel (small.cu).
#pragma once

#include "common.cuh"

namespace ksc {

// Halving exchange of 8 rows' partial sums over the warp (9 shuffles):
// afterwards every lane of quad `myrow` (lane bits 4, 3, 2) holds that row's
// total, summed in the same tree for every row.
__device__ __forceinline__ float exchange_rows8(float (&a)[8], int lane) {
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
    return a[0];
}

// FP32 partial sums of the 8 rows idv[] (-1: none) for this lane's 4
// coordinates, summed across the warp: every lane of quad `myrow` ends with
// that row's distance term (L2: the squared distance, IP: the dot product).
__device__ __forceinline__ float rerank_rows8(const float4& qv, const float* __restrict__ X, int d, int ip, bool inl,
                                              const int32_t (&idv)[8], int lane) {
    float4 xv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
        xv[u] = (idv[u] >= 0 && inl) ? __ldg(reinterpret_cast<const float4*>(X + (int64_t)idv[u] * d) + lane)
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
    float a[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        if (ip) {
            a[u] = qv.x * xv[u].x + qv.y * xv[u].y + qv.z * xv[u].z + qv.w * xv[u].w;
        } else {
            const float e0 = qv.x - xv[u].x, e1 = qv.y - xv[u].y, e2 = qv.z - xv[u].z, e3 = qv.w - xv[u].w;
            a[u] = fmaf(e0, e0, fmaf(e1, e1, fmaf(e2, e2, e3 * e3)));
        }
    }
    return exchange_rows8(a, lane);
}


// Keys up to which an order is found by counting ranks.  (1000 queries of 500k x
// 64, k 10: at R 257 243 us counted, 207 cut by radix refinement first; at R 512 310
// and 233; k = R = 400 286 counted, 246 sorted.)
constexpr int RR_RANK_R = 256;

// Keys of cta_rerank's kbuf: the k best, to a power of two where they are sorted.
__host__ __device__ inline int rerank_kbuf(int k) { return k > RR_RANK_R ? pow2_ceil(k) : k; }
// Shared bytes of cta_rerank's keys: R of them and, past RR_RANK_R, its kbuf.
inline size_t rerank_smem(int R, int k) {
    return sizeof(uint64_t) * ((size_t)R + (R > RR_RANK_R ? rerank_kbuf(k) : 0));
}

// Exact distance of each of the R candidates keys[] (KEY_NONE: none) of one
// query (qs, shared memory), by one CTA: L2 = sum (q_t - x_t)^2, IP = -<q, x>,
// a warp per row, 16-byte loads when d is a multiple of 4; then the k best by
// (distance, id) to out_ids / out_d (L2 distance ascending / IP similarity
// descending).  keys[] is overwritten; kbuf: rerank_kbuf(k) keys when R > RR_RANK_R.
// Bound by the rows' latency: a warp keeps 8 rows (d <= 128) or 4 in flight;
// up to 256 candidates are ordered by counting, for each, the smaller ones
// (one pass of broadcast reads, no barriers), more are cut to the k best by
// radix refinement first, and these sorted if they are more than 256 still.
template <int NT>
__device__ __forceinline__ void cta_rerank(uint64_t* keys, int R, uint64_t* kbuf, const float* qs,
                                           const float* __restrict__ X, int d, int ip, int k,
                                           int64_t* __restrict__ out_ids, float* __restrict__ out_d) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const bool vec4 = (d & 3) == 0;
    auto id_of = [&](int c) -> int32_t {
        const uint64_t kk = c < R ? keys[c] : KEY_NONE;
        return kk != KEY_NONE ? (int32_t)(kk & 0xffffffffu) : -1;
    };
    if (vec4 && d <= 128) {
        const bool inl = lane * 4 < d;
        const float4 qv = inl ? *reinterpret_cast<const float4*>(qs + lane * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
        const int myrow = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
        for (int c0 = w * 8; c0 < R; c0 += NW * 8) {
            int32_t idv[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) idv[u] = id_of(c0 + u);
            const float s = rerank_rows8(qv, X, d, ip, inl, idv, lane);
            const int c = c0 + myrow;
            const uint64_t kk = c < R ? keys[c] : KEY_NONE;
            __syncwarp();  // the step's keys are read before they are replaced
            if ((lane & 3) == 0 && kk != KEY_NONE)
                keys[c] = ((uint64_t)ordered_f32(ip ? -s : s) << 32) | (kk & 0xffffffffull);
        }
    } else {
        for (int c0 = w * 4; c0 < R; c0 += NW * 4) {
            int32_t idv[4];
            float s[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                idv[u] = id_of(c0 + u);
                s[u] = 0.f;
            }
            if (vec4) {
                for (int t = lane * 4; t < d; t += 128) {
                    const float4 qv = *reinterpret_cast<const float4*>(qs + t);
                    float4 xv[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        xv[u] = idv[u] >= 0 ? __ldg(reinterpret_cast<const float4*>(X + (int64_t)idv[u] * d + t))
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (ip) {
                            s[u] = fmaf(qv.x, xv[u].x, s[u]); s[u] = fmaf(qv.y, xv[u].y, s[u]);
                            s[u] = fmaf(qv.z, xv[u].z, s[u]); s[u] = fmaf(qv.w, xv[u].w, s[u]);
                        } else {
                            const float e0 = qv.x - xv[u].x, e1 = qv.y - xv[u].y, e2 = qv.z - xv[u].z,
                                        e3 = qv.w - xv[u].w;
                            s[u] = fmaf(e0, e0, s[u]); s[u] = fmaf(e1, e1, s[u]);
                            s[u] = fmaf(e2, e2, s[u]); s[u] = fmaf(e3, e3, s[u]);
                        }
                    }
                }
            } else {
                for (int t = lane; t < d; t += 32) {
                    const float qv = qs[t];
                    float xv[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) xv[u] = idv[u] >= 0 ? __ldg(X + (int64_t)idv[u] * d + t) : 0.f;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (ip) s[u] = fmaf(qv, xv[u], s[u]);
                        else { const float e = qv - xv[u]; s[u] = fmaf(e, e, s[u]); }
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
            __syncwarp();  // (every lane read the keys before they are replaced)
            if (lane < 4 && c0 + lane < R) {
                const float v = lane == 0 ? s[0] : (lane == 1 ? s[1] : (lane == 2 ? s[2] : s[3]));
                const uint64_t kk = keys[c0 + lane];
                if (kk != KEY_NONE) keys[c0 + lane] = ((uint64_t)ordered_f32(ip ? -v : v) << 32) | (kk & 0xffffffffull);
            }
        }
    }
    __syncthreads();
    // an empty slot i becomes KEY_NONE - i, which tells it from a candidate below
    // (a list given twice by the caller's probes repeats its keys: places of
    // equal keys go by position)
    for (int i = threadIdx.x; i < R; i += NT)
        if (keys[i] == KEY_NONE) keys[i] = KEY_NONE - (uint64_t)i;
    __syncthreads();
    auto put = [&](int r, uint64_t kk) {
        if (kk >= KEY_NONE - (uint64_t)R) {
            out_ids[r] = -1;
            out_d[r] = ip ? -INFINITY : INFINITY;
        } else {
            out_ids[r] = (int64_t)(kk & 0xffffffffu);
            const float dist = unordered_f32((uint32_t)(kk >> 32));
            out_d[r] = ip ? -dist : dist;
        }
    };
    if (R <= RR_RANK_R) {
        // a group of `parts` lanes per key (a power of two, all NT threads in
        // use), each counting every parts-th of the others
        int parts = 1;
        while (2 * parts * R <= NT && parts < 32) parts *= 2;
        for (int i0 = 0; i0 < R; i0 += NT / parts) {
            const int i = i0 + threadIdx.x / parts, o = threadIdx.x % parts;
            const uint64_t v = i < R ? keys[i] : 0ull;
            int rank = 0;
#pragma unroll 8
            for (int j = o; j < R; j += parts) {
                const uint64_t y = keys[j];
                rank += y < v || (y == v && j < i);
            }
            for (int s = parts >> 1; s > 0; s >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, s);
            if (i < R && o == 0 && rank < k) put(rank, v);
        }
    } else {
        __shared__ __align__(16) uint32_t hist[256];
        __shared__ uint64_t bb[32];
        const int kr = k < R ? k : R;  // (all of them: no refinement)
        if (k < R) {
            auto emit = [&](int i, uint64_t v) { kbuf[i] = v; };
            auto load = [&](int i) -> uint64_t { return keys[i]; };
            block_topk(load, R, k, emit, hist, bb);
        } else {
            for (int i = threadIdx.x; i < R; i += NT) kbuf[i] = keys[i];
        }
        __syncthreads();
        if (kr > RR_RANK_R) {
            // counting costs kr^2 reads: more keys are sorted (10,000 queries, k = R
            // 1000: the search 5547 us counted, 3010 sorted; 1000 queries 754 and 499)
            const int S = pow2_ceil(kr);
            for (int i = kr + threadIdx.x; i < S; i += NT) kbuf[i] = KEY_NONE;
            __syncthreads();
            block_bitonic_sort(kbuf, S);
            for (int i = threadIdx.x; i < kr; i += NT) put(i, kbuf[i]);
        } else for (int i = threadIdx.x; i < kr; i += NT) {
            const uint64_t v = kbuf[i];
            int rank = 0;
#pragma unroll 8
            for (int j = 0; j < kr; ++j) {
                const uint64_t y = kbuf[j];
                rank += y < v || (y == v && j < i);
            }
            put(rank, v);
        }
    }
    for (int r = R + threadIdx.x; r < k; r += NT) put(r, KEY_NONE);
}

}  // namespace ksc
