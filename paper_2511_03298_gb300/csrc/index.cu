// Index construction (Alg. 1), import / export and memory management.
//
// build: IVF k-means (Lloyd, Sec. 2.2) on a sample, list assignment by the
// ranking score, mean centroids for residuals (Sec. 4.6.1), PQ codebooks with
// K = 16 per subspace on residuals (Sec. 2.3), encoding, block packing
// (Alg. 1 BuildBlocks).  All on the GPU in FP32 (sums in FP64); the list
// ordering (a counting sort of the assignment) runs on the host.
#include <atomic>
#include <cstdarg>
#include <algorithm>
#include <functional>
#include <cstdio>
#include <cstring>
#include <vector>

#include "index.cuh"

namespace ksc {

// ------------------------------------------------------------------ errors
static thread_local char g_err[512] = "";

void set_error(const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}
const char* get_error() { return g_err; }

static std::atomic<unsigned long long> g_ws_gen{0};
unsigned long long workspace_generation() { return g_ws_gen.load(); }
void bump_workspace_generation() { g_ws_gen++; }

int ensure(Buffer& b, size_t bytes, cudaStream_t st) {
    if (bytes <= b.bytes && b.p) return KSC_OK;
    g_ws_gen++;
    if (b.p) {
        KSC_CUDA(cudaStreamSynchronize(st));
        KSC_CUDA(cudaFree(b.p));
        b.p = nullptr;
        b.bytes = 0;
    }
    size_t want = bytes < 256 ? 256 : bytes;
    want = (want + 255) & ~size_t(255);
    KSC_CUDA(cudaMalloc(&b.p, want));
    b.bytes = want;
    return KSC_OK;
}

void release(Buffer& b) {
    if (b.p) cudaFree(b.p);
    b.p = nullptr;
    b.bytes = 0;
}

int num_sms() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    return sms;
}

// ------------------------------------------------------------------ kernels
__global__ void k_gather_rows(const float* __restrict__ X, const int64_t* __restrict__ idx, int64_t cnt,
                              int d, float* __restrict__ out) {
    int64_t tot = cnt * d;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e / d;
        int t = (int)(e - r * d);
        out[e] = X[idx[r] * d + t];
    }
}

__global__ void k_row_sqnorm(const float* __restrict__ C, int L, int d, float* __restrict__ out) {
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= L) return;
    float s = 0.f;
    for (int t = 0; t < d; ++t) s = fmaf(C[(int64_t)c * d + t], C[(int64_t)c * d + t], s);
    out[c] = s;
}

__global__ void k_normalise_rows(float* __restrict__ C, int L, int d) {
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= L) return;
    double s = 0.0;
    for (int t = 0; t < d; ++t) s += (double)C[(int64_t)c * d + t] * C[(int64_t)c * d + t];
    if (s > 0.0) {
        double inv = 1.0 / sqrt(s);
        for (int t = 0; t < d; ++t) C[(int64_t)c * d + t] = (float)(C[(int64_t)c * d + t] * inv);
    }
}

// Nearest centroid of every row (or of the listed rows): score = ||c||^2 -
// 2<x,c> (L2) or -<x,c> (spherical); ties -> lower centroid id.  The rule of
// every assignment; where the data fit FP16 operands, assign_tc.cu decides
// most rows and this kernel the ones it lists.  64 rows x 64 centroids per tile,
// 256 threads, 4 x 4 outputs per thread, dims staged 32 at a time.
constexpr int AS_T = 64, AS_K = 32;
__global__ void __launch_bounds__(256) k_assign(const float* __restrict__ X, int64_t np, int d,
                                                const float* __restrict__ Cc, const float* __restrict__ cn,
                                                int L, int spherical, int32_t* __restrict__ assign,
                                                const int32_t* __restrict__ rows,
                                                const int32_t* __restrict__ nrows, int above) {
    __shared__ float xs[AS_K][AS_T + 4];
    __shared__ float cs[AS_K][AS_T + 4];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t row0 = (int64_t)blockIdx.x * AS_T;
    // every row, or (rows != NULL) the nrows[0] rows listed if those are more than `above`
    if (nrows) np = *nrows > above ? min(np, (int64_t)*nrows) : 0;
    if (row0 >= np) return;
    float best[4];
    int bid[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { best[i] = INFINITY; bid[i] = 0x7fffffff; }
    for (int c0 = 0; c0 < L; c0 += AS_T) {
        float acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
        for (int k0 = 0; k0 < d; k0 += AS_K) {
            for (int e = threadIdx.x; e < AS_T * AS_K; e += 256) {
                int r = e / AS_K, kk = e % AS_K;
                int64_t gr = row0 + r;
                int gk = k0 + kk;
                xs[kk][r] = (gr < np && gk < d) ? X[(rows ? rows[gr] : gr) * d + gk] : 0.f;
                int gc = c0 + r;
                cs[kk][r] = (gc < L && gk < d) ? Cc[(int64_t)gc * d + gk] : 0.f;
            }
            __syncthreads();
#pragma unroll 8
            for (int kk = 0; kk < AS_K; ++kk) {
                float a[4], b[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) a[i] = xs[kk][ty * 4 + i];
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
        for (int j = 0; j < 4; ++j) {
            int c = c0 + tx * 4 + j;
            if (c >= L) continue;
            float base = spherical ? 0.f : cn[c];
            float mul = spherical ? -1.f : -2.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float s = fmaf(mul, acc[i][j], base);
                if (s < best[i] || (s == best[i] && c < bid[i])) { best[i] = s; bid[i] = c; }
            }
        }
    }
    // reduce over the 16 threads (tx) that share these rows
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float ob = __shfl_xor_sync(0xffffffffu, best[i], off);
            int oi = __shfl_xor_sync(0xffffffffu, bid[i], off);
            if (ob < best[i] || (ob == best[i] && oi < bid[i])) { best[i] = ob; bid[i] = oi; }
        }
    }
    if (tx == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int64_t r = row0 + ty * 4 + i;
            if (r < np) assign[rows ? rows[r] : r] = bid[i];
        }
    }
}

// Accumulate rows into per-centroid FP64 sums (X rows, optional row index map).
__global__ void k_centroid_accum(const float* __restrict__ X, const int64_t* __restrict__ idx, int64_t np,
                                 int d, const int32_t* __restrict__ a, double* __restrict__ sums,
                                 unsigned long long* __restrict__ cnt) {
    int64_t tot = np * d;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e / d;
        int t = (int)(e - r * d);
        int64_t src = idx ? idx[r] : r;
        int c = a[r];
        atomicAdd(&sums[(int64_t)c * d + t], (double)X[src * d + t]);
        if (t == 0) atomicAdd(&cnt[c], 1ull);
    }
}

__global__ void k_centroid_finish(const double* __restrict__ sums, const unsigned long long* __restrict__ cnt,
                                  const float* __restrict__ fallback, int L, int d, float* __restrict__ out) {
    int64_t tot = (int64_t)L * d;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        int c = (int)(e / d);
        out[e] = cnt[c] > 0 ? (float)(sums[e] / (double)cnt[c]) : fallback[e];
    }
}

// residual rows r = x - c_mean[a(x)] (one fp32 subtraction)
__global__ void k_residual(const float* __restrict__ X, const int64_t* __restrict__ idx, int64_t cnt, int d,
                           const int32_t* __restrict__ assign, const float* __restrict__ c_mean,
                           float* __restrict__ out) {
    int64_t tot = cnt * d;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e / d;
        int t = (int)(e - r * d);
        int64_t src = idx ? idx[r] : r;
        out[e] = __fsub_rn(X[src * d + t], c_mean[(int64_t)assign[src] * d + t]);
    }
}

// ------------------------------------------------------------------ PQ, sub-vectors of a fixed width
// A thread keeps one subspace (j = thread % M) and its 16 codewords in
// registers and walks rows: a warp reads consecutive sub-vectors of a row, and
// an item costs 16 DS differences and FMAs and 16 compares.  (The kernels for
// any width below read the codebook and the row through L1 for every codeword:
// 517 us per 65,536 x 64 items of width 2 against 52 us here with the sums.)  Same
// operations and order for every (row, codeword), ties to the lower codeword.
// RG = 256 / M row groups share a CTA.
template <int DS>
struct PqRow {
    float v[DS];
};
template <int DS>
__device__ __forceinline__ PqRow<DS> pq_load(const float* __restrict__ p) {
    PqRow<DS> r;
    if constexpr (DS == 2) {
        const float2 x = __ldg(reinterpret_cast<const float2*>(p));
        r.v[0] = x.x;
        r.v[1] = x.y;
    } else if constexpr (DS % 4 == 0) {
#pragma unroll
        for (int t = 0; t < DS; t += 4) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(p + t));
            r.v[t] = x.x;
            r.v[t + 1] = x.y;
            r.v[t + 2] = x.z;
            r.v[t + 3] = x.w;
        }
    } else {
#pragma unroll
        for (int t = 0; t < DS; ++t) r.v[t] = __ldg(p + t);
    }
    return r;
}

template <int DS>
__device__ __forceinline__ int pq_nearest(const PqRow<DS>& r, const float (&w)[PQ_K][DS]) {
    float best = INFINITY;
    int bi = 0;
#pragma unroll
    for (int c = 0; c < PQ_K; ++c) {
        float s = 0.f;
#pragma unroll
        for (int t = 0; t < DS; ++t) {
            const float df = r.v[t] - w[c][t];
            s = fmaf(df, df, s);
        }
        if (s < best) {
            best = s;
            bi = c;
        }
    }
    return bi;
}

template <int DS>
__device__ __forceinline__ void pq_codewords(const float* __restrict__ cb, int j, float (&w)[PQ_K][DS]) {
#pragma unroll
    for (int c = 0; c < PQ_K; ++c)
#pragma unroll
        for (int t = 0; t < DS; ++t) w[c][t] = __ldg(cb + ((int64_t)j * PQ_K + c) * DS + t);
}

// Codes [np x M] of the rows of X, residuals to the mean of their list.
template <int DS>
__global__ void __launch_bounds__(256) k_pq_encode_w(const float* __restrict__ X, const int32_t* __restrict__ assign,
                                                     const float* __restrict__ c_mean, int64_t np, int M,
                                                     const float* __restrict__ cb, uint8_t* __restrict__ codes) {
    const int RG = 256 / M, rg = threadIdx.x / M, j = threadIdx.x - rg * M;
    if (rg >= RG) return;
    const int d = M * DS;
    float w[PQ_K][DS];
    pq_codewords<DS>(cb, j, w);
    for (int64_t r = (int64_t)blockIdx.x * RG + rg; r < np; r += (int64_t)gridDim.x * RG) {
        PqRow<DS> x = pq_load<DS>(X + r * d + j * DS);
        const PqRow<DS> c = pq_load<DS>(c_mean + (int64_t)assign[r] * d + j * DS);
#pragma unroll
        for (int t = 0; t < DS; ++t) x.v[t] = __fsub_rn(x.v[t], c.v[t]);
        codes[r * M + j] = (uint8_t)pq_nearest<DS>(x, w);
    }
}

// One k-means step on residual rows R [np x d]: every row's codewords, and the
// FP64 sums and counts of every codeword's rows.  A thread adds to its own
// sums (its subspace and row group: no atomics) in shared memory, laid out
// [codeword][t][subspace] so that a warp's updates fall in distinct banks
// whatever the codewords; each CTA leaves its sums in part [grid][16 DS M] and
// counts in pcnt [grid][16 M] (k_pq_finish_w adds them up in CTA order: the
// result does not depend on the scheduling).  Adding every element to 16 d
// global sums took 222 us per 65,536 x 128 elements in atomics.
template <int DS>
__global__ void __launch_bounds__(256) k_pq_step(const float* __restrict__ R, int64_t np, int M, int RG,
                                                 const float* __restrict__ cb, double* __restrict__ part,
                                                 uint32_t* __restrict__ pcnt) {
    extern __shared__ double pq_sm[];  // RG x 16 DS M sums, then RG x 16 M counts
    const int E = PQ_K * DS * M, EC = PQ_K * M;
    uint32_t* cnt = reinterpret_cast<uint32_t*>(pq_sm + (size_t)RG * E);
    for (int e = threadIdx.x; e < RG * E; e += 256) pq_sm[e] = 0.0;
    for (int e = threadIdx.x; e < RG * EC; e += 256) cnt[e] = 0u;
    __syncthreads();
    const int rg = threadIdx.x / M, j = threadIdx.x - rg * M;
    const int d = M * DS;
    if (rg < RG) {
        float w[PQ_K][DS];
        pq_codewords<DS>(cb, j, w);
        double* ms = pq_sm + (size_t)rg * E + j;
        uint32_t* mc = cnt + (size_t)rg * EC + j;
        const int64_t stride = (int64_t)gridDim.x * RG;
        for (int64_t r = (int64_t)blockIdx.x * RG + rg; r < np; r += 4 * stride) {
            PqRow<DS> x[4];  // four rows in flight
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (r + u * stride < np) x[u] = pq_load<DS>(R + (r + u * stride) * d + j * DS);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (r + u * stride >= np) break;
                const int c = pq_nearest<DS>(x[u], w);
                mc[c * M] += 1u;
#pragma unroll
                for (int t = 0; t < DS; ++t) ms[(c * DS + t) * M] += (double)x[u].v[t];
            }
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += 256) {
        double v = 0.0;
        for (int g = 0; g < RG; ++g) v += pq_sm[(size_t)g * E + e];
        part[(size_t)blockIdx.x * E + e] = v;
    }
    for (int e = threadIdx.x; e < EC; e += 256) {
        uint32_t v = 0;
        for (int g = 0; g < RG; ++g) v += cnt[(size_t)g * EC + e];
        pcnt[(size_t)blockIdx.x * EC + e] = v;
    }
}

// New codewords (one without rows keeps its value): 32 elements per CTA, 32
// slices of the partial sums each, so that a slice is about ten loads deep.
__global__ void __launch_bounds__(1024) k_pq_finish_w(const double* __restrict__ part,
                                                      const uint32_t* __restrict__ pcnt, int nparts, int M, int DS,
                                                      float* __restrict__ cb) {
    __shared__ double ss[32][32];
    __shared__ uint32_t sc[32][32];
    const int E = PQ_K * DS * M, EC = PQ_K * M;
    const int l = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + l;  // (c DS + t) M + j
    const int ct = e / M, j = e - ct * M, c = ct / DS, t = ct - c * DS;
    const int per = (nparts + 31) / 32, p0 = g * per, p1 = min(nparts, p0 + per);
    double s = 0.0;
    uint32_t n = 0;
    if (e < E) {
#pragma unroll 12
        for (int p = p0; p < p1; ++p) {
            s += part[(size_t)p * E + e];
            n += pcnt[(size_t)p * EC + c * M + j];
        }
    }
    ss[g][l] = s;
    sc[g][l] = n;
    __syncthreads();
    if (g == 0 && e < E) {
        for (int i = 1; i < 32; ++i) {
            s += ss[i][l];
            n += sc[i][l];
        }
        if (n > 0) cb[((int64_t)j * PQ_K + c) * DS + t] = (float)(s / (double)n);
    }
}

// PQ: nearest of the 16 codewords of subspace j for residual rows (one
// thread per (row, j)); rows either given as residuals R or computed from X.
__global__ void k_pq_encode(const float* __restrict__ R, const float* __restrict__ X,
                            const int32_t* __restrict__ assign, const float* __restrict__ c_mean, int64_t np,
                            int d, int M, int dsub, const float* __restrict__ cb, uint8_t* __restrict__ codes) {
    int64_t tot = np * M;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e / M;
        int j = (int)(e - r * M);
        float best = INFINITY;
        int bi = 0;
        for (int c = 0; c < PQ_K; ++c) {
            const float* w = cb + ((int64_t)j * PQ_K + c) * dsub;
            float s = 0.f;
            for (int t = 0; t < dsub; ++t) {
                int tt = j * dsub + t;
                float rv = R ? R[r * d + tt] : __fsub_rn(X[r * d + tt], c_mean[(int64_t)assign[r] * d + tt]);
                float df = rv - w[t];
                s = fmaf(df, df, s);
            }
            if (s < best) { best = s; bi = c; }
        }
        codes[e] = (uint8_t)bi;
    }
}

__global__ void k_pq_accum(const float* __restrict__ R, int64_t np, int d, int M, int dsub,
                           const uint8_t* __restrict__ codes, double* __restrict__ sums,
                           unsigned long long* __restrict__ cnt) {
    int64_t tot = np * d;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e / d;
        int tt = (int)(e - r * d);
        int j = tt / dsub, t = tt - j * dsub;
        int c = codes[r * M + j];
        atomicAdd(&sums[((int64_t)j * PQ_K + c) * dsub + t], (double)R[e]);
        if (t == 0) atomicAdd(&cnt[(int64_t)j * PQ_K + c], 1ull);
    }
}

__global__ void k_pq_finish(const double* __restrict__ sums, const unsigned long long* __restrict__ cnt, int M,
                            int dsub, float* __restrict__ cb) {
    int64_t tot = (int64_t)M * PQ_K * dsub;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t jc = e / dsub;
        if (cnt[jc] > 0) cb[e] = (float)(sums[e] / (double)cnt[jc]);
    }
}

__global__ void k_pq_init(const float* __restrict__ R, int d, int M, int dsub, float* __restrict__ cb) {
    // codeword c of subspace j = sub-vector j of sample row c
    int64_t tot = (int64_t)M * PQ_K * dsub;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        int t = (int)(e % dsub);
        int64_t jc = e / dsub;
        int c = (int)(jc % PQ_K), j = (int)(jc / PQ_K);
        cb[e] = R[(int64_t)c * d + j * dsub + t];
    }
}

// Pack unpacked codes [n x M] into the block layout given the block member ids.
__global__ void k_pack(const int32_t* __restrict__ blk_ids, int64_t nblocks, int M,
                       const uint8_t* __restrict__ codes, uint8_t* __restrict__ blk_codes) {
    int64_t tot = nblocks * M * 16;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        int i = (int)(e & 15);
        int64_t bj = e >> 4;
        int j = (int)(bj % M);
        int64_t b = bj / M;
        int32_t id0 = blk_ids[b * 32 + 2 * i], id1 = blk_ids[b * 32 + 2 * i + 1];
        uint32_t lo = id0 >= 0 ? codes[(int64_t)id0 * M + j] : 0u;
        uint32_t hi = id1 >= 0 ? codes[(int64_t)id1 * M + j] : 0u;
        blk_codes[e] = (uint8_t)(lo | (hi << 4));
    }
}

// Unpack the block layout back to codes [n x M].
__global__ void k_unpack(const int32_t* __restrict__ blk_ids, int64_t nblocks, int M,
                         const uint8_t* __restrict__ blk_codes, uint8_t* __restrict__ codes) {
    int64_t tot = nblocks * 32 * M;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        int j = (int)(e % M);
        int64_t bv = e / M;
        int v = (int)(bv & 31);
        int64_t b = bv >> 5;
        int32_t id = blk_ids[b * 32 + v];
        if (id < 0) continue;
        uint8_t byte = blk_codes[(b * M + j) * 16 + (v >> 1)];
        codes[(int64_t)id * M + j] = (v & 1) ? (byte >> 4) : (byte & 15);
    }
}

static int grid_for(int64_t work, int threads = 256) {
    int64_t g = (work + threads - 1) / threads;
    int64_t cap = (int64_t)num_sms() * 16;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

// ------------------------------------------------------------------ host helpers
static int alloc_copy(void** dst, const void* src, size_t bytes, cudaStream_t st, cudaMemcpyKind kind) {
    KSC_CUDA(cudaMalloc(dst, bytes < 16 ? 16 : bytes));
    if (src && bytes) KSC_CUDA(cudaMemcpyAsync(*dst, src, bytes, kind, st));
    return KSC_OK;
}

// The search workspace buffers of a handle.
static int workspace_buffers(ksc_index* ix, Buffer** out) {
    Buffer* bufs[] = {&ix->ws_scores, &ix->ws_probes, &ix->ws_lut, &ix->ws_bias, &ix->ws_scale, &ix->ws_range,
                      &ix->ws_thr, &ix->ws_cnt, &ix->ws_cand, &ix->ws_topr, &ix->ws_nprobe, &ix->ws_rerank,
                      &ix->ws_items, &ix->ws_misc, &ix->ws_qbf16, &ix->ws_err, &ix->ws_feat, &ix->ws_rscore,
                      &ix->ws_full, &ix->ws_topr2, &ix->ws_flag, &ix->ws_redo, &ix->ws_pprobes, &ix->ws_pn, &ix->ws_pprob, &ix->ws_qf};
    const int n = (int)(sizeof(bufs) / sizeof(bufs[0]));
    for (int i = 0; i < n; ++i) out[i] = bufs[i];
    return n;
}

int free_index_memory(ksc_index* ix) {
    Buffer* bufs[64];
    const int nb = workspace_buffers(ix, bufs);
    if (ix->parent) {
        // a view: its own workspace, status, counters and events, and what it
        // allocated lazily itself (not the same pointer as its source's)
        const ksc_index* s = ix->parent;
        void* own[] = {ix->status, ix->c_rank_bf16 != s->c_rank_bf16 ? ix->c_rank_bf16 : nullptr,
                       ix->c_rank_f8 != s->c_rank_f8 ? ix->c_rank_f8 : nullptr,
                       ix->c_rank_f8_scale != s->c_rank_f8_scale ? ix->c_rank_f8_scale : nullptr,
                       ix->X_bf16 != s->X_bf16 ? ix->X_bf16 : nullptr, ix->X_fp8 != s->X_fp8 ? ix->X_fp8 : nullptr,
                       ix->X_scale != s->X_scale ? ix->X_scale : nullptr,
                       ix->X_band != s->X_band ? ix->X_band : nullptr,
                       ix->X_u8 != s->X_u8 ? ix->X_u8 : nullptr};
        for (void* p : own)
            if (p) cudaFree(p);
        for (int i = 0; i < nb; ++i) release(*bufs[i]);
        for (int i = 0; i <= KSC_NUM_STAGES; ++i)
            if (ix->ev[i]) cudaEventDestroy(ix->ev[i]);
        return KSC_OK;
    }
    void* ptrs[] = {ix->X, ix->c_rank, ix->c_rank_sq, ix->c_mean, ix->codebook, ix->list_boff, ix->list_n,
                    ix->blk_ids, ix->blk_codes, ix->assign, ix->graph, ix->entry, ix->status,
                    ix->c_rank_bf16, ix->mlp_w, ix->blk_list, ix->nbr_pos, ix->nbr_codes, ix->entry_pos,
                    ix->X_bf16, ix->X_fp8, ix->X_scale, ix->pr_stats, ix->pr_vecs, ix->pr_model, ix->dims,
                    ix->X_rr, ix->c_rank_f8, ix->c_rank_f8_scale, ix->gids, ix->X_band, ix->X_u8};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    for (int i = 0; i < nb; ++i) release(*bufs[i]);
    for (int i = 0; i <= KSC_NUM_STAGES; ++i)
        if (ix->ev[i]) cudaEventDestroy(ix->ev[i]);
    return KSC_OK;
}

int pack_lists(ksc_index* ix, const uint8_t* codes_dev, const int32_t* assign_host, cudaStream_t st) {
    const int L = ix->L;
    const int64_t n = ix->n;
    std::vector<int64_t> cnt(L, 0);
    for (int64_t i = 0; i < n; ++i) {
        if (assign_host[i] < 0 || assign_host[i] >= L) {
            set_error("assignment of row %lld out of range", (long long)i);
            return KSC_EINVAL;
        }
        cnt[assign_host[i]]++;
    }
    ix->h_boff.assign(L + 1, 0);
    ix->h_n.assign(L, 0);
    int64_t maxl = 0;
    for (int c = 0; c < L; ++c) {
        ix->h_n[c] = (int32_t)cnt[c];
        ix->h_boff[c + 1] = ix->h_boff[c] + (cnt[c] + BLOCK_VECS - 1) / BLOCK_VECS;
        if (cnt[c] > maxl) maxl = cnt[c];
    }
    ix->max_list = (int32_t)maxl;
    ix->nblocks = ix->h_boff[L];
    ix->h_top_blocks.assign(L + 1, 0);
    for (int c = 0; c < L; ++c) ix->h_top_blocks[c + 1] = ix->h_boff[c + 1] - ix->h_boff[c];
    std::sort(ix->h_top_blocks.begin() + 1, ix->h_top_blocks.end(), std::greater<int64_t>());
    for (int c = 0; c < L; ++c) ix->h_top_blocks[c + 1] += ix->h_top_blocks[c];
    std::vector<int32_t> ids((size_t)ix->nblocks * BLOCK_VECS, -1);
    std::vector<int64_t> fill(L);
    for (int c = 0; c < L; ++c) fill[c] = ix->h_boff[c] * BLOCK_VECS;
    for (int64_t i = 0; i < n; ++i) ids[fill[assign_host[i]]++] = (int32_t)i;  // ascending id per list
    std::vector<int32_t> blist(ix->nblocks);
    for (int c = 0; c < L; ++c)
        for (int64_t bb = ix->h_boff[c]; bb < ix->h_boff[c + 1]; ++bb) blist[bb] = c;
    KSC_TRY(alloc_copy((void**)&ix->blk_list, blist.data(), sizeof(int32_t) * (ix->nblocks > 0 ? ix->nblocks : 1), st,
                       cudaMemcpyHostToDevice));
    KSC_TRY(alloc_copy((void**)&ix->list_boff, ix->h_boff.data(), sizeof(int64_t) * (L + 1), st, cudaMemcpyHostToDevice));
    KSC_TRY(alloc_copy((void**)&ix->list_n, ix->h_n.data(), sizeof(int32_t) * L, st, cudaMemcpyHostToDevice));
    KSC_TRY(alloc_copy((void**)&ix->blk_ids, ids.data(), sizeof(int32_t) * ids.size(), st, cudaMemcpyHostToDevice));
    KSC_CUDA(cudaMalloc(&ix->blk_codes, (size_t)ix->nblocks * ix->M * 16 + 16));
    k_pack<<<grid_for(ix->nblocks * ix->M * 16), 256, 0, st>>>(ix->blk_ids, ix->nblocks, ix->M, codes_dev,
                                                               ix->blk_codes);
    KSC_LAUNCH_CHECK();
    KSC_CUDA(cudaStreamSynchronize(st));  // `ids` goes out of scope
    return KSC_OK;
}

// splitmix64 (Steele, Lea, Flood 2014) driving a Fisher-Yates shuffle.
static uint64_t splitmix64(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

static void host_perm(int64_t n, uint64_t seed, std::vector<int64_t>& p) {
    p.resize(n);
    for (int64_t i = 0; i < n; ++i) p[i] = i;
    uint64_t s = seed;
    for (int64_t i = n - 1; i > 0; --i) {
        int64_t j = (int64_t)(splitmix64(s) % (uint64_t)(i + 1));
        int64_t t = p[i];
        p[i] = p[j];
        p[j] = t;
    }
}

// Row groups per CTA of k_pq_step and its shared bytes (at most 100 KB with
// more than one group, so that two CTAs fit an SM).
static size_t pq_step_smem(int M, int DS, int RG) { return (size_t)RG * M * PQ_K * (8 * DS + 4); }
static int pq_step_groups(int M, int DS) {
    int rg = 256 / M;
    while (rg > 1 && pq_step_smem(M, DS, rg) > 100 * 1024) --rg;
    return rg;
}

// k-means of the PQ codebooks cb [M x 16 x DS] on residual rows R [np x d],
// one kernel pair per iteration.
template <int DS>
static int pq_train_w(const float* R, int64_t np, int M, int iters, float* cb, cudaStream_t st) {
    const int RG = pq_step_groups(M, DS), E = PQ_K * DS * M, EC = PQ_K * M;
    const size_t smem = pq_step_smem(M, DS, RG);
    KSC_CUDA(cudaFuncSetAttribute(k_pq_step<DS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    KSC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pq_step<DS>, 256, smem));
    // 4 rows a group and CTA at least; 16 with few rounds, which do not win back what
    // allocating more partial sums costs (3000 rows x 96 in 96 subspaces: a round 52
    // and 50 us, two rounds' build 790 and 710; x 64 in 8: 48 and 57, 612 and 552)
    const int per = iters < 8 ? 16 : 4;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((np + per * RG - 1) / (per * RG),
                                                                 (int64_t)num_sms() * (per_sm > 0 ? per_sm : 1)));
    double* part = nullptr;
    KSC_CUDA(cudaMalloc(&part, (sizeof(double) * E + sizeof(uint32_t) * EC) * (size_t)grid));
    uint32_t* pcnt = reinterpret_cast<uint32_t*>(part + (size_t)grid * E);
    for (int it = 0; it < iters; ++it) {
        k_pq_step<DS><<<grid, 256, smem, st>>>(R, np, M, RG, cb, part, pcnt);
        k_pq_finish_w<<<(E + 31) / 32, 1024, 0, st>>>(part, pcnt, grid, M, DS, cb);
    }
    const cudaError_t e = cudaGetLastError();
    cudaFree(part);  // (waits for the kernels)
    KSC_CUDA(e);
    return KSC_OK;
}

// The widths that the register kernels serve (a row's sub-vectors then start
// on the loads' alignment: DS floats, d a multiple of DS); other widths take
// the kernels for any width.
static bool pq_width_w(int dsub) { return dsub == 1 || dsub == 2 || dsub == 3 || dsub == 4 || dsub == 8; }

static int pq_train(const float* R, int64_t np, int M, int dsub, int iters, float* cb, cudaStream_t st) {
    switch (dsub) {
        case 1: return pq_train_w<1>(R, np, M, iters, cb, st);
        case 2: return pq_train_w<2>(R, np, M, iters, cb, st);
        case 3: return pq_train_w<3>(R, np, M, iters, cb, st);
        case 4: return pq_train_w<4>(R, np, M, iters, cb, st);
        default: return pq_train_w<8>(R, np, M, iters, cb, st);
    }
}

static int pq_encode(const float* X, const int32_t* assign, const float* c_mean, int64_t n, int M, int dsub,
                     const float* cb, uint8_t* codes, cudaStream_t st) {
    const int RG = 256 / M;
    const int grid = (int)std::min<int64_t>((n + 4 * RG - 1) / (4 * RG), (int64_t)num_sms() * 8);
    switch (dsub) {
        case 1: k_pq_encode_w<1><<<grid, 256, 0, st>>>(X, assign, c_mean, n, M, cb, codes); break;
        case 2: k_pq_encode_w<2><<<grid, 256, 0, st>>>(X, assign, c_mean, n, M, cb, codes); break;
        case 3: k_pq_encode_w<3><<<grid, 256, 0, st>>>(X, assign, c_mean, n, M, cb, codes); break;
        case 4: k_pq_encode_w<4><<<grid, 256, 0, st>>>(X, assign, c_mean, n, M, cb, codes); break;
        default: k_pq_encode_w<8><<<grid, 256, 0, st>>>(X, assign, c_mean, n, M, cb, codes); break;
    }
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

// The assignment of T's rows to its centroids: tensor cores, then the FP32
// kernel for the rows left over.
static int assign_rows(AssignTc& T, int32_t* assign, cudaStream_t st) {
    KSC_TRY(T.run(assign, st));
    k_assign<<<(unsigned)((T.nrows + AS_T - 1) / AS_T), 256, 0, st>>>(T.X, T.nrows, T.d, T.C, T.cn, T.L, T.spherical,
                                                                      assign, T.redo, T.small, T.redo_rows());
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

// Whether the tensor cores pay off for a build's assignments (iters rounds of
// ns rows and one of n).  They score 256 centroids whatever L, from FP16 copies
// of the rows, in four launches; the FP32 kernel scores 64 at a time from the
// rows themselves.  Builds of 10 rounds in ms, FP32 / tensor cores: 20,000 x 128
// in 64 lists 2.0 / 2.3, in 192 2.6 / 2.4, in 256 2.9 / 2.5; 20,000 x 64 in 256
// (0.33 G multiply-adds a round) 2.1 / 2.1; 200,000 x 16 in 256 (0.32) 3.7 / 3.9;
// 1M x 128 in 64 14.8 / 16.0, in 128 15.4 / 16.0, in 192 17.0 / 15.8; 20,000 x 512 in
// 64 3.3 / 3.5, in 96 4.4 / 3.6.
static bool assign_tc_pays(int64_t n, int64_t ns, int d, int L, int iters) {
    return (L > 128 || (L > 64 && d >= 256)) && ((double)iters * ns + n) * L * d >= 0.35e9 * (iters + 1);
}

// Rows per pass of the final assignment (bounds the FP16 copy).
constexpr int64_t ASSIGN_CHUNK = 1 << 20;

// Lloyd on rows `sample` of X (device), init = first L sample rows.  T: the
// tensor-core assignment, or null (FP32 cores throughout).
static int lloyd(const float* X, const int64_t* sample_dev, int64_t ns, int d, int L, int iters, float* C,
                 AssignTc* T, float xmax, cudaStream_t st) {
    float* Xs = nullptr;
    float* cn = nullptr;
    int32_t* a = nullptr;
    double* sums = nullptr;
    unsigned long long* cnt = nullptr;
    int rc = KSC_OK;
    auto cleanup = [&]() {
        cudaFree(Xs); cudaFree(cn); cudaFree(a); cudaFree(sums); cudaFree(cnt);
    };
#define LL_CUDA(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) { set_error("%s: %s", #call, cudaGetErrorString(e_)); cleanup(); return KSC_ECUDA; } } while (0)
    LL_CUDA(cudaMalloc(&Xs, sizeof(float) * ns * d));
    LL_CUDA(cudaMalloc(&cn, sizeof(float) * L));
    LL_CUDA(cudaMalloc(&a, sizeof(int32_t) * ns));
    // an assignment on the tensor cores that gives up leaves rows undecided: they
    // then hold a list of an earlier round (or list 0) until the check below
    LL_CUDA(cudaMemsetAsync(a, 0, sizeof(int32_t) * ns, st));
    LL_CUDA(cudaMalloc(&sums, sizeof(double) * L * d));
    LL_CUDA(cudaMalloc(&cnt, sizeof(unsigned long long) * L));
    k_gather_rows<<<grid_for(ns * d), 256, 0, st>>>(X, sample_dev, ns, d, Xs);
    LL_CUDA(cudaMemcpyAsync(C, Xs, sizeof(float) * L * d, cudaMemcpyDeviceToDevice, st));
    LL_CUDA(cudaMemsetAsync(sums, 0, sizeof(double) * L * d, st));
    LL_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * L, st));
    if (T) rc = T->set_rows(Xs, ns, st);
    for (int it = 0; it < iters && rc == KSC_OK; ++it) {
        if (T) {
            // the means of the previous round are taken as the operands are made
            rc = T->set_centroids(C, it ? sums : nullptr, it ? cnt : nullptr, false, xmax, st);
            if (rc == KSC_OK) rc = assign_rows(*T, a, st);
            if (rc) break;
        } else {
            if (it) {
                k_centroid_finish<<<grid_for((int64_t)L * d), 256, 0, st>>>(sums, cnt, C, L, d, C);
                LL_CUDA(cudaMemsetAsync(sums, 0, sizeof(double) * L * d, st));
                LL_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * L, st));
            }
            k_row_sqnorm<<<(L + 255) / 256, 256, 0, st>>>(C, L, d, cn);
            k_assign<<<(unsigned)((ns + AS_T - 1) / AS_T), 256, 0, st>>>(Xs, ns, d, C, cn, L, 0, a, nullptr, nullptr, 0);
        }
        k_centroid_accum<<<grid_for(ns * d), 256, 0, st>>>(Xs, nullptr, ns, d, a, sums, cnt);
        LL_CUDA(cudaGetLastError());
    }
    if (rc == KSC_OK) {
        k_centroid_finish<<<grid_for((int64_t)L * d), 256, 0, st>>>(sums, cnt, C, L, d, C);
        LL_CUDA(cudaGetLastError());
    }
    LL_CUDA(cudaStreamSynchronize(st));
    if (T && rc == KSC_OK) rc = T->check(st);
    cleanup();
#undef LL_CUDA
    return rc;
}

}  // namespace ksc

using namespace ksc;

extern "C" {

const char* ksc_last_error(void) { return get_error(); }
const char* ksc_version(void) { return "kscann-gb300 0.1 (sm_103a)"; }

void ksc_index_free(ksc_index* ix) {
    if (!ix) return;
    free_index_memory(ix);
    delete ix;
}

int ksc_index_info(const ksc_index* ix, ksc_index_arrays* a) {
    KSC_CHECK_ARG(ix && a, "null argument");
    a->n = ix->n;
    a->d = ix->d;
    a->nlist = ix->L;
    a->M = ix->M;
    a->metric = ix->metric;
    a->spherical = ix->spherical;
    return KSC_OK;
}

static int finish_common(ksc_index* ix, cudaStream_t st) {
    if (!ix->c_rank_sq) KSC_CUDA(cudaMalloc(&ix->c_rank_sq, sizeof(float) * ix->L));
    k_row_sqnorm<<<(ix->L + 255) / 256, 256, 0, st>>>(ix->c_rank, ix->L, ix->d, ix->c_rank_sq);
    KSC_LAUNCH_CHECK();
    KSC_CUDA(cudaMalloc(&ix->status, STATUS_BYTES));
    ix->stats = (unsigned long long*)(ix->status + STATUS_STATS);
    KSC_CUDA(cudaMemsetAsync(ix->status, 0, STATUS_BYTES, st));
    KSC_CUDA(cudaStreamSynchronize(st));
    return KSC_OK;
}

static int check_shape(int64_t n, int32_t d, int32_t L, int32_t M, bool shard = false) {
    KSC_CHECK_ARG(n > 0 && n < (1ll << 31), "n must be in [1, 2^31)");
    KSC_CHECK_ARG(d > 0 && d <= KSC_MAX_DIM, "d must be in [1, %d]", KSC_MAX_DIM);
    // a shard holds every list (most of them empty): nlist may exceed its rows
    KSC_CHECK_ARG(L > 0 && L <= KSC_MAX_NLIST && (shard || L <= n), "nlist must be in [1, min(n, %d)]",
                  KSC_MAX_NLIST);
    KSC_CHECK_ARG(M > 0 && M <= KSC_MAX_M && d % M == 0, "M must divide d and be <= %d", KSC_MAX_M);
    return KSC_OK;
}

static int import_arrays(const ksc_index_arrays* a, void* stream, ksc_index** out, bool shard) {
    KSC_CHECK_ARG(a && out && a->X && a->c_rank && a->c_mean && a->codebook && a->codes && a->assign,
                  "null argument");
    KSC_TRY(check_shape(a->n, a->d, a->nlist, a->M, shard));
    KSC_CHECK_ARG(a->metric == KSC_L2 || a->metric == KSC_IP, "bad metric");
    // Every index the device code follows is checked here, on the host,
    // before any device work: codes address 16-entry tables, lists address
    // the list arrays, and the graph preparation and search take a neighbour
    // (or a list's entry) as a position inside its own list, so a neighbour
    // of another list would address codes and visited bits outside the list.
    const int64_t ncodes = a->n * a->M;
    for (int64_t i = 0; i < ncodes; ++i)
        KSC_CHECK_ARG(a->codes[i] < PQ_K, "code %lld is out of range", (long long)i);
    for (int64_t i = 0; i < a->n; ++i)
        KSC_CHECK_ARG(a->assign[i] >= 0 && a->assign[i] < a->nlist, "assignment of row %lld out of range",
                      (long long)i);
    if (a->graph && a->entry) {
        for (int64_t u = 0; u < a->n; ++u)
            for (int e = 0; e < 32; ++e) {
                const int32_t v = a->graph[u * 32 + e];
                KSC_CHECK_ARG(v >= -1 && v < a->n, "neighbour %d of row %lld is out of range", e, (long long)u);
                KSC_CHECK_ARG(v < 0 || a->assign[v] == a->assign[u],
                              "neighbour %d of row %lld is in another list", e, (long long)u);
            }
        for (int32_t p = 0; p < a->nlist; ++p) {
            const int32_t v = a->entry[p];
            KSC_CHECK_ARG(v >= -1 && v < a->n, "graph entry of list %d is out of range", p);
            KSC_CHECK_ARG(v < 0 || a->assign[v] == p, "graph entry of list %d is not in the list", p);
        }
    }
    cudaStream_t st = as_stream(stream);
    ksc_index* ix = new ksc_index();
    ix->n = a->n;
    ix->d = a->d;
    ix->L = a->nlist;
    ix->M = a->M;
    ix->dsub = a->d / a->M;
    ix->metric = a->metric;
    ix->spherical = (a->spherical || a->metric == KSC_IP) ? 1 : 0;
    int rc = KSC_OK;
    uint8_t* codes_dev = nullptr;
    do {
        if ((rc = alloc_copy((void**)&ix->X, a->X, sizeof(float) * ix->n * ix->d, st, cudaMemcpyHostToDevice))) break;
        if ((rc = alloc_copy((void**)&ix->c_rank, a->c_rank, sizeof(float) * ix->L * ix->d, st, cudaMemcpyHostToDevice))) break;
        if ((rc = alloc_copy((void**)&ix->c_mean, a->c_mean, sizeof(float) * ix->L * ix->d, st, cudaMemcpyHostToDevice))) break;
        if ((rc = alloc_copy((void**)&ix->codebook, a->codebook, sizeof(float) * ix->M * PQ_K * ix->dsub, st,
                             cudaMemcpyHostToDevice))) break;
        if ((rc = alloc_copy((void**)&ix->assign, a->assign, sizeof(int32_t) * ix->n, st, cudaMemcpyHostToDevice))) break;
        if ((rc = alloc_copy((void**)&codes_dev, a->codes, (size_t)ix->n * ix->M, st, cudaMemcpyHostToDevice))) break;
        if ((rc = pack_lists(ix, codes_dev, a->assign, st))) break;
        if (a->graph && a->entry) {
            if ((rc = alloc_copy((void**)&ix->graph, a->graph, sizeof(int32_t) * ix->n * 32, st, cudaMemcpyHostToDevice))) break;
            if ((rc = alloc_copy((void**)&ix->entry, a->entry, sizeof(int32_t) * ix->L, st, cudaMemcpyHostToDevice))) break;
            if ((rc = prepare_graph(ix, st))) break;
        }
        rc = finish_common(ix, st);
    } while (0);
    if (codes_dev) cudaFree(codes_dev);
    if (rc != KSC_OK) {
        ksc_index_free(ix);
        return rc;
    }
    *out = ix;
    return KSC_OK;
}

int ksc_index_import(const ksc_index_arrays* a, void* stream, ksc_index** out) {
    return import_arrays(a, stream, out, false);
}

// One shard of a list-partitioned index: the lists p with list_owner[p] ==
// shard keep their members (rows in ascending global id), every other list
// is empty; centroids and codebooks are replicated, so every shard ranks the
// lists and scales the tables (a_q over the whole probe set) as the whole
// index does.  gids maps local rows back to the global ids.
int ksc_index_import_shard(const ksc_index_arrays* full, const int32_t* list_owner, int32_t shard, void* stream,
                           ksc_index** out) {
    KSC_CHECK_ARG(full && list_owner && out && full->X && full->codes && full->assign, "null argument");
    KSC_CHECK_ARG(shard >= 0, "shard must be >= 0");
    KSC_TRY(check_shape(full->n, full->d, full->nlist, full->M));
    for (int32_t p = 0; p < full->nlist; ++p) KSC_CHECK_ARG(list_owner[p] >= 0, "owner of list %d is negative", p);
    std::vector<int32_t> rows;
    for (int64_t i = 0; i < full->n; ++i) {
        const int32_t p = full->assign[i];
        KSC_CHECK_ARG(p >= 0 && p < full->nlist, "assignment of row %lld out of range", (long long)i);
        if (list_owner[p] == shard) rows.push_back((int32_t)i);
    }
    KSC_CHECK_ARG(!rows.empty(), "shard %d holds no vector", shard);
    const int64_t ns = (int64_t)rows.size();
    const int d = full->d, M = full->M;
    std::vector<float> X((size_t)ns * d);
    std::vector<uint8_t> codes((size_t)ns * M);
    std::vector<int32_t> assign(ns);
    for (int64_t r = 0; r < ns; ++r) {
        const int64_t i = rows[r];
        std::copy(full->X + i * d, full->X + (i + 1) * d, X.begin() + r * d);
        std::copy(full->codes + i * M, full->codes + (i + 1) * M, codes.begin() + r * M);
        assign[r] = full->assign[i];
    }
    ksc_index_arrays a = *full;
    a.n = ns;
    a.X = X.data();
    a.codes = codes.data();
    a.assign = assign.data();
    a.graph = nullptr;
    a.entry = nullptr;
    ksc_index* ix = nullptr;
    KSC_TRY(import_arrays(&a, stream, &ix, true));
    if (alloc_copy((void**)&ix->gids, rows.data(), sizeof(int32_t) * ns, as_stream(stream),
                   cudaMemcpyHostToDevice) != KSC_OK ||
        cudaStreamSynchronize(as_stream(stream)) != cudaSuccess) {
        ksc_index_free(ix);
        set_error("shard id map: device copy failed");
        return KSC_ECUDA;
    }
    *out = ix;
    return KSC_OK;
}

int ksc_index_export(const ksc_index* ix, ksc_index_arrays* a) {
    KSC_CHECK_ARG(ix && a, "null argument");
    ksc_index_info(ix, a);
    if (a->X) KSC_CUDA(cudaMemcpy(a->X, ix->X, sizeof(float) * ix->n * ix->d, cudaMemcpyDeviceToHost));
    if (a->c_rank) KSC_CUDA(cudaMemcpy(a->c_rank, ix->c_rank, sizeof(float) * ix->L * ix->d, cudaMemcpyDeviceToHost));
    if (a->c_mean) KSC_CUDA(cudaMemcpy(a->c_mean, ix->c_mean, sizeof(float) * ix->L * ix->d, cudaMemcpyDeviceToHost));
    if (a->codebook)
        KSC_CUDA(cudaMemcpy(a->codebook, ix->codebook, sizeof(float) * ix->M * PQ_K * ix->dsub, cudaMemcpyDeviceToHost));
    if (a->assign) KSC_CUDA(cudaMemcpy(a->assign, ix->assign, sizeof(int32_t) * ix->n, cudaMemcpyDeviceToHost));
    if (a->codes) {
        uint8_t* codes_dev = nullptr;
        KSC_CUDA(cudaMalloc(&codes_dev, (size_t)ix->n * ix->M));
        k_unpack<<<grid_for(ix->nblocks * 32 * ix->M), 256>>>(ix->blk_ids, ix->nblocks, ix->M, ix->blk_codes,
                                                              codes_dev);
        cudaError_t e = cudaMemcpy(a->codes, codes_dev, (size_t)ix->n * ix->M, cudaMemcpyDeviceToHost);
        cudaFree(codes_dev);
        KSC_CUDA(e);
    }
    if (a->graph && ix->graph) KSC_CUDA(cudaMemcpy(a->graph, ix->graph, sizeof(int32_t) * ix->n * 32, cudaMemcpyDeviceToHost));
    if (a->entry && ix->entry) KSC_CUDA(cudaMemcpy(a->entry, ix->entry, sizeof(int32_t) * ix->L, cudaMemcpyDeviceToHost));
    return KSC_OK;
}

// Component filtration (Sec. 4.3; Alg. 1 FilterComponents): the index is
// built on the kept dimensions -- the sub-vector width d / M is kept, so the
// filtered index has ceil(kept / (d / M)) subspaces, the last completed with
// zero dimensions -- and holds the full vectors for the re-rank.
static int build_filtered(const float* X_dev, int64_t n, int32_t d, int32_t nlist, int32_t M, int32_t nbits,
                          ksc_metric metric, const ksc_build_opts* opts, void* stream, ksc_index** out) {
    KSC_TRY(check_shape(n, d, nlist, M));
    cudaStream_t st = as_stream(stream);
    const double thr = opts->filter_threshold;
    std::vector<double> frac(d);
    double* stats = nullptr;
    KSC_CUDA(cudaMalloc(&stats, sizeof(double) * 3 * d));
    int rc = component_stats(X_dev, n, d, stats, stats + d, stats + 2 * d, st);
    if (rc == KSC_OK && cudaMemcpy(frac.data(), stats + 2 * d, sizeof(double) * d, cudaMemcpyDeviceToHost) != cudaSuccess) {
        set_error("reading the component statistics failed");
        rc = KSC_ECUDA;
    }
    cudaFree(stats);
    KSC_TRY(rc);
    std::vector<int32_t> dims;
    for (int t = 0; t < d; ++t)
        if (frac[t] <= thr) dims.push_back(t);
    KSC_CHECK_ARG(!dims.empty(), "component filtration kept no dimension (threshold %g)", thr);
    const int dsub = d / M;
    const int Mf = (int)((dims.size() + dsub - 1) / dsub);
    while ((int)dims.size() < Mf * dsub) dims.push_back(-1);
    const int dw = Mf * dsub;
    float* Xw = nullptr;
    int32_t* dims_dev = nullptr;
    KSC_CUDA(cudaMalloc(&dims_dev, sizeof(int32_t) * dw));
    cudaError_t e = cudaMemcpy(dims_dev, dims.data(), sizeof(int32_t) * dw, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMalloc(&Xw, sizeof(float) * n * dw);
    if (e != cudaSuccess) {
        cudaFree(dims_dev);
        set_error("component filtration: %s", cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? KSC_ENOMEM : KSC_ECUDA;
    }
    rc = gather_dims(X_dev, n, d, dims_dev, dw, Xw, st);
    ksc_build_opts inner = *opts;
    inner.filter_threshold = 0.f;
    ksc_index* ix = nullptr;
    if (rc == KSC_OK) rc = ksc_build_index(Xw, n, dw, nlist, Mf, nbits, metric, &inner, stream, &ix);
    cudaStreamSynchronize(st);
    cudaFree(Xw);
    if (rc == KSC_OK) {
        ix->dims = dims_dev;
        dims_dev = nullptr;
        ix->h_dims = dims;
        ix->d_rr = d;
        e = cudaMalloc(&ix->X_rr, sizeof(float) * n * d);
        if (e == cudaSuccess) e = cudaMemcpyAsync(ix->X_rr, X_dev, sizeof(float) * n * d, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) {
            set_error("component filtration: %s", cudaGetErrorString(e));
            rc = e == cudaErrorMemoryAllocation ? KSC_ENOMEM : KSC_ECUDA;
            ksc_index_free(ix);
            ix = nullptr;
        }
    }
    if (dims_dev) cudaFree(dims_dev);
    if (rc == KSC_OK) *out = ix;
    return rc;
}

int ksc_build_index(const float* X_dev, int64_t n, int32_t d, int32_t nlist, int32_t M, int32_t nbits,
                    ksc_metric metric, const ksc_build_opts* opts, void* stream, ksc_index** out) {
    KSC_CHECK_ARG(X_dev && out, "null argument");
    if (opts && opts->filter_threshold > 0.f) return build_filtered(X_dev, n, d, nlist, M, nbits, metric, opts, stream, out);
    if (nbits != 4) {
        set_error("only 4-bit PQ codes (K = 16) are supported, got nbits = %d", nbits);
        return KSC_EUNSUPPORTED;
    }
    KSC_TRY(check_shape(n, d, nlist, M));
    KSC_CHECK_ARG(metric == KSC_L2 || metric == KSC_IP, "bad metric");
    cudaStream_t st = as_stream(stream);
    const int iters = (opts && opts->kmeans_iters > 0) ? opts->kmeans_iters : 20;
    const int spherical = (metric == KSC_IP || (opts && opts->spherical)) ? 1 : 0;
    std::vector<int64_t> perm;
    if (opts && opts->perm_host) {
        perm.assign(opts->perm_host, opts->perm_host + n);
    } else {
        host_perm(n, opts ? opts->seed : 0x5eed, perm);
    }
    ksc_index* ix = new ksc_index();
    ix->n = n; ix->d = d; ix->L = nlist; ix->M = M; ix->dsub = d / M;
    ix->metric = metric; ix->spherical = spherical;
    const int64_t ns = n < 256ll * nlist ? n : 256ll * nlist;
    const int64_t npq = n < 65536 ? n : 65536;
    int64_t* perm_dev = nullptr;
    uint8_t* codes_dev = nullptr;
    float* Rs = nullptr;
    double* sums = nullptr;
    unsigned long long* cnt = nullptr;
    uint8_t* pcodes = nullptr;
    int rc = KSC_OK;
    std::vector<int32_t> assign_host(n);
    AssignTc T;
    do {
#define B_CUDA(call) { cudaError_t e_ = (call); if (e_ != cudaSuccess) { set_error("%s: %s", #call, cudaGetErrorString(e_)); rc = e_ == cudaErrorMemoryAllocation ? KSC_ENOMEM : KSC_ECUDA; break; } }
        B_CUDA(cudaMalloc(&ix->X, sizeof(float) * n * d));
        B_CUDA(cudaMemcpyAsync(ix->X, X_dev, sizeof(float) * n * d, cudaMemcpyDeviceToDevice, st));
        B_CUDA(cudaMalloc(&perm_dev, sizeof(int64_t) * n));
        B_CUDA(cudaMemcpyAsync(perm_dev, perm.data(), sizeof(int64_t) * n, cudaMemcpyHostToDevice, st));
        B_CUDA(cudaMalloc(&ix->c_rank, sizeof(float) * nlist * d));
        B_CUDA(cudaMalloc(&ix->c_mean, sizeof(float) * nlist * d));
        B_CUDA(cudaMalloc(&ix->c_rank_sq, sizeof(float) * nlist));
        // 1. coarse quantiser
        float xmax = 0.f;
        bool tc = assign_tc_pays(n, ns, d, nlist, iters);
        if (tc && (rc = max_abs(ix->X, n * d, &xmax, st))) break;
        tc = tc && assign_tc_supported(xmax);
        // list of every row, and then the operands: where the device has no room for
        // them, or for the k-means beside them, the FP32 kernel needs neither
        B_CUDA(cudaMalloc(&ix->assign, sizeof(int32_t) * n));
        if (tc) {
            rc = T.init(std::max(ns, std::min(n, ASSIGN_CHUNK)), d, nlist, xmax, st);
            if (rc == KSC_OK) rc = lloyd(ix->X, perm_dev, ns, d, nlist, iters, ix->c_mean, &T, xmax, st);
            if (rc == KSC_ETIMEOUT) break;
            if (rc != KSC_OK) {
                cudaGetLastError();
                T.free();
                tc = false;
            }
        }
        if (!tc && (rc = lloyd(ix->X, perm_dev, ns, d, nlist, iters, ix->c_mean, nullptr, 0.f, st))) break;
        B_CUDA(cudaMemcpyAsync(ix->c_rank, ix->c_mean, sizeof(float) * nlist * d, cudaMemcpyDeviceToDevice, st));
        if (spherical) k_normalise_rows<<<(nlist + 255) / 256, 256, 0, st>>>(ix->c_rank, nlist, d);
        k_row_sqnorm<<<(nlist + 255) / 256, 256, 0, st>>>(ix->c_rank, nlist, d, ix->c_rank_sq);
        // 2. list of every vector by the ranking score
        if (tc) {
            rc = T.set_centroids(ix->c_rank, nullptr, nullptr, spherical, spherical ? 1.f : xmax, st);
            for (int64_t r0 = 0; r0 < n && rc == KSC_OK; r0 += ASSIGN_CHUNK) {
                if ((rc = T.set_rows(ix->X + r0 * d, std::min(n - r0, ASSIGN_CHUNK), st))) break;
                if (r0) B_CUDA(cudaMemsetAsync(T.small, 0, sizeof(int32_t) * 2, st));
                rc = assign_rows(T, ix->assign + r0, st);
            }
            if (rc == KSC_OK) rc = T.check(st);  // before anything indexes with the lists
            if (rc) break;
            T.free();
        } else {
            k_assign<<<(unsigned)((n + AS_T - 1) / AS_T), 256, 0, st>>>(ix->X, n, d, ix->c_rank, ix->c_rank_sq, nlist,
                                                                        spherical, ix->assign, nullptr, nullptr, 0);
        }
        // 3. mean centroids of the lists (Sec. 4.6.1)
        B_CUDA(cudaMalloc(&sums, sizeof(double) * (size_t)nlist * d));
        B_CUDA(cudaMalloc(&cnt, sizeof(unsigned long long) * nlist));
        B_CUDA(cudaMemsetAsync(sums, 0, sizeof(double) * (size_t)nlist * d, st));
        B_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * nlist, st));
        k_centroid_accum<<<grid_for(n * d), 256, 0, st>>>(ix->X, nullptr, n, d, ix->assign, sums, cnt);
        // (empty list: keeps its Lloyd centroid, already in c_mean)
        k_centroid_finish<<<grid_for((int64_t)nlist * d), 256, 0, st>>>(sums, cnt, ix->c_mean, nlist, d, ix->c_mean);
        B_CUDA(cudaGetLastError());
        // 4. PQ codebooks on the residuals of the first npq permuted rows
        B_CUDA(cudaMalloc(&Rs, sizeof(float) * npq * d));
        k_residual<<<grid_for(npq * d), 256, 0, st>>>(ix->X, perm_dev, npq, d, ix->assign, ix->c_mean, Rs);
        B_CUDA(cudaMalloc(&ix->codebook, sizeof(float) * M * PQ_K * ix->dsub));
        const bool wide = pq_width_w(ix->dsub);
        if (!wide) {
            B_CUDA(cudaMalloc(&pcodes, (size_t)npq * M));
            cudaFree(sums); sums = nullptr;
            cudaFree(cnt); cnt = nullptr;
            B_CUDA(cudaMalloc(&sums, sizeof(double) * M * PQ_K * ix->dsub));
            B_CUDA(cudaMalloc(&cnt, sizeof(unsigned long long) * M * PQ_K));
        }
        k_pq_init<<<grid_for((int64_t)M * PQ_K * ix->dsub), 256, 0, st>>>(Rs, d, M, ix->dsub, ix->codebook);
        if (wide && (rc = pq_train(Rs, npq, M, ix->dsub, iters, ix->codebook, st))) break;
        for (int it = 0; it < iters && !wide; ++it) {
            k_pq_encode<<<grid_for(npq * M), 256, 0, st>>>(Rs, nullptr, nullptr, nullptr, npq, d, M, ix->dsub,
                                                           ix->codebook, pcodes);
            B_CUDA(cudaMemsetAsync(sums, 0, sizeof(double) * M * PQ_K * ix->dsub, st));
            B_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * M * PQ_K, st));
            k_pq_accum<<<grid_for(npq * d), 256, 0, st>>>(Rs, npq, d, M, ix->dsub, pcodes, sums, cnt);
            k_pq_finish<<<grid_for((int64_t)M * PQ_K * ix->dsub), 256, 0, st>>>(sums, cnt, M, ix->dsub, ix->codebook);
        }
        B_CUDA(cudaGetLastError());
        if (rc) break;
        // 5. encode every vector and pack the lists into blocks
        B_CUDA(cudaMalloc(&codes_dev, (size_t)n * M));
        if (wide) rc = pq_encode(ix->X, ix->assign, ix->c_mean, n, M, ix->dsub, ix->codebook, codes_dev, st);
        else k_pq_encode<<<grid_for(n * M), 256, 0, st>>>(nullptr, ix->X, ix->assign, ix->c_mean, n, d, M, ix->dsub,
                                                          ix->codebook, codes_dev);
        if (rc) break;
        B_CUDA(cudaGetLastError());
        B_CUDA(cudaMemcpyAsync(assign_host.data(), ix->assign, sizeof(int32_t) * n, cudaMemcpyDeviceToHost, st));
        B_CUDA(cudaStreamSynchronize(st));
        if ((rc = pack_lists(ix, codes_dev, assign_host.data(), st))) break;
        if ((rc = finish_common(ix, st))) break;
        if (opts && opts->build_graph) {
            if ((rc = ksc::build_graph(ix, st))) break;
        }
#undef B_CUDA
    } while (0);
    cudaFree(perm_dev); cudaFree(codes_dev); cudaFree(Rs); cudaFree(sums); cudaFree(cnt); cudaFree(pcodes);
    if (rc != KSC_OK) {
        ksc_index_free(ix);
        return rc;
    }
    *out = ix;
    return KSC_OK;
}

}  // extern "C"

extern "C" int ksc_index_dims(ksc_index* ix, int32_t* dims_host, int32_t* d_full_host) {
    KSC_CHECK_ARG(ix && d_full_host, "null argument");
    *d_full_host = ix->X_rr ? ix->d_rr : ix->d;
    if (dims_host)
        for (int j = 0; j < ix->d; ++j) dims_host[j] = ix->X_rr ? ix->h_dims[j] : j;
    return KSC_OK;
}

extern "C" int ksc_component_stats(const float* X_dev, int64_t n, int32_t d, double* mu_dev, double* sd_dev,
                                   double* frac_dev, void* stream) {
    KSC_CHECK_ARG(X_dev && mu_dev && sd_dev && frac_dev && n > 0 && d > 0, "bad argument");
    return ksc::component_stats(X_dev, n, d, mu_dev, sd_dev, frac_dev, ksc::as_stream(stream));
}

// A second handle on the same index data with its own search workspace,
// status word, counters and stage events, so that searches on different
// streams can run at the same time (one handle each).
extern "C" int ksc_index_view(ksc_index* ix, ksc_index** out) {
    KSC_CHECK_ARG(ix && out, "null argument");
    ksc_index* v = new ksc_index(*ix);  // the shared arrays, models and host mirrors
    v->parent = ix;
    ksc::Buffer* bufs[64];
    const int nb = workspace_buffers(v, bufs);
    for (int i = 0; i < nb; ++i) *bufs[i] = ksc::Buffer{};
    for (int i = 0; i <= KSC_NUM_STAGES; ++i) {
        v->ev[i] = nullptr;
        v->ev_used[i] = false;
    }
    v->prof = false;
    v->launches = 0;
    v->u8_wanted = 0;
    v->status = nullptr;
    v->stats = nullptr;
    cudaError_t e = cudaMalloc(&v->status, STATUS_BYTES);
    if (e == cudaSuccess) {
        v->stats = (unsigned long long*)(v->status + STATUS_STATS);
        e = cudaMemset(v->status, 0, STATUS_BYTES);
    }
    if (e != cudaSuccess) {
        ksc::set_error("ksc_index_view: %s", cudaGetErrorString(e));
        ksc_index_free(v);
        return e == cudaErrorMemoryAllocation ? KSC_ENOMEM : KSC_ECUDA;
    }
    *out = v;
    return KSC_OK;
}
