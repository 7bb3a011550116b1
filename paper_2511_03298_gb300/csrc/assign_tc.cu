// Nearest centroid of every row (k-means assignment, Alg. 1) with the scores
// on the 5th-generation tensor cores and the decision in FP32.
//
// The FP32 rule (k_assign in index.cu): score = ||c||^2 - 2 <x, c> (or -<x, c>)
// with <x, c> summed by FMAs over ascending dimensions; the smallest score,
// ties to the lower centroid.  Here the scores of all centroids come from FP16
// operands with FP32 accumulation, within a proven bound of the FP32 rule's;
// a row's centroids within twice the bound of its best are re-scored by the
// FP32 rule itself, so the result is the rule's, bit for bit.  A row with more
// of them than its candidate list holds goes on a list for k_assign.
//
// Operands: rows and centroids scaled by powers of two (exact) so that their
// largest magnitude lies in [2^11, 2^12), each as the sum of two FP16 values
// h + l (l the rounding error of h, itself rounded: 22 bits together); the
// dot product is h_x h_c + h_x l_c + l_x h_c, the last only when some l_x is
// not zero (byte-valued rows need one value).  With h alone the bound (2^-10
// of |x| |c|) left about ten centroids a row to re-score on SIFT-shaped data
// and the kernel took 472 us; with h + l the accumulation's bound is left and
// few rows have a second candidate.
//
// One CTA per SM, persistent over 128-row tiles: warp 0 loads operand boxes
// (TMA, 64 elements of K, 2 stages), warp 1 issues the MMAs (128 x 256 tiles
// into one of two TMEM accumulators), and 16 warps read an accumulator back
// while the next tile's MMAs run: a thread per row and quarter of the columns
// (four warps alone left the schedulers waiting for instructions and operands:
// 507 us).  Rows with one centroid left are decided there; the others are
// queued and k_assign_pairs re-scores their candidates, all chains of the
// assignment in flight at once.  131,072 x 128 byte-valued rows against 512
// centroids: 93 us and 12 us for the queued and leftover rows; on the FP32 cores 698 us
// (25 TFLOP/s).
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "index.cuh"
#include "tc.cuh"

namespace ksc {

constexpr int AT_STAGES = 2;
constexpr int AT_A = TC_M * 128, AT_B = TC_N * 128;    // bytes of a box of rows, of centroids
constexpr int AT_STAGE_BYTES = 2 * (AT_A + AT_B);      // h and l of the centroids, h and l of the rows
constexpr int AT_Q = 4;      // epilogue warps per 32 rows, each a quarter of a tile's columns
constexpr int AT_CAND = 7;   // candidate centroids kept per row and quarter
constexpr int AT_ROWC = 16;  // candidates of a queued row
constexpr int AT_THREADS = 64 + 32 * 4 * AT_Q;
constexpr size_t AT_SMEM = (size_t)AT_STAGES * AT_STAGE_BYTES + sizeof(float2) * AT_Q * AT_CAND * TC_M + 1024;
constexpr int AT_REDO_ROWS = 2048;  // leftover rows up to which a CTA takes each (more: the FP32 tile kernel)

struct AssignArgs {
    const float* X;      // [rows x d]
    const float* C;      // [L x d]
    const float* base;   // [L up to a multiple of 256] ||c||^2 (0 spherical), +inf past L
    const float* cn;     // [L] ||c||^2
    const float* xnorm;  // [rows] upper bound of the row's norm
    const uint32_t* c2max;  // bits of max ||c||^2
    int64_t rows;
    int d, L, KB, spherical;
    float mul;           // -2 (L2) or -1 over both operand scales
    float rel;           // relative bound of the dot product
    float subx, subc;    // absolute bounds per unit of the row's and of the centroids' norm (subnormal FP16)
    int32_t* assign;
    const int32_t* xlow; // whether some row has an l part
    int32_t* redo;       // [rows] rows for the FP32 kernel
    int32_t* nredo;
    int32_t* queue;      // [rows] rows with several candidates, qcand [rows x AT_ROWC] their ids (-1: none)
    int32_t* qcand;
    int32_t* nqueue;
    int32_t* status;
};

// A bounded wait that also ends when another warp of the CTA has given up.
__device__ __forceinline__ bool at_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    for (uint32_t i = 0; i < 64; ++i) {
        if (mbar_wait(bar, parity, TC_WAIT_LIMIT / 64)) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// The FP32 rule's score of row x and centroid c.
__device__ __forceinline__ float assign_score(const float* __restrict__ x, const float* __restrict__ c, int d,
                                              bool vec, float mul, float base) {
    float acc = 0.f;
    if (vec) {
#pragma unroll 4
        for (int t = 0; t < d; t += 4) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(x + t));
            const float4 b = __ldg(reinterpret_cast<const float4*>(c + t));
            acc = fmaf(a.x, b.x, acc);
            acc = fmaf(a.y, b.y, acc);
            acc = fmaf(a.z, b.z, acc);
            acc = fmaf(a.w, b.w, acc);
        }
    } else {
#pragma unroll 4
        for (int t = 0; t < d; ++t) acc = fmaf(__ldg(x + t), __ldg(c + t), acc);
    }
    return fmaf(mul, acc, base);
}

// Drops the entries of a row's full list that a better score has since
// excluded; the number left.
__device__ __noinline__ int at_drop(float2* mine, float thr) {
    int k = 0;
    for (int u = 0; u < AT_CAND; ++u) {
        const float2 x = mine[u * TC_M];
        if (x.x <= thr) mine[k++ * TC_M] = x;
    }
    return k;
}

__global__ void __launch_bounds__(AT_THREADS, 1)
    k_assign_tc(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapAl,
                const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapBl, AssignArgs G) {
    extern __shared__ __align__(1024) uint8_t at_raw[];
    __shared__ __align__(8) uint64_t bars[2 * AT_STAGES + 5];
    __shared__ uint32_t tmem_base;
    __shared__ volatile int s_abort;
    __shared__ int s_stop[4];             // the abort flag as the four warps of 32 rows all see it
    __shared__ float q_best[AT_Q][TC_M];  // a quarter's best score of a row
    __shared__ int q_n[AT_Q][TC_M];       // its candidates kept (-1: more than fit)
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(at_raw) + 1023) & ~uintptr_t(1023));
    float2* cand = reinterpret_cast<float2*>(smem + (size_t)AT_STAGES * AT_STAGE_BYTES);  // [quarter][slot][row] (score, id)
    const uint32_t sbase = smem_u32(smem);
    auto full = [&](int s) { return smem_u32(&bars[s]); };
    auto empty = [&](int s) { return smem_u32(&bars[AT_STAGES + s]); };
    auto tfull = [&](int b) { return smem_u32(&bars[2 * AT_STAGES + b]); };
    auto tempty = [&](int b) { return smem_u32(&bars[2 * AT_STAGES + 2 + b]); };
    const uint32_t drain = smem_u32(&bars[2 * AT_STAGES + 4]);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t ntiles = (G.rows + TC_M - 1) / TC_M;
    const int NT = (G.L + TC_N - 1) / TC_N;
    if (threadIdx.x == 0) {
        for (int s = 0; s < AT_STAGES; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull(b), 1);
            mbar_init(tempty(b), 4 * AT_Q);
        }
        mbar_init(drain, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(2 * TC_N));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    const bool xlow = *G.xlow != 0;
    if (warp == 0) {
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int64_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x)
                for (int nt = 0; ok && nt < NT; ++nt)
                    for (int kb = 0; kb < G.KB; ++kb, ++it) {
                        const int s = it % AT_STAGES;
                        ok = at_wait(empty(s), ((it / AT_STAGES) & 1) ^ 1, &s_abort);
                        if (!ok) break;
                        const uint32_t sB = sbase + s * AT_STAGE_BYTES, sA = sB + 2 * AT_B;
                        mbar_expect_tx(full(s), 2 * AT_B + (xlow ? 2 : 1) * AT_A);
                        tma_load_2d(sA, &mapA, full(s), kb * TC_KB, (int)(tile * TC_M));
                        tma_load_2d(sB, &mapB, full(s), kb * TC_KB, nt * TC_N);
                        tma_load_2d(sB + AT_B, &mapBl, full(s), kb * TC_KB, nt * TC_N);
                        if (xlow) tma_load_2d(sA + AT_A, &mapAl, full(s), kb * TC_KB, (int)(tile * TC_M));
                    }
            if (!ok)  // given up: the copies in flight land before the CTA ends
                for (uint32_t i = it > AT_STAGES ? it - AT_STAGES : 0; i < it; ++i)
                    mbar_wait(full(i % AT_STAGES), (i / AT_STAGES) & 1, TC_WAIT_LIMIT);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            uint32_t it = 0, at = 0;
            bool ok = true;
            const uint32_t idesc = idesc_f16kind(0, TC_M, TC_N);
            for (int64_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x)
                for (int nt = 0; ok && nt < NT; ++nt, ++at) {
                    const int b = at & 1;
                    ok = at_wait(tempty(b), ((at >> 1) & 1) ^ 1, &s_abort);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    for (int kb = 0; kb < G.KB; ++kb, ++it) {
                        const int s = it % AT_STAGES;
                        ok = at_wait(full(s), (it / AT_STAGES) & 1, &s_abort);
                        if (!ok) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t sB = sbase + s * AT_STAGE_BYTES, sA = sB + 2 * AT_B;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            tc_mma(tmem + b * TC_N, smem_desc(sA + k * 32), smem_desc(sB + k * 32), idesc,
                                   (kb | k) != 0);
                            tc_mma(tmem + b * TC_N, smem_desc(sA + k * 32), smem_desc(sB + AT_B + k * 32), idesc, 1);
                            if (xlow)
                                tc_mma(tmem + b * TC_N, smem_desc(sA + AT_A + k * 32), smem_desc(sB + k * 32), idesc, 1);
                        }
                        tc_commit(empty(s));
                    }
                    if (ok) tc_commit(tfull(b));
                }
            if (!ok) {  // given up: the MMAs in flight end before TMEM is freed
                atomicOr(G.status, 2);
                tc_commit(drain);
                mbar_wait(drain, 0, TC_WAIT_LIMIT);
            }
        }
    } else {
        const int sub = warp & 3;          // the TMEM lanes a warp may read: 32 (warp % 4) ..
        const int quarter = (warp - 2) >> 2;
        const int row = sub * 32 + lane;
        const float cmax = sqrtf(__uint_as_float(*G.c2max)) * 1.0001f;
        float2* mine = cand + (size_t)quarter * AT_CAND * TC_M + row;
        uint32_t at = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
            const int64_t r = tile * TC_M + row;
            const bool in = r < G.rows;
            // twice the bound on |tensor-core score - FP32 score| of this row
            float e2;
            {
                const float xn = in ? G.xnorm[r] : 0.f;
                const float dot = (G.rel * xn * cmax + G.subx * xn + G.subc * cmax) * 1.0001f;
                const float rnd = (float)(G.d + 8) * 1.2e-7f * (xn + cmax) * (xn + cmax);
                e2 = 2.f * ((G.spherical ? dot : 2.f * dot) + rnd);
            }
            float best = INFINITY, thr = INFINITY;
            int n = 0;
            bool over = false;
            for (int nt = 0; ok && nt < NT; ++nt, ++at) {
                const int b = at & 1;
                ok = __all_sync(0xffffffffu, at_wait(tfull(b), (at >> 1) & 1, &s_abort));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int cq = quarter * (TC_N / AT_Q);
                const int cols = min(TC_N / AT_Q, G.L - nt * TC_N - cq);
                const float* bs = G.base + nt * TC_N + cq;
#pragma unroll 1
                for (int c0 = 0; c0 < cols; c0 += 16) {
                    uint32_t v[16];
                    __syncwarp();  // tcgen05.ld is a warp-collective instruction
                    tmem_ld16(tmem + b * TC_N + ((uint32_t)(sub * 32) << 16) + cq + c0, v);
                    float s[16], m = INFINITY;
#pragma unroll
                    for (int i = 0; i < 16; i += 4) {
                        const float4 bb = __ldg(reinterpret_cast<const float4*>(bs + c0 + i));
                        s[i] = fmaf(G.mul, __uint_as_float(v[i]), bb.x);
                        s[i + 1] = fmaf(G.mul, __uint_as_float(v[i + 1]), bb.y);
                        s[i + 2] = fmaf(G.mul, __uint_as_float(v[i + 2]), bb.z);
                        s[i + 3] = fmaf(G.mul, __uint_as_float(v[i + 3]), bb.w);
                        m = fminf(fminf(m, fminf(s[i], s[i + 1])), fminf(s[i + 2], s[i + 3]));
                    }
                    if (m <= thr) {
                        if (m < best) {
                            best = m;
                            thr = __fadd_ru(best, e2);
                        }
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (s[i] <= thr) {
                                if (n == AT_CAND) n = at_drop(mine, thr);
                                if (n < AT_CAND)
                                    mine[n++ * TC_M] = make_float2(s[i], __int_as_float(nt * TC_N + cq + c0 + i));
                                else
                                    over = true;
                            }
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty(b));
            }
            // (a warp that gave up still takes part in this tile's barriers; then
            // all four stop together)
            q_best[quarter][row] = best;
            q_n[quarter][row] = over ? -1 : n;
            __syncwarp();  // bar.sync is a warp-collective instruction
            asm volatile("bar.sync %0, %1;" ::"r"(1 + sub), "n"(32 * AT_Q) : "memory");  // the four warps of these rows
            if (quarter == 0 && lane == 0) s_stop[sub] = s_abort;
            if (quarter == 0 && in && ok) {
                float bt = best;
#pragma unroll
                for (int u = 1; u < AT_Q; ++u) bt = fminf(bt, q_best[u][row]);
                const float th = __fadd_ru(bt, e2);
                // the centroids that the bound cannot exclude
                int k = 0, first = -1;
                bool many = false;
                int32_t* qc = nullptr;
#pragma unroll 1
                for (int u = 0; u < AT_Q; ++u) {
                    if (!(q_best[u][row] <= th)) continue;  // (a quarter past the last centroid holds none)
                    const int nu = q_n[u][row];
                    many |= nu < 0;
                    for (int i = 0; i < nu; ++i) {
                        const float2 x = cand[((size_t)u * AT_CAND + i) * TC_M + row];
                        if (!(x.x <= th)) continue;
                        if (k == 0) {
                            first = __float_as_int(x.y);
                        } else {
                            if (k == 1) {
                                const int slot = atomicAdd(G.nqueue, 1);
                                G.queue[slot] = (int32_t)r;
                                qc = G.qcand + (int64_t)slot * AT_ROWC;
                                for (int j = 0; j < AT_ROWC; ++j) qc[j] = -1;
                                qc[0] = first;
                            }
                            if (k < AT_ROWC) qc[k] = __float_as_int(x.y);
                        }
                        ++k;
                    }
                }
                // too many candidates (or none: a NaN): the FP32 kernel
                if (many || k == 0 || k > AT_ROWC) G.redo[atomicAdd(G.nredo, 1)] = (int32_t)r;
                else if (k == 1) G.assign[r] = first;
            }
            __syncwarp();
            asm volatile("bar.sync %0, %1;" ::"r"(1 + sub), "n"(32 * AT_Q) : "memory");  // before the lists are reused
            ok = s_stop[sub] == 0;
        }
        if (!ok && lane == 0) atomicOr(G.status, 2);
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * TC_N));
}

// The rows with several candidates, by the FP32 rule: a thread per candidate,
// AT_ROWC threads per row.  A row that is also on the redo list is settled
// again there.
__global__ void __launch_bounds__(128) k_assign_pairs(AssignArgs G) {
    const int64_t p = (int64_t)blockIdx.x * (128 / AT_ROWC) + threadIdx.x / AT_ROWC;
    const int lane = threadIdx.x & 31, u = threadIdx.x % AT_ROWC;
    const int64_t n = *G.nqueue;
    const bool vec = (G.d & 3) == 0;
    for (int64_t q = p; q - threadIdx.x / AT_ROWC < n; q += (int64_t)gridDim.x * (128 / AT_ROWC)) {  // CTA-uniform
        const bool in = q < n;
        const int64_t r = in ? G.queue[q] : 0;
        const int c = in ? G.qcand[q * AT_ROWC + u] : -1;
        uint64_t key = KEY_NONE;
        if (c >= 0) {
            const float s = assign_score(G.X + r * G.d, G.C + (int64_t)c * G.d, G.d, vec, G.spherical ? -1.f : -2.f,
                                         G.spherical ? 0.f : __ldg(G.cn + c));
            // (+ 0: a score of -0 orders as +0, a tie)
            key = ((uint64_t)ordered_f32(s + 0.f) << 32) | (uint32_t)c;
        }
#pragma unroll
        for (int o = AT_ROWC / 2; o > 0; o >>= 1) {
            const uint64_t y = __shfl_xor_sync(0xffffffffu, key, o);
            key = y < key ? y : key;
        }
        if (in && (lane % AT_ROWC) == 0) G.assign[r] = (int32_t)(key & 0xffffffffu);
    }
}

// The leftover rows (up to AT_REDO_ROWS; the caller's tile kernel takes more),
// every centroid by the FP32 rule: a CTA per row, a thread per centroid.
__global__ void __launch_bounds__(256) k_assign_left(AssignArgs G) {
    __shared__ unsigned long long s_best;
    const int n = *G.nredo;
    if (n > AT_REDO_ROWS) return;
    const bool vec = (G.d & 3) == 0;
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        const int64_t r = G.redo[i];
        if (threadIdx.x == 0) s_best = ((unsigned long long)ordered_f32(INFINITY) << 32) | 0x7fffffffu;
        __syncthreads();
        for (int c = threadIdx.x; c < G.L; c += 256) {
            const float s = assign_score(G.X + r * G.d, G.C + (int64_t)c * G.d, G.d, vec, G.spherical ? -1.f : -2.f,
                                         G.spherical ? 0.f : __ldg(G.cn + c));
            if (s < INFINITY) atomicMin(&s_best, ((unsigned long long)ordered_f32(s + 0.f) << 32) | (uint32_t)c);
        }
        __syncthreads();
        if (threadIdx.x == 0) G.assign[r] = (int32_t)(s_best & 0xffffffffu);
        __syncthreads();
    }
}

// v (scaled) as FP16 h + l.
__device__ __forceinline__ void split16(float v, __half& h, __half& l) {
    h = __float2half_rn(v);
    l = __float2half_rn(v - __half2float(h));  // the difference is exact
}

// Rows of X [n x d] to FP16 operands h, l [n x Kp] (times scale, zero-padded K)
// and upper bounds of their norms; *low is set if some l is not zero.  A warp
// per row.
__global__ void k_rows16(const float* __restrict__ X, int64_t n, int d, int Kp, float scale, __half* __restrict__ oh,
                         __half* __restrict__ ol, float* __restrict__ norm, int32_t* __restrict__ low) {
    const int lane = threadIdx.x & 31;
    const int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= n) return;
    float s = 0.f;
    bool any = false;
    for (int t = 2 * lane; t < Kp; t += 64) {
        const float a = t < d ? X[r * d + t] : 0.f, b = t + 1 < d ? X[r * d + t + 1] : 0.f;
        s = fmaf(a, a, fmaf(b, b, s));
        __half2 h, l;
        split16(a * scale, h.x, l.x);
        split16(b * scale, h.y, l.y);
        *reinterpret_cast<__half2*>(oh + r * Kp + t) = h;
        *reinterpret_cast<__half2*>(ol + r * Kp + t) = l;
        any |= __half2float(l.x) != 0.f || __half2float(l.y) != 0.f;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    any = __any_sync(0xffffffffu, any);
    if (lane == 0) {
        norm[r] = sqrtf(s) * 1.0001f;
        if (any) *low = 1;
    }
}

// Largest magnitude of X [m], as bits (a NaN's are above infinity's).
__global__ void k_max_abs(const float* __restrict__ X, int64_t m, uint32_t* __restrict__ out) {
    uint32_t v = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        v = max(v, __float_as_uint(X[i]) & 0x7fffffffu);
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicMax(out, v);
}

// Centroids for the next assignment, 8 per CTA: the mean of their rows' sums
// (sums != NULL: FP64, cleared for the next round; one without rows keeps its
// value), ||c||^2 by FMAs over ascending dimensions (k_row_sqnorm's order), the
// epilogue's base scores, the FP16 operands and max ||c||^2.
__global__ void __launch_bounds__(256) k_centroid_prep(double* __restrict__ sums, unsigned long long* __restrict__ cnt,
                                                       float* __restrict__ C, int L, int d, int Kp, float scale,
                                                       int spherical, __half* __restrict__ C16,
                                                       __half* __restrict__ C16l, float* __restrict__ cn,
                                                       float* __restrict__ base, int Lpad,
                                                       uint32_t* __restrict__ c2max) {
    constexpr int CP = 8;
    __shared__ float tile[CP][129];
    const int c0 = blockIdx.x * CP;
    const int lane = threadIdx.x & 31;
    float s = 0.f;
    for (int k0 = 0; k0 < Kp; k0 += 128) {
        for (int e = threadIdx.x; e < CP * 128; e += 256) {
            const int r = e >> 7, t = k0 + (e & 127), c = c0 + r;
            float v = 0.f;
            if (c < L && t < d) {
                const int64_t at = (int64_t)c * d + t;
                if (sums) {
                    const unsigned long long n = cnt[c];
                    v = n > 0 ? (float)(sums[at] / (double)n) : C[at];
                    C[at] = v;
                    sums[at] = 0.0;
                } else {
                    v = C[at];
                }
            }
            tile[r][e & 127] = v;
            if (c < L && t < Kp) split16(v * scale, C16[(int64_t)c * Kp + t], C16l[(int64_t)c * Kp + t]);
        }
        __syncthreads();
        if (threadIdx.x < CP) {
            const int m = min(128, d - k0);
#pragma unroll 8
            for (int t = 0; t < m; ++t) s = fmaf(tile[lane][t], tile[lane][t], s);
        }
        __syncthreads();
    }
    if (threadIdx.x < 32) {
        const int c = c0 + lane;
        const bool in = lane < CP && c < L;
        if (in) {
            cn[c] = s;
            if (sums) cnt[c] = 0ull;
        }
        if (lane < CP && c < Lpad) base[c] = in ? (spherical ? 0.f : s) : INFINITY;
        const uint32_t m = __reduce_max_sync(0xffffffffu, in ? __float_as_uint(s) : 0u);
        if (lane == 0) atomicMax(c2max, m);
    }
}

static float pow2_scale(float mx) {  // mx * scale in [2^11, 2^12)
    if (!(mx > 0.f)) return 1.f;
    int e;
    std::frexp(mx, &e);  // mx = m 2^e, m in [1/2, 1)
    return std::ldexp(1.f, 12 - e);
}

int max_abs(const float* X, int64_t m, float* out, cudaStream_t st) {
    uint32_t* bits = nullptr;
    uint32_t h = 0;
    KSC_CUDA(cudaMalloc(&bits, sizeof(uint32_t)));
    cudaError_t e = cudaMemsetAsync(bits, 0, sizeof(uint32_t), st);
    if (e == cudaSuccess) {
        k_max_abs<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>((m + 1023) / 1024, 8 * (int64_t)num_sms())), 256, 0,
                    st>>>(X, m, bits);
        e = cudaMemcpyAsync(&h, bits, sizeof(h), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    cudaFree(bits);
    KSC_CUDA(e);
    memcpy(out, &h, sizeof(float));
    return KSC_OK;
}

bool assign_tc_supported(float xmax) { return xmax == 0.f || (xmax > 1e-12f && xmax < 1e15f); }

// Operands and scratch of assignments of up to `rows` rows to L centroids.
int AssignTc::init(int64_t rows_, int d_, int L_, float xmax, cudaStream_t st) {
    rows = rows_;
    d = d_;
    L = L_;
    Kp = (d + TC_KB - 1) / TC_KB * TC_KB;
    Lpad = (L + TC_N - 1) / TC_N * TC_N;
    xscale = pow2_scale(xmax);
    KSC_CUDA(cudaMalloc(&x16, sizeof(__half) * 2 * (size_t)rows * Kp));  // h, then l
    KSC_CUDA(cudaMalloc(&c16, sizeof(__half) * 2 * (size_t)L * Kp));
    KSC_CUDA(cudaMalloc(&xnorm, sizeof(float) * rows));
    KSC_CUDA(cudaMalloc(&cn, sizeof(float) * L));
    KSC_CUDA(cudaMalloc(&base, sizeof(float) * Lpad));
    KSC_CUDA(cudaMalloc(&redo, sizeof(int32_t) * (size_t)rows * (2 + AT_ROWC)));  // redo, queue, qcand
    // redo and queue counts, max ||c||^2, status, l part of the rows
    KSC_CUDA(cudaMalloc(&small, sizeof(int32_t) * 8));
    KSC_CUDA(cudaMemsetAsync(small, 0, sizeof(int32_t) * 8, st));
    return KSC_OK;
}

void AssignTc::free() {
    void* p[] = {x16, c16, xnorm, cn, base, redo, small};
    for (void* q : p)
        if (q) cudaFree(q);
    x16 = c16 = nullptr;
    xnorm = cn = base = nullptr;
    redo = small = nullptr;
}

int AssignTc::set_rows(const float* X_, int64_t n, cudaStream_t st) {
    X = X_;
    nrows = n;
    k_rows16<<<(unsigned)((n + 7) / 8), 256, 0, st>>>(X, n, d, Kp, xscale, (__half*)x16, (__half*)x16 + rows * Kp,
                                                      xnorm, small + 4);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

int AssignTc::set_centroids(float* C_, double* sums, unsigned long long* cnt, bool spherical_, float cmax_abs,
                            cudaStream_t st) {
    C = C_;
    spherical = spherical_;
    cscale = pow2_scale(cmax_abs);
    KSC_CUDA(cudaMemsetAsync(small, 0, sizeof(int32_t) * 3, st));
    k_centroid_prep<<<Lpad / 8, 256, 0, st>>>(sums, cnt, C_, L, d, Kp, cscale, spherical, (__half*)c16,
                                              (__half*)c16 + (size_t)L * Kp, cn, base, Lpad, (uint32_t*)small + 2);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

int AssignTc::redo_rows() { return AT_REDO_ROWS; }

int AssignTc::run(int32_t* assign, cudaStream_t st) {
    CUtensorMap mapA, mapAl, mapB, mapBl;
    KSC_TRY(make_map(&mapA, x16, nrows, Kp, TC_M, true));
    KSC_TRY(make_map(&mapAl, (__half*)x16 + rows * Kp, nrows, Kp, TC_M, true));
    KSC_TRY(make_map(&mapB, c16, L, Kp, TC_N, true));
    KSC_TRY(make_map(&mapBl, (__half*)c16 + (size_t)L * Kp, L, Kp, TC_N, true));
    AssignArgs G{};
    G.X = X;
    G.C = C;
    G.base = base;
    G.cn = cn;
    G.xnorm = xnorm;
    G.c2max = (const uint32_t*)small + 2;
    G.rows = nrows;
    G.d = d;
    G.L = L;
    G.KB = Kp / TC_KB;
    G.spherical = spherical;
    G.mul = (spherical ? -1.f : -2.f) / (xscale * cscale);
    // the rounding of both l parts and the missing l_x l_c (2^-22 each of |x|
    // |c|), and the FP32 accumulation, as for the list ranking's 16-bit scores
    G.rel = 1e-6f + (float)d * 4.8e-7f;
    // an element whose l falls below FP16's normal range: up to 2^-25 (scaled),
    // whatever its size, against the other operand's elements: 2^-25 sqrt(d)
    // of its norm
    const float sub = 0x1p-25f * std::sqrt((float)d) * 1.01f;
    G.subx = sub / cscale;
    G.subc = sub / xscale;
    G.assign = assign;
    G.xlow = small + 4;
    G.redo = redo;
    G.nredo = small;
    G.queue = redo + rows;
    G.qcand = redo + 2 * rows;
    G.nqueue = small + 1;
    G.status = small + 3;
    KSC_CUDA(cudaFuncSetAttribute(k_assign_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AT_SMEM));
    const int64_t tiles = (nrows + TC_M - 1) / TC_M;
    k_assign_tc<<<(unsigned)std::min<int64_t>(tiles, num_sms()), AT_THREADS, AT_SMEM, st>>>(mapA, mapAl, mapB, mapBl, G);
    k_assign_pairs<<<num_sms() * 8, 128, 0, st>>>(G);
    k_assign_left<<<num_sms() * 4, 256, 0, st>>>(G);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

// KSC_ETIMEOUT if a bounded wait of an assignment gave up.  Blocking.
int AssignTc::check(cudaStream_t st) {
    int32_t h = 0;
    KSC_CUDA(cudaMemcpyAsync(&h, small + 3, sizeof(h), cudaMemcpyDeviceToHost, st));
    KSC_CUDA(cudaStreamSynchronize(st));
    if (h) {
        set_error("assignment on the tensor cores: an operand copy or MMA never completed");
        return KSC_ETIMEOUT;
    }
    return KSC_OK;
}

}  // namespace ksc
