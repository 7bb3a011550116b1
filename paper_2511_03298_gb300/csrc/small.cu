// Searches of a few queries: a query's whole way is a chain of dependent
// kernels, and at one query each of the general path's 14 kernels and 5 memsets
// costs 3 to 12 us of launch, fill and drain for work of well under 1 us (97 us
// for one query of 1M x 128 at nprobe 7).  Here a cluster of 8 CTAs takes a
// query through ranking, tables and scan items in one kernel, and a CTA takes
// it through selection and re-rank in one more; between them run the scan, and
// the threshold with a second scan only when a query may probe more keys than
// the store holds.
#include <cooperative_groups.h>

#include "rerank.cuh"
#include "small.cuh"

namespace cg = cooperative_groups;

namespace ksc {

constexpr int SP_CL = 8;        // CTAs per query
constexpr int SP_T = 256;       // threads per CTA
constexpr int SP_ROWS = 4096;   // table rows whose minima are held at once

static size_t small_prep_smem(const SmallPrep& S) {
    const LutArgs& T = S.T;
    return sizeof(float) * ((((size_t)T.d + 3) & ~(size_t)3) + (((size_t)T.M * cb_ld(T.dsub) + 3) & ~(size_t)3) + SP_ROWS) +
           sizeof(int32_t) * (((size_t)T.Pmax + 3) & ~(size_t)3) +
           (S.c_rank ? sizeof(uint64_t) * ((size_t)T.L + SP_RANK_P) : 0);
}

// The lists [c0, c1) of one CTA, scored exactly (exact_list_score's operations
// and order, 8 lists in flight per warp when a row fits a warp's 16-byte
// loads), as keys into the leader's shared memory.
__device__ __forceinline__ void score_lists(const SmallPrep& S, const float* qs, int c0, int c1, uint64_t* lk) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, d = S.T.d;
    if ((d & 3) == 0 && d <= 128) {
        const bool inl = lane * 4 < d;
        const float4 qv = inl ? *reinterpret_cast<const float4*>(qs + lane * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
        const int myrow = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
        for (int i0 = c0 + 8 * w; i0 < c1; i0 += 8 * (SP_T / 32)) {
            float4 cv[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                cv[u] = inl && i0 + u < c1 ? __ldg(reinterpret_cast<const float4*>(S.c_rank + (int64_t)(i0 + u) * d) + lane)
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
            float a[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (S.spherical) {
                    a[u] = fmaf(qv.w, cv[u].w, fmaf(qv.z, cv[u].z, fmaf(qv.y, cv[u].y, qv.x * cv[u].x)));
                } else {
                    const float e0 = qv.x - cv[u].x, e1 = qv.y - cv[u].y, e2 = qv.z - cv[u].z, e3 = qv.w - cv[u].w;
                    a[u] = inl ? fmaf(e3, e3, fmaf(e2, e2, fmaf(e1, e1, e0 * e0))) : 0.f;
                }
            }
            const float s = exchange_rows8(a, lane);
            const int c = i0 + myrow;
            if ((lane & 3) == 0 && c < c1) lk[c] = ((uint64_t)ordered_f32(S.spherical ? -s : s) << 32) | (uint32_t)c;
        }
    } else {
        for (int c = c0 + w; c < c1; c += SP_T / 32) {
            const float s = exact_list_score(qs, S.c_rank + (int64_t)c * d, d, S.spherical, lane);
            if (lane == 0) lk[c] = ((uint64_t)ordered_f32(s) << 32) | (uint32_t)c;
        }
    }
}

// Scan items of one query (by one CTA): the end of the unfiltered part (the
// rule of k_count_parts), the places of its pairs in the store, and a record
// per tile of every probed list.  Each thread takes 4 consecutive ranks.
__device__ void query_items(const SmallPrep& S, int64_t q, const int32_t* prb, int P) {
    __shared__ uint32_t tot[32];
    __shared__ int s_split, s_base[2];
    const ScanArgs& A = S.A;
    const int r0 = 4 * threadIdx.x;
    int n[4];
    uint32_t mine = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        n[u] = r0 + u < P ? (int)list_size(A, prb[r0 + u]) : 0;
        mine += n[u];
    }
    const uint32_t before = block_exclusive_scan(mine, tot);
    if (threadIdx.x == SP_T - 1) s_base[0] = (int)(before + mine);
    if (threadIdx.x == 0) s_split = P;
    __syncthreads();
    const uint32_t total = (uint32_t)s_base[0];
    if (!S.all_near) {
        long long target = (long long)S.near_keys_per_r * rerank_of(A.rerank_q, A.Rfix, A.Rmin, S.Rmax, q);
        target = max(target, (long long)total / S.near_share_div);
        target = min(target, (long long)S.cap / 2);
        long long b = before;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = r0 + u;
            if (r > 0 && r < P && (b >= target || b + n[u] > S.cap)) {
                atomicMin(&s_split, r);
                break;
            }
            b += n[u];
        }
        __syncthreads();
    }
    const int split = s_split;
    uint32_t ta = 0, tb = 0, nearn = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int nb = (n[u] + 31) >> 5;
        if (r0 + u < split) {
            ta += (nb + S.TBa - 1) / S.TBa;
            nearn += n[u];
        } else {
            tb += (nb + S.TB - 1) / S.TB;
        }
    }
    const uint32_t oa = block_exclusive_scan(ta, tot);
    const uint32_t ob = block_exclusive_scan(tb, tot);
    const uint32_t on = block_exclusive_scan(nearn, tot);
    if (threadIdx.x == SP_T - 1) {
        s_base[0] = atomicAdd(&S.nrec[0], (int)(oa + ta));
        s_base[1] = atomicAdd(&S.nrec[1], (int)(ob + tb));
        S.cnt[q] = (int)(on + nearn);
    }
    __syncthreads();
    int ia = s_base[0] + (int)oa, ib = s_base[1] + (int)ob;
    uint32_t at = before;
    for (int u = 0; u < 4; ++u) {
        const int r = r0 + u;
        if (r >= P) break;
        const int e = (int)(q * A.Pmax + r), p = prb[r];
        const int nb = (n[u] + 31) >> 5;
        const bool near = r < split;
        const int nt = near ? (nb + S.TBa - 1) / S.TBa : (nb + S.TB - 1) / S.TB;
        if (near) S.noff[e] = (int)at;
        at += n[u];
        int4* out = near ? S.recsA + ia : S.recsB + ib;
        for (int t = 0; t < nt; ++t)
            out[t] = make_int4(e, (int)((int64_t)t * nb / nt), (int)((int64_t)(t + 1) * nb / nt), p);
        if (near) ia += nt;
        else ib += nt;
    }
    __syncthreads();
}

template <int DS>
__global__ void __cluster_dims__(SP_CL, 1, 1) __launch_bounds__(SP_T) k_small_prep(SmallPrep S) {
    extern __shared__ __align__(16) unsigned char sp_raw[];
    __shared__ uint32_t s_range, s_r, hist[256];
    __shared__ uint64_t bb[32];
    cg::cluster_group cl = cg::this_cluster();
    const int cr = (int)cl.block_rank();
    const LutArgs& T = S.T;
    const int64_t q = blockIdx.x / SP_CL;
    const int M = T.M, ld = cb_ld(T.dsub);
    float* qs = reinterpret_cast<float*>(sp_raw);
    float* cbs = qs + ((T.d + 3) & ~3);
    float* mins = cbs + ((M * ld + 3) & ~3);
    int32_t* prb = reinterpret_cast<int32_t*>(mins + SP_ROWS);
    uint64_t* keys = reinterpret_cast<uint64_t*>(prb + ((T.Pmax + 3) & ~3));  // (ranking) L list keys
    uint64_t* top = keys + T.L;                                               // and the P best
    const int P = probes_of(T, q);
    if (threadIdx.x == 0) {
        s_range = 0u;
        s_r = 0u;
    }
    for (int t = threadIdx.x; t < T.d; t += SP_T) qs[t] = T.Q[q * T.d + t];
    if (!S.c_rank)
        for (int r = threadIdx.x; r < P; r += SP_T) prb[r] = T.probes[q * T.Pmax + r];
    stage_codebook(T, cbs);  // ends with __syncthreads
    cl.sync();  // every CTA of the cluster runs: the leader's shared memory may be written
    if (S.c_rank) {
        const int Lc = (T.L + SP_CL - 1) / SP_CL;
        score_lists(S, qs, min(cr * Lc, T.L), min((cr + 1) * Lc, T.L), cl.map_shared_rank(keys, 0));
        cl.sync();
        if (cr == 0) {
            auto load = [&](int c) -> uint64_t { return keys[c]; };
            auto emit = [&](int i, uint64_t k) { top[i] = k; };
            const int K = min(P, T.L);
            if (K < T.L) block_topk(load, T.L, K, emit, hist, bb);
            else for (int c = threadIdx.x; c < K; c += SP_T) top[c] = keys[c];
            __syncthreads();
            for (int i = threadIdx.x; i < T.Pmax; i += SP_T) {
                int r = i;
                int32_t p = -1;
                if (i < K) {  // ranked by counting the smaller keys
                    const uint64_t k = top[i];
                    r = 0;
                    for (int j = 0; j < K; ++j) r += top[j] < k;
                    p = (int32_t)(k & 0xffffffffu);
                }
                prb[r] = p;
                S.probes_out[q * T.Pmax + r] = p;
            }
        }
        cl.sync();
        if (cr != 0) {
            const int32_t* lp = cl.map_shared_rank(prb, 0);
            for (int r = threadIdx.x; r < P; r += SP_T) prb[r] = lp[r];
            __syncthreads();
        }
    }
    if (cr == SP_CL - 1) query_items(S, q, prb, P);
    // tables of ranks cr, cr + 8, ...: the largest row range of the query first
    const int nr = P > cr ? (P - cr + SP_CL - 1) / SP_CL : 0;
    float R = 0.f;
    for (int row = threadIdx.x; row < nr * M; row += SP_T) {
        const int i = row / M, j = row - i * M, p = prb[cr + i * SP_CL];
        if (p < 0 || p >= T.L) continue;
        float Tv[PQ_K];
        row_table<DS>(T.dsub, T.ip, qs + j * T.dsub, T.c_mean + (int64_t)p * T.d + j * T.dsub, cbs + j * ld, Tv);
        float mn = Tv[0], mx = Tv[0];
#pragma unroll
        for (int c = 1; c < PQ_K; ++c) {
            mn = fminf(mn, Tv[c]);
            mx = fmaxf(mx, Tv[c]);
        }
        R = fmaxf(R, __fsub_rn(mx, mn));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) R = fmaxf(R, __shfl_xor_sync(0xffffffffu, R, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&s_r, __float_as_uint(R));
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(cl.map_shared_rank(&s_range, 0), s_r);
    cl.sync();
    const float Rq = __uint_as_float(*cl.map_shared_rank(&s_range, 0));
    const float a = (Rq == 0.f) ? 1.f : __fdiv_rn(255.f, Rq);
    const int group = SP_ROWS / M;
    for (int i0 = 0; i0 < nr; i0 += group) {
        const int ng = min(group, nr - i0);
        for (int row = threadIdx.x; row < ng * M; row += SP_T) {
            const int i = row / M, j = row - i * M, r = cr + (i0 + i) * SP_CL, p = prb[r];
            if (p < 0 || p >= T.L) continue;
            float Tv[PQ_K];
            row_table<DS>(T.dsub, T.ip, qs + j * T.dsub, T.c_mean + (int64_t)p * T.d + j * T.dsub, cbs + j * ld, Tv);
            float mn = Tv[0];
#pragma unroll
            for (int c = 1; c < PQ_K; ++c) mn = fminf(mn, Tv[c]);
            reinterpret_cast<uint4*>(S.lut + (q * T.Pmax + r) * (int64_t)M * PQ_K)[j] =
                make_uint4(quant4(Tv, mn, a), quant4(Tv + 4, mn, a), quant4(Tv + 8, mn, a), quant4(Tv + 12, mn, a));
            mins[row] = mn;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < ng; i += SP_T) {
            const int r = cr + (i0 + i) * SP_CL, p = prb[r];
            if (p >= 0 && p < T.L)
                S.bias[q * T.Pmax + r] = lut_bias(T, qs, T.c_mean + (int64_t)p * T.d, mins + i * M, a);
        }
        __syncthreads();
    }
    if (cr == 0 && threadIdx.x == 0) S.scale[q] = a;
    cl.sync();  // the leader's shared memory has been read
}

int launch_small_prep(const SmallPrep& S, cudaStream_t st) {
    const size_t smem = small_prep_smem(S);
    auto kern = S.T.dsub == 2 ? k_small_prep<2> : k_small_prep<0>;
    KSC_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<(unsigned)(S.T.nq * SP_CL), SP_T, smem, st>>>(S);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

// block_topk on keys held in registers: thread t has key t + u NT in kk[u]
// (KEY_NONE past N).
template <int NT, int U, class Emit>
__device__ void block_topk_regs(const uint64_t (&kk)[U], int N, int K, Emit emit, uint32_t* hist, uint64_t* bb) {
    __shared__ unsigned long long s_lo, s_hi;
    __shared__ int s_B, s_lt, s_inB, s_out, s_nb;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        s_lo = KEY_NONE;
        s_hi = 0ull;
        s_out = 0;
    }
    __syncthreads();
    uint64_t lo = KEY_NONE, hi = 0ull;
#pragma unroll
    for (int u = 0; u < U; ++u)
        if ((int)threadIdx.x + u * NT < N) {
            lo = kk[u] < lo ? kk[u] : lo;
            hi = kk[u] > hi ? kk[u] : hi;
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t a = __shfl_xor_sync(0xffffffffu, lo, o), b = __shfl_xor_sync(0xffffffffu, hi, o);
        lo = a < lo ? a : lo;
        hi = b > hi ? b : hi;
    }
    if (lane == 0) {
        atomicMin(&s_lo, (unsigned long long)lo);
        atomicMax(&s_hi, (unsigned long long)hi);
    }
    __syncthreads();
    lo = s_lo;
    hi = s_hi;
    int need = K;
    while (true) {
        const uint64_t width = hi - lo;
        const int shift = width < 256ull ? 0 : 56 - __clzll((long long)width);  // least with width >> shift < 256
        for (int b = threadIdx.x; b < 256; b += NT) hist[b] = 0u;
        if (threadIdx.x == 0) s_nb = 0;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < U; ++u)
            if ((int)threadIdx.x + u * NT < N && kk[u] >= lo && kk[u] <= hi)
                atomicAdd(&hist[(uint32_t)((kk[u] - lo) >> shift)], 1u);
        __syncthreads();
        if (threadIdx.x < 32) {
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
            if (excl < (uint32_t)need && (uint32_t)need <= incl) {
                uint32_t acc = excl;
                int B = -1;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (B < 0 && acc + c[j] >= (uint32_t)need) {
                        B = 8 * lane + j;
                        s_B = B;
                        s_lt = (int)acc;
                        s_inB = (int)c[j];
                    }
                    acc += c[j];
                }
            }
        }
        __syncthreads();
        const int lt = s_lt, inB = s_inB;
        const uint64_t blo = lo + ((uint64_t)s_B << shift);
        const uint64_t bhi = (hi - blo < (1ull << shift)) ? hi : blo + ((1ull << shift) - 1ull);
        const bool last = inB <= 32;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if ((int)threadIdx.x + u * NT >= N) break;
            if (kk[u] >= lo && kk[u] < blo) emit(atomicAdd(&s_out, 1), kk[u]);
            else if (last && kk[u] >= blo && kk[u] <= bhi) bb[atomicAdd(&s_nb, 1)] = kk[u];
        }
        __syncthreads();
        need -= lt;
        if (last) {
            if (threadIdx.x < 32) {
                const uint64_t v = warp_sort_key(lane < inB ? bb[lane] : KEY_NONE, lane);
                if (lane < need) emit(s_out + lane, v);
            }
            __syncthreads();
            return;
        }
        lo = blo;
        hi = bhi;
    }
}

template <int NT>
__global__ void __launch_bounds__(NT) k_select_rerank(ScanArgs A, int Rmax, const int32_t* __restrict__ cnt,
                                                      const uint64_t* __restrict__ cand, int cap, int nkeys,
                                                      int sel_cap, const float* __restrict__ Q,
                                                      const float* __restrict__ X, int d, int ip, int k,
                                                      int64_t* __restrict__ out_ids, float* __restrict__ out_d,
                                                      int32_t* __restrict__ status,
                                                      unsigned long long* __restrict__ stats) {
    extern __shared__ uint64_t sr_keys[];  // nkeys (at least Rmax; sel_cap when a store may overflow), then k
    __shared__ uint32_t hist[256];
    __shared__ uint64_t bb[32];
    __shared__ __align__(16) float qs[KSC_MAX_DIM];
    __shared__ int32_t s_pref[SP_MAX_P + 1];
    constexpr int U = SP_REG_KEYS / NT;
    const int64_t q = blockIdx.x;
    const int R = rerank_of(A.rerank_q, A.Rfix, A.Rmin, Rmax, q);
    const int n = cnt[q];
    const uint64_t* cq = cand + q * cap;
    for (int t = threadIdx.x; t < d; t += NT) qs[t] = Q[q * d + t];
    if (threadIdx.x == 0) {
        atomicAdd(&stats[1], (unsigned long long)n);
        atomicMax(&stats[2], (unsigned long long)n);
    }
    int K;
    auto emit = [&](int i, uint64_t v) { sr_keys[i] = v; };
    if (n > cap) {  // the store overflowed: every key again
        if (threadIdx.x == 0) {
            atomicAdd(&stats[0], 1ull);
            atomicOr(status, KSC_STATUS_CAND_OVERFLOW);
        }
        K = redo_select(A, q, R, sr_keys, sr_keys, sel_cap, hist, s_pref);
    } else {
        K = min(R, n);
        if (n <= K) {
            for (int i = threadIdx.x; i < n; i += NT) sr_keys[i] = cq[i];
        } else if (n <= SP_REG_KEYS) {
            uint64_t kk[U];
#pragma unroll
            for (int u = 0; u < U; ++u) kk[u] = (int)threadIdx.x + u * NT < n ? cq[threadIdx.x + u * NT] : KEY_NONE;
            block_topk_regs<NT, U>(kk, n, K, emit, hist, bb);
        } else {
            auto load = [&](int i) -> uint64_t { return cq[i]; };
            block_topk(load, n, K, emit, hist, bb);
        }
    }
    __syncthreads();
    for (int i = K + threadIdx.x; i < R; i += NT) sr_keys[i] = KEY_NONE;
    __syncthreads();
    cta_rerank<NT>(sr_keys, R, sr_keys + nkeys, qs, X, d, ip, k, out_ids + q * k, out_d + q * k);
}

int launch_select_rerank(const ScanArgs& A, int Rmax, const int32_t* cnt, const uint64_t* cand, int cap, int sel_cap,
                         const float* Q, const float* X, int d, int ip, int k, int64_t* ids, float* dists,
                         int32_t* status, unsigned long long* stats, cudaStream_t st) {
    const int nkeys = Rmax > sel_cap ? Rmax : sel_cap;
    const size_t smem = sizeof(uint64_t) * ((size_t)nkeys + (Rmax > RR_RANK_R ? k : 0));
    KSC_CUDA(cudaFuncSetAttribute(k_select_rerank<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_select_rerank<1024><<<(unsigned)A.nq, 1024, smem, st>>>(A, Rmax, cnt, cand, cap, nkeys, sel_cap, Q, X, d, ip, k,
                                                              ids, dists, status, stats);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

}  // namespace ksc
