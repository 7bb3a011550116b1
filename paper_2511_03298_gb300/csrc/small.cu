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
constexpr int SP_T = 512;       // threads per CTA
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

// Exclusive prefix sums over the CTA of three values at once; tot[96].
__device__ __forceinline__ void block_scan3(uint32_t& a, uint32_t& b, uint32_t& c, uint32_t* tot) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x[3] = {a, b, c};
    const uint32_t v[3] = {a, b, c};
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x[i], o);
            if (lane >= o) x[i] += y;
        }
    __syncthreads();  // tot is free
    if (lane == 31)
#pragma unroll
        for (int i = 0; i < 3; ++i) tot[32 * i + w] = x[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 3; ++i) {  // every warp sums the totals before its own
        uint32_t t = lane < w ? tot[32 * i + lane] : 0u;
        t = __reduce_add_sync(0xffffffffu, t);
        x[i] += t - v[i];
    }
    a = x[0];
    b = x[1];
    c = x[2];
}

// Scan items of one query (by one CTA): the end of the unfiltered part (the
// rule of k_count_parts), the places of its pairs in the store, and a record
// per tile of every probed list.  Each thread takes two consecutive ranks,
// then the tiles are dealt out to all threads.  size, ta, tb: SP_MAX_P + 1
// words each.
__device__ void query_items(const SmallPrep& S, int64_t q, const int32_t* prb, int P, uint32_t* size, uint32_t* ta,
                            uint32_t* tb) {
    constexpr int RT = SP_MAX_P / SP_T;
    __shared__ uint32_t tot[96];
    __shared__ int s_split, s_total, s_base[2];
    const ScanArgs& A = S.A;
    const int r0 = RT * threadIdx.x;
    uint32_t n[RT], mine = 0, z0 = 0, z1 = 0;
#pragma unroll
    for (int u = 0; u < RT; ++u) {
        n[u] = r0 + u < P ? (uint32_t)list_size(A, prb[r0 + u]) : 0u;
        mine += n[u];
    }
    uint32_t before = mine;
    if (threadIdx.x == 0) s_split = P;
    block_scan3(before, z0, z1, tot);
    int split = P;
    if (!S.all_near) {
        if (threadIdx.x == SP_T - 1) s_total = (int)(before + mine);
        __syncthreads();
        long long target = (long long)S.near_keys_per_r * rerank_of(A.rerank_q, A.Rfix, A.Rmin, S.Rmax, q);
        target = max(target, (long long)s_total / S.near_share_div);
        target = min(target, (long long)S.cap / 2);
        long long b = before;
#pragma unroll
        for (int u = 0; u < RT; ++u) {
            const int r = r0 + u;
            if (r > 0 && r < P && (b >= target || b + n[u] > S.cap)) {
                atomicMin(&s_split, r);
                break;
            }
            b += n[u];
        }
        __syncthreads();
        split = s_split;
    }
    uint32_t na = 0, nb = 0, nearn = 0;
#pragma unroll
    for (int u = 0; u < RT; ++u) {
        const uint32_t blk = (n[u] + 31) >> 5;
        if (r0 + u < split) {
            na += (blk + S.TBa - 1) / S.TBa;
            nearn += n[u];
        } else {
            nb += (blk + S.TB - 1) / S.TB;
        }
    }
    uint32_t oa = na, ob = nb, on = nearn;
    block_scan3(oa, ob, on, tot);
    if (threadIdx.x == SP_T - 1) {
        s_base[0] = atomicAdd(&S.nrec[0], (int)(oa + na));
        s_base[1] = atomicAdd(&S.nrec[1], (int)(ob + nb));
        S.cnt[q] = (int)(on + nearn);
        ta[SP_MAX_P] = oa + na;
        tb[SP_MAX_P] = ob + nb;
    }
    {  // first tile of each rank within its part
        uint32_t at = before, xa = oa, xb = ob;
#pragma unroll
        for (int u = 0; u < RT; ++u) {
            const int r = r0 + u;
            if (r < P) {
                const uint32_t blk = (n[u] + 31) >> 5;
                const bool near = r < split;
                size[r] = blk;
                ta[r] = xa;
                tb[r] = xb;
                if (near) {
                    S.noff[q * A.Pmax + r] = (int)at;
                    xa += (blk + S.TBa - 1) / S.TBa;
                } else {
                    xb += (blk + S.TB - 1) / S.TB;
                }
                at += n[u];
            }
        }
    }
    __syncthreads();
    for (int part = 0; part < 2; ++part) {
        const uint32_t* first = part ? tb : ta;
        const int lo0 = part ? split : 0, hi0 = part ? P : split, TB = part ? S.TB : S.TBa;
        const int nt = (int)first[SP_MAX_P];
        int4* out = (part ? S.recsB : S.recsA) + s_base[part];
        for (int t = threadIdx.x; t < nt; t += SP_T) {
            int lo = lo0, hi = hi0 - 1;  // the last rank whose first tile is at or before t
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if ((int)first[mid] <= t) lo = mid;
                else hi = mid - 1;
            }
            const int b0 = (t - (int)first[lo]) * TB;
            out[t] = make_int4((int)(q * A.Pmax + lo), b0, min((int)size[lo], b0 + TB), prb[lo]);
        }
    }
}

// stage_codebook by asynchronous copies (8 bytes, or 4 where rows are not that
// far aligned); wait with cp.async.wait_all and a barrier.
template <int DS>
__device__ __forceinline__ void stage_codebook_async(const LutArgs& T, float* cbs) {
    constexpr int V = DS == 2 ? 2 : 1;
    const int ld = cb_ld(T.dsub), rowlen = PQ_K * T.dsub;
    for (int e = V * threadIdx.x; e < T.M * rowlen; e += V * SP_T) {
        const int j = e / rowlen;
        const uint32_t dst = smem_addr(cbs + j * ld + (e - j * rowlen));
        if constexpr (V == 2) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(T.cb + e) : "memory");
        else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(T.cb + e) : "memory");
    }
}

template <int DS>
__global__ void __cluster_dims__(SP_CL, 1, 1) __launch_bounds__(SP_T) k_small_prep(SmallPrep S) {
    extern __shared__ __align__(16) unsigned char sp_raw[];
    __shared__ __align__(16) uint32_t hist[256];
    __shared__ uint32_t s_range, s_r;
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
    stage_codebook_async<DS>(T, cbs);  // waited for before the tables
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
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // the last CTA makes the scan items beside the others' tables (its table
    // buffers hold the ranks' sizes and first tiles); those take ranks cr, cr +
    // 7, ...: the largest row range of the query first
    constexpr int TC = SP_CL - 1;
    if (cr == TC) {
        uint32_t* iw = reinterpret_cast<uint32_t*>(mins);
        query_items(S, q, prb, P, iw, iw + SP_MAX_P + 1, iw + 2 * (SP_MAX_P + 1));
    }
    const int nr = cr < TC && P > cr ? (P - cr + TC - 1) / TC : 0;
    float R = 0.f;
    for (int row = threadIdx.x; row < nr * M; row += SP_T) {
        const int i = row / M, j = row - i * M, p = prb[cr + i * TC];
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
    cl.barrier_arrive();  // the leader's shared memory has been read (waited for at the end)
    const float a = (Rq == 0.f) ? 1.f : __fdiv_rn(255.f, Rq);
    const int group = SP_ROWS / M;
    for (int i0 = 0; i0 < nr; i0 += group) {
        const int ng = min(group, nr - i0);
        for (int row = threadIdx.x; row < ng * M; row += SP_T) {
            const int i = row / M, j = row - i * M, r = cr + (i0 + i) * TC, p = prb[r];
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
            const int r = cr + (i0 + i) * TC, p = prb[r];
            if (p >= 0 && p < T.L)
                S.bias[q * T.Pmax + r] = lut_bias(T, qs, T.c_mean + (int64_t)p * T.d, mins + i * M, a);
        }
        __syncthreads();
    }
    if (cr == 0 && threadIdx.x == 0) S.scale[q] = a;
    cl.barrier_wait();
}

int launch_small_prep(const SmallPrep& S, cudaStream_t st) {
    const size_t smem = small_prep_smem(S);
    auto kern = S.T.dsub == 2 ? k_small_prep<2> : (S.T.dsub == 4 ? k_small_prep<4> : k_small_prep<0>);
    KSC_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<(unsigned)(S.T.nq * SP_CL), SP_T, smem, st>>>(S);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

template <int NT>
__global__ void __launch_bounds__(NT) k_select_rerank(ScanArgs A, int Rmax, const int32_t* __restrict__ cnt,
                                                      uint64_t* cand, int cap, int nkeys,
                                                      int sel_cap, const float* __restrict__ Q,
                                                      const float* __restrict__ X, int d, int ip, int k,
                                                      int64_t* __restrict__ out_ids, float* __restrict__ out_d,
                                                      int32_t* __restrict__ status,
                                                      unsigned long long* __restrict__ stats) {
    extern __shared__ uint64_t sr_keys[];  // nkeys (at least Rmax; sel_cap when a store may overflow), then rerank_kbuf(k)
    __shared__ __align__(16) uint32_t hist[256];
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
        K = redo_select(A, q, R, cand + q * cap, cap, sr_keys, sr_keys, sel_cap, hist, bb, s_pref);
    } else {
        K = min(R, n);
        if (n <= K) {
            for (int i = threadIdx.x; i < n; i += NT) sr_keys[i] = cq[i];
        } else if (n <= SP_REG_KEYS) {
            uint64_t kk[U];
#pragma unroll
            for (int u = 0; u < U; ++u) kk[u] = (int)threadIdx.x + u * NT < n ? cq[threadIdx.x + u * NT] : KEY_NONE;
            auto each = [&](auto f) {
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (u * NT < n) f((int)threadIdx.x + u * NT < n, kk[u]);
            };
            block_topk_each(each, K, emit, hist, bb);
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

int launch_select_rerank(const ScanArgs& A, int Rmax, const int32_t* cnt, uint64_t* cand, int cap, int sel_cap,
                         const float* Q, const float* X, int d, int ip, int k, int64_t* ids, float* dists,
                         int32_t* status, unsigned long long* stats, cudaStream_t st) {
    const int nkeys = Rmax > sel_cap ? Rmax : sel_cap;
    const size_t smem = sizeof(uint64_t) * ((size_t)nkeys + (Rmax > RR_RANK_R ? rerank_kbuf(k) : 0));
    KSC_CUDA(cudaFuncSetAttribute(k_select_rerank<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_select_rerank<1024><<<(unsigned)A.nq, 1024, smem, st>>>(A, Rmax, cnt, cand, cap, nkeys, sel_cap, Q, X, d, ip, k,
                                                              ids, dists, status, stats);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

}  // namespace ksc
