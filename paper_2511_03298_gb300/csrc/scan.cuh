// Arguments and device helpers shared by the scan kernels: the byte-permute
// scans, thresholds and selections (search.cu) and the tensor-core scan
// (scan_tc.cu).  Work lists are cluster-major: pairs of (query, probe rank)
// grouped by list, items = (list, query group, tile of the list's blocks).
#pragma once

#include "index.cuh"

namespace ksc {

struct ScanArgs {
    int M;
    int Pmax;
    int64_t nq;
    const int32_t* probes;
    const int32_t* nprobe_q;
    int Pfix;
    const int32_t* rerank_q;
    int Rfix, Rmin;
    const uint8_t* lut;
    const int32_t* bias;
    const int64_t* boff;
    const int32_t* list_n;
    const uint8_t* codes;
    const int32_t* ids;
    int L;
};

__device__ __forceinline__ int nprobe_of(const ScanArgs& A, int64_t q) {
    int P = A.nprobe_q ? A.nprobe_q[q] : A.Pfix;
    return P < 1 ? 1 : (P > A.Pmax ? A.Pmax : P);
}

__device__ __forceinline__ int rerank_of(const int32_t* rerank_q, int Rfix, int Rmin, int Rmax, int64_t q) {
    int R = rerank_q ? rerank_q[q] : Rfix;
    return R < Rmin ? Rmin : (R > Rmax ? Rmax : R);
}

__device__ __forceinline__ int64_t list_size(const ScanArgs& A, int p) {
    return (p >= 0 && p < A.L) ? A.list_n[p] : 0;
}

// Place of the first key of probe rank r in query q's unfiltered store: the
// keys of its lower ranks come first.
__device__ __forceinline__ int64_t near_offset(const ScanArgs& A, int64_t q, int r) {
    const int32_t* pr = A.probes + q * A.Pmax;
    int64_t off = 0;
    for (int r2 = 0; r2 < r; ++r2) off += list_size(A, pr[r2]);
    return off;
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t s) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(s));
    return r;
}

// Packed FP32 pairs (sm_100 family): each half is the IEEE single-precision
// operation rounded to nearest, the same result as the scalar instruction,
// in one instruction for both.
__device__ __forceinline__ float2 f2_sub(float2 a, float2 b) {
    float2 d;
    asm("{.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "sub.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 f2_mul(float2 a, float2 b) {
    float2 d;
    asm("{.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 f2_add(float2 a, float2 b) {
    float2 d;
    asm("{.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}

__device__ __forceinline__ float2 f2_fma(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{.reg .b64 ra, rb, rc, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
        "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

struct ScanOut {
    const uint64_t* thr;
    int32_t* cnt;
    uint64_t* cand;
    int cap;
    // items given one by one (small batches): (pair e, first block, end block,
    // list), their number, and each pair's place in the unfiltered store
    const int4* recs = nullptr;
    const int32_t* nrec = nullptr;
    const int32_t* noff = nullptr;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

struct ScanItem {
    int p, b0, b1;
    int64_t g0, npairs;
};

// Item `it` of a work list, by the whole warp: the last list p with
// item_off[p] <= it is found by a 32-way search (each round one load per lane
// and a ballot; two rounds for 1024 lists), then the item's query group and
// tile.  All 32 lanes call and get the same item.
__device__ __forceinline__ ScanItem locate_item(const ScanArgs& A, const int64_t* __restrict__ pair_off,
                                                const int64_t* __restrict__ item_off, int L, int TB, int QG,
                                                int64_t it, int unit = 1) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = L - 1;  // invariant: item_off[lo] <= it < item_off[hi + 1]
    while (lo < hi) {
        const int step = (hi - lo + 32) / 32;  // ceil((hi - lo + 1) / 32)
        const int pos = min(lo + lane * step, hi);
        const uint32_t m = __ballot_sync(0xffffffffu, item_off[pos] <= it);  // a prefix of lanes; lane 0 holds
        const int last = 31 - __clz(m);
        const int nlo = min(lo + last * step, hi);
        hi = (last < 31 && lo + (last + 1) * step <= hi) ? lo + (last + 1) * step - 1 : hi;
        lo = nlo;
    }
    ScanItem r;
    r.p = lo;
    const int nb = (A.list_n[lo] + 31) >> 5;
    const int nt = (nb + TB - 1) / TB;
    const int64_t local = it - item_off[lo];
    const int64_t grp = local / nt;
    const int tile = (int)(local - grp * nt);
    // the list's nt tiles of near-equal length in whole units (no tile is
    // empty: there are at least nt units)
    const int nu = (nb + unit - 1) / unit;
    r.b0 = (int)((int64_t)tile * nu / nt) * unit;
    r.b1 = min(nb, (int)((int64_t)(tile + 1) * nu / nt) * unit);
    r.g0 = pair_off[lo] + grp * QG;
    r.npairs = pair_off[lo + 1] - r.g0;
    return r;
}

__device__ __forceinline__ int nibble_of(const uint8_t* __restrict__ blk, int M, int j, int v) {
    uint8_t byte = blk[j * 16 + (v >> 1)];
    return (v & 1) ? (byte >> 4) : (byte & 15);
}

__device__ __forceinline__ int32_t scalar_dist(const uint8_t* __restrict__ lutp, int32_t b,
                                               const uint8_t* __restrict__ blk, int M, int v) {
    int32_t D = b;
    for (int j = 0; j < M; ++j) D += lutp[j * 16 + nibble_of(blk, M, j, v)];
    return D;
}

// The keys of query q by position over all its probed lists, recomputed with
// scalar lookups; s_pref: one more shared word than the query's probes.
struct QueryKeys {
    const ScanArgs& A;
    int64_t q;
    int P;
    const int32_t* pref;
    __device__ __forceinline__ uint64_t operator()(int i) const {
        int lo = 0, hi = P - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (pref[mid] <= i) lo = mid; else hi = mid - 1;
        }
        const int64_t item = q * A.Pmax + lo;
        const int p = A.probes[item];
        const int m = i - pref[lo];
        const int64_t blk = A.boff[p] + (m >> 5);
        const int v = m & 31;
        int32_t D = scalar_dist(A.lut + item * A.M * PQ_K, A.bias[item], A.codes + blk * A.M * 16, A.M, v);
        return make_key(D, A.ids[blk * 32 + v]);
    }
};
__device__ __forceinline__ QueryKeys query_keys(const ScanArgs& A, int64_t q, int32_t* s_pref) {
    const int P = nprobe_of(A, q);
    __syncthreads();  // s_pref of the previous query is no longer read
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int r = 0; r < P; ++r) {
            s_pref[r] = acc;
            const int p = A.probes[q * A.Pmax + r];
            acc += (p >= 0 && p < A.L) ? A.list_n[p] : 0;
        }
        s_pref[P] = acc;
    }
    __syncthreads();
    return QueryKeys{A, q, P, s_pref};
}

// The R best keys of a query whose store (`row`, cap keys, all written)
// overflowed, in no particular order unless the last way is taken.  The row's
// keys are some of the query's, so their R-th smallest bounds the R-th of all:
// one pass over the recomputed keys gathers those at or below it in the row,
// from which the R best are selected.  Only where these overflow the row as
// well (or it holds R keys at most) the selection recomputes every key in each
// of its nine passes.  3 queries of 9100 keys (8192 stored, 50 subspaces): 2600 us before,
// 50 now.
// hist: 256 shared words, 16-byte aligned; bb: 32; sel: sel_cap keys for the last
// way (may be out).  All threads of the CTA; returns min(R, keys).
__device__ __forceinline__ int redo_select(const ScanArgs& A, int64_t q, int R, uint64_t* row, int cap, uint64_t* out,
                                           uint64_t* sel, int sel_cap, uint32_t* hist, uint64_t* bb, int32_t* s_pref) {
    __shared__ int s_kept;
    const QueryKeys key = query_keys(A, q, s_pref);
    const int N = s_pref[key.P];
    if (R < cap) {
        auto stored = [&](int i) -> uint64_t { return row[i]; };
        const uint64_t bound = block_topk(stored, cap, R, [](int, uint64_t) {}, hist, bb);
        if (threadIdx.x == 0) s_kept = 0;
        __syncthreads();  // (and the row has been read)
        for (int i = threadIdx.x; i < N; i += blockDim.x) {
            const uint64_t k = key(i);
            if (k > bound) continue;
            const int at = atomicAdd(&s_kept, 1);
            if (at < cap) row[at] = k;
        }
        __syncthreads();
        const int n = s_kept;  // at least R: the bound and the R - 1 stored keys below it are among them
        if (n == R) {
            for (int i = threadIdx.x; i < n; i += blockDim.x) out[i] = row[i];
            __syncthreads();
            return R;
        }
        if (n <= cap) {
            block_topk(stored, n, R, [&](int i, uint64_t k) { out[i] = k; }, hist, bb);
            __syncthreads();
            return R;
        }
    }
    const int K = min(R, N);
    block_select_smallest([&](int i) -> uint64_t { return key(i); }, N, K, out, sel, sel_cap, hist);
    return K;
}

// The exact FP32 score of list centroid c for the query qs (shared memory), by
// one warp.
__device__ __forceinline__ float exact_list_score(const float* __restrict__ qs, const float* __restrict__ c, int d,
                                                  int spherical, int lane) {
    float acc = 0.f;
    if ((d & 3) == 0) {
        for (int t = lane * 4; t < d; t += 128) {
            float4 cv = __ldg(reinterpret_cast<const float4*>(c + t));
            float4 qv = *reinterpret_cast<const float4*>(qs + t);
            if (spherical) {
                acc = fmaf(qv.x, cv.x, acc); acc = fmaf(qv.y, cv.y, acc);
                acc = fmaf(qv.z, cv.z, acc); acc = fmaf(qv.w, cv.w, acc);
            } else {
                float e0 = qv.x - cv.x, e1 = qv.y - cv.y, e2 = qv.z - cv.z, e3 = qv.w - cv.w;
                acc = fmaf(e0, e0, acc); acc = fmaf(e1, e1, acc); acc = fmaf(e2, e2, acc); acc = fmaf(e3, e3, acc);
            }
        }
    } else {
        for (int t = lane; t < d; t += 32) {
            float cv = __ldg(c + t);
            if (spherical) acc = fmaf(qs[t], cv, acc);
            else { float e = qs[t] - cv; acc = fmaf(e, e, acc); }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return spherical ? -acc : acc;
}

// The tensor-core scan (scan_tc.cu): queries per item for M subspaces (0: not
// supported), and one launch over a work list of items of at most nt queries
// and TB blocks (whole 4-block units).
int tcs_nt(int M);
constexpr int TCS_MAX_TILE = 2048;  // largest TB (a buffered key holds its vector of the tile in 16 bits)
int launch_scan_tc(const ScanArgs& A, const ScanOut& O, const int64_t* pair_off, const int64_t* item_off,
                   const uint32_t* pairs, int L, int TB, int nt, unsigned long long* next_item, int32_t* status,
                   cudaStream_t st);

}  // namespace ksc
