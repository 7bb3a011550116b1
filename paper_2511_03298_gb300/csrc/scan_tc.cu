// a3: the LUT16 scan on the 5th-generation tensor cores (Alg. 3's table lookups
// as a matrix product), for lists that many queries of the batch probe.
#include <algorithm>

#include "scan_ops.cuh"
#include "tc.cuh"

namespace ksc {

// The lookup sums of one list for a group of queries as one matrix product.
// A (row = vector, K = 16 M): entry 16 j + c is 1 when the vector's code in
// subspace j is c, else 0.  B holds two rows per query, the high and the low
// four bits of its u8 table of the list, entry 16 j + e.  All are e4m3 values,
// exact (1 and the integers 0 .. 15), and the sums are integers below 2^12 (15
// M), exact in the FP32 accumulator whatever the order of the additions: sum =
// 16 high + low, so the keys equal those of the byte-permute scan bit for bit.
//
// Roles of a CTA (one per SM, items from a global counter), each at its own
// pace behind mbarriers:
//  - one warp finds the next item: its list, tiles (128 vectors), queries and
//    thresholds;
//  - 8 warps stage its tables as B in the other of two buffers (K-major,
//    128-byte swizzle);
//  - one thread fetches the codes of the tiles, a bulk copy each;
//  - 8 warps expand codes into one-hot rows, straight into tensor memory (lane =
//    vector; a chunk of 8 subspaces is 32 columns; two groups of 4 chunks): 9
//    integer operations per code, no shared memory, no proxy fence;
//  - one warp issues the MMAs (A from tensor memory, M 128 x N 2 x queries x K
//    32) into one of two accumulators;
//  - 8 warps read the other (lane = vector, column = query), test the sums
//    against the queries' thresholds and append the passing ones to buffers (per
//    32 vectors of the tile and query, places from a ballot), 4 bytes each, and
//    write them to the store when they fill up and at the item's end.
//
// What bounds it: instruction fetch, then the MMAs' fixed cost.  The roles run
// different code at once, and with the loops unrolled for throughput (16 columns
// a step, tables and waits inlined wide; 78% hits in the instruction cache, an
// instruction per 10 cycles and warp) a tile of 128 vectors x 34 queries took
// 12000 cycles; short loops, one barrier per 4 chunks and 8 staging warps brought
// it to 4000 to 5500.  An MMA of these shapes takes 80 cycles whatever its N (32
// a tile).  The scan of 1M x 64 subspaces for 10k queries x 8 lists: 707 us with
// byte permutes, 327 us here; the search 1290 -> 899 us.
// Every wait is bounded; a failed one stops all roles.
constexpr int TS_NT = 64;      // queries per item at most
constexpr int TS_EXP = 8, TS_EPI = 8, TS_STG = 8;  // expanding, epilogue, staging warps
constexpr int TS_W_EPI = TS_EXP, TS_W_STG = TS_EXP + TS_EPI, TS_W_MMA = TS_W_STG + TS_STG,
              TS_W_LOAD = TS_W_MMA + 1, TS_W_ITEM = TS_W_LOAD + 1;
constexpr int TS_THREADS = 32 * (TS_W_ITEM + 1);
constexpr int TS_GRP = 4;      // A chunks per barrier; two such groups in tensor memory
constexpr int TS_KCAP = 24;    // keys buffered per query and 32-vector quarter of the tiles
constexpr int TS_KFLUSH = 12;  // ... from which buffers are written out before the next tile,
constexpr int TS_KMIN = 8;     // those of this many keys
constexpr uint32_t TS_A_COL = 4 * TS_NT;  // two accumulators of 2 TS_NT columns, then the ring
static_assert(TS_A_COL + 64 * TS_GRP <= 512, "tensor memory columns");

struct TsQuery {
    int64_t q;
    uint32_t e, thI;
    int32_t bias, lim;
};

struct TsItem {
    int p, b0, b1, nq, N2, ntile, listn, valid;
    int64_t gb, g0;
};
struct TsQueries {
    TsQuery query[TS_NT];
    __align__(16) float lim[TS_NT];  // largest passing sum + 2^23 (-1: none)
};

__host__ __device__ inline int ts_chunks(int M) { return (M + 7) / 8; }
static size_t ts_smem_bytes(int M, int nt) {
    const size_t C8 = ts_chunks(M);
    return 1024 + 2 * C8 * (2 * nt * 128) + 2 * 4 * C8 * 8 * 16 + (size_t)4 * nt * TS_KCAP * 4;
}

__device__ __forceinline__ void ts_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// A bounded wait that also ends when another role of the CTA has given up.
// (The roles' loops share the instruction cache, which bounds them when they are
// long: waits, and all code below, are kept short.)
__device__ __forceinline__ bool ts_wait(uint32_t bar, uint32_t parity, volatile int* fail) {
#pragma unroll 1
    for (uint32_t i = 0; i < TC_WAIT_LIMIT; ++i) {
        if (mbar_wait(bar, parity, 1)) return true;
        if (*fail) return false;
    }
    *fail = 1;
    return false;
}

// D[tmem d] (+)= A[tmem a] B[smem desc b]^T, e4m3 operands, by lane 0 of a
// converged warp.
__device__ __forceinline__ void ts_mma(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc, int lane) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.eq.b32 q, %5, 0;\n @q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], "
        "[%1], %2, %3, p;\n}" ::"r"(d),
        "r"(a), "l"(b), "r"(idesc), "r"(acc), "r"(lane)
        : "memory");
}

__device__ __forceinline__ void ts_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
        "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}

// tcgen05.ld of 8 columns (or 1) without its wait (ts_ld_wait names the
// registers it makes valid).
__device__ __forceinline__ void ts_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void ts_ld1(uint32_t taddr, uint32_t& r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr));
}
__device__ __forceinline__ void ts_ld_wait(uint32_t (&a)[8], uint32_t (&b)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                   "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])
                 :
                 : "memory");
}

// Sum of a column from its two accumulator words, plus 2^23 (exact: below 2^24;
// the sum is then the low bits of the word).
constexpr float TS_BIAS = 8388608.f;
__device__ __forceinline__ float ts_sum(uint32_t hi, uint32_t lo) {
    return fmaf(16.f, __uint_as_float(hi), __uint_as_float(lo) + TS_BIAS);
}
// The same read from tensor memory by the whole warp.
__device__ __forceinline__ float ts_column(uint32_t hi_addr, uint32_t lo_addr) {
    uint32_t h, l;
    __syncwarp();
    ts_ld1(hi_addr, h);
    ts_ld1(lo_addr, l);
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(h), "+r"(l) : : "memory");
    return ts_sum(h, l);
}

// Item `it` of the work list, by a whole warp (the 32-way search of
// locate_item; counts within a list fit 32 bits): its tiles' blocks and its
// query group, the groups of a list of near-equal size (multiples of 16).
__device__ __forceinline__ void ts_locate(const ScanArgs& A, const int64_t* __restrict__ pair_off,
                                          const int64_t* __restrict__ item_off, int L, int TB, int nt, int64_t it,
                                          TsItem& x) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = L - 1;
#pragma unroll 1
    while (lo < hi) {
        const int step = (hi - lo + 32) / 32;
        const uint32_t m = __ballot_sync(0xffffffffu, item_off[min(lo + lane * step, hi)] <= it);
        const int last = 31 - __clz(m);
        const int nlo = min(lo + last * step, hi);
        hi = (last < 31 && lo + (last + 1) * step <= hi) ? lo + (last + 1) * step - 1 : hi;
        lo = nlo;
    }
    const uint32_t local = (uint32_t)(it - item_off[lo]);
    const int64_t p0 = pair_off[lo];
    const uint32_t cnt = (uint32_t)(pair_off[lo + 1] - p0);
    x.listn = A.list_n[lo];
    x.gb = A.boff[lo];
    x.p = lo;
    const uint32_t nb = ((uint32_t)x.listn + 31u) >> 5, tiles = (nb + TB - 1) / TB, grp = local / tiles,
                   tile = local - grp * tiles, nu = (nb + 3) / 4;
    x.b0 = (int)((uint64_t)tile * nu / tiles) * 4;
    x.b1 = min((int)nb, (int)((uint64_t)(tile + 1) * nu / tiles) * 4);
    x.ntile = (x.b1 - x.b0 + 3) / 4;
    const uint32_t ng = (cnt + nt - 1) / nt, per = min((uint32_t)nt, ((cnt + ng - 1) / ng + 15u) & ~15u);
    x.g0 = p0 + (int64_t)grp * per;
    x.nq = (int)min(per, cnt - grp * per);
    x.N2 = (x.nq + 15) & ~15;
}

__global__ void __launch_bounds__(TS_THREADS, 1)
    k_scan_tc(ScanArgs A, ScanOut O, const int64_t* __restrict__ pair_off, const int64_t* __restrict__ item_off,
              const uint32_t* __restrict__ pairs, int L, int TB, int nt, unsigned long long* __restrict__ next_item,
              int32_t* __restrict__ status) {
    extern __shared__ __align__(1024) uint8_t ts_raw[];
    __shared__ __align__(8) uint64_t bars[17];
    __shared__ uint32_t s_tmem;
    __shared__ TsItem s_item[2];
    __shared__ TsQueries s_qry[2];
    __shared__ int s_stop[2];       // the staging warps' common decision
    __shared__ volatile int s_fail;
    __shared__ uint8_t s_pick[TS_EPI][32];
    __shared__ __align__(16) int s_kc[4][TS_NT];  // keys of each (quarter, query) in this item
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(ts_raw) + 1023) & ~uintptr_t(1023));
    const int M = A.M, C8 = ts_chunks(M), G = (C8 + TS_GRP - 1) / TS_GRP;
    const uint32_t box = (uint32_t)(2 * nt) * 128;  // bytes of a B box (8 subspaces)
    const uint32_t b_bytes = (uint32_t)C8 * box;    // bytes of a B buffer
    const int code_bytes = 4 * C8 * 8 * 16;         // a tile's codes
    uint8_t* pC = smem + 2 * (size_t)b_bytes;
    uint32_t* kbuf = reinterpret_cast<uint32_t*>(pC + 2 * code_bytes);  // [4][nt][TS_KCAP]
    const uint32_t sB = smem_addr(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto bar = [&](int i) { return smem_addr(&bars[i]); };
    auto a_full = [&](int s) { return bar(s); };
    auto a_free = [&](int s) { return bar(2 + s); };
    constexpr int B0 = 4;
    auto d_full = [&](int b) { return bar(B0 + b); };
    auto d_free = [&](int b) { return bar(B0 + 2 + b); };
    auto c_full = [&](int b) { return bar(B0 + 4 + b); };
    auto c_free = [&](int b) { return bar(B0 + 6 + b); };
    auto i_full = [&](int b) { return bar(B0 + 8 + b); };
    auto i_free = [&](int b) { return bar(B0 + 10 + b); };
    const uint32_t drain = bar(B0 + 12);
    if (tid == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(a_full(b), TS_EXP);
            mbar_init(a_free(b), 1);
            mbar_init(d_full(b), 1);
            mbar_init(d_free(b), TS_EPI);
            mbar_init(c_full(b), 1);
            mbar_init(c_free(b), TS_EXP);
            mbar_init(i_full(b), TS_STG);
            mbar_init(i_free(b), TS_EXP + TS_EPI + 2);
        }
        mbar_init(drain, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 4 * TS_NT) (&s_kc[0][0])[tid] = 0;
    // B's padding (subspaces past M) is zero for good; codes read past a
    // tile's end are some nibble, a valid one-hot row that is never used
    for (uint32_t e = tid; e < 2 * b_bytes / 16; e += TS_THREADS) reinterpret_cast<uint4*>(smem)[e] = make_uint4(0u, 0u, 0u, 0u);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    volatile int* fail = &s_fail;
    // every role counts items, tiles and groups of A chunks alike: n-th use of a buffer
    // waits for the phases of the uses before
    uint32_t ni = 0, nt_ = 0, ng = 0;
    // the item warp and the staging warps meet at a named barrier for each item
    auto sync = [&]() {
        __syncwarp();  // bar.sync is a warp-collective instruction
        asm volatile("bar.sync 1, %0;" ::"n"(32 * (TS_STG + 1)) : "memory");
    };
    if (warp == TS_W_ITEM) {
        // ---------------------------------------------------------------- items
        const int64_t total = item_off[L];
        for (;; ++ni) {
            TsItem& x = s_item[ni & 1u];
            TsQueries& y = s_qry[ni & 1u];
            // the next item in registers, then its place in shared memory
            long long it = 0;
            if (lane == 0) it = (long long)atomicAdd(next_item, 1ull);
            it = __shfl_sync(0xffffffffu, it, 0);
            TsItem r{};
            r.valid = it < total;
            TsQuery qi[TS_NT / 32];
            float lim[TS_NT / 32];
            if (r.valid) {
                ts_locate(A, pair_off, item_off, L, TB, nt, it, r);
#pragma unroll
                for (int u = 0; u < TS_NT / 32; ++u) {
                    lim[u] = -1.f;
                    if (lane + 32 * u < r.nq) {
                        qi[u].e = pairs[r.g0 + lane + 32 * u];
                        qi[u].q = qi[u].e / (uint32_t)A.Pmax;
                        qi[u].bias = A.bias[qi[u].e];
                        const uint64_t th = O.thr[qi[u].q];
                        qi[u].thI = (uint32_t)th;
                        const int64_t l = (int64_t)(th >> 32) - 2147483648ll - qi[u].bias;
                        qi[u].lim = (int32_t)(l < -1 ? -1 : (l > 65536 ? 65536 : l));
                        if (qi[u].lim >= 0) lim[u] = (float)qi[u].lim + TS_BIAS;
                    }
                }
            }
            const bool ok =
                __all_sync(0xffffffffu, ni < 2 || ts_wait(i_free(ni & 1u), ((ni >> 1) - 1) & 1u, fail));
            if (lane == 0) {
                s_stop[ni & 1u] = !ok;
                if (ok) x = r;
            }
            if (ok && r.valid)
#pragma unroll
                for (int u = 0; u < TS_NT / 32; ++u) {
                    if (lane + 32 * u < r.nq) y.query[lane + 32 * u] = qi[u];
                    y.lim[lane + 32 * u] = lim[u];
                }
            sync();
            if (!ok || !r.valid) break;
        }
    } else if (warp >= TS_W_STG && warp < TS_W_MMA) {
        // ---------------------------------------------------------------- staging
        const int st = tid - 32 * TS_W_STG;
        const uint4 f8 = make_uint4(0x44403800u, 0x4E4C4A48u, 0x53525150u, 0x57565554u);  // e4m3 of 0 .. 15
        const int dn = 32 * TS_STG / M, dj = 32 * TS_STG - dn * M;
        for (;; ++ni) {
            const TsItem& x = s_item[ni & 1u];
            const TsQueries& y = s_qry[ni & 1u];
            sync();
            if (s_stop[ni & 1u]) break;
            const bool valid = x.valid;
            if (valid) {
                // B: rows n (high nibbles) and N2 + n (low), 16 bytes per
                // subspace; four table rows per thread in flight
                const int nq = x.nq;
                const uint32_t low = (uint32_t)x.N2 * 128;
                uint8_t* pB = smem + (size_t)(ni & 1u) * b_bytes;
                int n = st / M, j = st - n * M;
#pragma unroll 1
                while (n < nq) {
                    uint4 t[4];
                    uint32_t at[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        at[u] = 0xffffffffu;
                        if (n < nq) {
                            t[u] = __ldg(reinterpret_cast<const uint4*>(A.lut + (int64_t)y.query[n].e * M * PQ_K) + j);
                            at[u] = (uint32_t)(j >> 3) * box + (n >> 3) * 1024 + (n & 7) * 128 + (((j ^ n) & 7) << 4);
                        }
                        n += dn;
                        j += dj;
                        if (j >= M) {
                            j -= M;
                            ++n;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (at[u] == 0xffffffffu) break;
                        const uint32_t w[4] = {t[u].x, t[u].y, t[u].z, t[u].w};
                        uint32_t hi[4], lo[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            uint32_t a, b;  // bytes: (low, high) nibble of entries 0, 1 and 2, 3
                            lut16x8(w[k], f8, a, b);
                            lo[k] = prmt(a, b, 0x6420u);
                            hi[k] = prmt(a, b, 0x7531u);
                        }
                        *reinterpret_cast<uint4*>(pB + at[u]) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                        *reinterpret_cast<uint4*>(pB + at[u] + low) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
            if (lane == 0) ts_arrive(i_full(ni & 1u));
            if (!valid) break;
        }
    } else if (warp < TS_EXP) {
        // ---------------------------------------------------------------- expansion
        // warp w: vectors 32 (w & 3) .. of a tile, chunks of parity w >> 2
        const int blk4 = warp & 3, par = warp >> 2;
        const uint32_t acol = tmem + TS_A_COL + ((uint32_t)(32 * blk4) << 16);
        const int rot = (4 * (lane & 7) - 3) & 31;  // the code to bits 3 .. 6
        bool ok = true;
        for (;; ++ni) {
            ok = __all_sync(0xffffffffu, ts_wait(i_full(ni & 1u), (ni >> 1) & 1u, fail));
            if (!ok) break;
            const TsItem& x = s_item[ni & 1u];
            if (!x.valid) break;
            const int ntile = x.ntile;
            for (int t = 0; t < ntile && ok; ++t, ++nt_) {
                ok = __all_sync(0xffffffffu, ts_wait(c_full(nt_ & 1u), (nt_ >> 1) & 1u, fail));
                if (!ok) break;
                const uint32_t* cw =
                    reinterpret_cast<const uint32_t*>(pC + (nt_ & 1u) * code_bytes + blk4 * M * 16) + (lane >> 3);
                for (int g = 0; g < G; ++g, ++ng) {
                    const uint32_t h = ng & 1u;
                    if (ng >= 2) {
                        ok = __all_sync(0xffffffffu, ts_wait(a_free(h), ((ng >> 1) - 1) & 1u, fail));
                        if (!ok) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    }
#pragma unroll 1
                    for (int c = TS_GRP * g + par; c < min(C8, TS_GRP * (g + 1)); c += 2) {
                        uint32_t r[32];
#pragma unroll
                        for (int k = 0; k < 8; ++k) r[4 * k] = cw[4 * (8 * c + k)];
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            // word i of the one-hot row: 1.0 (0x38) shifted by 8 code - 32 i
                            // bits, zero outside 0 .. 31
                            const uint32_t c8 = __funnelshift_r(r[4 * k], r[4 * k], rot) & 0x78u;
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                asm("shl.b32 %0, %1, %2;" : "=r"(r[4 * k + i]) : "r"(0x38u), "r"(c8 - 32u * i));
                        }
                        __syncwarp();  // tcgen05.st is a warp-collective instruction
                        ts_st32(acol + 32 * (TS_GRP * h + (c & (TS_GRP - 1))), r);
                    }
                    __syncwarp();
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) ts_arrive(a_full(h));
                }
                if (!ok) break;
                if (lane == 0) ts_arrive(c_free(nt_ & 1u));
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0) ts_arrive(i_free(ni & 1u));
        }
    } else if (warp == TS_W_LOAD) {
        // ---------------------------------------------------------------- codes
        // one thread fetches every tile's codes in order, two tiles ahead at most
        // (a second loader would wait for phases two behind its own)
        if (lane == 0) {
            bool ok = true;
            for (;; ++ni) {
                ok = ts_wait(i_full(ni & 1u), (ni >> 1) & 1u, fail);
                if (!ok) break;
                const TsItem& x = s_item[ni & 1u];
                if (!x.valid) break;
                const int ntile = x.ntile, b0 = x.b0, b1 = x.b1;
                const int64_t gb = x.gb;
                for (int t = 0; t < ntile; ++t, ++nt_) {
                    const uint32_t b = nt_ & 1u;
                    ok = nt_ < 2 || ts_wait(c_free(b), ((nt_ >> 1) - 1) & 1u, fail);
                    if (!ok) break;
                    const int c0 = b0 + 4 * t, c1 = min(b1, c0 + 4);
                    const uint32_t bytes = (uint32_t)(c1 - c0) * M * 16;
                    ok = c1 > c0 && bytes <= (uint32_t)code_bytes;  // (always: a tile holds 1 to 4 blocks)
                    if (!ok) break;
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    mbar_expect_tx(c_full(b), bytes);
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                            smem_addr(pC + b * code_bytes)),
                        "l"(A.codes + (gb + c0) * (int64_t)M * 16), "r"(bytes), "r"(c_full(b))
                        : "memory");
                }
                if (!ok) break;
                ts_arrive(i_free(ni & 1u));
            }
            if (!ok) *fail = 1;
            // the copies in flight land before the CTA ends, also after a failure
            for (uint32_t T = nt_ < 2 ? 0 : nt_ - 2; T < nt_; ++T) mbar_wait(c_full(T & 1u), (T >> 1) & 1u, TC_WAIT_LIMIT);
        }
        __syncwarp();
    } else if (warp == TS_W_MMA) {
        // ---------------------------------------------------------------- MMAs
        // the warp runs the loop, its lane 0 issues: the operands stay warp-uniform
        {
            bool ok = true;
            for (;; ++ni) {
                ok = __all_sync(0xffffffffu, ts_wait(i_full(ni & 1u), (ni >> 1) & 1u, fail));
                if (!ok) break;
                const TsItem& x = s_item[ni & 1u];
                if (!x.valid) break;
                const int ntile = x.ntile;
                if (x.N2 < 16 || x.N2 > nt || (x.N2 & 15)) {  // (never: groups of 1 to nt queries)
                    *fail = 1;
                    break;
                }
                const uint32_t idesc = idesc_f16kind(0, 128, 2 * x.N2);
                const uint32_t sBi = sB + (ni & 1u) * b_bytes;
                for (int t = 0; t < ntile && ok; ++t, ++nt_) {
                    const uint32_t b = nt_ & 1u;
                    if (nt_ >= 2) ok = __all_sync(0xffffffffu, ts_wait(d_free(b), ((nt_ >> 1) - 1) & 1u, fail));
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    for (int g = 0; g < G; ++g, ++ng) {
                        const uint32_t h = ng & 1u;
                        ok = __all_sync(0xffffffffu, ts_wait(a_full(h), (ng >> 1) & 1u, fail));
                        if (!ok) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
                        for (int c = TS_GRP * g; c < min(C8, TS_GRP * (g + 1)); ++c) {
                            const uint32_t a = tmem + TS_A_COL + 32 * (TS_GRP * h + (c & (TS_GRP - 1)));
                            const uint64_t bd = smem_desc(sBi + c * box);
#pragma unroll
                            for (int k = 0; k < 4; ++k)  // (32 bytes on: 2 in the descriptor's address field)
                                ts_mma(tmem + b * (2 * TS_NT), a + 8 * k, bd + 2 * k, idesc, (c | k) != 0, lane);
                        }
                        if (lane == 0) tc_commit(a_free(h));
                        __syncwarp();
                    }
                    if (ok && lane == 0) tc_commit(d_full(b));
                    __syncwarp();
                }
                if (!ok) break;
                if (lane == 0) tc_commit(i_free(ni & 1u));  // B has been read
                __syncwarp();
            }
        }
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- epilogue
        // warp: TMEM lanes 32 (warp % 4) .., column groups of parity hf
        const int sub = warp & 3, hf = (warp - TS_W_EPI) >> 2;
        const uint32_t below = (1u << lane) - 1u;
        uint32_t* mybuf = kbuf + (size_t)sub * nt * TS_KCAP;
        int* mykc = s_kc[sub];
        bool ok = true;
        for (;; ++ni) {
            ok = __all_sync(0xffffffffu, ts_wait(i_full(ni & 1u), (ni >> 1) & 1u, fail));
            if (!ok) break;
            const TsItem& x = s_item[ni & 1u];
            if (!x.valid) break;
            const TsQueries& y = s_qry[ni & 1u];
            const int ntile = x.ntile, nq = x.nq, N2 = x.N2;
            if (nq < 1 || N2 > nt || nq > N2) {
                *fail = 1;
                break;
            }
            int most = 0;  // keys in the fullest buffer
            for (int t = 0; t < ntile; ++t, ++nt_) {
                const uint32_t b = nt_ & 1u;
                ok = __all_sync(0xffffffffu, ts_wait(d_full(b), (nt_ >> 1) & 1u, fail));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int blk = x.b0 + 4 * t + sub;
                const bool valid = blk < x.b1 && blk * 32 + lane < x.listn;
                const uint32_t idx = (uint32_t)((blk - x.b0) * 32 + lane);
                const uint32_t base = tmem + b * (2 * TS_NT) + ((uint32_t)(sub * 32) << 16);
#pragma unroll 1
                for (int n0 = 8 * hf; n0 < nq; n0 += 16) {
                    uint32_t hi[8], lo[8];
                    __syncwarp();  // tcgen05.ld is a warp-collective instruction
                    ts_ld8(base + n0, hi);
                    ts_ld8(base + N2 + n0, lo);
                    const float4 l0 = *reinterpret_cast<const float4*>(&y.lim[n0]);
                    const float4 l1 = *reinterpret_cast<const float4*>(&y.lim[n0 + 4]);
                    const int4 k0 = *reinterpret_cast<const int4*>(&mykc[n0]);
                    const int4 k1 = *reinterpret_cast<const int4*>(&mykc[n0 + 4]);
                    const float lv[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
                    int kv[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
                    uint32_t* kb = mybuf + n0 * TS_KCAP;
                    int over = 0;
                    ts_ld_wait(hi, lo);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float s = ts_sum(hi[i], lo[i]);
                        const bool in = valid && s <= lv[i];
                        const uint32_t m = __ballot_sync(0xffffffffu, in);
                        const int at = kv[i] + __popc(m & below);
                        if (in && at < TS_KCAP) kb[i * TS_KCAP + at] = prmt(idx, __float_as_uint(s), 0x5410u);
                        kv[i] += __popc(m);
                        over = max(over, kv[i]);
                    }
                    most = max(most, over);
                    if (lane == 0) {
                        *reinterpret_cast<int4*>(&mykc[n0]) = make_int4(kv[0], kv[1], kv[2], kv[3]);
                        *reinterpret_cast<int4*>(&mykc[n0 + 4]) = make_int4(kv[4], kv[5], kv[6], kv[7]);
                    }
                    __syncwarp();
                    if (over <= TS_KCAP) continue;
                    // full buffers: the keys past them straight to the store (a key that
                    // ties with the threshold's distance only if its id is in): which
                    // lanes, one reservation for all columns, the keys
                    const uint32_t id = valid ? (uint32_t)A.ids[(x.gb + blk) * 32 + lane] : 0u;
                    uint32_t mine = 0u;  // lane i: the lanes of column n0 + i
#pragma unroll 1
                    for (int i = 0; i < 8; ++i) {
                        const int kn = mykc[n0 + i];
                        if (kn <= TS_KCAP) continue;
                        const float s = ts_column(base + n0 + i, base + N2 + n0 + i);
                        const bool in = valid && s <= y.lim[n0 + i];
                        const uint32_t m = __ballot_sync(0xffffffffu, in);
                        const TsQuery& qi = y.query[n0 + i];
                        const bool out = in && kn - __popc(m) + __popc(m & below) >= TS_KCAP &&
                                         ((int32_t)(s - TS_BIAS) != qi.lim || id <= qi.thI);
                        const uint32_t mo = __ballot_sync(0xffffffffu, out);
                        if (lane == i) mine = mo;
                    }
                    __syncwarp();
                    int at0 = 0;
                    if (lane < 8) {
                        if (mine) at0 = atomicAdd(&O.cnt[y.query[n0 + lane].q], __popc(mine));
                        mykc[n0 + lane] = min(mykc[n0 + lane], TS_KCAP);
                    }
#pragma unroll 1
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t mo = __shfl_sync(0xffffffffu, mine, i);
                        const int at = __shfl_sync(0xffffffffu, at0, i) + __popc(mo & below);
                        if (!mo) continue;
                        const int32_t sum = (int32_t)(ts_column(base + n0 + i, base + N2 + n0 + i) - TS_BIAS);
                        const TsQuery& qi = y.query[n0 + i];
                        if (((mo >> lane) & 1u) && at < O.cap)
                            O.cand[qi.q * O.cap + at] = ((uint64_t)((uint32_t)(qi.bias + sum) ^ 0x80000000u) << 32) | id;
                    }
                    __syncwarp();
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) ts_arrive(d_free(b));
                if (t + 1 < ntile && most < TS_KFLUSH) continue;
                // this warp's buffered keys to the store, at the item's end all,
                // before it only the fuller buffers: one reservation per query (lane
                // = query of the warp's groups), then 4 lanes per query, 8 queries at
                // a time.  (A buffered key may tie with the threshold's distance and
                // lie above it by its id: one more candidate for the selection, none
                // lost.)
                const int col = (lane >> 3) * 16 + 8 * hf + (lane & 7);  // lane -> column
                int cnt = col < nq ? min(mykc[col], TS_KCAP) : 0, at0 = 0;
                const bool sel = cnt >= (t + 1 < ntile ? TS_KMIN : 1);
                const uint32_t ms = __ballot_sync(0xffffffffu, sel);
                if (sel) {
                    at0 = atomicAdd(&O.cnt[y.query[col].q], cnt);
                    mykc[col] = 0;
                    s_pick[warp - TS_W_EPI][__popc(ms & below)] = (uint8_t)lane;
                }
                __syncwarp();  // s_pick is read by other lanes (votes and reductions order no memory)
                most = __reduce_max_sync(0xffffffffu, sel ? 0 : cnt);
                const int32_t* idp = A.ids + (x.gb + x.b0) * 32;
#pragma unroll 1
                for (int k = lane >> 2; k - (lane >> 2) < __popc(ms); k += 8) {
                    const int src = k < __popc(ms) ? s_pick[warp - TS_W_EPI][k] : lane;
                    const int c = (src >> 3) * 16 + 8 * hf + (src & 7);
                    int m = __shfl_sync(0xffffffffu, cnt, src);
                    if (k >= __popc(ms)) m = 0;
                    uint32_t e[TS_KCAP / 4], id[TS_KCAP / 4];
#pragma unroll
                    for (int u = 0; u < TS_KCAP / 4; ++u) e[u] = 4 * u + (lane & 3) < m ? mybuf[c * TS_KCAP + 4 * u + (lane & 3)] : 0u;
#pragma unroll
                    for (int u = 0; u < TS_KCAP / 4; ++u) id[u] = 4 * u + (lane & 3) < m ? (uint32_t)idp[e[u] & 0xffffu] : 0u;
                    const int at = __shfl_sync(0xffffffffu, at0, src);
                    if (m > 0) {
                        const uint32_t bias = (uint32_t)y.query[c].bias ^ 0x80000000u;
                        uint64_t* dst = O.cand + y.query[c].q * O.cap;
#pragma unroll
                        for (int u = 0; u < TS_KCAP / 4; ++u) {
                            const int i = 4 * u + (lane & 3);
                            if (i < m && at + i < O.cap) dst[at + i] = ((uint64_t)(bias + (e[u] >> 16)) << 32) | id[u];
                        }
                    }
                }
                __syncwarp();
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0) ts_arrive(i_free(ni & 1u));
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (s_fail && tid == 0) atomicOr(status, 8);
    // every MMA issued by this CTA has completed before the tensor memory is freed
    if (tid == 32 * TS_W_MMA) {
        tc_commit(drain);
        if (!mbar_wait(drain, 0, TC_WAIT_LIMIT)) atomicOr(status, 8);
    }
    __syncwarp();
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// Queries per item of the tensor-core scan for M subspaces: two buffers of
// their tables (32 M bytes each) and the rest fit in 220 KB of shared memory; 0:
// not supported.
int tcs_nt(int M) {
    if (M < 1 || M > 128) return 0;
    for (int nt = TS_NT; nt >= 16; nt -= 16)
        if (ts_smem_bytes(M, nt) <= 220 * 1024) return nt;
    return 0;
}

// One CTA per SM (at least 120 KB of shared memory keeps a second one off).
int launch_scan_tc(const ScanArgs& A, const ScanOut& O, const int64_t* pair_off, const int64_t* item_off,
                   const uint32_t* pairs, int L, int TB, int nt, unsigned long long* next_item, int32_t* status,
                   cudaStream_t st) {
    const size_t smem = std::max<size_t>(ts_smem_bytes(A.M, nt), 120 * 1024);
    KSC_CUDA(cudaFuncSetAttribute(k_scan_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_scan_tc<<<num_sms(), TS_THREADS, smem, st>>>(A, O, pair_off, item_off, pairs, L, TB, nt, next_item, status);
    KSC_LAUNCH_CHECK();
    return KSC_OK;
}

}  // namespace ksc
