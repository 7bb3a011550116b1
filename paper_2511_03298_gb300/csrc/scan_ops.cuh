// Lookup, widening and reduction steps of the byte-permute scans (search.cu); the
// tensor-core scan (scan_tc.cu) splits its tables by the same lookups.
#pragma once

#include "scan.cuh"

namespace ksc {

// Eight lookups of one 16-entry u8 table t (4 registers, entry e in byte e)
// for the eight 4-bit codes of w (code of vector n in bits 4n..4n+3):
// lo = bytes T[c0..c3], hi = bytes T[c4..c7].  Two byte permutes fetch
// T[c & 7] and T[8 + (c & 7)], a third picks per byte by bit 3 of c.  A byte
// permute reads only the low 16 bits of its selector, so both halves come
// from one masked word and a shift.
__device__ __forceinline__ void lut16x8(uint32_t w, const uint4& t, uint32_t& lo, uint32_t& hi) {
    const uint32_t s0 = w & 0x77777777u;                            // entry index within a half
    const uint32_t s1 = s0 >> 16;
    const uint32_t k0 = ((w >> 1) & 0x44444444u) | 0x32103210u;     // byte n of a (n) or of b (4 + n)
    const uint32_t k1 = k0 >> 16;
    lo = prmt(prmt(t.x, t.y, s0), prmt(t.z, t.w, s0), k0);
    hi = prmt(prmt(t.x, t.y, s1), prmt(t.z, t.w, s1), k1);
}

// Add the 16 lookups of one (subspace, 16-byte code chunk) into the u16x2
// lane sums acc[m] = (vector 2m, vector 2m+1).
__device__ __forceinline__ void accum_chunk(const uint4& c, const uint4& t, uint32_t (&acc)[16]) {
    const uint32_t w[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t lo, hi;
        lut16x8(w[k], t, lo, hi);
        acc[4 * k + 0] += prmt(lo, 0u, 0x4140u);
        acc[4 * k + 1] += prmt(lo, 0u, 0x4342u);
        acc[4 * k + 2] += prmt(hi, 0u, 0x4140u);
        acc[4 * k + 3] += prmt(hi, 0u, 0x4342u);
    }
}

// Two subspaces at once: each lane sum takes both widened lookups in one
// three-input add.
__device__ __forceinline__ void accum_pair(const uint4& c0, const uint4& t0, const uint4& c1, const uint4& t1,
                                           uint32_t (&acc)[16]) {
    const uint32_t w0[4] = {c0.x, c0.y, c0.z, c0.w};
    const uint32_t w1[4] = {c1.x, c1.y, c1.z, c1.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t lo0, hi0, lo1, hi1;
        lut16x8(w0[k], t0, lo0, hi0);
        lut16x8(w1[k], t1, lo1, hi1);
        acc[4 * k + 0] += prmt(lo0, 0u, 0x4140u) + prmt(lo1, 0u, 0x4140u);
        acc[4 * k + 1] += prmt(lo0, 0u, 0x4342u) + prmt(lo1, 0u, 0x4342u);
        acc[4 * k + 2] += prmt(hi0, 0u, 0x4140u) + prmt(hi1, 0u, 0x4140u);
        acc[4 * k + 3] += prmt(hi0, 0u, 0x4342u) + prmt(hi1, 0u, 0x4342u);
    }
}

// The same lookups with the widening done by byte dot products (dp4a with a
// one-hot byte selector adds byte b of the looked-up word to a 32-bit sum):
// acc[v] is the sum of vector v.  The dot products issue on the FMA pipe, so
// the integer pipe keeps only the selector and permute work.
__device__ __forceinline__ void widen_add4(uint32_t x, uint32_t* acc) {
    acc[0] = __dp4a(x, 0x00000001u, acc[0]);
    acc[1] = __dp4a(x, 0x00000100u, acc[1]);
    acc[2] = __dp4a(x, 0x00010000u, acc[2]);
    acc[3] = __dp4a(x, 0x01000000u, acc[3]);
}

__device__ __forceinline__ void accum_chunk32(const uint4& c, const uint4& t, uint32_t (&acc)[32]) {
    const uint32_t w[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t lo, hi;
        lut16x8(w[k], t, lo, hi);
        widen_add4(lo, acc + 8 * k);
        widen_add4(hi, acc + 8 * k + 4);
    }
}

__device__ __forceinline__ void accum_pair32(const uint4& c0, const uint4& t0, const uint4& c1, const uint4& t1,
                                             uint32_t (&acc)[32]) {
    accum_chunk32(c0, t0, acc);
    accum_chunk32(c1, t1, acc);
}

// Selectors of one code word w (eight 4-bit codes, vector n in bits 4n..4n+3)
// for lut16x8, computed once per word and shared by every query slot of a
// warp: (s0, s1, k0, k1).
__device__ __forceinline__ uint4 lut16_selectors(uint32_t w) {
    const uint32_t s0 = w & 0x77777777u;
    const uint32_t k0 = ((w >> 1) & 0x44444444u) | 0x32103210u;
    return make_uint4(s0, s0 >> 16, k0, k0 >> 16);
}

// The lookups of one word from its selectors: lo = T[c0..c3], hi = T[c4..c7].
__device__ __forceinline__ void lut16x8_sel(const uint4& s, const uint4& t, uint32_t& lo, uint32_t& hi) {
    lo = prmt(prmt(t.x, t.y, s.x), prmt(t.z, t.w, s.x), s.z);
    hi = prmt(prmt(t.x, t.y, s.y), prmt(t.z, t.w, s.y), s.w);
}

// Two subspaces j0, j1 from shared selectors (sel[k M + j]: word k of
// subspace j): the looked-up bytes of the same vector from both subspaces
// are interleaved by one byte permute, so one byte dot product adds two
// lookups to the vector's 32-bit sum (acc[v], v the vector of the block).
__device__ __forceinline__ void accum_pair_sel(const uint4* __restrict__ sel, int M, int j0, int j1, const uint4& t0,
                                               const uint4& t1, uint32_t (&acc)[32]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t lo0, hi0, lo1, hi1;
        lut16x8_sel(sel[k * M + j0], t0, lo0, hi0);
        lut16x8_sel(sel[k * M + j1], t1, lo1, hi1);
        uint32_t* a = acc + 8 * k;
        uint32_t x = prmt(lo0, lo1, 0x5140u), y = prmt(lo0, lo1, 0x7362u);
        a[0] = __dp4a(x, 0x00000101u, a[0]);
        a[1] = __dp4a(x, 0x01010000u, a[1]);
        a[2] = __dp4a(y, 0x00000101u, a[2]);
        a[3] = __dp4a(y, 0x01010000u, a[3]);
        x = prmt(hi0, hi1, 0x5140u);
        y = prmt(hi0, hi1, 0x7362u);
        a[4] = __dp4a(x, 0x00000101u, a[4]);
        a[5] = __dp4a(x, 0x01010000u, a[5]);
        a[6] = __dp4a(y, 0x00000101u, a[6]);
        a[7] = __dp4a(y, 0x01010000u, a[7]);
    }
}

__device__ __forceinline__ void accum_chunk_sel(const uint4* __restrict__ sel, int M, int j, const uint4& t,
                                                uint32_t (&acc)[32]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t lo, hi;
        lut16x8_sel(sel[k * M + j], t, lo, hi);
        widen_add4(lo, acc + 8 * k);
        widen_add4(hi, acc + 8 * k + 4);
    }
}

// Reduce-scatter of the 16 u16x2 sums over the G lanes of a group: after it,
// group lane g holds the full sums of vectors V*g .. V*g+V-1 (V = 32/G) in
// out[0..V) (u16 values).
template <int G>
__device__ __forceinline__ void reduce_scatter(uint32_t (&acc)[16], int lane, uint32_t (&out)[32 / G]) {
    constexpr int V = 32 / G;
    int nreg = 16;
#pragma unroll
    for (int o = G / 2; o >= 1; o >>= 1) {
        if (nreg == 1) break;
        const int h = nreg >> 1;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (i < h) {
                uint32_t send = up ? acc[i] : acc[i + h];
                uint32_t keep = up ? acc[i + h] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        nreg = h;
    }
    if constexpr (V == 1) {
        // G = 32: one register of two vectors left; split it over lane bit 0
        const bool odd = lane & 1;
        uint32_t send = odd ? (acc[0] & 0xffffu) : (acc[0] >> 16);
        uint32_t keep = odd ? (acc[0] >> 16) : (acc[0] & 0xffffu);
        out[0] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
    } else {
#pragma unroll
        for (int i = 0; i < V / 2; ++i) {
            out[2 * i] = acc[i] & 0xffffu;
            out[2 * i + 1] = acc[i] >> 16;
        }
    }
}

constexpr uint32_t SCAN_WAIT_LIMIT = 1u << 22;

// Poll an mbarrier phase at most SCAN_WAIT_LIMIT times; false if it never completed.
__device__ __forceinline__ bool scan_wait(uint32_t bar, uint32_t parity) {
    for (uint32_t i = 0; i < SCAN_WAIT_LIMIT; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

}  // namespace ksc
