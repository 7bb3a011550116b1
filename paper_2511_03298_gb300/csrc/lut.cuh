// The quantised residual tables (a2): the FP32 rule of a table row, its 8-bit
// entries and the integer bias, shared by the table kernels (search.cu) and the
// small-batch kernel (small.cu).
//
// FP32 rule of the table entries, every op separately rounded:
//   L2: u_t = q_t - c_t, acc += (u_t - C_jit)^2 over t ascending
//   IP: u_t = q_t,       acc += u_t C_jit,                        T = -acc
// The row operand u (the dsub values of subspace j) is formed once per row;
// each entry is then the same sequence of rounded ops as written above.
#pragma once

#include "scan.cuh"

namespace ksc {

struct LutArgs {
    const float* Q;
    int64_t nq;
    int d, M, dsub, ip, Pmax;
    const int32_t* probes;
    const int32_t* nprobe_q;
    int Pfix;
    const float* c_mean;
    const float* cb;
    int L;
    // optional compact work: pairs e = q * Pmax + r, two ranges (NULL: every
    // (q, r < P_q))
    const uint32_t* pairs0;
    const int64_t* npairs0;
    const uint32_t* pairs1;
    const int64_t* npairs1;
};

// Item i of the LUT pass: its (query, rank) flat index, or -1 if it does no work.
__device__ __forceinline__ int64_t lut_item(const LutArgs& A, int64_t i, int64_t n0) {
    if (A.pairs0) return i < n0 ? (int64_t)A.pairs0[i] : (int64_t)A.pairs1[i - n0];
    return i;
}

__device__ __forceinline__ int64_t lut_items(const LutArgs& A, int64_t* n0) {
    if (A.pairs0) {
        *n0 = *A.npairs0;
        return *n0 + *A.npairs1;
    }
    *n0 = 0;
    return A.nq * A.Pmax;
}

__device__ __forceinline__ int probes_of(const LutArgs& A, int64_t q) {
    int P = A.nprobe_q ? A.nprobe_q[q] : A.Pfix;
    return P < 1 ? 1 : (P > A.Pmax ? A.Pmax : P);
}

// Codebook row stride in shared memory.  dsub = 2: 34 floats (codewords
// 8-byte aligned; a half-warp reading 16 consecutive rows with 8-byte loads
// covers all 32 banks once); dsub = 4: 68 (16-byte aligned; 8 consecutive rows
// of a 16-byte load cover all banks once); else 16 dsub + 1 (odd: 32
// consecutive rows fall in distinct banks).
__host__ __device__ __forceinline__ int cb_ld(int dsub) {
    return dsub == 2 ? 34 : (dsub == 4 ? 68 : PQ_K * dsub + 1);
}

__device__ __forceinline__ void stage_codebook(const LutArgs& A, float* cbs) {
    const int ld = cb_ld(A.dsub), rowlen = PQ_K * A.dsub;
    for (int e = threadIdx.x; e < A.M * rowlen; e += blockDim.x) {
        const int j = e / rowlen;
        cbs[j * ld + (e - j * rowlen)] = A.cb[e];
    }
    __syncthreads();
}

// The 16 FP32 entries of one subspace: qj, cj = the query's and the list
// centroid's values of the subspace, cw = its codebook row in shared memory.
// DS = dsub when fixed at compile time (2: 8-byte loads, 4: 16-byte loads; qj
// and cj aligned to that), 0 = read from dsub.  (60k x 784, M 196, 10,000
// queries at nprobe 4: 419 us with width 4 read from dsub, 367 us fixed.)
template <int DS>
__device__ __forceinline__ void row_table(int dsub, int ip, const float* __restrict__ qj,
                                          const float* __restrict__ cj, const float* cw, float (&T)[PQ_K]) {
    if constexpr (DS == 2) {
        const float2 qv = *reinterpret_cast<const float2*>(qj);
        float u0 = qv.x, u1 = qv.y;
        if (!ip) {
            const float2 cv = *reinterpret_cast<const float2*>(cj);
            u0 = __fsub_rn(u0, cv.x);
            u1 = __fsub_rn(u1, cv.y);
        }
#pragma unroll
        for (int i = 0; i < PQ_K; ++i) {
            const float2 c = *reinterpret_cast<const float2*>(cw + 2 * i);
            float acc = 0.f;
            if (ip) {
                acc = __fadd_rn(acc, __fmul_rn(u0, c.x));
                acc = __fadd_rn(acc, __fmul_rn(u1, c.y));
                T[i] = -acc;
            } else {
                // 0 + e0^2 is e0^2 exactly (a square is +0 or more), so the sum
                // from 0 needs one addition; both differences and both squares
                // as packed pairs
                const float2 e = f2_sub(make_float2(u0, u1), c);
                const float2 e2 = f2_mul(e, e);
                T[i] = __fadd_rn(e2.x, e2.y);
            }
        }
    } else if constexpr (DS == 4) {
        // 16-byte loads, differences, products and squares as packed pairs, the
        // sums in ascending t (0 + the first term is the term)
        const float4 qv = *reinterpret_cast<const float4*>(qj);
        float2 u01 = make_float2(qv.x, qv.y), u23 = make_float2(qv.z, qv.w);
        if (!ip) {
            const float4 cv = *reinterpret_cast<const float4*>(cj);
            u01 = f2_sub(u01, make_float2(cv.x, cv.y));
            u23 = f2_sub(u23, make_float2(cv.z, cv.w));
        }
#pragma unroll
        for (int i = 0; i < PQ_K; ++i) {
            const float4 c = *reinterpret_cast<const float4*>(cw + 4 * i);
            float2 e01, e23;
            if (ip) {
                e01 = f2_mul(u01, make_float2(c.x, c.y));
                e23 = f2_mul(u23, make_float2(c.z, c.w));
                e01.x = __fadd_rn(0.f, e01.x);
            } else {
                e01 = f2_sub(u01, make_float2(c.x, c.y));
                e23 = f2_sub(u23, make_float2(c.z, c.w));
                e01 = f2_mul(e01, e01);
                e23 = f2_mul(e23, e23);
            }
            const float s = __fadd_rn(__fadd_rn(__fadd_rn(e01.x, e01.y), e23.x), e23.y);
            T[i] = ip ? -s : s;
        }
    } else {
#pragma unroll
        for (int i = 0; i < PQ_K; ++i) T[i] = 0.f;
        for (int t = 0; t < dsub; ++t) {
            const float u = ip ? qj[t] : __fsub_rn(qj[t], cj[t]);
#pragma unroll
            for (int i = 0; i < PQ_K; ++i) {
                const float c = cw[i * dsub + t];
                if (ip) {
                    T[i] = __fadd_rn(T[i], __fmul_rn(u, c));
                } else {
                    const float e = __fsub_rn(u, c);
                    T[i] = __fadd_rn(T[i], __fmul_rn(e, e));
                }
            }
        }
        if (ip) {
#pragma unroll
            for (int i = 0; i < PQ_K; ++i) T[i] = -T[i];
        }
    }
}

// u8 entry min(255, floor((T - m) a + 1/2)) of four table entries, packed.
// T >= m, so the argument of floor is positive (or NaN, which converts to 0
// either way) and a conversion rounding down gives floor directly.
__device__ __forceinline__ uint32_t quant4(const float* T, float mn, float a) {
    uint32_t v[4];
#pragma unroll
    for (int i = 0; i < 4; i += 2) {  // (T - m) a + 1/2 of two entries as packed pairs
        const float2 x = f2_add(f2_mul(f2_sub(make_float2(T[i], T[i + 1]), make_float2(mn, mn)), make_float2(a, a)),
                                make_float2(0.5f, 0.5f));
        v[i] = min(__float2uint_rd(x.x), 255u);
        v[i + 1] = min(__float2uint_rd(x.y), 255u);
    }
    return __byte_perm(__byte_perm(v[0], v[1], 0x0040), __byte_perm(v[2], v[3], 0x0040), 0x5410);
}

// Integer bias floor(S a + 1/2) of one (query, list), S = sum_j m_j in
// ascending j (+ -<q, c_p> first for IP), clamped to +-2^30.
__device__ __forceinline__ int32_t lut_bias(const LutArgs& A, const float* __restrict__ qv, const float* __restrict__ cp,
                                            const float* mins, float a) {
    float S = 0.f;
    if (A.ip) {
        float dot = 0.f;
        for (int t = 0; t < A.d; ++t) dot = __fadd_rn(dot, __fmul_rn(qv[t], cp[t]));
        S = -dot;
    }
    for (int j = 0; j < A.M; ++j) S = __fadd_rn(S, mins[j]);
    float bf = floorf(__fadd_rn(__fmul_rn(S, a), 0.5f));
    bf = fminf(fmaxf(bf, -1073741824.f), 1073741823.f);
    return (int32_t)bf;
}

}  // namespace ksc
