// RACE feature helpers shared by the tensor-core kernels (tc.cu, tc_ws.cu).
#pragma once

#include "device_common.cuh"
#include "tc_common.cuh"

namespace elsaa {
namespace tc {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

__device__ __forceinline__ uint32_t align1k(uint32_t x) {
    return (x + 1023u) & ~1023u;
}

// Two threads share each row (warps w and w + 4 read the same TMEM lanes).
// The RACE tables of a row are split between them at table `split`, chosen
// so that each half's buckets start on a 32-bucket boundary (whole TMEM
// store groups) and each half reads at most 32 projection columns.
__host__ __device__ inline int table_split(int L, int G) {
    const int R = 1 << G;
    const int unit = R >= 32 ? 1 : 32 / R;  // tables per 32 buckets
    int split = ((L + 1) / 2 + unit - 1) / unit * unit;
    return split > L ? L : split;
}

// Per-bit factors sp[j] = sigmoid(2 beta tanh(a_j)) of the projection
// columns [col0, col0 + 32) of this thread's TMEM lane; entries past `ncols`
// are set to 1/2 and not used.
__device__ __forceinline__ void race_bits32(uint32_t taddr, int ncols,
                                           float beta, float (&sp)[32]) {
    uint32_t pr[32];
    tmem_ld32(taddr, pr);
    tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        if (j < ncols) {
            float t = tanh_approx(beta * tanh_approx(__uint_as_float(pr[j])));
            sp[j] = fmaf(0.5f, t, 0.5f);  // 1/2 + tanh(beta u)/2
        } else {
            sp[j] = 0.5f;
        }
    }
}

// The per-bit factors of n projections already loaded from TMEM (fp32 bits
// in pr). Columns past the last table give values that nothing reads.
template <int n>
__device__ __forceinline__ void race_factors(const uint32_t *pr, float beta,
                                             float *sp) {
#pragma unroll
    for (int j = 0; j < n; ++j)
        sp[j] = fmaf(0.5f,
                     tanh_approx(beta * tanh_approx(__uint_as_float(pr[j]))),
                     0.5f);
}

// Features of table l from its G per-bit factors: phi[r] = prod_b (bit b of
// r ? sp[b] : 1 - sp[b]), r < 2^G.
template <int G>
__device__ __forceinline__ void table_phi(const float *sp, float *phi,
                                          float init = 1.0f) {
    phi[0] = init;  // a common factor of the whole table (1 or a scale)
#pragma unroll
    for (int b = 0; b < G; ++b) {
        const float p = sp[b], q = 1.0f - p;
#pragma unroll
        for (int r = 0; r < (1 << b); ++r) {
            phi[r + (1 << b)] = phi[r] * p;
            phi[r] *= q;
        }
    }
}


// gamma = 4: the 16 features of one table factor as an outer product,
// phi[i + 4 j] = u[i] * w[j], with u over hash bits 0-1 and w over bits 2-3:
// u = (q0 q1, p0 q1, q0 p1, p0 p1), w = (q2 q3, p2 q3, q2 p3, p2 p3),
// p_b = sp[b], q_b = 1 - p_b. `scale` multiplies every feature.
__device__ __forceinline__ void table_uw4(const float *sp, float scale,
                                          float (&u)[4], float (&w)[4]) {
    const float p0 = sp[0], q0 = 1.0f - p0, p1 = sp[1], q1 = 1.0f - p1;
    const float p2 = sp[2], q2 = 1.0f - p2, p3 = sp[3], q3 = 1.0f - p3;
    const float a = q1 * scale, c = p1 * scale;
    u[0] = q0 * a;
    u[1] = p0 * a;
    u[2] = q0 * c;
    u[3] = p0 * c;
    w[0] = q2 * q3;
    w[1] = p2 * q3;
    w[2] = q2 * p3;
    w[3] = p2 * p3;
}

// sum_r phi_r A_r of one gamma = 4 table = sum_j w_j (u . A[4 j .. 4 j + 3]).
__device__ __forceinline__ float table_dot4(const float (&u)[4],
                                            const float (&w)[4],
                                            const float4 (&A)[4]) {
    const float2 u01 = make_float2(u[0], u[1]), u23 = make_float2(u[2], u[3]);
    float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 t = fma2(u23, make_float2(A[j].z, A[j].w),
                              mul2(u01, make_float2(A[j].x, A[j].y)));
        s = fma2(make_float2(w[j], w[j]), t, s);
    }
    return s.x + s.y;
}
// The same with A (16 floats, 16-byte aligned) in shared memory.
__device__ __forceinline__ float table_dot4(const float (&u)[4],
                                            const float (&w)[4],
                                            const float *A) {
    float4 a[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
        a[j] = *reinterpret_cast<const float4 *>(A + 4 * j);
    return table_dot4(u, w, a);
}

// Packed bf16 features of one gamma = 4 table: out[k] holds buckets
// (2k, 2k + 1), k < 8.
__device__ __forceinline__ void table_pack4(const float (&u)[4],
                                            const float (&w)[4],
                                            uint32_t *out) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 wj = make_float2(w[j], w[j]);
        const float2 a = mul2(make_float2(u[0], u[1]), wj);
        const float2 b = mul2(make_float2(u[2], u[3]), wj);
        out[2 * j] = pack_bf16x2(a.x, a.y);
        out[2 * j + 1] = pack_bf16x2(b.x, b.y);
    }
}

// sum_r phi_r A_r of one gamma = 4 table from its per-bit factors, bit by
// bit from the highest: A[i] <- q A[i] + p A[i + half], all terms positive as
// in table_dot4. Fewer operations (7 + 7 in pairs against 8 single and 12 in
// pairs) in a longer chain. The block kernel takes it where one query buffer
// is in flight and no window is walked. us with table_dot4 and with this, 32
// heads of 16384 rows, d = 128, r = 256: c3 133 and 128, top-k of one block 164
// and 161, of two, three and four 226 and 225, 312 and 311, 390 and 391,
// r = 128 with b = 128, 64 110 and 110, 109 and 109; but a window of three
// blocks 244 and 255. 48 heads of 8192 rows, d = 64, b = 256: r = 128 105 and
// 107, r = 256 126 and 124. With three query buffers c2 37 and 39, c5 106 and
// 110; the pair kernel 584 with both.
// A: 16 floats, 16-byte aligned, in shared memory.
__device__ __forceinline__ float table_den4(const float *sp, const float *A) {
    float4 a[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
        a[j] = *reinterpret_cast<const float4 *>(A + 4 * j);
    const float2 p3 = make_float2(sp[3], sp[3]),
                 p2 = make_float2(sp[2], sp[2]),
                 p1 = make_float2(sp[1], sp[1]);
    const float2 q3 = make_float2(1.0f - sp[3], 1.0f - sp[3]),
                 q2 = make_float2(1.0f - sp[2], 1.0f - sp[2]),
                 q1 = make_float2(1.0f - sp[1], 1.0f - sp[1]);
    auto lo = [](const float4 &x) { return make_float2(x.x, x.y); };
    auto hi = [](const float4 &x) { return make_float2(x.z, x.w); };
    const float2 c0 = fma2(p3, lo(a[2]), mul2(q3, lo(a[0]))),
                 c1 = fma2(p3, hi(a[2]), mul2(q3, hi(a[0]))),
                 c2 = fma2(p3, lo(a[3]), mul2(q3, lo(a[1]))),
                 c3 = fma2(p3, hi(a[3]), mul2(q3, hi(a[1])));
    const float2 b0 = fma2(p2, c2, mul2(q2, c0)),
                 b1 = fma2(p2, c3, mul2(q2, c1));
    const float2 t = fma2(p1, b1, mul2(q1, b0));
    return fmaf(sp[0], t.y, (1.0f - sp[0]) * t.x);
}

// sum over tables t < nt of phi_t . A_t for the tables of one 64-bucket
// chunk (at most TT of them; per-bit factors sp[t * G ..], A of the chunk's
// first table at A). Four independent partial sums in acc. FOLD: which of the
// two forms gamma = 4 takes.
template <int G, int TT, bool FOLD = false>
__device__ __forceinline__ void chunk_den(const float *sp, int nt,
                                          const float *A, float (&acc)[4]) {
    constexpr int R = 1 << G;
#pragma unroll
    for (int t = 0; t < TT; ++t) {
        if (t < nt) {
            if constexpr (G == 4) {
                if constexpr (FOLD) {
                    acc[t & 3] += table_den4(&sp[t * G], A + t * R);
                } else {
                    float u[4], w[4];
                    table_uw4(&sp[t * G], 1.0f, u, w);
                    acc[t & 3] += table_dot4(u, w, A + t * R);
                }
            } else {
                float phi[R];
                table_phi<G>(&sp[t * G], phi);
#pragma unroll
                for (int q = 0; q < R; ++q)
                    acc[q & 3] = fmaf(phi[q], A[t * R + q], acc[q & 3]);
            }
        }
    }
}

// Writes the features phi * scale of the nt (<= TT) tables of one 64-bucket
// chunk as packed bf16 pairs into TMEM: bucket pair (2k, 2k + 1) of the
// chunk at column taddr + k, k < 32, in two stores of 16 columns (the second
// only when the chunk holds more than 32 buckets). Pairs past the chunk's
// last table are zero.
template <int G, int TT>
__device__ __forceinline__ void write_phi_chunk(const float *sp, int nt,
                                                float scale, uint32_t taddr) {
    constexpr int R = 1 << G;
    static_assert(TT * R == 64, "a chunk is 64 buckets");
    uint32_t buf[16];
#pragma unroll
    for (int t = 0; t < TT; ++t) {
        uint32_t pk[R / 2];
        if (t < nt) {
            if constexpr (G == 4) {
                float u[4], w[4];
                table_uw4(&sp[t * G], scale, u, w);
                table_pack4(u, w, pk);
            } else {
                float phi[R];
                table_phi<G>(&sp[t * G], phi, scale);
#pragma unroll
                for (int q = 0; q < R; q += 2)
                    pk[q >> 1] = pack_bf16x2(phi[q], phi[q + 1]);
            }
        } else {
#pragma unroll
            for (int q = 0; q < R / 2; ++q) pk[q] = 0u;
        }
#pragma unroll
        for (int q = 0; q < R / 2; ++q) {
            const int k = t * (R / 2) + q;
            buf[k & 15] = pk[q];
            if ((k & 15) == 15 && (k < 16 || nt * R > 32))
                tmem_st16(taddr + (uint32_t)(k - 15), buf);
        }
    }
}

// TMEM column of K-step k (16 keys or buckets = 8 packed bf16 columns) of
// the quarter pair starting at col0: quarters (col0, col0 + 64) of 32
// columns each, the A operand of the P V and Phi'B products in the block
// kernels' slots.
__device__ __forceinline__ uint32_t quarter_col(int k, int col0) {
    return (uint32_t)(col0 + (k < 4 ? 8 * k : 64 + 8 * (k - 4)));
}

}  // namespace tc
}  // namespace elsaa
