// Device code shared by the decoders that keep a codeword on chip (flooding slots, two-SM
// clusters, layered sum-product): the check rule in the product (tanh) domain.
#pragma once

#include "ldpc_internal.h"

namespace ldpc {

// The approximate base-2 exponential and logarithm of the special-function units.
__device__ __forceinline__ float s_ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float s_lg2(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
constexpr float kSLog2e = 1.4426950408889634f;
constexpr float kSLn2 = 0.6931471805599453f;

// phi(X) log2 e, the lower end [phi(X), X] of the clamp of |Q| in base-2 units (once per
// kernel): log2((1 + t)/(1 - t)) with t = e^-X, as two logarithms of opposite sign below
// X = 3 and from the series 2t + 2t^3/3 (relative accuracy) above.
__device__ __forceinline__ float s_phi_b2(float X)
{
    const float t = s_ex2(-X * kSLog2e);
    return X > 3.0f ? t * fmaf(t * t, (2.0f / 3.0f) * kSLog2e, 2.0f * kSLog2e) : s_lg2(1.0f + t) - s_lg2(1.0f - t);
}

// Degree dispatch: the checks of one block row all have the same degree, so every lane of
// a warp takes the same branch.  Degrees up to 8 get an exact, guard-free body; larger
// degrees share buckets of four (edges past the degree are skipped under a uniform guard).
__host__ __device__ constexpr int next_degree(int d) { return d < 8 ? d + 1 : d + 4; }

template <typename T>
__device__ __forceinline__ const T *at(const char *base, int off) { return reinterpret_cast<const T *>(base + off); }
template <typename T>
__device__ __forceinline__ T *at(char *base, int off) { return reinterpret_cast<T *>(base + off); }

// The check rule of the sum-product algorithm,
//   R'_k = prod_{j != k} sgn Q_j * min(X, phi(sum_{j != k} phi(a_j))),  a_j = |Q_j| clamped to [phi(X), X],
// in the product (tanh) domain.  With d_j = e^-a_j, tanh(a_j / 2) = (1 - d_j) / (1 + d_j), and
// the exclusive product P_k of the other edges' tanh gives R_k = ln((1 + P_k) / (1 - P_k)),
// which is phi(sum_{j != k} phi(a_j)) exactly (phi(x) = -ln tanh(x / 2) is its own inverse).
// With B = prod (1 + d_j) and A = prod (1 - d_j), the pair alpha = (B + A) / 2,
// beta = (B - A) / 2 gives (1 + P) / (1 - P) = alpha / beta, and one more factor d maps it
// to (alpha + d beta, beta + d alpha): every term is non-negative, so neither 1 - P nor the
// exclusion of edge k cancels (the exclusion combines prefix and suffix pairs as the product
// of the two maps).  Per edge this is one ex2 (of |Q|) and two lg2 (of alpha and beta).
// The clamp of a_j to [phi(X), X] is a clamp of the ex2 argument to [-Xb, -Pb]
// (Xb = X log2 e, Pb = phi(X) log2 e); the clamp min(X, .) of the result never binds, as
// phi(sum_{j != k} phi(a_j)) <= min_{j != k} a_j <= X, so it is not applied.
// B2: Q and R in base-2 units (LLR x log2 e), where neither the ex2 argument nor the lg2
// difference needs a scaling multiply; else natural units (FP16 messages, whose stored value
// is the natural one rounded to binary16).
template <bool B2>
__device__ __forceinline__ float tanh_d(float q, float Xb, float Pb)
{
    return s_ex2(fminf(fmaxf(B2 ? -fabsf(q) : fabsf(q) * -kSLog2e, -Xb), -Pb));
}
template <bool B2>
__device__ __forceinline__ float tanh_mag(float al, float be)
{
    const float l = s_lg2(al) - s_lg2(be);
    return B2 ? l : l * kSLn2;
}

// The exclusive pair of an edge from its prefix and suffix pairs.
__device__ __forceinline__ void tanh_combine(float pa, float pb, float sa, float sb, float &al, float &be)
{
    al = fmaf(pb, sb, pa * sa);
    be = fmaf(pb, sa, pa * sb);
}

// The product-domain rule for a row of degree dc <= D with D > 8, in groups of 8 edges,
// holding no per-edge state between its two passes (the registers of D pairs would spill):
//   pass 1 forms every d_k and each group's pair (the product of its edges' maps);
//   pass 2, group by group, forms the group's d_k again, its suffix pairs, and a prefix
//   that starts from the product of the other groups' pairs.
// Every term stays non-negative, as in the prefix / suffix form of rows up to degree 8.
// qof(k, first) returns Q_k of edge k (`first`: pass 1, where the caller also takes what it
// needs once per edge); put(k, R, Q) writes the signed message R of edge k (Q: its Q_k).
__device__ __forceinline__ void pair_mul(float a1, float b1, float a2, float b2, float &a, float &b)
{
    a = fmaf(b1, b2, a1 * a2);
    b = fmaf(b1, a2, a1 * b2);
}

template <int D, bool B2, typename QF, typename PF>
__device__ __forceinline__ void tanh_check_wide(int dc, float Xb, float Pb, QF qof, PF put)
{
    constexpr uint32_t kSign = 0x80000000u;
    constexpr int G = (D + 7) / 8;
    float ga[G], gb[G];
    uint32_t sg = 0;
#pragma unroll
    for (int g = 0; g < G; g++) {
        ga[g] = 1.0f;
        gb[g] = 0.0f;
    }
    // the loops leave at the row's degree (a warp-uniform test) rather than predicate the
    // edges of the body past it
#pragma unroll
    for (int g = 0; g < G; g++) {
        if (8 * g >= dc) break;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int k = 8 * g + i;
            if (k >= D || k >= dc) break;
            {
                const float q = qof(k, true);
                sg ^= __float_as_uint(q);
                const float d = tanh_d<B2>(q, Xb, Pb);
                if (i == 0) {
                    gb[g] = d;
                } else {
                    const float t = fmaf(d, gb[g], ga[g]);
                    gb[g] = fmaf(d, ga[g], gb[g]);
                    ga[g] = t;
                }
            }
        }
    }
#pragma unroll
    for (int g = 0; g < G; g++) {
        if (8 * g >= dc) break;
        // the other groups' product
        float pa = 1.0f, pb = 0.0f;
        bool first = true;
#pragma unroll
        for (int h = 0; h < G; h++) {
            if (h == g) continue;
            if (first) {
                pa = ga[h];
                pb = gb[h];
                first = false;
            } else {
                pair_mul(pa, pb, ga[h], gb[h], pa, pb);
            }
        }
        float d[8];
        uint32_t qb[8];
#pragma unroll
        for (int i = 0; i < 8; i++) {
            d[i] = 0.0f;  // a missing edge is the identity map
            qb[i] = 0;
        }
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int k = 8 * g + i;
            if (k >= D || k >= dc) break;
            {
                const float q = qof(k, false);
                qb[i] = __float_as_uint(q);
                d[i] = tanh_d<B2>(q, Xb, Pb);
            }
        }
        float sa[9], sb[9];
        sa[8] = 1.0f;
        sb[8] = 0.0f;
        sa[7] = 1.0f;
        sb[7] = d[7];
#pragma unroll
        for (int i = 6; i >= 1; i--) {
            sa[i] = fmaf(d[i], sb[i + 1], sa[i + 1]);
            sb[i] = fmaf(d[i], sa[i + 1], sb[i + 1]);
        }
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int k = 8 * g + i;
            if (k >= D || k >= dc) break;
            float al, be;
            if (i == 7)
                al = pa, be = pb;
            else
                pair_mul(pa, pb, sa[i + 1], sb[i + 1], al, be);
            {
                const float mag = tanh_mag<B2>(al, be);
                put(k, __uint_as_float(__float_as_uint(mag) | ((qb[i] ^ sg) & kSign)), __uint_as_float(qb[i]));
            }
            if (i < 7) {
                const float t = fmaf(d[i], pb, pa);
                pb = fmaf(d[i], pa, pb);
                pa = t;
            }
        }
    }
}

// The grouped rule holding each edge's factor between its two passes (d_k in a register,
// the sign of Q_k in d_k's own sign bit): pass 2 then needs no second load of the edge's
// operands and no second ex2.  put(k, R) writes the signed message of edge k.
template <int D, bool B2, typename QF, typename PF>
__device__ __forceinline__ void tanh_check_wide_held(int dc, float Xb, float Pb, QF qof, PF put)
{
    constexpr uint32_t kSign = 0x80000000u;
    constexpr int G = (D + 7) / 8;
    float ga[G], gb[G];
    uint32_t dq[D];  // d_k with the sign of Q_k
    uint32_t sg = 0;
#pragma unroll
    for (int g = 0; g < G; g++) {
        ga[g] = 1.0f;
        gb[g] = 0.0f;
    }
#pragma unroll
    for (int k = 0; k < D; k++) dq[k] = 0;
#pragma unroll
    for (int g = 0; g < G; g++) {
        if (8 * g >= dc) break;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int k = 8 * g + i;
            if (k >= D || k >= dc) break;
            const float q = qof(k);
            const uint32_t qs = __float_as_uint(q) & kSign;
            sg ^= qs;
            const float d = tanh_d<B2>(q, Xb, Pb);
            dq[k] = __float_as_uint(d) | qs;
            if (i == 0) {
                gb[g] = d;
            } else {
                const float t = fmaf(d, gb[g], ga[g]);
                gb[g] = fmaf(d, ga[g], gb[g]);
                ga[g] = t;
            }
        }
    }
#pragma unroll
    for (int g = 0; g < G; g++) {
        if (8 * g >= dc) break;
        float pa = 1.0f, pb = 0.0f;
        bool first = true;
#pragma unroll
        for (int h = 0; h < G; h++) {
            if (h == g) continue;
            if (first) {
                pa = ga[h];
                pb = gb[h];
                first = false;
            } else {
                pair_mul(pa, pb, ga[h], gb[h], pa, pb);
            }
        }
        float d[8];
#pragma unroll
        for (int i = 0; i < 8; i++) d[i] = (8 * g + i < D) ? __uint_as_float(dq[8 * g + i] & ~kSign) : 0.0f;
        float sa[9], sb[9];
        sa[8] = 1.0f;
        sb[8] = 0.0f;
        sa[7] = 1.0f;
        sb[7] = d[7];
#pragma unroll
        for (int i = 6; i >= 1; i--) {
            sa[i] = fmaf(d[i], sb[i + 1], sa[i + 1]);
            sb[i] = fmaf(d[i], sa[i + 1], sb[i + 1]);
        }
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int k = 8 * g + i;
            if (k >= D || k >= dc) break;
            float al, be;
            if (i == 7)
                al = pa, be = pb;
            else
                pair_mul(pa, pb, sa[i + 1], sb[i + 1], al, be);
            put(k, __uint_as_float(__float_as_uint(tanh_mag<B2>(al, be)) | ((dq[k] ^ sg) & kSign)));
            if (i < 7) {
                const float t = fmaf(d[i], pb, pa);
                pb = fmaf(d[i], pa, pb);
                pa = t;
            }
        }
    }
}

// Whether the flooding slot decoder stores FP32 messages in base-2 units (R log2 e) while
// APP stays in natural units: Q in base-2 units is then one FMA (APP log2 e - R), the ex2
// argument and the lg2 difference need no scaling multiply, and the variable-node sum
// adds R ln 2 with an FMA; two multiplies fewer per edge update at no other cost.  (FP16
// messages stay natural: the stored binary16 value is the natural one rounded.)
#ifndef LDPC_SLOTS_B2
#define LDPC_SLOTS_B2 1
#endif
template <typename MsgT>
constexpr bool kSlotB2 = LDPC_SLOTS_B2 && sizeof(MsgT) == 4;

}  // namespace ldpc
