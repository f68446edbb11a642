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
//
// Whether the flooding slot decoder stores FP32 messages in base-2 units (R log2 e) while
// APP stays in natural units: Q in base-2 units is then one FMA (APP log2 e - R), the ex2
// argument and the lg2 difference need no scaling multiply, and the variable-node sum
// adds R ln 2 with an FMA; two multiplies fewer per edge update at no other cost.  (FP16
// messages stay natural: the stored binary16 value is the natural one rounded.)
template <typename MsgT>
constexpr bool kSlotB2 = sizeof(MsgT) == 4;

}  // namespace ldpc
