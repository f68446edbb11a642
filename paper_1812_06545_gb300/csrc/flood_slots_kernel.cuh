// The kernel of the flooding slot decoder (see flood_slots.cu for the schedule and the host
// side); its instances are compiled one translation unit per message type and clamp form
// (flood_slots_f32.cu, ...).
#pragma once

#include "flood_slots.h"
#include "slot_common.cuh"

namespace ldpc {

// Channel values a thread loads at once when a slot takes a codeword.
constexpr int kRefillChunk = 8;
// Columns whose channel values a thread requests at once in the variable-node phase (4: 915 us
// against 907 on the N = 1944 rate-1/2 FP32 launch, 655 against 645 FP16).
constexpr int kVnChunk = 3;

// ------------------------------------------------------------------ V codewords per thread
//
// A value of a thread is a float (one codeword) or a float2 (two codewords, whose multiplies
// and adds issue as packed pairs; each half is rounded exactly as the scalar operation).
template <int V>
struct Vec;
template <>
struct Vec<1> {
    using T = float;
};
template <>
struct Vec<2> {
    using T = float2;
};
template <int V>
using VT = typename Vec<V>::T;
__device__ __forceinline__ float vset(float, float c) { return c; }
__device__ __forceinline__ float2 vset(float2, float c) { return make_float2(c, c); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
// apply f(element, element index) to the elements
template <typename F>
__device__ __forceinline__ void each(float &x, F f) { f(x, 0); }
template <typename F>
__device__ __forceinline__ void each(float2 &x, F f)
{
    f(x.x, 0);
    f(x.y, 1);
}

// Shared-memory access of V consecutive codewords' values at a byte offset of the dynamic
// shared memory.
template <typename MsgT, int V>
struct Sm;
template <>
struct Sm<float, 1> {
    static __device__ __forceinline__ float ld(const char *p) { return *reinterpret_cast<const float *>(p); }
    static __device__ __forceinline__ void st(char *p, float x) { *reinterpret_cast<float *>(p) = x; }
};
template <>
struct Sm<float, 2> {
    static __device__ __forceinline__ float2 ld(const char *p) { return *reinterpret_cast<const float2 *>(p); }
    static __device__ __forceinline__ void st(char *p, float2 x) { *reinterpret_cast<float2 *>(p) = x; }
};
template <>
struct Sm<__half, 1> {
    static __device__ __forceinline__ float ld(const char *p)
    {
        return __half2float(*reinterpret_cast<const __half *>(p));
    }
    static __device__ __forceinline__ void st(char *p, float x)
    {
        *reinterpret_cast<__half *>(p) = __float2half_rn(x);
    }
};
template <>
struct Sm<__half, 2> {
    static __device__ __forceinline__ float2 ld(const char *p)
    {
        return __half22float2(*reinterpret_cast<const __half2 *>(p));
    }
    static __device__ __forceinline__ void st(char *p, float2 x)
    {
        *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(x.x, x.y);
    }
};

// ------------------------------------------------------------------ the check rule
//
// Messages are stored negated (N = -R): Q = APP + N needs no negation and the variable-node
// sum adds -N (a multiply-add by a negative constant).  The rule itself is slot_common.cuh's:
// d = e^-a per edge, prefix and suffix products of the maps (alpha, beta) <- (alpha + d beta,
// beta + d alpha), R = ln(alpha / beta) with the sign of the other edges.

// d of each codeword.  HC: the upper clamp a >= phi(X) is applied; without it the clamp is
// known not to change d (phi(X) so small that ex2 rounds e^-phi(X) to 1, see flood_slots.cu).
template <bool B2, bool HC>
__device__ __forceinline__ float form_d(float q, float Xb, float Pb)
{
    const float x = fmaxf(B2 ? -fabsf(q) : fabsf(q) * -kSLog2e, -Xb);
    return s_ex2(HC ? fminf(x, -Pb) : x);
}
template <bool B2, bool HC>
__device__ __forceinline__ float2 form_d(float2 q, float Xb, float Pb)
{
    if constexpr (!B2) q = __fmul2_rn(q, make_float2(kSLog2e, kSLog2e));  // |q| -log2 e = -|q log2 e| exactly
    return make_float2(form_d<true, HC>(q.x, Xb, Pb), form_d<true, HC>(q.y, Xb, Pb));
}

// -ln(alpha / beta) in the message's unit
template <bool B2>
__device__ __forceinline__ float neg_mag(float al, float be)
{
    const float l = s_lg2(be) - s_lg2(al);
    return B2 ? l : l * kSLn2;
}
template <bool B2>
__device__ __forceinline__ float2 neg_mag(float2 al, float2 be)
{
    const float2 l = __ffma2_rn(make_float2(s_lg2(al.x), s_lg2(al.y)), make_float2(-1.0f, -1.0f),
                                make_float2(s_lg2(be.x), s_lg2(be.y)));
    return B2 ? l : __fmul2_rn(l, make_float2(kSLn2, kSLn2));
}

// A thread's place: byte offsets of its row's position in the slot's APP and messages, plain
// and less one block (for the edges whose row wraps), and its row.
template <int V>
struct Place {
    uint32_t a0, a1, r0, r1;
    int r;
    bool own;  // an idle lane of a slot's last warp repeats the last row's loads and stores nothing
};

// The edge's operand offsets.  With one element size for APP and messages the two regions of
// a slot are at a fixed distance (already in the descriptor's .y), so one select serves both.
template <int V, typename MsgT>
__device__ __forceinline__ void edge_at(const int4 &e, const Place<V> &p, uint32_t &ao, uint32_t &ro)
{
    const bool w = p.r >= e.z;
    const uint32_t a = w ? p.a1 : p.a0;
    ao = a + (uint32_t)e.x;
    if constexpr (sizeof(MsgT) == sizeof(float))
        ro = a + (uint32_t)e.y;
    else
        ro = (w ? p.r1 : p.r0) + (uint32_t)e.y;
}

// Rows up to degree 8: every edge's state in registers.
template <int D, int V, typename MsgT, bool HC>
__device__ __forceinline__ void check_narrow(const int4 *__restrict__ ed, char *sm, const Place<V> &p, float Xb,
                                             float Pb, uint32_t (&pbad)[V])
{
    constexpr bool B2 = kSlotB2<MsgT>;
    constexpr uint32_t kSign = 0x80000000u;
    using T = VT<V>;
    const T one = vset(T(), 1.0f), zero = vset(T(), 0.0f);
    T d[D];
    uint32_t ro[D], par[V];
    uint32_t sg[V];  // the signs of Q: edge k's in bit D - 1 - k (a word per codeword, not one per edge)
#pragma unroll
    for (int v = 0; v < V; v++) sg[v] = par[v] = 0;
#pragma unroll
    for (int k = 0; k < D; k++) {
        uint32_t ao;
        edge_at<V, MsgT>(ed[k], p, ao, ro[k]);
        T ap = Sm<float, V>::ld(sm + ao);
        const T n = Sm<MsgT, V>::ld(sm + ro[k]);
        T q = B2 ? vfma(ap, vset(T(), kSLog2e), n) : vadd(ap, n);
        each(ap, [&](float x, int v) { par[v] ^= __float_as_uint(x); });
        each(q, [&](float x, int v) { sg[v] = __funnelshift_l(__float_as_uint(x), sg[v], 1); });
        d[k] = form_d<B2, HC>(q, Xb, Pb);
    }
#pragma unroll
    for (int v = 0; v < V; v++) sg[v] ^= 0u - (__popc(sg[v]) & 1u);  // the product of the other edges' signs
    T sa[D + 1], sb[D + 1];  // suffix maps of edges k..D-1 applied to (1, 0)
    sa[D - 1] = one;
    sb[D - 1] = d[D - 1];
#pragma unroll
    for (int k = D - 2; k >= 1; k--) {
        sa[k] = vfma(d[k], sb[k + 1], sa[k + 1]);
        sb[k] = vfma(d[k], sa[k + 1], sb[k + 1]);
    }
    T pa = one, pb = zero;
#pragma unroll
    for (int k = 0; k < D; k++) {
        T al, be;
        if (k == 0) {
            al = sa[1];
            be = sb[1];
        } else if (k == D - 1) {
            al = pa;
            be = pb;
        } else if (k == D - 2) {  // the suffix is one edge's map (1, d): one rounding less
            al = vfma(pb, sb[D - 1], pa);
            be = vfma(pa, sb[D - 1], pb);
        } else {
            al = vfma(pb, sb[k + 1], vmul(pa, sa[k + 1]));
            be = vfma(pb, sa[k + 1], vmul(pa, sb[k + 1]));
        }
        T n = neg_mag<B2>(al, be);
        each(n, [&](float &x, int v) { x = __uint_as_float(__float_as_uint(x) & ~((sg[v] << (32 - D + k)) & kSign)); });
        if (p.own) Sm<MsgT, V>::st(sm + ro[k], n);
        if (k == 0) {
            pb = d[0];
        } else if (k < D - 1) {
            const T t = vfma(d[k], pb, pa);
            pb = vfma(d[k], pa, pb);
            pa = t;
        }
    }
#pragma unroll
    for (int v = 0; v < V; v++) pbad[v] |= par[v];
}

// Rows above degree 8 in groups of 8 edges: pass 1 forms every edge's factor d and each
// group's pair (the product of its edges' maps); pass 2, group by group, the group's suffix
// pairs and a prefix that starts from the product of the other groups' pairs.  Full groups have
// straight-line code (their loads overlap); a row's last group leaves its edge loops at the row's
// degree (warp-uniform tests).

// d of a group's edges (0 past its end: the identity map), the suffix pairs, and every edge's
// message from them and the others' product (pa, pb).  sg: the signs, edge i's in bit 31 - i;
// store(i, N) writes the message.
template <bool FULL, bool B2, int V, typename ST>
__device__ __forceinline__ void group_out(int n, const VT<V> (&d)[8], VT<V> pa, VT<V> pb, const uint32_t (&sg)[V], ST store)
{
    constexpr uint32_t kSign = 0x80000000u;
    using T = VT<V>;
    T sa[8], sb[8];
    sa[7] = vset(T(), 1.0f);
    sb[7] = d[7];
#pragma unroll
    for (int i = 6; i >= 1; i--) {
        sa[i] = vfma(d[i], sb[i + 1], sa[i + 1]);
        sb[i] = vfma(d[i], sa[i + 1], sb[i + 1]);
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
        if (!FULL && i >= n) break;
        T al, be;
        if (i == 7) {
            al = pa;
            be = pb;
        } else if (i == 6) {  // the suffix is one edge's map (1, d): one rounding less
            al = vfma(pb, sb[7], pa);
            be = vfma(pa, sb[7], pb);
        } else {
            al = vfma(pb, sb[i + 1], vmul(pa, sa[i + 1]));
            be = vfma(pb, sa[i + 1], vmul(pa, sb[i + 1]));
        }
        T x = neg_mag<B2>(al, be);
        each(x, [&](float &y, int v) { y = __uint_as_float(__float_as_uint(y) & ~((sg[v] << i) & kSign)); });
        store(i, x);
        if (i < 7) {
            const T t = vfma(d[i], pb, pa);
            pb = vfma(d[i], pa, pb);
            pa = t;
        }
    }
}

template <bool B>
struct Const {
    static constexpr bool value = B;
};

// Degree 9..12: the factors held in registers between the passes.
template <int V, typename MsgT, bool HC>
__device__ __forceinline__ void check_12(int dc, const int4 *__restrict__ ed, char *sm, const Place<V> &p, float Xb,
                                         float Pb, uint32_t (&pbad)[V])
{
    constexpr bool B2 = kSlotB2<MsgT>;
    using T = VT<V>;
    T d[12], ga[2], gb[2];
    uint32_t sg[V], par[V];
#pragma unroll
    for (int v = 0; v < V; v++) sg[v] = par[v] = 0;
#pragma unroll
    for (int k = 0; k < 12; k++) {
        d[k] = vset(T(), 0.0f);
        if (k < 9 || k < dc) {
            uint32_t ao, ro;
            edge_at<V, MsgT>(ed[k], p, ao, ro);
            T ap = Sm<float, V>::ld(sm + ao);
            const T n = Sm<MsgT, V>::ld(sm + ro);
            T q = B2 ? vfma(ap, vset(T(), kSLog2e), n) : vadd(ap, n);
            each(ap, [&](float x, int v) { par[v] ^= __float_as_uint(x); });
            each(q, [&](float x, int v) { sg[v] = __funnelshift_l(__float_as_uint(x), sg[v], 1); });
            d[k] = form_d<B2, HC>(q, Xb, Pb);
            const int g = k / 8;
            if (k % 8 == 0) {
                ga[g] = vset(T(), 1.0f);
                gb[g] = d[k];
            } else {
                const T t = vfma(d[k], gb[g], ga[g]);
                gb[g] = vfma(d[k], ga[g], gb[g]);
                ga[g] = t;
            }
        }
    }
#pragma unroll
    for (int v = 0; v < V; v++) {
        sg[v] ^= 0u - (__popc(sg[v]) & 1u);  // the product of the other edges' signs
        sg[v] <<= 32 - dc;
        pbad[v] |= par[v];
    }
#pragma unroll
    for (int g = 0; g < 2; g++) {
        T e[8];
        uint32_t s8[V];
#pragma unroll
        for (int i = 0; i < 8; i++) e[i] = 8 * g + i < 12 ? d[8 * g + i] : vset(T(), 0.0f);
#pragma unroll
        for (int v = 0; v < V; v++) s8[v] = sg[v] << (8 * g);
        auto put = [&](int i, T x) {
            uint32_t ao, ro;
            edge_at<V, MsgT>(ed[8 * g + i], p, ao, ro);
            if (p.own) Sm<MsgT, V>::st(sm + ro, x);
        };
        if (g == 0)
            group_out<true, B2, V>(8, e, ga[1], gb[1], s8, put);
        else
            group_out<false, B2, V>(dc - 8, e, ga[0], gb[0], s8, put);
    }
}

// Degree 13..32.  Between the passes an FP32 message's word holds its edge's d (N is dead once
// Q is formed); with FP16 messages d is formed again from APP and N, or held in registers
// (one codeword per thread, degree <= 16).  Two codewords per thread (G = 0) run the groups
// in a loop, so that the code of all these degrees is one group's: unrolled, the bodies of a
// mixed-code launch overflow the instruction cache (its share of stalls was 1.6 per issue).
// One codeword per thread, the form of small batches, unrolls G groups, whose loads then
// overlap.
template <int G, int V, typename MsgT, bool HC>
__device__ __forceinline__ void check_wide(int dc, const int4 *__restrict__ ed, char *sm, const Place<V> &p, float Xb,
                                           float Pb, uint32_t (&pbad)[V])
{
    constexpr bool B2 = kSlotB2<MsgT>, HOLD = G == 2, INPLACE = !HOLD && sizeof(MsgT) == sizeof(float);
    constexpr int GM = G > 0 ? G : 4;
    using T = VT<V>;
    const T one = vset(T(), 1.0f), zero = vset(T(), 0.0f);
    T ga[GM], gb[GM];
    T held[HOLD ? 8 * GM : 1];
    uint32_t sg[V], par[V];
#pragma unroll
    for (int v = 0; v < V; v++) sg[v] = par[v] = 0;
#pragma unroll
    for (int g = 0; g < GM; g++) {
        ga[g] = one;
        gb[g] = zero;
    }
    if constexpr (HOLD) {
#pragma unroll
        for (int k = 0; k < 8 * GM; k++) held[k] = zero;
    }
    auto q_of = [&](int k, uint32_t &ro, bool first) -> T {
        uint32_t ao;
        edge_at<V, MsgT>(ed[k], p, ao, ro);
        T ap = Sm<float, V>::ld(sm + ao);
        const T n = Sm<MsgT, V>::ld(sm + ro);
        if (first) each(ap, [&](float x, int v) { par[v] ^= __float_as_uint(x); });
        return B2 ? vfma(ap, vset(T(), kSLog2e), n) : vadd(ap, n);
    };
    auto pass1 = [&](int k0, auto full) {
        constexpr bool FULL = decltype(full)::value;
        T a = one, b = zero;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            if (!FULL && k0 + i >= dc) break;
            uint32_t ro;
            T q = q_of(k0 + i, ro, true);
            each(q, [&](float x, int v) { sg[v] = __funnelshift_l(__float_as_uint(x), sg[v], 1); });
            const T d = form_d<B2, HC>(q, Xb, Pb);
            if constexpr (HOLD) held[k0 + i] = d;
            if (INPLACE && p.own) Sm<float, V>::st(sm + ro, d);
            if (i == 0) {
                b = d;
            } else {
                const T t = vfma(d, b, a);
                b = vfma(d, a, b);
                a = t;
            }
        }
#pragma unroll
        for (int g = 0; g < GM; g++)
            if (k0 == 8 * g) {
                ga[g] = a;
                gb[g] = b;
            }
    };
    auto pass2 = [&](int k0, auto full) {
        constexpr bool FULL = decltype(full)::value;
        T pa = one, pb = zero;  // the other groups' product (its first factor is taken exactly)
#pragma unroll
        for (int h = 0; h < GM; h++) {
            if (k0 == 8 * h || 8 * h >= dc) continue;
            const T a1 = pa, b1 = pb;
            pa = vfma(b1, gb[h], vmul(a1, ga[h]));
            pb = vfma(b1, ga[h], vmul(a1, gb[h]));
        }
        T d[8];
        uint32_t ro[8];
#pragma unroll
        for (int i = 0; i < 8; i++) {
            d[i] = zero;
            ro[i] = 0;
        }
#pragma unroll
        for (int i = 0; i < 8; i++) {
            if (!FULL && k0 + i >= dc) break;
            if constexpr (INPLACE || HOLD) {
                uint32_t ao;
                edge_at<V, MsgT>(ed[k0 + i], p, ao, ro[i]);
                if constexpr (HOLD)
                    d[i] = held[k0 + i];
                else
                    d[i] = Sm<float, V>::ld(sm + ro[i]);
            } else {
                d[i] = form_d<B2, HC>(q_of(k0 + i, ro[i], false), Xb, Pb);
            }
        }
        group_out<FULL, B2, V>(dc - k0, d, pa, pb, sg, [&](int i, T x) {
            if (p.own) Sm<MsgT, V>::st(sm + ro[i], x);
        });
#pragma unroll
        for (int v = 0; v < V; v++) sg[v] <<= 8;
    };
    if constexpr (G > 0) {
#pragma unroll
        for (int g = 0; g < G - 1; g++) pass1(8 * g, Const<true>());
        pass1(8 * (G - 1), Const<false>());
    } else {
        int k0 = 0;
#pragma unroll 1
        for (; k0 + 8 <= dc; k0 += 8) pass1(k0, Const<true>());
        if (k0 < dc) pass1(k0, Const<false>());
    }
#pragma unroll
    for (int v = 0; v < V; v++) {
        sg[v] ^= 0u - (__popc(sg[v]) & 1u);  // the product of the other edges' signs
        sg[v] <<= 32 - dc;
        pbad[v] |= par[v];
    }
    if constexpr (G > 0) {
#pragma unroll
        for (int g = 0; g < G - 1; g++) pass2(8 * g, Const<true>());
        pass2(8 * (G - 1), Const<false>());
    } else {
        int k0 = 0;
#pragma unroll 1
        for (; k0 + 8 <= dc; k0 += 8) pass2(k0, Const<true>());
        if (k0 < dc) pass2(k0, Const<false>());
    }
}

// The check-node phase of one thread: its row of every W-th block row, in ascending degree
// (one loop per degree class, so that a row needs no dispatch; flooding checks are
// independent, so the order of the rows changes no result).  Row group w0 takes rows w0,
// 2W-1-w0, 2W+w0, ... (back and forth), which evens out the degrees.
template <int CLS, int DMAX, int V, typename MsgT, bool HC>
__device__ __forceinline__ void rows_of(const FloodGroup &gd, const int4 *__restrict__ tab,
                                        const int32_t *__restrict__ rows, char *sm, const Place<V> &p, float Xb,
                                        float Pb, uint32_t (&pbad)[V], int i, int step, int W2)
{
    constexpr int D = flood_class_degree(CLS);
    if constexpr (D <= DMAX) {
        constexpr bool LAST = CLS + 1 == FLOOD_CLASSES || (V == 2 && D == 16);  // (one body for all wide rows)
        const int end = gd.rend[LAST ? FLOOD_CLASSES - 1 : CLS];
        for (; i < end; i += step, step = W2 - step) {
            const int hd = rows[i];
            if constexpr (D <= 8)
                check_narrow<D, V, MsgT, HC>(tab + (hd >> 8), sm, p, Xb, Pb, pbad);
            else if constexpr (D == 12)
                check_12<V, MsgT, HC>(hd & 255, tab + (hd >> 8), sm, p, Xb, Pb, pbad);
            else
                check_wide<V == 1 ? D / 8 : 0, V, MsgT, HC>(hd & 255, tab + (hd >> 8), sm, p, Xb, Pb, pbad);
        }
        if constexpr (!LAST)
            rows_of<CLS + 1, DMAX, V, MsgT, HC>(gd, tab, rows, sm, p, Xb, Pb, pbad, i, step, W2);
    }
}

// Add one message to a variable's sum (messages are stored negated; in base-2 units when
// kSlotB2).
template <int V, typename MsgT>
__device__ __forceinline__ VT<V> vn_add(VT<V> s, int off, uint32_t r0, const char *sm)
{
    using T = VT<V>;
    const T n = Sm<MsgT, V>::ld(sm + (r0 + (uint32_t)off));
    return vfma(n, vset(T(), kSlotB2<MsgT> ? -kSLn2 : -1.0f), s);
}

// The variable-node phase of one thread: position r of every W-th block column, in ascending
// degree with one loop per degree 1..4 and one for the rest: APP = L + the column's messages
// in block-row order.  A column's element holds its first four message offsets (a column of
// degree above 4: three, and in .w the element of the others); its place in the posteriors
// follows from its list position through the cols words.
template <int V>
struct VnArgs {
    const float *L[V];  // the codewords' channel values at the thread's position of block column 0
    uint32_t a0, r0;    // the thread's posterior and message offsets
    int ZL, ZA;         // a block's step in L (elements) and in the posteriors (bytes)
    bool st[V], all;    // whether the thread stores each codeword's posterior, and both
};
template <int DV, int V, typename MsgT>
__device__ __forceinline__ void vn_cols(const FloodGroup &gd, const int4 *__restrict__ tab,
                                        const int32_t *__restrict__ cols, char *sm, const VnArgs<V> &q, int i, int W)
{
    using T = VT<V>;
    const int end = gd.cend[DV - 1];
    for (; i < end;) {
        T lv[kVnChunk];
        int jc[kVnChunk];
#pragma unroll
        for (int c = 0; c < kVnChunk; c++) {
            lv[c] = vset(T(), 0.0f);
            jc[c] = 0;
            if (c == 0 || i + c * W < end) {
                jc[c] = cols[i + c * W];
                each(lv[c], [&](float &x, int v) { x = __ldg(q.L[v] + jc[c] * q.ZL); });
            }
        }
#pragma unroll
        for (int c = 0; c < kVnChunk; c++) {
            if (c == 0 || i < end) {
                const int4 o = tab[gd.t_col + i];
                T s = vn_add<V, MsgT>(lv[c], o.x, q.r0, sm);
                if constexpr (DV > 1) s = vn_add<V, MsgT>(s, o.y, q.r0, sm);
                if constexpr (DV > 2) s = vn_add<V, MsgT>(s, o.z, q.r0, sm);
                if constexpr (DV == 4) s = vn_add<V, MsgT>(s, o.w, q.r0, sm);
                if constexpr (DV == 5) {
                    const int4 *m = tab + (o.w >> 8);
                    for (int k = o.w & 255; k > 0; k -= 4, m++) {
                        s = vn_add<V, MsgT>(s, m->x, q.r0, sm);
                        if (k > 1) s = vn_add<V, MsgT>(s, m->y, q.r0, sm);
                        if (k > 2) s = vn_add<V, MsgT>(s, m->z, q.r0, sm);
                        if (k > 3) s = vn_add<V, MsgT>(s, m->w, q.r0, sm);
                    }
                }
                s = vadd(s, vset(T(), 0.0f));  // -0 -> +0: the sign bit is the decision
                const uint32_t ao = q.a0 + (uint32_t)(jc[c] * q.ZA);
                if (q.all) Sm<float, V>::st(sm + ao, s);
                if constexpr (V > 1)
                    each(s, [&](float x, int v) {
                        if (q.st[v] && !q.all) *reinterpret_cast<float *>(sm + (ao + 4 * v)) = x;
                    });
                i += W;
            }
        }
    }
    if constexpr (DV < 5) vn_cols<DV + 1, V, MsgT>(gd, tab, cols, sm, q, i, W);
}

template <int DMAX, int V, typename MsgT, bool HC>
__global__ void __launch_bounds__(flood_threads_max(DMAX, V, sizeof(MsgT) == 2), 1) k_flood_slots(const __grid_constant__ FloodArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    char *sm = reinterpret_cast<char *>(smem_raw);
    int32_t *misc = reinterpret_cast<int32_t *>(sm);                // [4] code-group hand-over
    FloodBook *books = reinterpret_cast<FloodBook *>(sm + 16);      // [slots]
    int4 *tab = reinterpret_cast<int4 *>(sm + a.tab0);              // the code's tables
    using T = VT<V>;
    const int tid = threadIdx.x, nth = blockDim.x;
    const float Xb = a.X * kSLog2e, Pb = s_phi_b2(a.X);  // the clamp [phi(X), X] in base-2 units
    constexpr uint32_t kSign = 0x80000000u;
    constexpr int SA = (int)sizeof(float) * V, SR = (int)sizeof(MsgT) * V;
    int grp = 0;
    {
        const float u = (blockIdx.x + 0.5f) / gridDim.x;
        while (grp < a.n_groups - 1 && a.groups[grp].cumw < u) grp++;
    }

    for (;;) {
        const FloodGroup &gd = a.groups[grp];
        const int N = gd.N, Z = gd.Z, nb = gd.nb, nnz = gd.nnz;
        // Thread slot g (V codewords) is run by its own W row groups of WT threads (whole warps):
        // thread r < Z of row group w0 owns row r of block rows and columns w0, w0 + W, ...  A
        // warp works on one block row at a time, and a thread slot synchronises only its own
        // warps.
        const int W = gd.W, TPG = gd.TPG, WT = TPG / W;
        // (g and w0 are the same for a warp's lanes: taken from a warp reduction, the loops over
        // block rows and columns compile to uniform branches)
        const int gw = (int)__reduce_min_sync(0xffffffffu, (unsigned)(tid / WT));
        const int g = gw / W, w0 = gw - g * W, ru = tid - gw * WT;
        const bool member = g < gd.G;            // the thread's warp belongs to a thread slot
        const bool mine = member && ru < Z;      // a row of it (else an idle lane of the last warp)
        const int r = ru < Z ? ru : Z - 1;
        const bool lead = mine && ru == 0 && w0 == 0;  // the thread that takes codewords for the slot
        FloodBook *book = books + (member ? g : 0) * V;
        const int32_t *rows = reinterpret_cast<const int32_t *>(tab + gd.t_row);

        // a slot's leader takes the group's next codeword and finds its request
        auto grab = [&](int v) {
            const unsigned long long k = atomicAdd(a.next + grp, 1ull);
            int64_t loc = -1;
            int rq = -1;
            if (k < (unsigned long long)gd.n_items) {
                for (rq = gd.req_begin; rq < gd.req_end - 1; rq++)
                    if ((int64_t)k < a.reqs[rq + 1].item0) break;
                loc = (int64_t)k - a.reqs[rq].item0;
            }
            book[v].cw = loc;
            book[v].req = rq;
        };
        for (int i = tid; i < gd.n_tab; i += nth) tab[i] = gd.tab[i];
        if (lead) {
#pragma unroll
            for (int v = 0; v < V; v++) {
                grab(v);
                book[v].bad[0] = book[v].bad[1] = 0;
            }
        }
        __syncthreads();

        Place<V> p;
        p.r = r;
        p.own = mine;
        p.a0 = (uint32_t)(a.slots0 + (member ? g : 0) * gd.strA + r * SA);
        p.a1 = p.a0 - (uint32_t)(Z * SA);
        p.r0 = (uint32_t)(a.slots0 + gd.offR + (member ? g : 0) * gd.strR + r * SR);
        p.r1 = p.r0 - (uint32_t)(Z * SR);
        float *A = reinterpret_cast<float *>(sm + p.a0);   // position r of block column 0
        MsgT *R = reinterpret_cast<MsgT *>(sm + p.r0);     // position r of block 0
        // every thread of the slot's warps keeps its codewords' state (idle lanes too)
        int64_t cw[V];  // request-local codeword (-1: none)
        int rq[V];      // its request
        int t[V];       // iterations completed on it
#pragma unroll
        for (int v = 0; v < V; v++) {
            cw[v] = member ? book[v].cw : -1;
            rq[v] = member ? book[v].req : -1;
            t[v] = 0;
        }

        // load a new codeword into lane v, this thread's columns: APP = L (+0 for -0), messages 0
        auto refill = [&](int v) {
            const float *Lr = a.reqs[rq[v]].llr + cw[v] * N;
            constexpr int CH = kRefillChunk;
            for (int j0 = w0; j0 < nb; j0 += CH * W) {
                float x[CH];
#pragma unroll
                for (int c = 0; c < CH; c++)
                    if (j0 + c * W < nb) x[c] = __ldg(Lr + (j0 + c * W) * Z + r);
#pragma unroll
                for (int c = 0; c < CH; c++)
                    if (j0 + c * W < nb) {
                        if (!isfinite(x[c])) atomicOr(gd.status, IN_NONFINITE);
                        A[(j0 + c * W) * Z * V + v] = x[c] + 0.0f;
                    }
            }
            for (int b = w0; b < nnz; b += W) R[b * Z * V + v] = MsgT(0.0f);
        };
        // the barrier of the thread slot's warps (named barriers 1..15; barrier 0 is the CTA's)
        auto gsync = [&]() {
            if (TPG == 32)
                __syncwarp();
            else
                asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(TPG) : "memory");
        };

        bool any = false;
#pragma unroll
        for (int v = 0; v < V; v++) {
            if (mine && cw[v] >= 0) refill(v);
            any |= cw[v] >= 0;
        }
        // (votes over the warp: conditions that are the same for all its lanes, said so)
        any = __any_sync(0xffffffffu, any);
        if (any) gsync();

        for (int ph = 0; any; ph ^= 1) {
            // ---------------- check-node phase: row r of this row group's block rows, all V codewords at once
            {
                uint32_t pbad[V];
#pragma unroll
                for (int v = 0; v < V; v++) pbad[v] = 0;
                rows_of<0, DMAX, V, MsgT, HC>(gd, tab, rows, sm, p, Xb, Pb, pbad, w0, 2 * (W - w0) - 1, 2 * W);
#pragma unroll
                for (int v = 0; v < V; v++)
                    if (mine && (pbad[v] & kSign)) book[v].bad[ph] = 1;
            }
            gsync();

            // ---------------- decision, variable-node phase, output
            bool done[V], act[V];
            bool anyact = false, anydone = false;
#pragma unroll
            for (int v = 0; v < V; v++) {
                done[v] = cw[v] >= 0 && t[v] >= 1 && a.early_exit && book[v].bad[ph] == 0;  // converged
                act[v] = cw[v] >= 0 && !done[v];
                anyact |= act[v];
            }
            if (lead) {
                // the other flag was last read before this round's first barrier
#pragma unroll
                for (int v = 0; v < V; v++) book[v].bad[ph ^ 1] = 0;
            }
            if (__any_sync(0xffffffffu, anyact)) {
                VnArgs<V> q;
                q.all = true;
#pragma unroll
                for (int v = 0; v < V; v++) {  // an idle lane of a pair reads the other's channel values
                    const int rx = act[v] ? rq[v] : rq[V - 1 - v];
                    const int64_t cx = act[v] ? cw[v] : cw[V - 1 - v];
                    q.L[v] = a.reqs[rx].llr + cx * N + r;
                    q.st[v] = mine && act[v];
                    q.all &= q.st[v];
                }
                q.a0 = p.a0;
                q.r0 = p.r0;
                q.ZL = Z;
                q.ZA = Z * SA;
                vn_cols<1, V, MsgT>(gd, tab, rows + gd.mb, sm, q, w0, W);
            }
#pragma unroll
            for (int v = 0; v < V; v++) {
                if (act[v]) {
                    t[v]++;
                    done[v] = t[v] >= a.max_iter;
                }
                anydone |= done[v];
                if (__any_sync(0xffffffffu, done[v]) && mine) {
                    const FloodReq &q = a.reqs[rq[v]];
                    uint8_t *Bo = q.bits + cw[v] * N;
                    float *Ao = q.app ? q.app + cw[v] * N : nullptr;
                    const int32_t *cols = rows + gd.mb;
                    for (int i = w0; i < nb; i += W) {  // the columns this thread has just updated
                        const int j = cols[i];
                        const float x = A[j * Z * V + v];
                        Bo[j * Z + r] = x < 0.0f ? 1 : 0;
                        if (Ao) Ao[j * Z + r] = x;
                    }
                    if (lead) {
                        q.iters[cw[v]] = t[v];
                        grab(v);
                    }
                }
            }
            gsync();

            // ---------------- refill finished slots
            if (__any_sync(0xffffffffu, anydone)) {
                any = false;
#pragma unroll
                for (int v = 0; v < V; v++) {
                    if (done[v]) {
                        cw[v] = book[v].cw;
                        rq[v] = book[v].req;
                        t[v] = 0;
                        if (mine && cw[v] >= 0) refill(v);
                    }
                    any |= cw[v] >= 0;
                }
                any = __any_sync(0xffffffffu, any);
                gsync();
            }
        }

        // this group is dry here and every slot has drained: move to the group with the
        // most codewords left, or stop
        if (a.n_groups == 1) return;
        if (tid == 0) {
            int best = -1;
            long long most = 0;
            for (int q = 0; q < a.n_groups; q++) {
                const long long left = a.groups[q].n_items - (long long)atomicAdd(a.next + q, 0ull);
                if (left > most) {
                    most = left;
                    best = q;
                }
            }
            misc[0] = best;
        }
        __syncthreads();
        grp = (int)__reduce_max_sync(0xffffffffu, misc[0]);  // (uniform, as gw)
        __syncthreads();
        if (grp < 0) return;
    }
}

template <int DMAX, int V, typename MsgT, bool HC>
static cudaError_t launch_one(const FloodArgs &a, size_t smem, int threads, int ctas, cudaStream_t s)
{
    cudaError_t e = ensure_smem<k_flood_slots<DMAX, V, MsgT, HC>>(smem);
    if (e != cudaSuccess) return e;
    LaunchScope ls(F_SLOTS, s);
    k_flood_slots<DMAX, V, MsgT, HC><<<(unsigned)ctas, threads, smem, s>>>(a);
    return cudaGetLastError();
}

template <typename MsgT, bool HC>
cudaError_t flood_slots_launch(int dmax, int V, const FloodArgs &a, size_t smem, int threads, int ctas,
                               cudaStream_t s)
{
    if (dmax <= 8)
        return V == 2 ? launch_one<8, 2, MsgT, HC>(a, smem, threads, ctas, s)
                      : launch_one<8, 1, MsgT, HC>(a, smem, threads, ctas, s);
    return V == 2 ? launch_one<32, 2, MsgT, HC>(a, smem, threads, ctas, s)
                  : launch_one<32, 1, MsgT, HC>(a, smem, threads, ctas, s);
}

}  // namespace ldpc
