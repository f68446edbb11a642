// The flooding check-node update of one check row, for one or two codewords per thread
// (flooding slot decoder) or of two check rows of one codeword (two-SM cluster decoder).
#pragma once

#include "slot_common.cuh"

namespace ldpc {

// ------------------------------------------------------------------ V rows per thread
//
// A value of a thread is a float (one codeword) or a float2 (two codewords, or two check rows
// of one block row, whose multiplies and adds issue as packed pairs; each half is rounded
// exactly as the scalar operation).
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

// Where the operands of a check lie: posteriors and messages both in the CTA's own shared
// memory, at byte offsets from its start.
template <int V, typename MsgT>
struct OwnMem {
    char *sm;
    __device__ __forceinline__ VT<V> app(uint32_t o) const { return Sm<float, V>::ld(sm + o); }
    __device__ __forceinline__ VT<V> msg(uint32_t o) const { return Sm<MsgT, V>::ld(sm + o); }
    template <typename PL>
    __device__ __forceinline__ void put(const PL &p, uint32_t o, VT<V> x) const
    {
        if (p.own) Sm<MsgT, V>::st(sm + o, x);
    }
    // a message's word as the place of a float (FP32 messages)
    __device__ __forceinline__ VT<V> word(uint32_t o) const { return Sm<float, V>::ld(sm + o); }
    template <typename PL>
    __device__ __forceinline__ void put_word(const PL &p, uint32_t o, VT<V> x) const
    {
        if (p.own) Sm<float, V>::st(sm + o, x);
    }
};

// ------------------------------------------------------------------ the check rule
//
// Messages are stored negated (N = -R): Q = APP + N needs no negation and the variable-node
// sum adds -N (a multiply-add by a negative constant).  The rule itself is slot_common.cuh's:
// d = e^-a per edge, prefix and suffix products of the maps (alpha, beta) <- (alpha + d beta,
// beta + d alpha), R = ln(alpha / beta) with the sign of the other edges.

// d of each codeword.  HC: the upper clamp a >= phi(X) is applied; without it the clamp is
// known not to change d (phi(X) so small that ex2 rounds e^-phi(X) to 1, see FLOOD_CLAMP_X).
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
    using Ref = uint32_t;  // an operand's offset
    uint32_t a0, a1, r0, r1;
    int r;
    bool own;  // an idle lane of a slot's last warp repeats the last row's loads and stores nothing
};

// The edge's operand offsets.  With one element size for APP and messages the two regions of
// a slot are at a fixed distance (already in the descriptor's .y), so one select serves both.
template <typename MsgT, int V>
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
template <int D, int V, typename MsgT, bool B2, bool HC, typename MEM, typename PL>
__device__ __forceinline__ void check_narrow(const int4 *__restrict__ ed, const MEM mem, const PL &p, float Xb,
                                             float Pb, uint32_t (&pbad)[V])
{
    constexpr uint32_t kSign = 0x80000000u;
    using T = VT<V>;
    const T one = vset(T(), 1.0f), zero = vset(T(), 0.0f);
    T d[D];
    typename PL::Ref ro[D];
    uint32_t par[V];
    uint32_t sg[V];  // the signs of Q: edge k's in bit D - 1 - k (a word per codeword, not one per edge)
#pragma unroll
    for (int v = 0; v < V; v++) sg[v] = par[v] = 0;
#pragma unroll
    for (int k = 0; k < D; k++) {
        typename PL::Ref ao;
        edge_at<MsgT>(ed[k], p, ao, ro[k]);
        T ap = mem.app(ao);
        const T n = mem.msg(ro[k]);
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
        mem.put(p, ro[k], n);
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
template <int V, typename MsgT, bool B2, bool HC, typename MEM, typename PL>
__device__ __forceinline__ void check_12(int dc, const int4 *__restrict__ ed, const MEM mem, const PL &p,
                                         float Xb, float Pb, uint32_t (&pbad)[V])
{
    using T = VT<V>;
    T d[12], ga[2], gb[2];
    uint32_t sg[V], par[V];
#pragma unroll
    for (int v = 0; v < V; v++) sg[v] = par[v] = 0;
#pragma unroll
    for (int k = 0; k < 12; k++) {
        d[k] = vset(T(), 0.0f);
        if (k < 9 || k < dc) {
            typename PL::Ref ao, ro;
            edge_at<MsgT>(ed[k], p, ao, ro);
            T ap = mem.app(ao);
            const T n = mem.msg(ro);
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
            typename PL::Ref ao, ro;
            edge_at<MsgT>(ed[8 * g + i], p, ao, ro);
            mem.put(p, ro, x);
        };
        if (g == 0)
            group_out<true, B2, V>(8, e, ga[1], gb[1], s8, put);
        else
            group_out<false, B2, V>(dc - 8, e, ga[0], gb[0], s8, put);
    }
}

// Degree 13..32.  Between the passes an FP32 message's word holds its edge's d (N is dead once
// Q is formed); with FP16 messages d is formed again from APP and N, or held in registers
// (G = 2: degree <= 16).  Two codewords per thread (G = 0) run the groups
// in a loop, so that the code of all these degrees is one group's: unrolled, the bodies of a
// mixed-code launch overflow the instruction cache (its share of stalls was 1.6 per issue).
// One codeword per thread, the form of small batches, and the cluster decoder, whose loads come
// from the other SM, unroll G groups, whose loads then overlap.
template <int G, int V, typename MsgT, bool B2, bool HC, typename MEM, typename PL>
__device__ __forceinline__ void check_wide(int dc, const int4 *__restrict__ ed, const MEM mem, const PL &p,
                                           float Xb, float Pb, uint32_t (&pbad)[V])
{
    constexpr bool HOLD = G == 2, INPLACE = !HOLD && sizeof(MsgT) == sizeof(float);
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
    auto q_of = [&](int k, typename PL::Ref &ro, bool first) -> T {
        typename PL::Ref ao;
        edge_at<MsgT>(ed[k], p, ao, ro);
        T ap = mem.app(ao);
        const T n = mem.msg(ro);
        if (first) each(ap, [&](float x, int v) { par[v] ^= __float_as_uint(x); });
        return B2 ? vfma(ap, vset(T(), kSLog2e), n) : vadd(ap, n);
    };
    auto pass1 = [&](int k0, auto full) {
        constexpr bool FULL = decltype(full)::value;
        T a = one, b = zero;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            if (!FULL && k0 + i >= dc) break;
            typename PL::Ref ro;
            T q = q_of(k0 + i, ro, true);
            each(q, [&](float x, int v) { sg[v] = __funnelshift_l(__float_as_uint(x), sg[v], 1); });
            const T d = form_d<B2, HC>(q, Xb, Pb);
            if constexpr (HOLD) held[k0 + i] = d;
            if constexpr (INPLACE) mem.put_word(p, ro, d);
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
        typename PL::Ref ro[8];
#pragma unroll
        for (int i = 0; i < 8; i++) {
            d[i] = zero;
            ro[i] = typename PL::Ref();
        }
#pragma unroll
        for (int i = 0; i < 8; i++) {
            if (!FULL && k0 + i >= dc) break;
            if constexpr (INPLACE || HOLD) {
                typename PL::Ref ao;
                edge_at<MsgT>(ed[k0 + i], p, ao, ro[i]);
                if constexpr (HOLD)
                    d[i] = held[k0 + i];
                else
                    d[i] = mem.word(ro[i]);
            } else {
                d[i] = form_d<B2, HC>(q_of(k0 + i, ro[i], false), Xb, Pb);
            }
        }
        group_out<FULL, B2, V>(dc - k0, d, pa, pb, sg, [&](int i, T x) {
            mem.put(p, ro[i], x);
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

// ------------------------------------------------------------------ rows end to end over warps
//
// A warp whose lanes are at rows of different degree takes them in turns of one body each, agreed on by
// a vote; a lane without a row for that body repeats another's loads and stores nothing.

constexpr unsigned kFullWarp = 0xffffffffu;
constexpr int kNoRow = 255;  // above any degree

// The body that rows of degree dc share: exact up to 8, then up to 12, 16, 24, 32.
__device__ __forceinline__ int body_of(int dc) { return dc <= 8 ? dc : dc <= 12 ? 12 : dc <= 16 ? 16 : dc <= 24 ? 24 : dc <= 32 ? 32 : dc; }

// The first body any lane is at (kNoRow: none has a row left); hd: a lane's row << 8 | degree (kNoRow: none),
// afterwards a row for that body; on: whether it is the lane's own.
__device__ __forceinline__ int vote_body(int &hd, bool &on)
{
    const int mine = body_of(hd & 255);
    const int body = (int)__reduce_min_sync(kFullWarp, (unsigned)mine);
    on = mine == body && body != kNoRow;
    const unsigned m = __ballot_sync(kFullWarp, on);
    const int hs = __shfl_sync(kFullWarp, hd, m ? __ffs(m) - 1 : 0);
    if (!on) hd = hs;
    return body;
}

__device__ __forceinline__ float pick(bool c, float a, float b) { return c ? a : b; }
__device__ __forceinline__ float2 pick(bool c, float2 a, float2 b) { return make_float2(c ? a.x : b.x, c ? a.y : b.y); }

}  // namespace ldpc
