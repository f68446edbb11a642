// Horizontal layered sum-product decoding with the decoder state on chip (Sec. II
// "Algorithm 2" schedule with the sum-product check rule of Sec. I).
//
// A persistent grid of one CTA per SM.  Each CTA holds thread slots of V codewords (two, packed in
// float2 operands, where the messages are FP16, or one); a thread slot keeps its codewords'
// posteriors APP [N] (fp32) and check-to-variable messages R [E] (fp32 or fp16, stored negated)
// in shared memory for their whole decode.  Thread r of a thread slot's warps owns check row r
// of every block row (layer): the Z checks of a QC layer touch disjoint variables (each block
// is one circulant), so the row threads update a layer at once, and the thread slot's own
// barrier (a named barrier, or the warp itself) separates consecutive layers; the thread slots
// of a CTA run independently (narrow codes: several thread slots to a barrier, see
// k_layered_spa_packed).  Messages are in check-row order, edge (b, r) at b*Z + r: the
// layered schedule has no variable-node pass, so a warp reads and writes them contiguously.
// Per check (the arithmetic of the flooding slot decoder, only the schedule differs):
//   Q_k   = APP_n - R_k                                   over the check's edges
//   R'_k  = prod_{other} sgn Q * min(X, phi( sum_{other} phi(clampX |Q|) ))
//           in the product (tanh) domain (slot_common.cuh), stored as fp16 when the
//           messages are half precision
//   APP_n = Q_k + R'_k   with R'_k the stored value, so that the next Q = APP - R removes
//                        exactly what was added
// After every full iteration each slot's hard decisions are checked against its checks, layer
// by layer until every codeword has shown an unsatisfied one; a codeword that converged (early
// exit) or reached max_iter is written out and the slot takes the next one from the global
// work counter.
//
// What bounds it (GB300): instruction issue (71-83 %).  8192 codewords of the N = 1944 rate-1/2
// code, FP32, 2.0 dB: 605 -> 502 us per launch, 45 -> 39 warp instructions per edge update;
// 7281 codewords of the N = 2304 code, FP16, 5 fixed iterations: 355 -> 298 us.  What went: the
// syndrome pass over all layers in every iteration (15 % of the instructions; most codewords
// show an unsatisfied check in the first layer), divergent control, one barrier of two per
// iteration's end, the upper clamp of |Q| where it cannot bind.
//
// APP is never -0: the refill adds +0 to the (scaled) channel value and Q + R' is -0 only when both
// are -0, which cannot happen while APP is not -0 (then Q = APP - R is not -0).  The sign
// bit therefore is the hard decision [APP < 0] and sgn(0) = +1, as the oracle reads it.
#include <math.h>

#include "flood_check.cuh"

namespace ldpc {

// The FP32-message form keeps APP, Q and R in base-2 units (LLR x log2 e, set at the refill
// and undone at the output), which spares the check rule its scaling multiplies; the
// FP16-message form stays in natural units, so that its stored binary16 message is the
// natural-unit value rounded, as the oracle's binary16 mode rounds it.
// (Measured on the 8192-codeword N = 1944 rate-1/2 sweep: base-2 units 9.22 info Gbit/s,
// natural units 8.98.)
template <typename MsgT>
constexpr bool kBase2 = sizeof(MsgT) == 4;

// Bookkeeping of one slot in shared memory.
struct LspaBook {
    int64_t cw;      // its next codeword (-1: none)
    int32_t bad[2];  // unsatisfied check seen, by iteration parity
};

struct LayeredSpaArgs {
    const float *llr;
    int64_t n_cw;
    uint8_t *bits;
    int32_t *iters;
    float *app_out;
    unsigned long long *next;
    // sizes and layer lists from here, not from the code's device tables: known to be warp-uniform
    int N, Z, mb, nb, nnz;
    int G, TPG;        // thread slots per CTA, threads of a barrier group (whole warps)
    int K;             // thread slots of a barrier group (1 unless packed)
    int tab0, slots0;  // tables and first slot, bytes from the start of shared memory
    int strA, strR, offR;  // bytes from one thread slot's posteriors / messages to the next one's; first messages
    int max_iter, early_exit;
    float X;
    uint8_t deg[MB_MAX];    // degree of each layer
    uint16_t first[MB_MAX]; // its first block
};

// Edge descriptor of block b = (row l, column j, shift s): .x = byte offset of the posterior
// j*Z + s, .y of the message row b*Z, .z = Z - s.  Check row r reaches variable position
// (r + s) mod Z: .x from the thread's posterior base (position r), less one block when r >= .z;
// its message is .y from its message base (row r), with no wrap.
template <int V>
__device__ __forceinline__ void lspa_at(const int4 &e, const Place<V> &p, uint32_t &ao, uint32_t &ro)
{
    ao = (p.r >= e.z ? p.a1 : p.a0) + (uint32_t)e.x;
    ro = p.r0 + (uint32_t)e.y;
}

// Store the negated message n of an edge and the posterior Q - n, with n as stored.
template <typename MsgT>
__device__ __forceinline__ void lspa_put(char *sm, bool own, uint32_t ao, uint32_t ro, float q, float n)
{
    if constexpr (sizeof(MsgT) == 2) {
        const __half h = __float2half_rn(n);
        if (own) *reinterpret_cast<__half *>(sm + ro) = h;
        n = __half2float(h);
    } else {
        if (own) *reinterpret_cast<float *>(sm + ro) = n;
    }
    if (own) *reinterpret_cast<float *>(sm + ao) = q - n;
}
template <typename MsgT>
__device__ __forceinline__ void lspa_put(char *sm, bool own, uint32_t ao, uint32_t ro, float2 q, float2 n)
{
    if constexpr (sizeof(MsgT) == 2) {
        const __half2 h = __floats2half2_rn(n.x, n.y);
        if (own) *reinterpret_cast<__half2 *>(sm + ro) = h;
        n = __half22float2(h);
    } else {
        if (own) *reinterpret_cast<float2 *>(sm + ro) = n;
    }
    const float2 a = __ffma2_rn(n, make_float2(-1.0f, -1.0f), q);
    if (own) *reinterpret_cast<float2 *>(sm + ao) = a;
}

// One check of degree D <= 8: every edge's state in registers.
template <int D, int V, typename MsgT, bool HC>
__device__ __forceinline__ void layer_narrow(const int4 *__restrict__ ed, char *sm, const Place<V> &p, float Xb, float Pb)
{
    constexpr bool B2 = kBase2<MsgT>;
    constexpr uint32_t kSign = 0x80000000u;
    using T = VT<V>;
    const T one = vset(T(), 1.0f), zero = vset(T(), 0.0f);
    T d[D], q[D];
    uint32_t ao[D], sg[V];
#pragma unroll
    for (int v = 0; v < V; v++) sg[v] = 0;
#pragma unroll
    for (int k = 0; k < D; k++) {
        uint32_t ro;
        lspa_at<V>(ed[k], p, ao[k], ro);
        q[k] = vadd(Sm<float, V>::ld(sm + ao[k]), Sm<MsgT, V>::ld(sm + ro));
        each(q[k], [&](float x, int v) { sg[v] ^= __float_as_uint(x); });
        d[k] = form_d<B2, HC>(q[k], Xb, Pb);
    }
    T sa[D + 1], sb[D + 1];
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
        T qk = q[k];
        each(qk, [&](float x, int v) {
            float &y = reinterpret_cast<float *>(&n)[v];
            y = __uint_as_float(__float_as_uint(y) & ~((__float_as_uint(x) ^ sg[v]) & kSign));
        });
        lspa_put<MsgT>(sm, p.own, ao[k], p.r0 + (uint32_t)ed[k].y, q[k], n);
        if (k == 0) {
            pb = d[0];
        } else if (k < D - 1) {
            const T t = vfma(d[k], pb, pa);
            pb = vfma(d[k], pa, pb);
            pa = t;
        }
    }
}

// One check of degree 9..32 in groups of 8 edges (see flood_check.cuh): pass 1 forms each
// group's pair, pass 2 each group's messages; Q is formed from APP and N in both (neither is
// written before its own edge is).
template <int G, int V, typename MsgT, bool HC>
__device__ __forceinline__ void layer_wide(int dc, const int4 *__restrict__ ed, char *sm, const Place<V> &p, float Xb,
                                           float Pb)
{
    constexpr bool B2 = kBase2<MsgT>;
    using T = VT<V>;
    const T one = vset(T(), 1.0f), zero = vset(T(), 0.0f);
    T ga[G], gb[G];
    uint32_t sg[V];
#pragma unroll
    for (int v = 0; v < V; v++) sg[v] = 0;
#pragma unroll
    for (int g = 0; g < G; g++) {
        ga[g] = one;
        gb[g] = zero;
    }
    auto q_of = [&](int k, uint32_t &ao, uint32_t &ro) -> T {
        lspa_at<V>(ed[k], p, ao, ro);
        return vadd(Sm<float, V>::ld(sm + ao), Sm<MsgT, V>::ld(sm + ro));
    };
    auto pass1 = [&](int k0, auto full) {
        constexpr bool FULL = decltype(full)::value;
        T a = one, b = zero;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            if (!FULL && k0 + i >= dc) break;
            uint32_t ao, ro;
            T q = q_of(k0 + i, ao, ro);
            each(q, [&](float x, int v) { sg[v] = __funnelshift_l(__float_as_uint(x), sg[v], 1); });
            const T d = form_d<B2, HC>(q, Xb, Pb);
            if (i == 0) {
                b = d;
            } else {
                const T t = vfma(d, b, a);
                b = vfma(d, a, b);
                a = t;
            }
        }
#pragma unroll
        for (int g = 0; g < G; g++)
            if (k0 == 8 * g) {
                ga[g] = a;
                gb[g] = b;
            }
    };
    auto pass2 = [&](int k0, auto full) {
        constexpr bool FULL = decltype(full)::value;
        T pa = one, pb = zero;  // the other groups' product (its first factor is taken exactly)
#pragma unroll
        for (int h = 0; h < G; h++) {
            if (k0 == 8 * h || 8 * h >= dc) continue;
            const T a1 = pa, b1 = pb;
            pa = vfma(b1, gb[h], vmul(a1, ga[h]));
            pb = vfma(b1, ga[h], vmul(a1, gb[h]));
        }
        T d[8], q[8];
        uint32_t ao[8], ro[8];
#pragma unroll
        for (int i = 0; i < 8; i++) {
            d[i] = q[i] = zero;
            ao[i] = ro[i] = 0;
        }
#pragma unroll
        for (int i = 0; i < 8; i++) {
            if (!FULL && k0 + i >= dc) break;
            q[i] = q_of(k0 + i, ao[i], ro[i]);
            d[i] = form_d<B2, HC>(q[i], Xb, Pb);
        }
        group_out<FULL, B2, V>(dc - k0, d, pa, pb, sg,
                               [&](int i, T n) { lspa_put<MsgT>(sm, p.own, ao[i], ro[i], q[i], n); });
#pragma unroll
        for (int v = 0; v < V; v++) sg[v] <<= 8;
    };
#pragma unroll
    for (int g = 0; g < G - 1; g++) pass1(8 * g, Const<true>());
    pass1(8 * (G - 1), Const<false>());
#pragma unroll
    for (int v = 0; v < V; v++) {
        sg[v] ^= 0u - (__popc(sg[v]) & 1u);  // the product of the other edges' signs
        sg[v] <<= 32 - dc;
    }
#pragma unroll
    for (int g = 0; g < G - 1; g++) pass2(8 * g, Const<true>());
    pass2(8 * (G - 1), Const<false>());
}

// One layer (the degree is warp-uniform).
template <int DMAX, int V, typename MsgT, bool HC>
__device__ __forceinline__ void layer_check(int dc, const int4 *__restrict__ ed, char *sm, const Place<V> &p, float Xb,
                                            float Pb)
{
    switch (dc) {
    case 2: layer_narrow<2, V, MsgT, HC>(ed, sm, p, Xb, Pb); break;
    case 3: layer_narrow<3, V, MsgT, HC>(ed, sm, p, Xb, Pb); break;
    case 4: layer_narrow<4, V, MsgT, HC>(ed, sm, p, Xb, Pb); break;
    case 5: layer_narrow<5, V, MsgT, HC>(ed, sm, p, Xb, Pb); break;
    case 6: layer_narrow<6, V, MsgT, HC>(ed, sm, p, Xb, Pb); break;
    case 7: layer_narrow<7, V, MsgT, HC>(ed, sm, p, Xb, Pb); break;
    case 8: layer_narrow<8, V, MsgT, HC>(ed, sm, p, Xb, Pb); break;
    default:
        if constexpr (DMAX > 8) {
            if (dc <= 16)
                layer_wide<2, V, MsgT, HC>(dc, ed, sm, p, Xb, Pb);
            else if (dc <= 24)
                layer_wide<3, V, MsgT, HC>(dc, ed, sm, p, Xb, Pb);
            else
                layer_wide<4, V, MsgT, HC>(dc, ed, sm, p, Xb, Pb);
        }
    }
}

// XOR of the posterior sign bits of the thread's check row of one layer, per codeword.
template <int V>
__device__ __forceinline__ void lspa_parity(int dc, const int4 *__restrict__ ed, const char *sm, const Place<V> &p,
                                            uint32_t (&par)[V])
{
#pragma unroll
    for (int v = 0; v < V; v++) par[v] = 0;
    auto take = [&](int k) {
        uint32_t ao, ro;
        lspa_at<V>(ed[k], p, ao, ro);
        VT<V> a = Sm<float, V>::ld(sm + ao);
        each(a, [&](float x, int v) { par[v] ^= __float_as_uint(x); });
    };
    int k = 0;
    for (; k + 4 <= dc; k += 4) {
        take(k);
        take(k + 1);
        take(k + 2);
        take(k + 3);
    }
    for (; k < dc; k++) take(k);
}

// Threads per CTA for an instance.
__host__ __device__ constexpr int lspa_threads(int dmax, int V, bool f16)
{
    if (V == 2) return 640;
    return f16 ? (dmax <= 8 ? 1024 : 768) : 672;
}

template <int DMAX, int V, typename MsgT, bool HC>
__global__ void __launch_bounds__(lspa_threads(DMAX, V, sizeof(MsgT) == 2), 1)
    k_layered_spa(const CodeDev *__restrict__ cd, const __grid_constant__ LayeredSpaArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    char *sm = reinterpret_cast<char *>(smem_raw);
    LspaBook *books = reinterpret_cast<LspaBook *>(sm);
    int4 *tab = reinterpret_cast<int4 *>(sm + a.tab0);
    constexpr int SA = (int)sizeof(float) * V, SR = (int)sizeof(MsgT) * V;
    constexpr uint32_t kSign = 0x80000000u;
    const int N = a.N, Z = a.Z, mb = a.mb, nb = a.nb, nnz = a.nnz, TPG = a.TPG;
    const int tid = threadIdx.x, nth = blockDim.x;
    const float Xb = a.X * kSLog2e, Pb = s_phi_b2(a.X);  // the clamp [phi(X), X] in base-2 units
    for (int i = tid; i < nnz; i += nth) {
        const int e = cd->ent[i], sh = e & 0xffff;
        tab[i] = make_int4(SA * ((e >> 16) * Z + sh), SR * i * Z, Z - sh, 0);
    }
    // thread slot g (a warp reduction: known to be warp-uniform), row ru of its layers
    const int g = (int)__reduce_min_sync(0xffffffffu, (unsigned)(tid / TPG)), ru = tid - g * TPG;
    const bool own = ru < Z, lead = ru == 0;  // (idle lanes of the last warp repeat row Z - 1 and store nothing)
    LspaBook *book = books + g * V;
    // the next codeword; without a work counter every codeword has a slot from the start
    auto grab = [&](int v, bool first) {
        const unsigned long long k = a.next  ? atomicAdd(a.next, 1ull)
                                     : first ? blockIdx.x + (unsigned long long)gridDim.x * (g * V + v)
                                             : ~0ull;
        book[v].cw = k < (unsigned long long)a.n_cw ? (int64_t)k : -1;
    };
    if (lead) {
#pragma unroll
        for (int v = 0; v < V; v++) {
            grab(v, true);
            book[v].bad[0] = book[v].bad[1] = 0;
        }
    }
    __syncthreads();
    Place<V> p;
    p.own = own;
    p.r = own ? ru : Z - 1;
    p.a0 = (uint32_t)(a.slots0 + g * a.strA + p.r * SA);
    p.a1 = p.a0 - (uint32_t)(Z * SA);
    p.r0 = (uint32_t)(a.slots0 + a.offR + g * a.strR + p.r * SR);
    p.r1 = p.r0;
    const int r = p.r;
    float *A = reinterpret_cast<float *>(sm + p.a0);
    MsgT *R = reinterpret_cast<MsgT *>(sm + p.r0);
    auto gsync = [&]() {
        if (TPG == 32)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(TPG) : "memory");
    };

    // lane v takes codeword k: APP = L (+0: no -0 in APP), messages 0; the channel values of a chunk
    // are all requested before any is used
    auto refill = [&](int v, int64_t k) {
        const float *L = a.llr + k * N + r;
        constexpr int CH = 4;
        for (int j0 = 0; j0 < nb; j0 += CH) {
            float x[CH];
#pragma unroll
            for (int w = 0; w < CH; w++)
                if (j0 + w < nb) x[w] = __ldg(L + (j0 + w) * Z);
#pragma unroll
            for (int w = 0; w < CH; w++)
                if (j0 + w < nb) {
                    if (!isfinite(x[w])) atomicOr(cd->status, IN_NONFINITE);
                    A[(j0 + w) * Z * V + v] = kBase2<MsgT> ? fmaf(x[w], kSLog2e, 0.0f) : x[w] + 0.0f;
                }
        }
        for (int b = 0; b < nnz; b++) R[b * Z * V + v] = MsgT(0.0f);
    };

    int64_t cw[V];
    int t[V];
    bool any = false;
#pragma unroll
    for (int v = 0; v < V; v++) {
        cw[v] = book[v].cw;
        t[v] = 0;
        if (cw[v] >= 0 && own) refill(v, cw[v]);
        any |= cw[v] >= 0;
    }
    any = __any_sync(0xffffffffu, any);  // (votes: conditions known to be warp-uniform)
    gsync();

    for (int ph = 0; any; ph ^= 1) {
#pragma unroll 1
        for (int l = 0; l < mb; l++) {
            layer_check<DMAX, V, MsgT, HC>(a.deg[l], tab + a.first[l], sm, p, Xb, Pb);
            gsync();
        }
        bool busy[V], done[V];
        bool anydone = false;
#pragma unroll
        for (int v = 0; v < V; v++) {
            busy[v] = cw[v] >= 0;
            t[v] += busy[v];
        }
        if (a.early_exit) {
            // syndrome of the hard decisions (APP sign bits), until each codeword of the slot has
            // shown this warp an unsatisfied check
            bool seen[V];
#pragma unroll
            for (int v = 0; v < V; v++) seen[v] = !busy[v];
#pragma unroll 1
            for (int l = 0; l < mb; l++) {
                uint32_t par[V];
                lspa_parity<V>(a.deg[l], tab + a.first[l], sm, p, par);
                bool rest = false;
#pragma unroll
                for (int v = 0; v < V; v++) {
                    const bool u = __any_sync(0xffffffffu, (par[v] & kSign) != 0);
                    if (busy[v] && u) seen[v] = true;
                    rest |= !seen[v];
                }
                if (!__any_sync(0xffffffffu, rest)) break;
            }
            if ((tid & 31) == 0) {
#pragma unroll
                for (int v = 0; v < V; v++)
                    if (seen[v]) book[v].bad[ph] = 1;
            }
            gsync();
        }
#pragma unroll
        for (int v = 0; v < V; v++) {
            done[v] = busy[v] && ((a.early_exit && book[v].bad[ph] == 0) || t[v] >= a.max_iter);
            anydone |= done[v];
        }
        if (a.early_exit && lead) {
            // the other flag was last read in the iteration before
#pragma unroll
            for (int v = 0; v < V; v++) book[v].bad[ph ^ 1] = 0;
        }
        if (__any_sync(0xffffffffu, anydone)) {
#pragma unroll
            for (int v = 0; v < V; v++) {
                if (done[v] && own) {
                    uint8_t *Bo = a.bits + cw[v] * N + r;
                    float *Ao = a.app_out ? a.app_out + cw[v] * N + r : nullptr;
                    for (int j = 0; j < nb; j++) {
                        const float x = A[j * Z * V + v];
                        Bo[j * Z] = x < 0.0f ? 1 : 0;
                        if (Ao) Ao[j * Z] = kBase2<MsgT> ? x * kSLn2 : x;
                    }
                    if (lead) {
                        a.iters[cw[v]] = t[v];
                        grab(v, false);
                    }
                }
            }
            gsync();
            any = false;
#pragma unroll
            for (int v = 0; v < V; v++) {
                if (done[v]) {
                    cw[v] = book[v].cw;
                    t[v] = 0;
                    if (cw[v] >= 0 && own) refill(v, cw[v]);
                }
                any |= cw[v] >= 0;
            }
            any = __any_sync(0xffffffffu, any);
            gsync();
        }
    }
}

// The same for widths that whole warps fit badly (Z of a few lanes, or just above a multiple of 32): the
// rows of K thread slots lie end to end over ceil(K Z / 32) warps.  They share a barrier and run their
// layers in step, so that layers, degrees and tables stay the same for all lanes of a warp and only
// the slot is a lane's own; each codeword still ends, is written out and refilled by itself.  The state
// of the group's codewords is kept by every warp, codeword i in lane i (so K V <= 32), and what a warp
// does next is decided by votes, alike in all warps of the group.  Results are bit-equal.
template <int DMAX, int V, typename MsgT, bool HC>
__global__ void __launch_bounds__(lspa_threads(DMAX, V, sizeof(MsgT) == 2), 1)
    k_layered_spa_packed(const CodeDev *__restrict__ cd, const __grid_constant__ LayeredSpaArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    char *sm = reinterpret_cast<char *>(smem_raw);
    LspaBook *books = reinterpret_cast<LspaBook *>(sm);
    int4 *tab = reinterpret_cast<int4 *>(sm + a.tab0);
    constexpr int SA = (int)sizeof(float) * V, SR = (int)sizeof(MsgT) * V;
    constexpr uint32_t kSign = 0x80000000u;
    constexpr unsigned kFull = 0xffffffffu;
    const int N = a.N, Z = a.Z, mb = a.mb, nb = a.nb, nnz = a.nnz, TPG = a.TPG, K = a.K, KV = K * V;
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31;
    const float Xb = a.X * kSLog2e, Pb = s_phi_b2(a.X);  // the clamp [phi(X), X] in base-2 units
    for (int i = tid; i < nnz; i += nth) {
        const int e = cd->ent[i], sh = e & 0xffff;
        tab[i] = make_int4(SA * ((e >> 16) * Z + sh), SR * i * Z, Z - sh, 0);
    }
    // barrier group g (a warp reduction: known to be warp-uniform); a lane's thread slot k and row r
    const int g = (int)__reduce_min_sync(kFull, (unsigned)(tid / TPG)), x = tid - g * TPG;
    const bool own = x < K * Z;  // (else an idle lane of the group's last warp)
    const int k = own ? x / Z : 0, r = own ? x - k * Z : 0, slot = g * K + k;
    const bool lead = own && r == 0;
    LspaBook *gbook = books + g * KV, *book = gbook + k * V;
    const unsigned peers = __match_any_sync(kFull, own ? k : -1);  // the warp's lanes of the same thread slot
    auto grab = [&](int v, bool first) {
        const unsigned long long n = a.next  ? atomicAdd(a.next, 1ull)
                                     : first ? blockIdx.x + (unsigned long long)gridDim.x * (slot * V + v)
                                             : ~0ull;
        book[v].cw = n < (unsigned long long)a.n_cw ? (int64_t)n : -1;
    };
    if (lead) {
#pragma unroll
        for (int v = 0; v < V; v++) {
            grab(v, true);
            book[v].bad[0] = book[v].bad[1] = 0;
        }
    }
    __syncthreads();
    Place<V> p;
    p.own = own;
    p.r = r;
    p.a0 = (uint32_t)(a.slots0 + slot * a.strA + r * SA);
    p.a1 = p.a0 - (uint32_t)(Z * SA);
    p.r0 = (uint32_t)(a.slots0 + a.offR + slot * a.strR + r * SR);
    p.r1 = p.r0;
    float *A = reinterpret_cast<float *>(sm + p.a0);
    MsgT *R = reinterpret_cast<MsgT *>(sm + p.r0);
    auto gsync = [&]() {
        if (TPG == 32)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(TPG) : "memory");
    };
    auto refill = [&](int v, int64_t n) {  // as k_layered_spa's
        const float *L = a.llr + n * N + r;
        constexpr int CH = 4;
        for (int j0 = 0; j0 < nb; j0 += CH) {
            float y[CH];
#pragma unroll
            for (int w = 0; w < CH; w++)
                if (j0 + w < nb) y[w] = __ldg(L + (j0 + w) * Z);
#pragma unroll
            for (int w = 0; w < CH; w++)
                if (j0 + w < nb) {
                    if (!isfinite(y[w])) atomicOr(cd->status, IN_NONFINITE);
                    A[(j0 + w) * Z * V + v] = kBase2<MsgT> ? fmaf(y[w], kSLog2e, 0.0f) : y[w] + 0.0f;
                }
        }
        for (int b = 0; b < nnz; b++) R[b * Z * V + v] = MsgT(0.0f);
    };
    int64_t cw[V];  // the lane's codewords
#pragma unroll
    for (int v = 0; v < V; v++) {
        cw[v] = book[v].cw;
        if (cw[v] >= 0 && own) refill(v, cw[v]);
    }
    // codeword `lane` of the group: whether there is one, and iterations completed on it
    bool has = lane < KV && gbook[lane].cw >= 0;
    int t = 0;
    unsigned busy = __ballot_sync(kFull, has);
    auto bit = [&](unsigned m, int v) -> bool { return (m >> (k * V + v)) & 1u; };
    gsync();

    for (int ph = 0; busy != 0; ph ^= 1) {
#pragma unroll 1
        for (int l = 0; l < mb; l++) {
            layer_check<DMAX, V, MsgT, HC>(a.deg[l], tab + a.first[l], sm, p, Xb, Pb);
            gsync();
        }
        t += has;
        if (a.early_exit) {
            // syndrome of the hard decisions, until each codeword with rows in this warp has shown an
            // unsatisfied check
            bool seen[V];
#pragma unroll
            for (int v = 0; v < V; v++) seen[v] = !own || !bit(busy, v);
#pragma unroll 1
            for (int l = 0; l < mb; l++) {
                uint32_t par[V];
                lspa_parity<V>(a.deg[l], tab + a.first[l], sm, p, par);
                bool rest = false;
#pragma unroll
                for (int v = 0; v < V; v++) {
                    seen[v] |= (__ballot_sync(kFull, (par[v] & kSign) != 0) & peers) != 0;
                    rest |= !seen[v];
                }
                if (!__any_sync(kFull, rest)) break;
            }
            if (own && lane == __ffs(peers) - 1) {
#pragma unroll
                for (int v = 0; v < V; v++)
                    if (seen[v]) book[v].bad[ph] = 1;
            }
            gsync();
        }
        const bool end = has && ((a.early_exit && gbook[lane].bad[ph] == 0) || t >= a.max_iter);
        const unsigned done = __ballot_sync(kFull, end);
        // the other flag was last read in the iteration before
        if (a.early_exit && x < KV) gbook[x].bad[ph ^ 1] = 0;
        if (done != 0) {
#pragma unroll
            for (int v = 0; v < V; v++) {
                const int tv = __shfl_sync(kFull, t, k * V + v);
                if (own && bit(done, v)) {
                    uint8_t *Bo = a.bits + cw[v] * N + r;
                    float *Ao = a.app_out ? a.app_out + cw[v] * N + r : nullptr;
                    for (int j = 0; j < nb; j++) {
                        const float y = A[j * Z * V + v];
                        Bo[j * Z] = y < 0.0f ? 1 : 0;
                        if (Ao) Ao[j * Z] = kBase2<MsgT> ? y * kSLn2 : y;
                    }
                    if (lead) {
                        a.iters[cw[v]] = tv;
                        grab(v, false);
                    }
                }
            }
            gsync();
            if (end) {
                has = gbook[lane].cw >= 0;
                t = 0;
            }
            busy = __ballot_sync(kFull, has);
#pragma unroll
            for (int v = 0; v < V; v++)
                if (bit(done, v)) {
                    cw[v] = book[v].cw;
                    if (cw[v] >= 0 && own) refill(v, cw[v]);
                }
            gsync();
        }
    }
}

static size_t lspa_slot_bytes(const CodeDev &h, int msg)
{
    return (size_t)((h.N + 3) & ~3) * sizeof(float) +
           (size_t)((h.E + 7) & ~7) * (msg == LDPC_MSG_F16 ? sizeof(__half) : sizeof(float));
}

static size_t lspa_smem(const CodeDev &h, int msg, int C)
{
    return slots_smem_head(4 * h.nnz + h.mb + 1) + (size_t)C * lspa_slot_bytes(h, msg);
}

static size_t lspa_limit()
{
    int dev = 0, lim = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return lim > 0 ? (size_t)lim : 227 * 1024;
}

// Whether the decoder serves a code: one slot in shared memory (beside tables of the size it
// once needed, so that the line stays where it is) and its rows in a CTA's threads.
int layered_spa_slots_per_cta(const CodeDev &h, int msg)
{
    if (h.dc_max > 32 || h.N >= 65536) return 0;
    const int tmax = msg == LDPC_MSG_F16 ? (h.dc_max <= 8 ? 1024 : h.dc_max <= 16 ? 768 : 512)
                                         : (h.dc_max <= 16 ? 672 : 512);
    return ((h.Z + 31) / 32) * 32 <= tmax && lspa_smem(h, msg, 1) <= lspa_limit() ? 1 : 0;
}

// Strides congruent to Z modulo the 32 banks, so that rows of neighbouring slots do not collide.
static int lspa_stride(int n, int Z) { return n + ((Z % 32) - (n % 32) + 32) % 32; }

// Thread slots of V codewords per CTA, at most cap, that the bookkeeping and shared memory allow.
static int lspa_room(const CodeDev &h, int msg, int V, int cap)
{
    int G = cap * V > SLOTS_MAX ? SLOTS_MAX / V : cap;
    const size_t slot = (size_t)V * (4 * (size_t)lspa_stride(h.N, h.Z) +
                                     (msg == LDPC_MSG_F16 ? 2 : 4) * (size_t)lspa_stride(h.E, h.Z)), limit = lspa_limit();
    while (G > 0 && (size_t)G * V * sizeof(LspaBook) + (size_t)h.nnz * 16 + 64 + G * slot > limit) G--;
    return G;
}

// Thread slots of whole warps.
static int lspa_fit(const CodeDev &h, int msg, int V, int cap)
{
    const int wt = ((h.Z + 31) / 32) * 32, dmax = h.dc_max <= 8 ? 8 : 32;
    int G = lspa_threads(dmax, V, msg == LDPC_MSG_F16) / wt;
    if (G > cap) G = cap;
    if (wt > 32 && G > 15) G = 15;  // named barriers
    return lspa_room(h, msg, V, G);
}

// What n codewords cost an SM with G thread slots in groups of K and so many warps, in warps times
// turns: fewer than 20 warps take as long as 20 (latency), a few times the resident codewords take
// whole turns of them, a row of two codewords takes 1.6 times as long as a row of one, and K slots in
// step 5 % and 2 % each, as some of many codewords end in every iteration and hold up the others.
static double lspa_cost(int64_t n, int G, int K, int V, int warps)
{
    double turns = (double)((n + V - 1) / V) / G;
    turns = turns < 8.0 ? ceil(turns) : turns + 0.5;
    return turns * (warps > 20 ? warps : 20) * (V == 2 ? 1.6 : 1.0) * (K > 1 ? 1.05 + 0.02 * (K - 1) : 1.0);
}

template <int DMAX, int V, typename MsgT, bool HC>
static cudaError_t launch_lspa(const CodeDev *d, const LayeredSpaArgs &a, size_t smem, int64_t ctas, cudaStream_t s)
{
    const unsigned threads = a.G / a.K * a.TPG;
    if (a.K > 1) {
        cudaError_t e = ensure_smem<k_layered_spa_packed<DMAX, V, MsgT, HC>>(smem);
        if (e != cudaSuccess) return e;
        LaunchScope ls(F_LAYERED_SPA, s);
        k_layered_spa_packed<DMAX, V, MsgT, HC><<<(unsigned)ctas, threads, smem, s>>>(d, a);
        return cudaGetLastError();
    }
    cudaError_t e = ensure_smem<k_layered_spa<DMAX, V, MsgT, HC>>(smem);
    if (e != cudaSuccess) return e;
    LaunchScope ls(F_LAYERED_SPA, s);
    k_layered_spa<DMAX, V, MsgT, HC><<<(unsigned)ctas, threads, smem, s>>>(d, a);
    return cudaGetLastError();
}

template <typename MsgT, bool HC>
static cudaError_t launch_lspa_d(const CodeDev &h, const CodeDev *d, const LayeredSpaArgs &a, size_t smem,
                                 int64_t ctas, cudaStream_t s)
{
    return h.dc_max <= 8 ? launch_lspa<8, 1, MsgT, HC>(d, a, smem, ctas, s)
                         : launch_lspa<32, 1, MsgT, HC>(d, a, smem, ctas, s);
}

cudaError_t layered_spa_decode(const CodeDev &h, const CodeDev *d, const ldpc_decode_params &p, const float *llr,
                               int64_t n_cw, uint8_t *bits, int32_t *iters, float *app_out, void *counter,
                               cudaStream_t s)
{
    const bool f16 = p.msg == LDPC_MSG_F16;
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int64_t per_sm = (n_cw + nsm - 1) / nsm;  // a small batch spreads over the SMs
    const int cap1 = (int)(per_sm < SLOTS_MAX ? per_sm : SLOTS_MAX), cap2 = (cap1 + 1) / 2;
    const int g1 = lspa_fit(h, p.msg, 1, cap1), g2 = lspa_fit(h, p.msg, 2, cap2);
    // two codewords per thread where that holds more codewords per CTA than the threads allow one
    // to a thread: FP16 messages, rows of degree <= 8.  (8192 codewords on GB300, one against two:
    // N = 1944 rate 1/2 FP16 507 / 467 us, 10 slots against 6 pairs; FP32 502 / 626, 7 against 3;
    // rate 5/6 FP16 489 / 545: there single slots of more warps win.)
    const bool pairs = f16 && h.dc_max <= 8;
    int V = pairs && per_sm > g1 && 2 * g2 > g1 ? 2 : 1;
    const int wt = (h.Z + 31) & ~31;
    LayeredSpaArgs a;
    a.G = V == 2 ? g2 : g1;
    a.K = 1;
    a.TPG = wt;
    if (a.G < 1) return cudaErrorInvalidValue;
    // thread slots end to end in a warp where two fifths of the lanes would be idle and that is estimated
    // 5 % cheaper.  (GB300, 12 x 24 code, us per launch, whole warps / packed: Z = 8 FP32 65536 codewords
    // 2226 / 910, Z = 16 FP16 41472 1345 / 1071, Z = 33 FP32 20107 1826 / 1454, Z = 36 FP32 18432 1498 /
    // 1282; with fewer lanes idle whole warps win, as codewords do not wait for one another: Z = 24 FP32
    // 1003 / 1129, Z = 70 FP32 1202 / 1547.)
    if (5 * h.Z <= 3 * wt && per_sm > 1) {
        double cost = lspa_cost(per_sm, a.G, 1, V, a.G * wt / 32) / 1.05;
        for (int v = 1; v <= (pairs ? 2 : 1); v++) {
            const int tmax = lspa_threads(h.dc_max <= 8 ? 8 : 32, v, f16), room = lspa_room(h, p.msg, v, v == 2 ? cap2 : cap1);
            for (int K = 2; K <= room && K * v <= 32 && K * h.Z <= tmax; K++) {
                const int tpg = (K * h.Z + 31) & ~31;
                int n = tmax / tpg < room / K ? tmax / tpg : room / K;
                if (tpg > 32 && n > 15) n = 15;  // named barriers
                const double c = lspa_cost(per_sm, n * K, K, v, n * tpg / 32);
                if (c < cost * 0.999) {
                    cost = c;
                    V = v;
                    a.G = n * K;
                    a.K = K;
                    a.TPG = tpg;
                }
            }
        }
    }
    a.llr = llr;
    a.n_cw = n_cw;
    a.bits = bits;
    a.iters = iters;
    a.app_out = app_out;
    a.next = static_cast<unsigned long long *>(counter);
    a.N = h.N;
    a.Z = h.Z;
    a.mb = h.mb;
    a.nb = h.nb;
    a.nnz = h.nnz;
    const int SA = 4 * V, SR = (f16 ? 2 : 4) * V;
    a.tab0 = (a.G * V * (int)sizeof(LspaBook) + 15) & ~15;
    a.slots0 = a.tab0 + 16 * h.nnz;
    a.strA = SA * lspa_stride(h.N, h.Z);
    a.strR = SR * lspa_stride(h.E, h.Z);
    a.offR = (a.G * a.strA + 15) & ~15;
    const size_t smem = (size_t)a.slots0 + a.offR + (size_t)a.G * a.strR;
    a.max_iter = p.max_iter;
    a.early_exit = p.early_exit;
    a.X = p.phi_clamp;
    for (int l = 0; l < h.mb; l++) {
        a.first[l] = (uint16_t)h.rowptr[l];
        a.deg[l] = (uint8_t)(h.rowptr[l + 1] - h.rowptr[l]);
    }
    const int64_t need = (n_cw + a.G * V - 1) / (a.G * V), ctas = need < nsm ? need : nsm;
    if (n_cw <= ctas * a.G * V) a.next = nullptr;  // no refills: no counter
    else if (!counter) return cudaErrorInvalidValue;
    if (a.next) {
        const cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned long long), s);
        if (e != cudaSuccess) return e;
    }
    const bool hc = p.phi_clamp < FLOOD_CLAMP_X;
    if (V == 2)
        return hc ? launch_lspa<8, 2, __half, true>(d, a, smem, ctas, s)
                  : launch_lspa<8, 2, __half, false>(d, a, smem, ctas, s);
    if (f16)
        return hc ? launch_lspa_d<__half, true>(h, d, a, smem, ctas, s)
                  : launch_lspa_d<__half, false>(h, d, a, smem, ctas, s);
    return hc ? launch_lspa_d<float, true>(h, d, a, smem, ctas, s)
              : launch_lspa_d<float, false>(h, d, a, smem, ctas, s);
}

}  // namespace ldpc
