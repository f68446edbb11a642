// Horizontal layered normalised min-sum with two codewords per thread (Sec. II "Algorithm 2":
// the checks of a layer are computed from the current variable values, which are updated at
// once; Sec. III-A frame-level parallelism), bit-exact with the integer definition.
//
// Every quantity of the integer min-sum is an integer of magnitude below 2048, which binary16
// represents exactly, and the packed half-precision instructions (add, min/max, compare,
// fused multiply-add) act on two such values at once and round only when the exact result
// is not representable.  So a thread carries the same check row of two codewords in the two
// halves of each 32-bit register and runs every step of the check once for both:
//   Q_k   = sat(APP_n - R_k, msg_sat)                      sub, min, max
//   min1, min2 over |Q_k| (duplicates counted)             3 x min/max per edge
//   S     = XOR of the sign bits of Q_k                    xor of the whole words
//   mag_k = alpha * (|Q_k| == min1 ? min2 : min1)          compare mask, select
//   R_k   = mag_k with sign S xor sign(Q_k)                xor of the sign bits
//   APP_n = sat(Q_k + R_k, app_sat)                        add (+ min, max if it can bind)
// The edge whose |Q| equals min1 takes min2; when two edges share min1, min2 = min1 and the
// choice is immaterial, so no argmin is tracked.  alpha * m = floor(alpha_num * m /
// 2^alpha_shift) is formed per check as round(alpha m - delta) with delta = 1/2 -
// 2^-(alpha_shift + 1): the fractions of alpha m are multiples of 2^-alpha_shift, so alpha m -
// delta lies strictly within 1/2 of floor(alpha m), and adding 1536 (binary16 spacing 1 in
// [1024, 2048)) rounds it there; the host admits only parameters for which alpha m - delta is
// itself exact (layered_pairs_exact).
//
// Storage (shared memory, one CTA per SM, persistent): APP and R as one byte per codeword, each
// the value + 128, the two codewords of a variable or edge in one 16-bit word.  A byte placed under the
// exponent of 1024 (one byte permute for two) is the binary16 number 1024 + 128 + value: the
// biases of APP and R cancel in APP - R, and Q + (R + 1152) is the new APP in the same form, so
// one permute of the low bytes stores both values.  Bit 7 of a byte is set when the value is >= 0:
// the hard decision, and XORing the words of a check gives both codewords' parities at once.
// Messages are in check-row order, edge (b, r) at b*Z + r.  Messages are not cleared when a lane
// takes a codeword: its bytes read as 128 through a mask in its first iteration.
//
// Thread r of a thread slot's warps owns check row r of every layer; the thread slot's own
// barrier separates layers; each lane (codeword) of a thread slot converges, writes its outputs
// and is refilled from the work counter independently.  After each iteration the syndrome is
// taken layer by layer until every lane has shown the warp an unsatisfied check.
//
// What bounds it (GB300): instruction issue (74 %).  65536 codewords of the N = 1944 rate-5/6
// code, 4.0 dB: 1858 -> 1429 us per launch, 66 -> 51 warp instructions per edge of two codewords;
// 4193 codewords of the N = 4000 code, 10 iterations: 421 -> 325 us.  What went: APP as half2
// (bytes now, whose bias cancels in APP - R), the degree test at every edge (blocks of four, and
// exact bodies up to degree 8), divergent control around stores and layers, the descriptor, select and
// add per operand (the offset table: 1667 -> 1429 us), clearing the messages of a new codeword.
// Four codewords per thread (32-bit words) took 41 instructions per edge of two, but left 15
// warps instead of 24: 1644 us.
#include <cuda_fp16.h>
#include <string.h>

#include "ldpc_internal.h"
#include "layered_pairs.h"

namespace ldpc {

constexpr int kPairRefillChunk = 4;  // channel values a thread requests at once when a lane takes a codeword

// Bookkeeping of one lane (codeword) of a thread slot in shared memory.
struct PairBook {
    int64_t cw;      // its next codeword (request-local, -1: none)
    int32_t req;     // and the request
    int32_t cur;     // the request of the codeword it decodes
    int32_t bad[2];  // unsatisfied check seen, by iteration parity
};

// One launch decodes every codeword of up to MULTI_MAX_REQS requests of one code: the
// codewords are the items of one work sequence (request i's codewords are items item0 ..
// item0 + n_cw - 1), taken from a global work counter.
struct LayeredPairArgs {
    int llr_type;
    float scale;
    int n_req;
    int64_t n_items;
    // sizes and layer lists from here, not from the code's device tables: known to be warp-uniform
    int N, Z, mb, nb, nnz;
    int G, TPG;            // thread slots per CTA, threads of one (whole warps)
    int tab0, slots0;      // tables and first slot, bytes from the start of shared memory
    int strA, strR, offR;  // bytes from one thread slot's posteriors / messages to the next one's; first messages
    int max_iter, early_exit, msg_sat, app_sat;
    // binary16 pairs: +-msg_sat, +-app_sat + 1152, alpha = alpha_num / 2^alpha_shift and -delta =
    // 2^-(alpha_shift + 1) - 1/2, in both halves
    uint32_t sat, nsat, appmax, appmin, alpha, ndelta;
    unsigned long long *next;
    uint8_t deg[MB_MAX];    // degree of each layer
    uint16_t first[MB_MAX]; // its first block
    ReqDev reqs[MULTI_MAX_REQS];
};

__device__ __forceinline__ uint32_t h2u(__half2 x) { return *reinterpret_cast<uint32_t *>(&x); }
__device__ __forceinline__ __half2 u2h(uint32_t x) { return *reinterpret_cast<__half2 *>(&x); }

constexpr uint32_t kH1152 = 0x64806480u;    // binary16 1152 in both halves
constexpr uint32_t kH1536 = 0x66006600u;    // 1536
constexpr uint32_t kHm1536 = 0xE600E600u;   // -1536
constexpr uint32_t kHInf = 0x7C007C00u;     // +infinity
constexpr uint32_t kSign2 = 0x80008000u;
constexpr uint32_t kZero2 = 0x8080u;        // the value 0 in both bytes

// the two bytes of a word -> 1024 + byte in each half; and back: the low bytes of the halves
__device__ __forceinline__ __half2 widen(uint32_t w) { return u2h(__byte_perm(w, 0x64646464u, 0x5140)); }
__device__ __forceinline__ uint16_t narrow(__half2 x) { return (uint16_t)__byte_perm(h2u(x), 0u, 0x0020); }

// Shared-memory stores under a predicate: an `if` around them compiles to a divergent region of its
// own (three control instructions per edge).
__device__ __forceinline__ void store_if(bool on, uint32_t addr, uint16_t x)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p st.shared.u16 [%0], %1;\n\t}" ::"r"(addr), "h"(x),
                 "r"((int)on)
                 : "memory");
}
// Edges of a check: EXACT, all D; else edges 4b .. 4b + 3 as one straight-line block and the last
// dc mod 4 one by one: few (warp-uniform) tests of the degree, and a block's loads overlap.
// f(k, slot): edge k, whose state lives in register slot `slot` (a constant).
template <int D, bool EXACT, typename F>
__device__ __forceinline__ void for_edges(int dc, F f)
{
    if constexpr (EXACT) {
#pragma unroll
        for (int k = 0; k < D; k++) f(k, k);
    } else {
        const int nb4 = dc >> 2;
#pragma unroll
        for (int b = 0; b < D / 4; b++) {
            if (b >= nb4) break;
#pragma unroll
            for (int i = 0; i < 4; i++) f(4 * b + i, 4 * b + i);
        }
        const int k0 = nb4 << 2, rem = dc & 3;
        if (rem > 0) f(k0, D);
        if (rem > 1) f(k0 + 1, D + 1);
        if (rem > 2) f(k0 + 2, D + 2);
    }
}

// The posterior offsets of a layer's edges for the thread's row, in one of two forms.  TABLE: a
// 16-bit entry per (block, row), shared by all thread slots: one load, whose address and
// result take warp-uniform offsets (k blocks further; the slot).  Else from the edge descriptors
// (.x = offset of position s, .y = Z - s): row r reaches position r + s, less Z when r >= Z - s.
template <bool TABLE>
struct PairAt;
template <>
struct PairAt<true> {
    const char *sm;
    uint32_t t0;    // the thread's entry of the layer's first block (bytes)
    uint32_t tz;    // bytes of a block's entries
    uint32_t slot;  // the slot's posteriors
    __device__ __forceinline__ uint32_t operator()(int k) const
    {
        return slot + *reinterpret_cast<const uint16_t *>(sm + (t0 + (uint32_t)k * tz));
    }
    __device__ __forceinline__ void again() { asm volatile("" : "+r"(t0)); }
};
template <>
struct PairAt<false> {
    const char *sm;
    uint32_t eo;      // the layer's first descriptor
    uint32_t a0, a1;  // the thread's posterior of block column 0, plain and less one block
    int r;
    __device__ __forceinline__ uint32_t operator()(int k) const
    {
        const int2 e = *reinterpret_cast<const int2 *>(sm + (eo + 8u * (uint32_t)k));
        return (r >= e.y ? a1 : a0) + (uint32_t)e.x;
    }
    __device__ __forceinline__ void again() { asm volatile("" : "+r"(eo), "+r"(a0), "+r"(a1)); }
};

// One check row of a layer for the two codewords of a thread slot.  at: the edges' posteriors; rr:
// offset of the first edge's message; zb: bytes of a block of messages; keep: mask of the lanes
// whose messages are valid; own: whether the thread stores.
template <int D, bool SATAPP, bool EXACT, typename AT>
__device__ __forceinline__ void pair_check(int dc, AT at, char *sm, bool own, uint32_t rr, uint32_t zb, uint32_t keep,
                                           const LayeredPairArgs &k_)
{
    uint32_t q[EXACT ? D : D + 3];
    __half2 mn1 = u2h(kHInf), mn2 = u2h(kHInf);
    uint32_t S = 0;
    for_edges<D, EXACT>(dc, [&](int k, int slot) {
        const uint32_t aw = *reinterpret_cast<const uint16_t *>(sm + at(k));
        uint32_t rw = *reinterpret_cast<const uint16_t *>(sm + (rr + (uint32_t)k * zb));
        rw = (rw & keep) | (kZero2 & ~keep);
        __half2 qq = __hsub2(widen(aw), widen(rw));
        qq = __hmax2(__hmin2(qq, u2h(k_.sat)), u2h(k_.nsat));
        const __half2 mag = __habs2(qq);
        mn2 = __hmin2(mn2, __hmax2(mn1, mag));
        mn1 = __hmin2(mn1, mag);
        S ^= h2u(qq);
        q[slot] = h2u(qq);
    });
    // alpha * min1, min2 as floor(alpha m), carrying the sign of the whole check
    const __half2 m1 = __hadd2(__hadd2(__hfma2(mn1, u2h(k_.alpha), u2h(k_.ndelta)), u2h(kH1536)), u2h(kHm1536));
    const __half2 m2 = __hadd2(__hadd2(__hfma2(mn2, u2h(k_.alpha), u2h(k_.ndelta)), u2h(kH1536)), u2h(kHm1536));
    const uint32_t Sm = S & kSign2;
    const uint32_t A1 = h2u(m1) ^ Sm, A2 = h2u(m2) ^ Sm;
    // (the second pass forms the offsets again: held across the passes they spill)
    if constexpr (!EXACT) {
        at.again();
        asm volatile("" : "+r"(rr));
    }
    const uint32_t sb = (uint32_t)__cvta_generic_to_shared(sm);
    for_edges<D, EXACT>(dc, [&](int k, int slot) {
        const uint32_t qb = q[slot];
        const uint32_t eq = __heq2_mask(__habs2(u2h(qb)), mn1);
        const uint32_t m = ((eq & A2) | (~eq & A1)) ^ (qb & kSign2);
        const __half2 t = __hadd2(u2h(m), u2h(kH1152));  // R + 1152 (and -0 becomes 1152)
        __half2 a = __hadd2(u2h(qb), t);
        if constexpr (SATAPP) a = __hmax2(__hmin2(a, u2h(k_.appmax)), u2h(k_.appmin));
        store_if(own, sb + (rr + (uint32_t)k * zb), narrow(t));
        store_if(own, sb + at(k), narrow(a));
    });
}

// One layer (the degree is warp-uniform): exact bodies up to degree 8.
template <int D, int DMAX, bool SATAPP, typename AT>
__device__ __forceinline__ void pair_layer(int dc, const AT &at, char *sm, bool own, uint32_t rr, uint32_t zb,
                                           uint32_t keep, const LayeredPairArgs &k_)
{
    if constexpr (D <= 8) {
        if (dc == D)
            pair_check<D, SATAPP, true>(dc, at, sm, own, rr, zb, keep, k_);
        else
            pair_layer<D + 1, DMAX, SATAPP>(dc, at, sm, own, rr, zb, keep, k_);
    } else if constexpr (DMAX > 8) {
        pair_check<DMAX, SATAPP, false>(dc, at, sm, own, rr, zb, keep, k_);
    }
}

// XOR of the posterior words of check row r of one layer: bit 7 of each byte is the parity of the
// codeword's decisions [APP >= 0].
template <typename AT>
__device__ __forceinline__ uint32_t pair_parity(int dc, const AT &at, const char *sm)
{
    auto word = [&](uint32_t o) -> uint32_t { return *reinterpret_cast<const uint16_t *>(sm + o); };
    uint32_t par = (dc & 1) ? kZero2 : 0u;  // of [APP < 0] then
    int k = 0;
#pragma unroll 1
    for (; k + 4 <= dc; k += 4) {
        const uint32_t x0 = at(k), x1 = at(k + 1), x2 = at(k + 2), x3 = at(k + 3);
        par ^= word(x0) ^ word(x1);
        par ^= word(x2) ^ word(x3);
    }
#pragma unroll 1
    for (; k < dc; k++) par ^= word(at(k));
    return par;
}

__device__ __forceinline__ int sat_q(int x, int s) { return max(-s, min(s, x)); }

// Load codeword k of request rq into a lane (A: its byte of position r of block column 0; two bytes
// to a variable): APP = quantised LLRs; the channel values of a chunk are all requested before any is used.
__device__ __forceinline__ void lpair_refill(const LayeredPairArgs &a, const CodeDev *__restrict__ cd, uint8_t *A, int rq,
                                             int64_t k, int r)
{
    const void *llr = a.reqs[rq].llr;
    const int N = a.N, Z = a.Z, nb = a.nb;
    constexpr int CH = kPairRefillChunk;
    for (int j0 = 0; j0 < nb; j0 += CH) {
        int q[CH];
        if (a.llr_type == LDPC_LLR_I8) {
            int raw[CH];
#pragma unroll
            for (int w = 0; w < CH; w++)
                if (j0 + w < nb) raw[w] = static_cast<const int8_t *>(llr)[k * N + (j0 + w) * Z + r];
#pragma unroll
            for (int w = 0; w < CH; w++)
                if (j0 + w < nb) {
                    if (raw[w] < -a.msg_sat || raw[w] > a.msg_sat) atomicOr(cd->status, IN_I8_RANGE);
                    q[w] = sat_q(raw[w], a.msg_sat);
                }
        } else {
            float in[CH];
#pragma unroll
            for (int w = 0; w < CH; w++)
                if (j0 + w < nb) in[w] = __ldg(static_cast<const float *>(llr) + k * N + (j0 + w) * Z + r);
#pragma unroll
            for (int w = 0; w < CH; w++)
                if (j0 + w < nb) {
                    if (!isfinite(in[w])) atomicOr(cd->status, IN_NONFINITE);
                    const float rr = rintf(__fmul_rn(a.scale, in[w]));
                    q[w] = rr > (float)a.msg_sat ? a.msg_sat : (rr < -(float)a.msg_sat ? -a.msg_sat : (int)rr);
                }
        }
#pragma unroll
        for (int w = 0; w < CH; w++)
            if (j0 + w < nb) A[(j0 + w) * Z * 2] = (uint8_t)(q[w] + 128);
    }
}

// Threads per CTA of an instance: its registers hold the Q words of up to dmax edges.  (65536
// codewords of the N = 1944 rate-5/6 code, dmax 24: 768 threads 1432 us, 896 1549, 1024 1615, which
// spill; 4193 of the N = 4000 code, dmax 16: 896 326 us, 1024 353.)
__host__ __device__ constexpr int lpairs_threads(int dmax) { return dmax <= 8 ? 1024 : dmax <= 16 ? 896 : 768; }

template <int DMAX, bool SATAPP, bool TABLE, int THREADS>
__global__ void __launch_bounds__(THREADS, 1)
    k_layered_pairs(const CodeDev *__restrict__ cd, const __grid_constant__ LayeredPairArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    char *sm = reinterpret_cast<char *>(smem_raw);
    constexpr int V = 2;  // lanes of a thread slot, and bytes of a word
    PairBook *books = reinterpret_cast<PairBook *>(sm);
    const int N = a.N, Z = a.Z, mb = a.mb, nb = a.nb, nnz = a.nnz, TPG = a.TPG;
    const int tid = threadIdx.x, nth = blockDim.x;
    for (int i = tid; !TABLE && i < nnz; i += nth) {
        const int e = cd->ent[i], sh = e & 0xffff;
        if constexpr (!TABLE) reinterpret_cast<int2 *>(sm + a.tab0)[i] = make_int2(V * ((e >> 16) * Z + sh), Z - sh);
    }
    if constexpr (TABLE)
        for (int i = tid; i < nnz * Z; i += nth) {
            const int b = i / Z, x = i - b * Z + (cd->ent[b] & 0xffff);
            reinterpret_cast<uint16_t *>(sm + a.tab0)[i] = (uint16_t)(V * ((cd->ent[b] >> 16) * Z + (x >= Z ? x - Z : x)));
        }
    // thread slot g (a warp reduction: known to be warp-uniform), row ru of its layers
    const int g = (int)__reduce_min_sync(0xffffffffu, (unsigned)(tid / TPG)), ru = tid - g * TPG;
    const bool lead = ru == 0;
    PairBook *book = books + g * V;
    // a lane's leader takes the next item of the work sequence and finds its request; without a
    // work counter every item has a lane from the start
    auto grab = [&](int v, bool first) {
        const unsigned long long k = a.next  ? atomicAdd(a.next, 1ull)
                                     : first ? blockIdx.x + (unsigned long long)gridDim.x * (g * V + v)
                                             : ~0ull;
        int64_t loc = -1;
        int rq = -1;
        if (k < (unsigned long long)a.n_items) {
            for (rq = 0; rq < a.n_req - 1; rq++)
                if ((int64_t)k < a.reqs[rq].item0 + a.reqs[rq].n_cw) break;
            loc = (int64_t)k - a.reqs[rq].item0;
        }
        book[v].cw = loc;
        book[v].req = rq;
    };
    if (lead) {
#pragma unroll
        for (int v = 0; v < V; v++) {
            grab(v, true);
            book[v].bad[0] = book[v].bad[1] = 0;
        }
    }
    __syncthreads();
    // (an idle lane of a slot's last warp repeats the last row's loads and stores nothing)
    const bool own = ru < Z;
    const int r = own ? ru : Z - 1;
    const uint32_t slot = (uint32_t)(a.slots0 + g * a.strA);  // the slot's posteriors
    const uint32_t r0 = (uint32_t)(a.slots0 + a.offR + g * a.strR + r * V);  // row r of its messages
    uint8_t *A = reinterpret_cast<uint8_t *>(sm + slot + r * V);
    auto edges = [&](int b0) {  // of the layer whose first block is b0
        if constexpr (TABLE)
            return PairAt<true>{sm, (uint32_t)(a.tab0 + 2 * r) + (uint32_t)(2 * b0 * Z), (uint32_t)(2 * Z), slot};
        else
            return PairAt<false>{sm, (uint32_t)(a.tab0 + 8 * b0), slot + (uint32_t)(r * V),
                                 slot + (uint32_t)((r - Z) * V), r};
    };
    auto gsync = [&]() {
        if (TPG == 32)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(TPG) : "memory");
    };

    // a lane's codeword (request-local; requests hold at most 2^31), -1: none; its request is kept in
    // shared memory (read again at the output), not in registers
    int cw[V], t[V];
    uint32_t keep = 0;  // lanes past their first iteration (a byte each): their messages are valid
    bool any = false;
    auto take = [&](int v) {
        const int64_t c = book[v].cw;
        cw[v] = (int)c;
        t[v] = 0;
        keep &= ~(0xffu << (8 * v));
        if (c >= 0) {
            const int rq = book[v].req;
            if (lead) book[v].cur = rq;
            if (own) lpair_refill(a, cd, A + v, rq, c, r);
        }
        any |= c >= 0;
    };
#pragma unroll
    for (int v = 0; v < V; v++) take(v);
    any = __any_sync(0xffffffffu, any);  // (votes: conditions known to be warp-uniform)
    gsync();

    const uint32_t zb = (uint32_t)(Z * V);
    for (int ph = 0; any; ph ^= 1) {
#pragma unroll 1
        for (int l = 0; l < mb; l++) {
            const int b0 = a.first[l];
            pair_layer<2, DMAX, SATAPP>(a.deg[l], edges(b0), sm, own, r0 + (uint32_t)b0 * zb, zb, keep, a);
            gsync();
        }
        keep = 0xffffffffu;
        bool busy[V], done[V];
        bool anydone = false;
        uint32_t busym = 0;
#pragma unroll
        for (int v = 0; v < V; v++) {
            busy[v] = cw[v] >= 0;
            t[v] += busy[v];
            busym |= busy[v] ? 0x80u << (8 * v) : 0u;
        }
        if (a.early_exit) {
            // syndrome of the lanes' hard decisions, until each busy lane has shown this warp an
            // unsatisfied check
            uint32_t seen = 0;
#pragma unroll 1
            for (int l = 0; l < mb; l++) {
                seen |= __reduce_or_sync(0xffffffffu, pair_parity(a.deg[l], edges(a.first[l]), sm) & kZero2);
                if (__all_sync(0xffffffffu, (seen & busym) == busym)) break;
            }
            if ((tid & 31) == 0) {
#pragma unroll
                for (int v = 0; v < V; v++)
                    if (seen & (0x80u << (8 * v))) book[v].bad[ph] = 1;
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
                    const ReqDev &q = a.reqs[book[v].cur];
                    uint8_t *Bo = q.bits + (int64_t)cw[v] * N + r;
                    float *Ao = q.app ? q.app + (int64_t)cw[v] * N + r : nullptr;
                    for (int j = 0; j < nb; j++) {
                        const int x = A[j * Z * V + v];
                        Bo[j * Z] = x < 128 ? 1 : 0;
                        if (Ao) Ao[j * Z] = (float)(x - 128);
                    }
                    if (lead) {
                        q.iters[cw[v]] = t[v];
                        grab(v, false);
                    }
                }
            }
            gsync();
            any = false;
#pragma unroll
            for (int v = 0; v < V; v++) {
                if (done[v])
                    take(v);
                else
                    any |= cw[v] >= 0;
            }
            any = __any_sync(0xffffffffu, any);
            gsync();
        }
    }
}

// ------------------------------------------------------------------ host side

// Whether the half-precision form computes the integer min-sum exactly for these parameters:
// every message magnitude floor(alpha_num * m / 2^alpha_shift) <= 127 (one biased byte), and
// alpha m - delta exact in binary16 for every m <= msg_sat (its numerator 2 alpha_num m -
// 2^alpha_shift + 1 over 2^(alpha_shift + 1) below 2^11).
bool layered_pairs_exact(const ldpc_decode_params &p)
{
    if (p.msg_sat < 1 || p.msg_sat > 127 || p.app_sat < p.msg_sat || p.app_sat > 127) return false;
    if (p.nms_alpha_shift < 0 || p.nms_alpha_shift > 10 || p.nms_alpha_num < 0) return false;
    const long long top = ((long long)p.nms_alpha_num * p.msg_sat) >> p.nms_alpha_shift;
    if (top > 127) return false;
    return 2LL * p.nms_alpha_num * p.msg_sat + (1LL << p.nms_alpha_shift) <= 2047;
}

static int lpairs_dmax(const CodeDev &h) { return h.dc_max <= 8 ? 8 : h.dc_max <= 16 ? 16 : h.dc_max <= 24 ? 24 : 32; }

// Strides congruent to Z modulo the 32 banks' width in elements (of bytes bytes), so that rows of
// neighbouring slots do not collide; whole 16 bytes.
static int lpairs_stride(int n, int Z, int bytes)
{
    const int m = 128 / bytes;
    const int s = (n + (((Z % m) - (n % m)) % m + m) % m) * bytes;
    return (s + 15) & ~15;
}

// The tables' bytes: 16-bit offsets per (block, row), or 8-byte descriptors per block.
static size_t lpairs_tab(const CodeDev &h, bool table) { return table ? 2 * (size_t)h.nnz * h.Z : 8 * (size_t)h.nnz; }

// Thread slots of two codewords per CTA of so many threads, at most cap.
static int lpairs_fit(const CodeDev &h, int cap, bool table, int threads)
{
    if (h.dc_max > 32 || 4 * h.N > 65535) return 0;
    const int wt = ((h.Z + 31) / 32) * 32, V = 2;
    int G = threads / wt;
    if (G > cap) G = cap;
    if (G * V > SLOTS_MAX) G = SLOTS_MAX / V;
    if (wt > 32 && G > 15) G = 15;  // named barriers
    const size_t slot = (size_t)lpairs_stride(h.N, h.Z, V) + lpairs_stride(h.E, h.Z, V);
    while (G > 0 && (size_t)G * V * sizeof(PairBook) + lpairs_tab(h, table) + 64 + G * slot > 227 * 1024) G--;
    return G;
}

// Codewords per CTA (0: code too large: a pair's 4-byte posteriors and 2-byte messages beside
// tables as they once were, so that the line stays where it is).
int layered_pairs_per_cta(const CodeDev &h)
{
    const size_t tables = 4 * (size_t)(2 * SLOTS_MAX + h.mb + 1 + 2 * h.nnz + (h.dc_max <= 8 ? (h.nnz * h.Z + 1) / 2 : 0));
    const size_t head = ((size_t)SLOTS_MAX * 16 + 16 + tables + 15) & ~(size_t)15;
    auto stride = [&](int n, int m) { return (size_t)(n + (((h.Z % m) - (n % m)) % m + m) % m); };
    if (head + stride(h.N, 32) * 4 + stride(h.E, 64) * 2 + 16 > 227 * 1024) return 0;
    return 2 * lpairs_fit(h, SLOTS_MAX / 2, false, lpairs_threads(lpairs_dmax(h)));
}

template <int DMAX, bool SATAPP, bool TABLE, int THREADS = lpairs_threads(DMAX)>
static cudaError_t launch_lpairs(const CodeDev *d, const LayeredPairArgs &a, size_t smem, int ctas, cudaStream_t s)
{
    cudaError_t e = ensure_smem<k_layered_pairs<DMAX, SATAPP, TABLE, THREADS>>(smem);
    if (e != cudaSuccess) return e;
    LaunchScope ls(F_LAYERED, s);
    k_layered_pairs<DMAX, SATAPP, TABLE, THREADS><<<(unsigned)ctas, a.G * a.TPG, smem, s>>>(d, a);
    return cudaGetLastError();
}

template <bool SATAPP, bool TABLE>
static cudaError_t launch_lpairs_d(const CodeDev &h, const CodeDev *d, const LayeredPairArgs &a, size_t smem, int ctas,
                                   cudaStream_t s)
{
    switch (lpairs_dmax(h)) {
    case 8: return launch_lpairs<8, SATAPP, TABLE>(d, a, smem, ctas, s);
    case 16:  // (1024 threads only where 896 hold fewer slots)
        return a.G * a.TPG > lpairs_threads(16) ? launch_lpairs<16, SATAPP, TABLE, 1024>(d, a, smem, ctas, s)
                                                : launch_lpairs<16, SATAPP, TABLE>(d, a, smem, ctas, s);
    case 24: return launch_lpairs<24, SATAPP, TABLE>(d, a, smem, ctas, s);
    default: return launch_lpairs<32, SATAPP, TABLE>(d, a, smem, ctas, s);
    }
}

// Decode the codewords of n requests of one code (reqs[i].code all the same) in one launch.
cudaError_t layered_pairs_decode(const CodeDev &h, const CodeDev *d, const ldpc_decode_params &p,
                                 const HostReq *reqs, int n, int llr_type, void *counter, cudaStream_t s)
{
    if (!layered_pairs_exact(p) || n < 1 || n > MULTI_MAX_REQS) return cudaErrorInvalidValue;
    LayeredPairArgs a;
    memset(&a, 0, sizeof a);
    int64_t items = 0;
    for (int i = 0; i < n; i++) {
        if (reqs[i].n_cw <= 0) continue;
        ReqDev &q = a.reqs[a.n_req++];
        q.llr = reqs[i].llr;
        q.bits = reqs[i].bits;
        q.iters = reqs[i].iters;
        q.app = reqs[i].app;
        q.n_cw = reqs[i].n_cw;
        q.item0 = items;
        items += reqs[i].n_cw;
    }
    if (items == 0) return cudaSuccess;
    a.n_items = items;
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    // a small batch spreads over the SMs rather than filling a few CTAs' slots
    const int64_t per_cta = (items + nsm - 1) / nsm;
    const int cap = per_cta < SLOTS_MAX ? (int)((per_cta + 1) / 2) : SLOTS_MAX / 2;
    // the offset table where it costs no thread slot
    int threads = lpairs_threads(lpairs_dmax(h)), g = lpairs_fit(h, cap, false, threads);
    // rows of 9 to 16 edges in 1024 threads, which spill, where their further thread slots save more than that:
    // 896 hold one slot of Z in 449..512 and 1024 two (4 x 16 code of Z = 500, 10 iterations, 600 codewords
    // 149 against 127 us, 12000 2842 against 2367; but Z = 250, 4000 codewords, five turns against four:
    // 404 against 421)
    if (threads == 896) {
        const int wide = lpairs_fit(h, cap, false, 1024);
        auto turns = [&](int G) { return (int)(((per_cta + 1) / 2 + G - 1) / G); };
        if (g < 1 || 1.3 * turns(wide) < turns(g)) {
            threads = 1024;
            g = wide;
        }
    }
    const bool table = lpairs_fit(h, cap, true, threads) == g;
    constexpr int V = 2;
    a.G = g;
    if (a.G < 1) return cudaErrorInvalidValue;
    a.TPG = ((h.Z + 31) / 32) * 32;
    a.llr_type = llr_type;
    a.scale = p.llr_scale;
    a.N = h.N;
    a.Z = h.Z;
    a.mb = h.mb;
    a.nb = h.nb;
    a.nnz = h.nnz;
    a.tab0 = (a.G * V * (int)sizeof(PairBook) + 15) & ~15;
    a.slots0 = (a.tab0 + (int)lpairs_tab(h, table) + 15) & ~15;
    a.strA = lpairs_stride(h.N, h.Z, V);
    a.strR = lpairs_stride(h.E, h.Z, V);
    a.offR = a.G * a.strA;
    const size_t smem = (size_t)a.slots0 + a.offR + (size_t)a.G * a.strR;
    for (int l = 0; l < h.mb; l++) {
        a.first[l] = (uint16_t)h.rowptr[l];
        a.deg[l] = (uint8_t)(h.rowptr[l + 1] - h.rowptr[l]);
    }
    a.max_iter = p.max_iter;
    a.early_exit = p.early_exit;
    a.msg_sat = p.msg_sat;
    a.app_sat = p.app_sat;
    auto pair = [](float x) {
        const unsigned short hb = __half_as_ushort(__float2half_rn(x));  // exact for these values
        return (uint32_t)hb | ((uint32_t)hb << 16);
    };
    a.sat = pair((float)p.msg_sat);
    a.nsat = pair(-(float)p.msg_sat);
    a.appmax = pair(1152.0f + (float)p.app_sat);
    a.appmin = pair(1152.0f - (float)p.app_sat);
    a.alpha = pair((float)p.nms_alpha_num / (float)(1 << p.nms_alpha_shift));
    a.ndelta = pair(1.0f / (float)(2 << p.nms_alpha_shift) - 0.5f);
    a.next = static_cast<unsigned long long *>(counter);
    const int64_t need = (items + a.G * V - 1) / (a.G * V);
    const int ctas = (int)(need < nsm ? need : nsm);
    if (items <= (int64_t)ctas * a.G * V) a.next = nullptr;  // no refills: no counter
    else if (!counter) return cudaErrorInvalidValue;
    if (a.next) {
        const cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned long long), s);
        if (e != cudaSuccess) return e;
    }
    const long long top = ((long long)p.nms_alpha_num * p.msg_sat) >> p.nms_alpha_shift;
    const bool sat = p.msg_sat + top > p.app_sat;
    if (table)
        return sat ? launch_lpairs_d<true, true>(h, d, a, smem, ctas, s)
                   : launch_lpairs_d<false, true>(h, d, a, smem, ctas, s);
    return sat ? launch_lpairs_d<true, false>(h, d, a, smem, ctas, s)
               : launch_lpairs_d<false, false>(h, d, a, smem, ctas, s);
}

}  // namespace ldpc
