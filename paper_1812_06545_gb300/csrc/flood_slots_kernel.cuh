// The kernel of the flooding slot decoder (see flood_slots.cu for the schedule and the host
// side); its instances are compiled one translation unit per message type and clamp form
// (flood_slots_f32.cu, ...).
#pragma once

#include "flood_check.cuh"
#include "flood_slots.h"

namespace ldpc {

// Channel values a thread loads at once when a slot takes a codeword.
constexpr int kRefillChunk = 8;
// Columns whose channel values a thread requests at once in the variable-node phase (4: 915 us
// against 907 on the N = 1944 rate-1/2 FP32 launch, 655 against 645 FP16).
constexpr int kVnChunk = 3;

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
    constexpr bool B2 = kSlotB2<MsgT>;
    const OwnMem<V, MsgT> mem{sm};
    if constexpr (D <= DMAX) {
        constexpr bool LAST = CLS + 1 == FLOOD_CLASSES || (V == 2 && D == 16);  // (one body for all wide rows)
        const int end = gd.rend[LAST ? FLOOD_CLASSES - 1 : CLS];
        for (; i < end; i += step, step = W2 - step) {
            const int hd = rows[i];
            if constexpr (D <= 8)
                check_narrow<D, V, MsgT, B2, HC>(tab + (hd >> 8), mem, p, Xb, Pb, pbad);
            else if constexpr (D == 12)
                check_12<V, MsgT, B2, HC>(hd & 255, tab + (hd >> 8), mem, p, Xb, Pb, pbad);
            else
                check_wide<V == 1 ? D / 8 : 0, V, MsgT, B2, HC>(hd & 255, tab + (hd >> 8), mem, p, Xb, Pb, pbad);
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
// degree above 4: three, and in .w the element of the others); its first variable, in the
// channel values and the posteriors alike, is the cols word.  All lanes' posteriors are stored
// (converged codewords have been written out before): N = 1944 rate 1/2, FP32 901 -> 887 us, FP16
// 643 -> 629, rate 5/6 311 -> 304 against a store per active lane and a multiply per address.
template <int V>
struct VnArgs {
    const float *L[V];  // the codewords' channel values at the thread's position of block column 0
    uint32_t a0, r0;    // the thread's posterior and message offsets
    bool st;            // not an idle lane of the slot's last warp
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
            lv[c] = vset(T(), 0.0f);  // (left unset the values of a chunk spill: 1033 us against 887)
            jc[c] = 0;
            if (c == 0 || i + c * W < end) {
                jc[c] = cols[i + c * W];
                each(lv[c], [&](float &x, int v) { x = __ldg(q.L[v] + jc[c]); });
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
                if (q.st) Sm<float, V>::st(sm + (q.a0 + (uint32_t)(jc[c] * (int)sizeof(T))), s);
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
        FloodBook *book = reinterpret_cast<FloodBook *>(sm + gd.book0) + (member ? g : 0) * V;
        const int32_t *rows = reinterpret_cast<const int32_t *>(tab + gd.t_row);

        // a slot's leader takes the group's next codeword and finds its request; without a work
        // counter every codeword has a slot from the start
        auto grab = [&](int v, bool first) {
            const unsigned long long k = a.next  ? atomicAdd(a.next + grp, 1ull)
                                         : first ? blockIdx.x + (unsigned long long)gridDim.x * (g * V + v)
                                                 : ~0ull;
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
                grab(v, true);
                book[v].bad[0] = book[v].bad[1] = 0;
            }
        }
        __syncthreads();

        Place<V> p;
        p.r = r;
        p.own = mine;
        p.a0 = (uint32_t)(gd.slots0 + (member ? g : 0) * gd.strA + r * SA);
        p.a1 = p.a0 - (uint32_t)(Z * SA);
        p.r0 = (uint32_t)(gd.slots0 + gd.offR + (member ? g : 0) * gd.strR + r * SR);
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
            // first the converged codewords are written out (after which their posteriors may be
            // overwritten: the variable-node phase stores all lanes), then, after the
            // variable-node phase, those at the iteration limit
            auto output = [&](int v, bool out) {
                if (__any_sync(0xffffffffu, out) && mine) {
                    const FloodReq &q = a.reqs[rq[v]];
                    uint8_t *Bo = q.bits + cw[v] * N;
                    float *Ao = q.app ? q.app + cw[v] * N : nullptr;
                    const int32_t *cols = rows + gd.mb;
                    for (int i = w0; i < nb; i += W) {  // the columns this thread updates
                        const int n = cols[i];
                        const float x = A[n * V + v];
                        Bo[n + r] = x < 0.0f ? 1 : 0;
                        if (Ao) Ao[n + r] = x;
                    }
                    if (lead) {
                        q.iters[cw[v]] = t[v];
                        grab(v, false);
                    }
                }
            };
#pragma unroll
            for (int v = 0; v < V; v++) output(v, done[v]);
            if (__any_sync(0xffffffffu, anyact)) {
                VnArgs<V> q;
#pragma unroll
                for (int v = 0; v < V; v++) {  // an idle lane of a pair reads the other's channel values
                    const int rx = act[v] ? rq[v] : rq[V - 1 - v];
                    const int64_t cx = act[v] ? cw[v] : cw[V - 1 - v];
                    q.L[v] = a.reqs[rx].llr + cx * N + r;
                }
                q.a0 = p.a0;
                q.r0 = p.r0;
                q.st = mine;
                vn_cols<1, V, MsgT>(gd, tab, rows + gd.mb, sm, q, w0, W);
            }
#pragma unroll
            for (int v = 0; v < V; v++) {
                if (act[v]) t[v]++;
                const bool last = act[v] && t[v] >= a.max_iter;
                output(v, last);
                done[v] |= last;
                anydone |= done[v];
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
static cudaError_t launch_one(const FloodPlan &q, cudaStream_t s)
{
    cudaError_t e = ensure_smem<k_flood_slots<DMAX, V, MsgT, HC>>(q.smem);
    if (e != cudaSuccess) return e;
    LaunchScope ls(F_SLOTS, s);
    k_flood_slots<DMAX, V, MsgT, HC><<<(unsigned)q.ctas, q.threads, q.smem, s>>>(q.a);
    return cudaGetLastError();
}

template <typename MsgT, bool HC>
cudaError_t flood_slots_launch(const FloodPlan &q, cudaStream_t s)
{
    if (q.dmax <= 8) return q.V == 2 ? launch_one<8, 2, MsgT, HC>(q, s) : launch_one<8, 1, MsgT, HC>(q, s);
    return q.V == 2 ? launch_one<32, 2, MsgT, HC>(q, s) : launch_one<32, 1, MsgT, HC>(q, s);
}

}  // namespace ldpc
