// The flooding slot decoder for widths that whole warps fit badly (Z of a few lanes, or just above a
// multiple of 32).
//
// In k_flood_slots (flood_slots_kernel.cuh) a block row of a thread slot takes ceil(Z / 32) warps,
// which for Z = 8 leaves three lanes of four idle.  Here the rows of K thread slots lie end to end over
// ceil(K Z / 32) warps, which still work on one block row at a time: loops, degrees and tables stay the
// same for all lanes of a warp, and only the slot is a lane's own.  The K thread slots share a
// barrier and run in step; each codeword still ends, is written out and refilled by itself.  The state
// of the group's codewords is kept by every warp, codeword i in lane i (so K V <= 32), and what a
// warp does next is decided by votes, alike in all warps of the group.
// flood_slots.cu has the rule for it and what it measured.
//
// SPREAD (one codeword per thread): the row groups lie end to end too, lane x of a barrier group at row
// x mod Z of thread slot (x / Z) mod K in row group x / (K Z), for small batches and codes of which
// few codewords fit an SM, where there are no K thread slots to fill the warps.  A warp's lanes then
// can be at rows of different degree: it takes rows and columns in turns whose body it agrees on by
// a vote (a lane without a row for that body repeats another's loads and stores nothing), and tables
// are read at per-lane addresses.
//
// Operations and order of every message are those of k_flood_slots: results are bit-equal.
#pragma once

#include "flood_slots_kernel.cuh"

namespace ldpc {

// The check-node phase of one thread: list positions i, i + step, ... (back and forth, as rows_of) below mb.
// In each turn the warp takes the first body any of its lanes is at.
template <int DMAX, int V, typename MsgT, bool HC>
__device__ __forceinline__ void rows_spread(const int4 *__restrict__ tab, const int32_t *__restrict__ rows, int mb,
                                            const OwnMem<V, MsgT> mem, const Place<V> &p, float Xb, float Pb,
                                            uint32_t (&pbad)[V], int i, int step, int W2)
{
    constexpr bool B2 = kSlotB2<MsgT>;
    for (;;) {
        int hd = i < mb ? rows[i] : kNoRow;
        bool on;
        const int body = vote_body(hd, on), dc = hd & 255;
        if (body == kNoRow) break;
        const int4 *ed = tab + (hd >> 8);
        Place<V> q = p;
        q.own = p.own && on;
        // (the parity of the row a lane repeats is one of its own codeword's checks too)
        switch (body) {
        case 2: check_narrow<2, V, MsgT, B2, HC>(ed, mem, q, Xb, Pb, pbad); break;
        case 3: check_narrow<3, V, MsgT, B2, HC>(ed, mem, q, Xb, Pb, pbad); break;
        case 4: check_narrow<4, V, MsgT, B2, HC>(ed, mem, q, Xb, Pb, pbad); break;
        case 5: check_narrow<5, V, MsgT, B2, HC>(ed, mem, q, Xb, Pb, pbad); break;
        case 6: check_narrow<6, V, MsgT, B2, HC>(ed, mem, q, Xb, Pb, pbad); break;
        case 7: check_narrow<7, V, MsgT, B2, HC>(ed, mem, q, Xb, Pb, pbad); break;
        case 8: check_narrow<8, V, MsgT, B2, HC>(ed, mem, q, Xb, Pb, pbad); break;
        default:
            if constexpr (DMAX > 8) {
                if (body == 12)
                    check_12<V, MsgT, B2, HC>(dc, ed, mem, q, Xb, Pb, pbad);
                else if (body == 16)
                    check_wide<2, V, MsgT, B2, HC>(dc, ed, mem, q, Xb, Pb, pbad);
                else if (body == 24)
                    check_wide<3, V, MsgT, B2, HC>(dc, ed, mem, q, Xb, Pb, pbad);
                else
                    check_wide<4, V, MsgT, B2, HC>(dc, ed, mem, q, Xb, Pb, pbad);
            }
        }
        if (on) {
            i += step;
            step = W2 - step;
        }
    }
}

// The variable-node phase of one thread: columns i, i + W, ... below nb of the degree-ordered list.
template <int V, typename MsgT>
__device__ __forceinline__ void cols_spread(const FloodGroup &gd, const int4 *__restrict__ tab,
                                           const int32_t *__restrict__ cols, char *sm, const VnArgs<V> &q, int i, int W)
{
    using T = VT<V>;
    const int nb = gd.nb, e1 = gd.cend[0], e2 = gd.cend[1], e3 = gd.cend[2], e4 = gd.cend[3];
    for (; __any_sync(kFullWarp, i < nb); i += kVnChunk * W) {
        T lv[kVnChunk];
        int at[kVnChunk], jc[kVnChunk];
#pragma unroll
        for (int c = 0; c < kVnChunk; c++) {
            at[c] = i + c * W < nb ? i + c * W : nb - 1;
            jc[c] = cols[at[c]];
            lv[c] = vset(T(), 0.0f);
            each(lv[c], [&](float &x, int v) { x = __ldg(q.L[v] + jc[c]); });
        }
#pragma unroll
        for (int c = 0; c < kVnChunk; c++) {
            const bool ok = i + c * W < nb;
            const int dv = 1 + (at[c] >= e1) + (at[c] >= e2) + (at[c] >= e3) + (at[c] >= e4);  // 5: above 4
            const int top = (int)__reduce_max_sync(kFullWarp, ok ? (unsigned)dv : 0u);
            if (top == 0) break;
            const int4 o = tab[gd.t_col + at[c]];
            T s = vn_add<V, MsgT>(lv[c], o.x, q.r0, sm);
            if (top > 1) s = pick(dv > 1, vn_add<V, MsgT>(s, o.y, q.r0, sm), s);
            if (top > 2) s = pick(dv > 2, vn_add<V, MsgT>(s, o.z, q.r0, sm), s);
            if (top > 3) s = pick(dv == 4, vn_add<V, MsgT>(s, dv == 4 ? o.w : 0, q.r0, sm), s);
            if (top > 4) {
                int k = dv == 5 ? o.w & 255 : 0;
                const int4 *m = tab + (dv == 5 ? o.w >> 8 : 0);
                for (; __any_sync(kFullWarp, k > 0); k -= 4, m++) {
                    const int4 e = k > 0 ? *m : make_int4(0, 0, 0, 0);
                    s = pick(k > 0, vn_add<V, MsgT>(s, e.x, q.r0, sm), s);
                    s = pick(k > 1, vn_add<V, MsgT>(s, e.y, q.r0, sm), s);
                    s = pick(k > 2, vn_add<V, MsgT>(s, e.z, q.r0, sm), s);
                    s = pick(k > 3, vn_add<V, MsgT>(s, e.w, q.r0, sm), s);
                }
            }
            s = vadd(s, vset(T(), 0.0f));  // -0 -> +0: the sign bit is the decision
            if (ok && q.st) Sm<float, V>::st(sm + (q.a0 + (uint32_t)(jc[c] * (int)sizeof(T))), s);
        }
    }
}

template <int DMAX, int V, typename MsgT, bool HC, bool SPREAD>
__global__ void __launch_bounds__(flood_threads_max(DMAX, V, sizeof(MsgT) == 2), 1) k_flood_packed(const __grid_constant__ FloodArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    char *sm = reinterpret_cast<char *>(smem_raw);
    int32_t *misc = reinterpret_cast<int32_t *>(sm);    // [4] code-group hand-over
    int4 *tab = reinterpret_cast<int4 *>(sm + a.tab0);  // the code's tables
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31;
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
        const int N = gd.N, Z = gd.Z, nb = gd.nb, nnz = gd.nnz, W = gd.W, K = gd.K, TPG = gd.TPG;
        const int KV = K * V;  // codewords of a barrier group (at most a warp's lanes)
        // barrier group g and, unless SPREAD, row group w0 of a warp (from a reduction: known to be
        // warp-uniform); the thread slot k of the group and the row r of a lane
        const int WT = SPREAD ? TPG : TPG / W, gw = (int)__reduce_min_sync(kFullWarp, (unsigned)(tid / WT));
        const int g = SPREAD ? gw : gw / W, x = tid - gw * WT;
        const bool member = g * K < gd.G;                            // the warp belongs to a barrier group
        const bool mine = member && x < K * Z * (SPREAD ? W : 1);  // (else an idle lane of a last warp)
        const int kw = mine ? x / Z : 0, r = mine ? x - kw * Z : 0;
        const int w0 = SPREAD ? kw / K : gw - g * W, k = SPREAD ? kw - w0 * K : kw;
        const int slot = member ? g * K + k : 0;
        const bool lead = mine && r == 0 && w0 == 0;  // the thread that takes codewords for its slot
        FloodBook *gbook = reinterpret_cast<FloodBook *>(sm + gd.book0) + (member ? g : 0) * KV;
        FloodBook *book = gbook + k * V;
        const int32_t *rows = reinterpret_cast<const int32_t *>(tab + gd.t_row), *cols = rows + gd.mb;

        auto grab = [&](int v, bool first) {
            const unsigned long long n = a.next  ? atomicAdd(a.next + grp, 1ull)
                                         : first ? blockIdx.x + (unsigned long long)gridDim.x * (slot * V + v)
                                                 : ~0ull;
            int64_t loc = -1;
            int rq = -1;
            if (n < (unsigned long long)gd.n_items) {
                for (rq = gd.req_begin; rq < gd.req_end - 1; rq++)
                    if ((int64_t)n < a.reqs[rq + 1].item0) break;
                loc = (int64_t)n - a.reqs[rq].item0;
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
        p.a0 = (uint32_t)(gd.slots0 + slot * gd.strA + r * SA);
        p.a1 = p.a0 - (uint32_t)(Z * SA);
        p.r0 = (uint32_t)(gd.slots0 + gd.offR + slot * gd.strR + r * SR);
        p.r1 = p.r0 - (uint32_t)(Z * SR);
        float *A = reinterpret_cast<float *>(sm + p.a0);  // position r of block column 0
        MsgT *R = reinterpret_cast<MsgT *>(sm + p.r0);    // position r of block 0
        int cw[V];  // the thread's codewords (request-local; requests hold at most 2^31) and their requests
        int rq[V];
#pragma unroll
        for (int v = 0; v < V; v++) {
            cw[v] = member ? (int)book[v].cw : -1;
            rq[v] = member ? book[v].req : -1;
        }
        // codeword `lane` of the group: whether there is one, and iterations completed on it
        bool has = member && lane < KV && gbook[lane].cw >= 0;
        int t = 0;
        auto bit = [&](unsigned m, int v) -> bool { return (m >> (k * V + v)) & 1u; };

        // load a new codeword into lane v, this thread's columns: APP = L (+0 for -0), messages 0
        auto refill = [&](int v) {
            const float *Lr = a.reqs[rq[v]].llr + (int64_t)cw[v] * N;
            constexpr int CH = kRefillChunk;
            for (int j0 = w0; j0 < nb; j0 += CH * W) {
                float y[CH];
#pragma unroll
                for (int c = 0; c < CH; c++)
                    if (j0 + c * W < nb) y[c] = __ldg(Lr + (j0 + c * W) * Z + r);
#pragma unroll
                for (int c = 0; c < CH; c++)
                    if (j0 + c * W < nb) {
                        if (!isfinite(y[c])) atomicOr(gd.status, IN_NONFINITE);
                        A[(j0 + c * W) * Z * V + v] = y[c] + 0.0f;
                    }
            }
            for (int b = w0; b < nnz; b += W) R[b * Z * V + v] = MsgT(0.0f);
        };
        auto gsync = [&]() {  // the barrier of the group's warps
            if (TPG == 32)
                __syncwarp();
            else
                asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(TPG) : "memory");
        };

        bool any = __any_sync(kFullWarp, has);
        if (any) {
#pragma unroll
            for (int v = 0; v < V; v++)
                if (mine && cw[v] >= 0) refill(v);
            gsync();
        }

        for (int ph = 0; any; ph ^= 1) {
            // ---------------- check-node phase
            {
                uint32_t pbad[V];
#pragma unroll
                for (int v = 0; v < V; v++) pbad[v] = 0;
                if constexpr (SPREAD)
                    rows_spread<DMAX, V, MsgT, HC>(tab, rows, gd.mb, OwnMem<V, MsgT>{sm}, p, Xb, Pb, pbad,
                                                   mine ? w0 : gd.mb, 2 * (W - w0) - 1, 2 * W);
                else
                    rows_of<0, DMAX, V, MsgT, HC>(gd, tab, rows, sm, p, Xb, Pb, pbad, w0, 2 * (W - w0) - 1, 2 * W);
#pragma unroll
                for (int v = 0; v < V; v++)
                    if (mine && (pbad[v] & kSign)) book[v].bad[ph] = 1;
            }
            gsync();

            // ---------------- decision: the group's converged and its active codewords
            const bool conv = has && t >= 1 && a.early_exit && gbook[lane].bad[ph] == 0;
            unsigned done = __ballot_sync(kFullWarp, conv);
            const unsigned act = __ballot_sync(kFullWarp, has && !conv);
            // the other flag was last read before this round's first barrier
            if (x < KV && (SPREAD || w0 == 0)) gbook[x].bad[ph ^ 1] = 0;
            // converged codewords are written out first, after which their posteriors may be overwritten
            auto output = [&](unsigned m) {
                if (m == 0) return;
#pragma unroll
                for (int v = 0; v < V; v++) {
                    const int tv = __shfl_sync(kFullWarp, t, k * V + v);
                    if (mine && bit(m, v)) {
                        const FloodReq &q = a.reqs[rq[v]];
                        uint8_t *Bo = q.bits + (int64_t)cw[v] * N;
                        float *Ao = q.app ? q.app + (int64_t)cw[v] * N : nullptr;
                        for (int i = w0; i < nb; i += W) {  // the columns this thread updates
                            const int n = cols[i];
                            const float y = A[n * V + v];
                            Bo[n + r] = y < 0.0f ? 1 : 0;
                            if (Ao) Ao[n + r] = y;
                        }
                        if (lead) {
                            q.iters[cw[v]] = tv;
                            grab(v, false);
                        }
                    }
                }
            };
            output(done);
            // ---------------- variable-node phase
            if (act != 0) {
                VnArgs<V> q;
#pragma unroll
                for (int v = 0; v < V; v++) {  // a lane without a codeword reads the other's channel values, or the first's
                    const int u = bit(act, v) ? v : V - 1 - v;
                    const bool own = bit(act, u);
                    q.L[v] = (own ? a.reqs[u == v ? rq[v] : rq[V - 1 - v]].llr + (int64_t)(u == v ? cw[v] : cw[V - 1 - v]) * N
                                  : a.reqs[gd.req_begin].llr) + r;
                }
                q.a0 = p.a0;
                q.r0 = p.r0;
                q.st = mine;
                if constexpr (SPREAD)
                    cols_spread<V, MsgT>(gd, tab, cols, sm, q, mine ? w0 : nb, W);
                else
                    vn_cols<1, V, MsgT>(gd, tab, cols, sm, q, w0, W);
            }
            const bool on = (act >> lane) & 1u;
            t += on;
            const unsigned last = __ballot_sync(kFullWarp, on && t >= a.max_iter);
            output(last);
            done |= last;
            gsync();

            // ---------------- refill finished slots
            if (done != 0) {
                if ((done >> lane) & 1u) {
                    has = gbook[lane].cw >= 0;
                    t = 0;
                }
                any = __any_sync(kFullWarp, has);
#pragma unroll
                for (int v = 0; v < V; v++)
                    if (bit(done, v)) {
                        cw[v] = (int)book[v].cw;
                        rq[v] = book[v].req;
                        if (mine && cw[v] >= 0) refill(v);
                    }
                gsync();
            }
        }

        // this group is dry here and every slot has drained: move to the group with the most
        // codewords left, or stop
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
        grp = (int)__reduce_max_sync(kFullWarp, misc[0]);
        __syncthreads();
        if (grp < 0) return;
    }
}

template <int DMAX, int V, typename MsgT, bool HC, bool SPREAD>
static cudaError_t launch_packed(const FloodPlan &q, cudaStream_t s)
{
    cudaError_t e = ensure_smem<k_flood_packed<DMAX, V, MsgT, HC, SPREAD>>(q.smem);
    if (e != cudaSuccess) return e;
    LaunchScope ls(F_SLOTS, s);
    k_flood_packed<DMAX, V, MsgT, HC, SPREAD><<<(unsigned)q.ctas, q.threads, q.smem, s>>>(q.a);
    return cudaGetLastError();
}

template <int DMAX, typename MsgT, bool HC>
static cudaError_t launch_packed_v(const FloodPlan &q, cudaStream_t s)
{
    if (q.form == FLOOD_SPREAD) return launch_packed<DMAX, 1, MsgT, HC, true>(q, s);
    return q.V == 2 ? launch_packed<DMAX, 2, MsgT, HC, false>(q, s) : launch_packed<DMAX, 1, MsgT, HC, false>(q, s);
}

template <typename MsgT, bool HC>
cudaError_t flood_packed_launch(const FloodPlan &q, cudaStream_t s)
{
    return q.dmax <= 8 ? launch_packed_v<8, MsgT, HC>(q, s) : launch_packed_v<32, MsgT, HC>(q, s);
}

}  // namespace ldpc
