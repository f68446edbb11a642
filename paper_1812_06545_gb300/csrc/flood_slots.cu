// Flooding sum-product decoding with the decoder state on chip: the slot decoder.
//
// A persistent grid of one CTA per SM.  Each CTA holds thread slots of V codewords (two, packed
// in float2 operands, or one for small batches); a thread slot keeps its codewords' posteriors
// APP [N] (fp32) and check-to-variable messages R [E] (fp32 or fp16, stored negated) in shared
// memory for their whole decode, so HBM/L2 traffic per iteration is the channel LLRs only
// (re-read from the caller's buffer, L2-resident while the slot is busy).
//
// Threads: a thread slot is run by W row groups of whole warps.  Thread r of row group w owns row
// r (the Z checks of a QC block row touch disjoint variables) of every W-th block row and
// position r of every W-th block column, both taken in ascending degree, so that a warp runs
// one straight-line body of exact degree at a time, and control and table indexes are the same
// for all its lanes.  Only the thread slot's own warps synchronise (a named barrier): the
// thread slots of a CTA run their rounds independently.
// Where whole warps would leave many lanes idle (Z below a warp, or just above a multiple of 32), the
// rows of several thread slots, or of several row groups, lie end to end (flood_packed_kernel.cuh).
//
// One round of a thread slot (Sec. II two-phase message passing, Algorithm 1 loop order):
//   check-node phase   Q = APP - R, R' from the check rule in the product (tanh) domain
//                      (slot_common.cuh), written in place; the parity of the hard decisions
//                      (APP sign bits) over each check marks a codeword whose previous
//                      iteration left an unsatisfied check
//   barrier
//   decision           a codeword with >= 1 iteration done and no unsatisfied check has
//                      converged: its APP (from that iteration) is final
//   output             converged codewords write bits / APP / iteration count; one thread per
//                      slot takes the next codeword index from the global work counter
//   variable-node phase the others: APP = L + sum of the new R (block-row order,
//                      deterministic); a codeword reaching max_iter is final and written out
//   barrier
//   refill             (only after an output) APP = L, R = 0 of the new codeword; barrier
// Codewords therefore leave as soon as they converge and slots are refilled at once: early
// exit saves whole rounds of work instead of idling lanes of a tile.
//
// One launch serves several requests (mixed codes): requests of the same code form a
// group with its own work counter; each CTA starts on a group chosen in proportion to the
// groups' work, and when its group runs dry and its slots have drained it reloads the code
// tables and layout of the group with the most codewords left.  A single batch is the
// one-group case.
//
// What bounds it, and what the shape measured (GB300, 8192 codewords of the N = 1944 rate-1/2
// code, 1.75 dB FP32 / 2.25 dB FP16, per launch): instruction issue and its latencies, not the
// special-function units (0.35 of their ceiling) nor shared memory.
//   one codeword per thread, lock-step over the CTA          1225 us FP32
//   two per thread and barrier groups of three slots                        790 us FP16
//   two per thread, two row groups, one slot per barrier       964            679
//   + degree-ordered loops, uniform control, signs in a word   906            645
//   + output ahead of the variable-node phase                  887            629
// FP32: 18 warps of 3 thread slots (57 warp instructions per edge of two codewords, was 2 x 40);
// FP16: 24 warps of 4 (six slots of one row group each, 18 warps, took 718).
#include <math.h>
#include <string.h>

#include "flood_slots.h"

namespace ldpc {

// Per-slot strides of APP and messages (elements): at least the length, and congruent to Z
// modulo the 32 shared-memory banks, so that a warp whose rows run from the end of one slot
// into the start of the next sees the two slots' rows as one contiguous bank sequence.
static int slot_stride(int n, int Z) { return n + ((Z % 32) - (n % 32) + 32) % 32; }

// ------------------------------------------------------------------ host side

static int g_sm_count[64];

static int sm_count()
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 1;
    if (!g_sm_count[dev]) {
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        g_sm_count[dev] = n > 0 ? n : 1;
    }
    return g_sm_count[dev];
}

static size_t max_smem_optin()  // (asked for once per device)
{
    static int cached[64];
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && (v = __atomic_load_n(&cached[dev], __ATOMIC_RELAXED)) > 0) return (size_t)v;
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (dev >= 0 && dev < 64 && v > 0) __atomic_store_n(&cached[dev], v, __ATOMIC_RELAXED);
    return v > 0 ? (size_t)v : 227 * 1024;
}

// Bytes of one thread slot (V codewords) and where its parts lie.  FP32 messages follow their
// own slot's posteriors (one base and one wrap select per edge serve both); FP16 messages
// lie after all slots' posteriors.
struct SlotLayout {
    int strA, strR, offR;
    size_t bytes;  // of G thread slots
};
static SlotLayout slot_layout(const CodeDev &h, int msg, int V, int G)
{
    SlotLayout l;
    const int sa = 4 * V * slot_stride(h.N, h.Z);
    if (msg == LDPC_MSG_F16) {
        l.strA = sa;
        l.strR = 2 * V * slot_stride(h.E, h.Z);
        l.offR = (G * l.strA + 15) & ~15;
        l.bytes = (size_t)l.offR + (size_t)G * l.strR;
    } else {
        l.strA = l.strR = 4 * V * slot_stride(h.N + h.E, h.Z);
        l.offR = 4 * V * h.N;
        l.bytes = (size_t)G * l.strA;
    }
    return l;
}

// Shared memory ahead of a code's slots: the group hand-over, the code's tables and its slots'
// bookkeeping.  Each code of a launch is laid out by its own sizes (a CTA that takes up another code lays
// all of it out anew), so that a code which fits alone fits beside any other.
static int book_offset(int n_tab) { return FLOOD_TAB0 + n_tab * (int)sizeof(int4); }
static int slots_offset(int n_tab, int slots)
{
    return (book_offset(n_tab) + slots * (int)sizeof(FloodBook) + 15) & ~15;
}

// Thread slots of a code per CTA, the row groups each is spread over, and the barrier groups they
// form: K thread slots of TPG threads together.
struct SlotShape {
    int G, W, TPG, K;
};

// The most thread slots, up to cap, that shared memory and the bookkeeping allow.
static int slots_fit(const CodeDev &h, int msg, int V, size_t limit, int cap)
{
    if (h.dc_max > 32 || h.N >= 65536) return 0;
    int G = cap * V > SLOTS_MAX ? SLOTS_MAX / V : cap;
    while (G > 0 && slots_offset(h.n_ftab, G * V) + slot_layout(h, msg, V, G).bytes > limit) G--;
    return G;
}

// The shape of whole-warp rows (k_flood_slots) for V codewords per thread with at most `cap` thread
// slots: the most warps that the instance's threads (dmax: the launch's largest row degree), the named
// barriers and shared memory allow, with no more than two row groups unless that leaves fewer than
// 16 warps: each further row group adds its share of the round's fixed work (N = 1944 rate-1/2 FP32:
// 3 slots x 2 row groups 906 us, 2 x 4 928 us).
static SlotShape slot_shape(const CodeDev &h, int msg, int V, int dmax, size_t limit, int cap)
{
    SlotShape best = {0, 1, 32, 1};
    const int wt = ((h.Z + 31) / 32) * 32, tmax = flood_threads_max(dmax, V, msg == LDPC_MSG_F16);
    const int gmax = slots_fit(h, msg, V, limit, tmax / wt < cap ? tmax / wt : cap);
    for (int W = 1; W <= h.mb && W * wt <= tmax; W++) {
        int G = tmax / (W * wt);
        if (G > gmax) G = gmax;
        if (W * wt > 32 && G > FLOOD_BARRIERS) G = FLOOD_BARRIERS;
        if (G * W > best.G * best.W && (W <= 2 || best.G * best.TPG < 512)) best = {G, W, W * wt, 1};
    }
    return best;
}

// What n codewords cost an SM in a shape of V codewords per thread, as warps times check rows:
//   a round takes ceil(mb / W) block rows of every warp, and as long as 14 more edges for the rest of it;
//   fewer than 20 warps take as long as 20 (`least`; 8 where far fewer warps of spread rows above degree 12
//     stand against whole ones, as such a row has many independent edges);
//   a few times the resident codewords take whole turns of them;
//   a row of two codewords takes 1.35 times as long as a row of one (FP16, rows above degree 12, which
//     spill: 1.55, packed 1.9);
//   K thread slots in step: 3 % and 2 % each, as some of many codewords end in every round and hold up
//     the others;
//   spread row groups: a vote per row, and a warp covers 1 + (32 - gcd) / (K Z) of them on average,
//     whose rows need different bodies with the share `change` of the degree-ordered list's neighbours.
// Measured (us, whole warps / packed / spread, 10 iterations): at widths without idle lanes, N = 768 rate 1/2,
// FP32 675 / 711 / 881, rate 5/6 1000 / 1048 / 1190; 600 codewords of a 12 x 24 code of Z = 3 42 / 27 / 27;
// 39 of a 46 x 92 code of Z = 9 112 / - / 54; 16588 of a rate-5/6 code of Z = 20, FP16 733 / 600 / 712.
static double shape_cost(const CodeDev &h, int msg, const SlotShape &s, int V, int64_t n, FloodForm form, double change,
                         double least = 20.0)
{
    const double warps = s.G / s.K * (s.TPG / 32.0), degree = (double)h.nnz / h.mb;
    double turns = (double)((n + V - 1) / V) / s.G;
    turns = turns < 8.0 ? ceil(turns) : turns + 0.5;
    double rows = (h.mb + s.W - 1) / s.W;
    if (form == FLOOD_SPREAD) {
        const int block = s.K * h.Z, two = block & -block;  // (its largest power of two)
        double span = 1.0 + (32 - (two < 32 ? two : 32)) / (double)block;
        if (span > s.W) span = s.W;
        rows *= 1.0 + 0.25 * (span - 1.0) * change;
    }
    double c = (rows + 14.0 / degree) * turns * (warps > least ? warps : least);
    if (V == 2) c *= h.dc_max <= 12 || msg != LDPC_MSG_F16 ? 1.35 : form == FLOOD_WHOLE ? 1.55 : 1.9;
    if (form != FLOOD_WHOLE) c *= (form == FLOOD_SPREAD ? 1.0 + 2.1 / degree : 1.03) + 0.02 * (s.K - 1);
    return c;
}

// The share of neighbouring rows of the degree-ordered list that have different bodies.
static double body_changes(const CodeDev &h)
{
    int n = 0;
    for (int c = 0, end = 0; c < FLOOD_CLASSES; end = h.rend[c++]) n += h.rend[c] > end;
    return h.mb > 1 ? (n - 1.0) / (h.mb - 1.0) : 0.0;
}

// The cheapest shape with the rows of K thread slots end to end (k_flood_packed), or with those of the
// row groups too (spread).
static SlotShape packed_shape(const CodeDev &h, int msg, int V, int dmax, size_t limit, int cap, int64_t n, FloodForm form)
{
    SlotShape best = {0, 1, 32, 1};
    double cost = 0.0;
    const int tmax = flood_threads_max(dmax, V, msg == LDPC_MSG_F16);
    const int gmax = slots_fit(h, msg, V, limit, cap);
    const bool spread = form == FLOOD_SPREAD;
    const double change = spread ? body_changes(h) : 0.0;
    // (of narrow rows, which have many shapes, 1, 2, 3, 4, 6, 8, 12, 16, ...)
    auto next = [&](int x) { return h.Z >= 16 || x < 4 ? x + 1 : x % 3 ? x / 2 * 3 : x / 3 * 4; };
    for (int K = spread ? 1 : 2; K <= gmax && K * V <= 32 && K * h.Z <= tmax; K = next(K)) {
        for (int W = 1; W <= h.mb; W = W == h.mb ? W + 1 : next(W) < h.mb ? next(W) : h.mb) {
            const int tpg = spread ? (K * W * h.Z + 31) & ~31 : W * ((K * h.Z + 31) & ~31);
            if (tpg > tmax) break;
            int groups = tmax / tpg < gmax / K ? tmax / tpg : gmax / K;
            if (tpg > 32 && groups > FLOOD_BARRIERS) groups = FLOOD_BARRIERS;
            const SlotShape s = {groups * K, W, tpg, K};
            const double c = shape_cost(h, msg, s, V, n, form, change);
            if (best.G == 0 || c < cost * 0.999) {
                best = s;
                cost = c;
            }
        }
    }
    return best;
}

// Whether the slot decoder serves a code (V = 1), or pairs its slots (V = 2): one thread slot
// with its posteriors, messages and the code's tables in shared memory.
static bool fits_slot(const CodeDev &h, int msg, int V, size_t limit)
{
    if (h.dc_max > 32 || h.N >= 65536 || h.Z > (V == 2 ? 512 : 640)) return false;
    const size_t head = ((size_t)SLOTS_MAX * 16 + 16 + (size_t)4 * (5 * h.nnz + 2 * h.mb + h.nb + 11) + 15) & ~(size_t)15;
    const size_t sa = ((size_t)V * slot_stride(h.N, h.Z) * 4 + 15) & ~(size_t)15;
    return head + sa + (size_t)V * slot_stride(h.E, h.Z) * (msg == LDPC_MSG_F16 ? 2 : 4) <= limit &&
           slot_shape(h, msg, V, h.dc_max, limit, 1).G > 0;
}

int slots_supported(const CodeDev &h, int msg) { return fits_slot(h, msg, 1, 227 * 1024); }

int slots_pairable(const CodeDev &h, int msg) { return fits_slot(h, msg, 2, max_smem_optin()); }

static int table_words(const CodeDev &h) { return (h.mb + h.nb + 3) / 4; }

int flood_table_size(const CodeDev &h)
{
    int n = h.nnz + h.nb + table_words(h);
    for (int j = 0; j < h.nb; j++) {
        const int dv = h.colptr[j + 1] - h.colptr[j];
        if (dv > 4) n += dv / 4;  // the entries past the third, four to an element
    }
    return n;
}

void flood_build_table(CodeDev &h, int msg, int V, int4 *tab)
{
    const int SA = 4 * V, SR = (msg == LDPC_MSG_F16 ? 2 : 4) * V;
    const int base_r = msg == LDPC_MSG_F16 ? 0 : slot_layout(h, msg, V, 1).offR;
    int32_t *rows = reinterpret_cast<int32_t *>(tab + h.n_ftab - table_words(h)), *cols = rows + h.mb;
    int ne = 0, nr = 0;
    for (int c = 0; c < FLOOD_CLASSES; c++) {
        const int lo = c ? flood_class_degree(c - 1) : 0, hi = flood_class_degree(c);
        for (int d = lo + 1; d <= hi; d++)
            for (int l = 0; l < h.mb; l++) {
                const int b0 = h.rowptr[l], dc = h.rowptr[l + 1] - b0;
                if (dc != d) continue;
                rows[nr++] = (ne << 8) | dc;
                for (int k = 0; k < dc; k++) {
                    const int b = b0 + k, j = h.ent[b] >> 16, sh = h.ent[b] & 0xffff;
                    tab[ne++] = make_int4(SA * (j * h.Z + sh), base_r + SR * (b * h.Z + sh), h.Z - sh, 0);
                }
            }
        h.rend[c] = (uint8_t)nr;
    }
    int4 *col = tab + h.nnz;
    int nc = 0, nx = h.nnz + h.nb;
    for (int c = 1; c <= 5; c++) {
        for (int d = c; d <= (c < 5 ? c : h.mb); d++)
            for (int j = 0; j < h.nb; j++) {
                const int i0 = h.colptr[j], dv = h.colptr[j + 1] - i0;
                if (dv != d) continue;
                auto off = [&](int i) { return i < dv ? SR * (h.colent[i0 + i] >> 16) * h.Z : 0; };
                const int take = dv > 4 ? 3 : 4;
                col[nc] = make_int4(off(0), off(1), off(2), dv > 4 ? (nx << 8) | (dv - 3) : off(3));
                cols[nc++] = j * h.Z;
                for (int i = take; i < dv; i += 4) tab[nx++] = make_int4(off(i), off(i + 1), off(i + 2), off(i + 3));
            }
        h.cend[c - 1] = (uint8_t)nc;
    }
}

// Group the requests by code object and size every group's slots for one persistent grid over all of
// them.
cudaError_t flood_plan(const HostReq *reqs, int n, const ldpc_decode_params &p, void *counters, size_t limit, int nsm,
                       FloodPlan &out)
{
    FloodArgs &a = out.a;  // ~7 KB, passed by value as the kernel parameter
    const ldpc_code *codes[MULTI_MAX_GROUPS];
    int ng = 0;
    for (int i = 0; i < n; i++) {
        if (reqs[i].n_cw <= 0) continue;
        int g = 0;
        while (g < ng && codes[g] != reqs[i].code) g++;
        if (g == ng) {
            if (ng == MULTI_MAX_GROUPS) return cudaErrorInvalidValue;
            codes[ng++] = reqs[i].code;
        }
    }
    out.ctas = 0;
    if (ng == 0) return cudaSuccess;
    int dmax = 0;
    int64_t items_of[MULTI_MAX_GROUPS] = {};
    for (int g = 0; g < ng; g++) {
        dmax = codes[g]->host.dc_max > dmax ? codes[g]->host.dc_max : dmax;
        for (int i = 0; i < n; i++)
            if (reqs[i].n_cw > 0 && reqs[i].code == codes[g]) items_of[g] += reqs[i].n_cw;
    }
    const int tuned = codes[0]->tuned_flood[p.msg == LDPC_MSG_F16 ? 1 : 0];
    // shapes with V codewords per thread; a small batch spreads over the SMs rather than
    // filling a few CTAs' slots
    SlotShape shape[MULTI_MAX_GROUPS];
    int64_t per_sm[MULTI_MAX_GROUPS];
    for (int g = 0; g < ng; g++) per_sm[g] = (items_of[g] + nsm - 1) / nsm;
    // (in s; returns the launch's estimated cost, 0: some code has no slot)
    auto shapes = [&](int V, FloodForm form, SlotShape *s) {
        double cost = 0.0;
        for (int g = 0; g < ng; g++) {
            const CodeDev &h = codes[g]->host;
            const int64_t want = (per_sm[g] + V - 1) / V;
            const int cap = want < SLOTS_MAX ? (int)want : SLOTS_MAX;
            s[g] = form == FLOOD_WHOLE ? slot_shape(h, p.msg, V, dmax, limit, cap)
                                       : packed_shape(h, p.msg, V, dmax, limit, cap, per_sm[g], form);
            if (s[g].G < 1) return 0.0;
            cost += h.nnz / (double)h.mb *
                    shape_cost(h, p.msg, s[g], V, per_sm[g], form, body_changes(h));
        }
        return cost;
    };
    SlotShape pair[MULTI_MAX_GROUPS];
    const double one = tuned == SCHED_SLOTS_V2 ? 0.0 : shapes(1, FLOOD_WHOLE, shape);
    int V = tuned == SCHED_SLOTS_V1 ? 1 : 2;
    double whole = one;
    if (!tuned && one > 0.0) {
        // one codeword per thread where every code's codewords are all resident at once with two
        // row groups or more each, or one to an SM; with rows above degree 16 (few block rows, long
        // serial rows) also with one, up to 12 warps.  Per launch on GB300, one against two codewords per thread, 3 / 4
        // / 6 codewords per SM: N = 1944 rate 1/2 FP32 82 / 100, 116 / 100, 140 / 127 us; rate 5/6
        // 126 / 178, 156 / 181, 226 / 211; N = 648 rate 1/2 46 / 66, 55 / 68, 66 / 75 (and 12: 113 / 110).
        bool single = true;
        for (int g = 0; g < ng && single; g++)
            single = per_sm[g] <= shape[g].G && (shape[g].W >= 2 || per_sm[g] == 1 ||
                                                 (codes[g]->host.dc_max > 16 && per_sm[g] * shape[g].TPG <= 400));
        if (single) V = 1;
    }
    if (V == 2) {
        whole = shapes(2, FLOOD_WHOLE, pair);
        if (whole == 0.0 || (p.msg != LDPC_MSG_F16 && one > 0.0 && one * 1.2 < whole)) {  // (too few pairs fit)
            V = 1;
            whole = tuned == SCHED_SLOTS_V2 ? shapes(1, FLOOD_WHOLE, shape) : one;
        } else {
            memcpy(shape, pair, sizeof shape);
        }
    }
    if (whole == 0.0) return cudaErrorInvalidValue;
    // rows end to end where that is estimated 5 % cheaper: packed if a quarter of some code's lanes would be
    // idle, spread if a twentieth would be and a thread of one codeword has several rows
    out.form = FLOOD_WHOLE;
    bool quarter = false, some = false, several = false;
    int64_t most = 0;  // (one codeword to an SM has nothing to be packed with)
    for (int g = 0; g < ng; g++) {
        const int Z = codes[g]->host.Z, wt = (Z + 31) & ~31;
        quarter |= 4 * Z <= 3 * wt;
        some |= 20 * Z <= 19 * wt;
        several |= shape[g].W < codes[g]->host.mb;
        most = per_sm[g] > most ? per_sm[g] : most;
    }
    if (!quarter && (ng > 1 || V == 2 || !several)) some = false;  // (not worth the host's time for many codes)
    const struct { FloodForm form; int V; } other[3] = {{FLOOD_PACKED, 1}, {FLOOD_PACKED, 2}, {FLOOD_SPREAD, 1}};
    for (int i = 0; i < 3 && some; i++) {
        SlotShape s[MULTI_MAX_GROUPS];
        if ((tuned && other[i].V != V) || (other[i].form == FLOOD_PACKED && (!quarter || most < 2 * other[i].V))) continue;
        const double cost = shapes(other[i].V, other[i].form, s);
        bool take = cost > 0.0 && cost * (out.form ? 1.0 : 1.05) < whole;
        if (cost > 0.0 && !take && !out.form && V == 1 && other[i].form == FLOOD_SPREAD) {
            double a = 0.0, b = 0.0;
            take = true;
            for (int g = 0; g < ng; g++) {
                const CodeDev &h = codes[g]->host;
                take &= h.dc_max > 12;
                a += h.nnz / (double)h.mb * shape_cost(h, p.msg, shape[g], 1, per_sm[g], FLOOD_WHOLE, 0.0, 8.0);
                b += h.nnz / (double)h.mb * shape_cost(h, p.msg, s[g], 1, per_sm[g], FLOOD_SPREAD, body_changes(h), 8.0);
            }
            take &= b * 1.3 < a;
        }
        if (take) {
            out.form = other[i].form;
            whole = cost;
            V = other[i].V;
            memcpy(shape, s, sizeof shape);
        }
    }
    size_t smem = 0;
    int threads = 32, nr = 0;
    double wsum = 0.0, acc = 0.0;
    int64_t min_ctas = 0;
    for (int g = 0; g < ng; g++) wsum += (double)items_of[g] * codes[g]->host.E;
    for (int g = 0; g < ng; g++) {
        const CodeDev &h = codes[g]->host;
        FloodGroup &gd = a.groups[g];
        gd.N = h.N;
        gd.Z = h.Z;
        gd.nb = h.nb;
        gd.nnz = h.nnz;
        gd.status = h.status;
        gd.req_begin = nr;
        int64_t items = 0;
        for (int i = 0; i < n; i++) {
            if (reqs[i].n_cw <= 0 || reqs[i].code != codes[g]) continue;
            FloodReq &q = a.reqs[nr++];
            q.llr = static_cast<const float *>(reqs[i].llr);
            q.bits = reqs[i].bits;
            q.iters = reqs[i].iters;
            q.app = reqs[i].app;
            q.item0 = items;
            items += reqs[i].n_cw;
        }
        gd.req_end = nr;
        gd.n_items = items;
        gd.G = shape[g].G;
        gd.W = shape[g].W;
        gd.TPG = shape[g].TPG;
        gd.K = shape[g].K;
        const SlotLayout l = slot_layout(h, p.msg, V, gd.G);
        gd.strA = l.strA;
        gd.strR = l.strR;
        gd.offR = l.offR;
        gd.book0 = book_offset(h.n_ftab);
        gd.slots0 = slots_offset(h.n_ftab, gd.G * V);
        smem = gd.slots0 + l.bytes > smem ? gd.slots0 + l.bytes : smem;
        gd.tab = codes[g]->ftab + (size_t)h.n_ftab * ((p.msg == LDPC_MSG_F16 ? 2 : 0) + V - 1);
        gd.n_tab = h.n_ftab;
        gd.t_col = h.nnz;
        gd.t_row = h.n_ftab - table_words(h);
        gd.mb = h.mb;
        memcpy(gd.rend, h.rend, sizeof gd.rend);
        memcpy(gd.cend, h.cend, sizeof gd.cend);
        threads = gd.G / gd.K * gd.TPG > threads ? gd.G / gd.K * gd.TPG : threads;
        min_ctas += (items + gd.G * V - 1) / (gd.G * V);
        acc += (double)items * h.E;
        gd.cumw = g == ng - 1 ? 1.0f : (float)(acc / wsum);
    }
    a.n_groups = ng;
    a.tab0 = FLOOD_TAB0;
    a.next = static_cast<unsigned long long *>(counters);
    a.max_iter = p.max_iter;
    a.early_exit = p.early_exit;
    a.X = p.phi_clamp;
    int ctas = nsm;
    if (min_ctas < ctas) ctas = (int)min_ctas;
    if (ng == 1 && items_of[0] <= (int64_t)ctas * a.groups[0].G * V) a.next = nullptr;  // no refills: no counter
    else if (!counters) return cudaErrorInvalidValue;
    out.dmax = dmax;
    out.V = V;
    out.threads = threads;
    out.ctas = ctas;
    out.smem = smem;
    return cudaSuccess;
}

template <typename MsgT, bool HC>
static cudaError_t launch(const FloodPlan &q, cudaStream_t s)
{
    return q.form == FLOOD_WHOLE ? flood_slots_launch<MsgT, HC>(q, s) : flood_packed_launch<MsgT, HC>(q, s);
}

cudaError_t flood_multi_decode(const HostReq *reqs, int n, const ldpc_decode_params &p, void *counters, cudaStream_t s)
{
    FloodPlan q;
    cudaError_t e = flood_plan(reqs, n, p, counters, max_smem_optin(), sm_count(), q);
    if (e != cudaSuccess || q.ctas == 0) return e;
    if (q.a.next) {
        e = cudaMemsetAsync(counters, 0, sizeof(unsigned long long) * q.a.n_groups, s);
        if (e != cudaSuccess) return e;
    }
    const bool hc = p.phi_clamp < FLOOD_CLAMP_X;
    if (p.msg == LDPC_MSG_F16) return hc ? launch<__half, true>(q, s) : launch<__half, false>(q, s);
    return hc ? launch<float, true>(q, s) : launch<float, false>(q, s);
}

}  // namespace ldpc
