// Flooding sum-product decoding of codes too large for one SM: the cluster slot decoder.
//
// A thread-block cluster of CL CTAs (CL SMs) holds one codeword for the whole decode, split
// between its CTAs: CTA q owns a contiguous range of block rows (their checks and the
// messages R of their edges) and a contiguous range of block columns (their posteriors
// APP).  The two ranges are balanced by block count.  A check of CTA q reads the posteriors
// of its variables wherever they live (distributed shared memory of the cluster); a variable
// of CTA q reads the messages of its edges wherever they live.  One round (Sec. II two-phase
// message passing, Algorithm 1 loop order), each phase closed by a cluster barrier:
//   check-node phase   every owned check: Q = APP - R, R' from the check rule in the product
//                      (tanh) domain of the slot decoders, written in place; the parity of the APP sign
//                      bits over the check flags an unsatisfied check of the previous
//                      iteration's decisions
//   decision           no CTA of the cluster flagged a check and >= 1 iteration done: the
//                      codeword has converged (its APP from that iteration is final)
//   variable-node phase otherwise every owned variable: APP = L + sum of the new R
// A finished codeword is written out and the cluster's leader takes the next codeword from
// the global work counter.  Messages are stored negated at the variable's position inside the
// block, edge (b, r) of the owned block b at (b - first owned block) * Z + (r + s) mod Z;
// posteriors at (place of column j) * Z + c.
//
// Check-node threads: W row groups of whole warps; thread r of a row group owns rows r and
// r + ceil(Z / 2) of the block rows that fall to its group in ascending degree, so that a warp runs
// one straight-line body at a time (flood_check.cuh) with two rows' arithmetic packed and one read
// of each edge descriptor.  One CTA has several times more rows than threads, so that pairing them
// costs no parallelism.  Rows above degree 12 have their groups of edges unrolled, whose remote loads
// then overlap (600 codewords of a 42 x 84 code, Z = 136, FP16: rows of 13 to 15 edges 1628 -> 1017 us, of
// 19 to 21 2054 -> 1364).  Variable-node threads: W4 groups; a thread owns four consecutive positions
// of its group's columns, one access per block (where Z is a multiple of 4; else its two rows'
// positions).  Rows and columns are dealt to the groups by weight on the host, because a phase ends
// at a cluster barrier.  Where groups of whole warps would leave too many lanes idle, rows and columns lie
// end to end over the threads instead (cl_rows_spread).  The table entries hold complete shared::cluster addresses (own CTA or the other),
// so an operand in either CTA costs one add.
// Measured on 2048 codewords of the N = 26112 code, FP16, 2.0 dB, per launch, and warp
// instructions per edge update (both phases): one row and one position per thread 5378 us, 57; two
// rows 5087 us, 49; and four positions 4706 us, 43; dealt by weight (not back and forth) 4609 us.
// Bound by instruction issue (58 %) and the waits at the two cluster barriers of a round (15 % of a
// warp's time).
#include <math.h>
#include <string.h>

#include <new>

#include "flood_check.cuh"

namespace ldpc {

constexpr int CLUSTER_CTAS = 2;
constexpr int CL_CLASSES = 11;  // row degree classes: 2..8 exact, then up to 12, 16, 24, 32
__host__ __device__ constexpr int cl_class_degree(int c)
{
    return c < 7 ? c + 2 : c == 7 ? 12 : c == 8 ? 16 : c == 9 ? 24 : 32;
}

constexpr int CL_GROUPS = 24;  // groups of whole warps a CTA can have

// One launch decodes every codeword of up to MULTI_MAX_REQS requests of one code: the codewords
// are the items of one work sequence (request i's are items item0 .. item0 + n_cw - 1).
struct ClusterArgs {
    int n_req;
    // from here (neither loaded nor divided in the kernel) these are known to be warp-uniform: the
    // code's sizes, and W row groups of WT threads
    int Z, H, N, W, WT;
    // the variable-node phase in quads: W4 groups of WT4 threads (W4 = 0: Z is no multiple of 4)
    int W4, WT4, wide_L;
    int spread;  // rows and columns end to end over the threads instead
    int64_t n_items;
    unsigned long long *next;
    int row_split[CLUSTER_CTAS + 1];  // block rows [row_split[q], row_split[q+1]) belong to CTA q
    int ncols[CLUSTER_CTAS];          // block columns CTA q holds the posteriors of
    int col_owner[NB_MAX];            // owner of block column j
    int col_slot[NB_MAX];             // its place among the owner's columns
    // CTA q's rows and columns group by group (a group's share in ascending degree), where each
    // group's share starts and the ends of its degree classes, the rows' first edge
    // descriptors, and the elements of the CTA's table
    uint8_t row_list[CLUSTER_CTAS][MB_MAX], col_list[CLUSTER_CTAS][NB_MAX];
    uint8_t rstart[CLUSTER_CTAS][CL_GROUPS], cstart[CLUSTER_CTAS][CL_GROUPS];
    uint8_t rend[CLUSTER_CTAS][CL_GROUPS][CL_CLASSES], cend[CLUSTER_CTAS][CL_GROUPS][5];
    uint16_t row_e0[CLUSTER_CTAS][MB_MAX], col_x0[CLUSTER_CTAS][NB_MAX];
    int n_edge[CLUSTER_CTAS], n_tab[CLUSTER_CTAS];
    int off_app, off_r;  // posteriors and messages, bytes from the start of shared memory
    int max_iter, early_exit;
    float X;
    ReqDev reqs[MULTI_MAX_REQS];
};

// 32-bit shared::cluster addresses: the address of shared variable p in CTA `rank` of the
// cluster, and loads through such an address (the CTA's own memory or the other's).
__device__ __forceinline__ uint32_t cl_map(const void *p, unsigned rank)
{
    uint32_t out;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(out)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return out;
}
__device__ __forceinline__ float cl_ld(const float *, uint32_t addr)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ float cl_ld(const __half *, uint32_t addr)
{
    unsigned short v;
    asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return __half2float(__ushort_as_half(v));
}
// four consecutive messages (aligned)
__device__ __forceinline__ void cl_ld4(const float *, uint32_t addr, float2 (&m)[2])
{
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(m[0].x), "=f"(m[0].y), "=f"(m[1].x), "=f"(m[1].y)
                 : "r"(addr));
}
__device__ __forceinline__ void cl_ld4(const __half *, uint32_t addr, float2 (&m)[2])
{
    uint32_t u, v;
    asm volatile("ld.shared::cluster.v2.b32 {%0, %1}, [%2];" : "=r"(u), "=r"(v) : "r"(addr));
    m[0] = __half22float2(*reinterpret_cast<const __half2 *>(&u));
    m[1] = __half22float2(*reinterpret_cast<const __half2 *>(&v));
}
__device__ __forceinline__ void cl_st(uint32_t addr, int x)
{
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(x) : "memory");
}

// The cluster barrier, in its aligned form (all threads of a warp together): the compiler then
// knows that warps leave it converged, which uniform branches after it need.
__device__ __forceinline__ void cl_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__host__ __device__ inline int cl_owner(const int *split, int x)
{
    int q = 0;
    while (q < CLUSTER_CTAS - 1 && x >= split[q + 1]) q++;
    return q;
}

// A thread's place: two rows r and s = r + H of its block row (H = ceil(Z / 2)), plain and less
// one block.  An idle lane of a group's last warp repeats the last rows, and row Z (odd Z) is row
// Z - 1 once more; neither stores anything.
struct PairPlace {
    struct Ref {  // the two rows' operands
        uint32_t x, y;
    };
    int r, rw, s, sw;
    bool own, own2;
};
template <typename MsgT>
__device__ __forceinline__ void edge_at(const int4 &e, const PairPlace &p, PairPlace::Ref &ao, PairPlace::Ref &ro)
{
    const int t = p.r >= e.z ? p.rw : p.r, u = p.s >= e.z ? p.sw : p.s;
    ao = {(uint32_t)(e.x + 4 * t), (uint32_t)(e.x + 4 * u)};
    ro = {(uint32_t)(e.y + (int)sizeof(MsgT) * t), (uint32_t)(e.y + (int)sizeof(MsgT) * u)};
}

// Two checks' operands: the posteriors at shared::cluster addresses, the messages in the own CTA.
template <typename MsgT>
struct ClusterMem {
    using Ref = PairPlace::Ref;
    char *sm;
    __device__ __forceinline__ float2 app(Ref o) const
    {
        return make_float2(cl_ld((const float *)nullptr, o.x), cl_ld((const float *)nullptr, o.y));
    }
    __device__ __forceinline__ float2 msg(Ref o) const
    {
        return make_float2(Sm<MsgT, 1>::ld(sm + o.x), Sm<MsgT, 1>::ld(sm + o.y));
    }
    __device__ __forceinline__ void put(const PairPlace &p, Ref o, float2 x) const
    {
        if constexpr (sizeof(MsgT) == 2) {
            const __half2 h = __floats2half2_rn(x.x, x.y);
            if (p.own) *reinterpret_cast<__half *>(sm + o.x) = __low2half(h);
            if (p.own2) *reinterpret_cast<__half *>(sm + o.y) = __high2half(h);
        } else {
            put_word(p, o, x);
        }
    }
    __device__ __forceinline__ float2 word(Ref o) const
    {
        return make_float2(Sm<float, 1>::ld(sm + o.x), Sm<float, 1>::ld(sm + o.y));
    }
    __device__ __forceinline__ void put_word(const PairPlace &p, Ref o, float2 x) const
    {
        if (p.own) Sm<float, 1>::st(sm + o.x, x.x);
        if (p.own2) Sm<float, 1>::st(sm + o.y, x.y);
    }
};

// The thread's two rows of its group's block rows from list position i, in ascending degree (see
// rows_of of the slot decoder).
template <int CLS, int DMAX, typename MsgT, bool HC>
__device__ __forceinline__ void cl_rows(const uint8_t *rend, const int4 *__restrict__ tab,
                                        const int32_t *__restrict__ rows, const ClusterMem<MsgT> mem,
                                        const PairPlace &p, float Xb, float Pb, uint32_t (&pbad)[2], int i)
{
    constexpr int D = cl_class_degree(CLS);
    if constexpr (D <= DMAX) {
        const int end = rend[CLS];
        for (; i < end; i++) {
            const int hd = rows[i];
            if constexpr (D <= 8)
                check_narrow<D, 2, MsgT, false, HC>(tab + (hd >> 8), mem, p, Xb, Pb, pbad);
            else if constexpr (D == 12)
                check_12<2, MsgT, false, HC>(hd & 255, tab + (hd >> 8), mem, p, Xb, Pb, pbad);
            else
                check_wide<D / 8, 2, MsgT, false, HC>(hd & 255, tab + (hd >> 8), mem, p, Xb, Pb, pbad);
        }
        if constexpr (CLS + 1 < CL_CLASSES)
            cl_rows<CLS + 1, DMAX, MsgT, HC>(rend, tab, rows, mem, p, Xb, Pb, pbad, i);
    }
}

// The positions of a column that a thread of the variable-node phase owns, and their values in
// packed pairs.  rb: byte offsets in a block of messages; L: channel values of block column 0;
// A: posteriors of place 0.
//   VarPair  positions r and s = r + H, the thread's rows of the check-node phase
//   VarQuad  four consecutive positions, whose messages and posteriors are one access each
//            (Z a multiple of 4)
template <typename MsgT>
struct VarPair {
    static constexpr int NV = 1;
    const float *L, *L2;
    uint32_t rb, rb2;
    float *A, *A2;
    bool own, own2;
    __device__ __forceinline__ void channel(int o, float2 (&x)[1]) const { x[0] = make_float2(__ldg(L + o), __ldg(L2 + o)); }
    __device__ __forceinline__ void add(float2 (&s)[1], int addr) const
    {
        const float2 m = make_float2(cl_ld((const MsgT *)nullptr, rb + (uint32_t)addr),
                                     cl_ld((const MsgT *)nullptr, rb2 + (uint32_t)addr));
        s[0] = __ffma2_rn(m, make_float2(-1.0f, -1.0f), s[0]);
    }
    __device__ __forceinline__ void put(int a, const float2 (&s)[1]) const
    {
        if (own) A[a] = s[0].x + 0.0f;  // -0 -> +0: the sign bit is the decision
        if (own2) A2[a] = s[0].y + 0.0f;
    }
};
template <typename MsgT>
struct VarQuad {
    static constexpr int NV = 2;
    const float *L;
    uint32_t rb;
    float *A;
    bool own, wide;  // wide: the channel values are 16-byte aligned
    __device__ __forceinline__ void channel(int o, float2 (&x)[2]) const
    {
        float4 v;
        if (wide)
            v = __ldg(reinterpret_cast<const float4 *>(L + o));
        else
            v = make_float4(__ldg(L + o), __ldg(L + o + 1), __ldg(L + o + 2), __ldg(L + o + 3));
        x[0] = make_float2(v.x, v.y);
        x[1] = make_float2(v.z, v.w);
    }
    __device__ __forceinline__ void add(float2 (&s)[2], int addr) const
    {
        float2 m[2];
        cl_ld4((const MsgT *)nullptr, rb + (uint32_t)addr, m);
#pragma unroll
        for (int i = 0; i < 2; i++) s[i] = __ffma2_rn(m[i], make_float2(-1.0f, -1.0f), s[i]);
    }
    __device__ __forceinline__ void put(int a, const float2 (&s)[2]) const
    {
        const float2 z = make_float2(0.0f, 0.0f), u = __fadd2_rn(s[0], z), v = __fadd2_rn(s[1], z);
        if (own) *reinterpret_cast<float4 *>(A + a) = make_float4(u.x, u.y, v.x, v.y);
    }
};

// A thread's positions of its group's columns from list position i, in ascending degree:
// APP = L + the column's messages in block-row order.
constexpr int kClChunk = 2;  // columns whose channel values a thread requests at once
template <int DV, typename VAR>
__device__ __forceinline__ void cl_cols(const uint8_t *cend, const int4 *__restrict__ ctab,
                                        const int4 *__restrict__ tab, const int32_t *__restrict__ cols, const VAR p,
                                        int Z, int i)
{
    const int end = cend[DV - 1];
    for (; i < end;) {
        float2 s[kClChunk][VAR::NV];
        int jc[kClChunk];
#pragma unroll
        for (int c = 0; c < kClChunk; c++) {
#pragma unroll
            for (int v = 0; v < VAR::NV; v++) s[c][v] = make_float2(0.0f, 0.0f);
            jc[c] = 0;
            if (c == 0 || i + c < end) {
                jc[c] = cols[i + c];
                p.channel((jc[c] & 255) * Z, s[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < kClChunk; c++) {
            if (c == 0 || i < end) {
                const int4 o = ctab[i];
                p.add(s[c], o.x);
                if constexpr (DV > 1) p.add(s[c], o.y);
                if constexpr (DV > 2) p.add(s[c], o.z);
                if constexpr (DV == 4) p.add(s[c], o.w);
                if constexpr (DV == 5) {
                    const int4 *m = tab + (o.w >> 8);
                    for (int k = o.w & 255; k > 0; k -= 4, m++) {
                        p.add(s[c], m->x);
                        if (k > 1) p.add(s[c], m->y);
                        if (k > 2) p.add(s[c], m->z);
                        if (k > 3) p.add(s[c], m->w);
                    }
                }
                p.put((jc[c] >> 8) * Z, s[c]);
                i++;
            }
        }
    }
    if constexpr (DV < 5) cl_cols<DV + 1>(cend, ctab, tab, cols, p, Z, i);
}

// Rows and positions end to end over the CTA's threads (SPREAD), for widths that whole warps fit badly:
// thread x has rows r and r + H of list row i, where i H + r = x, x + threads, ...; a warp's lanes can
// be at two or more rows (flood_check.cuh, vote_body).
template <int DMAX, typename MsgT, bool HC>
__device__ __forceinline__ void cl_rows_spread(const int4 *__restrict__ tab, const int32_t *__restrict__ rows, int n_rows,
                                               const ClusterMem<MsgT> mem, int Z, int H, int tid, int nth, float Xb,
                                               float Pb, uint32_t (&pbad)[2])
{
    int i = tid / H, r = tid - i * H;
    const int di = nth / H, dr = nth - di * H;
    for (;;) {
        int hd = i < n_rows ? rows[i] : kNoRow;
        bool on;
        const int body = vote_body(hd, on), dc = hd & 255;
        if (body == kNoRow) break;
        const int4 *ed = tab + (hd >> 8);
        PairPlace p;
        p.own = on;
        p.own2 = on && r + H < Z;
        p.r = r;
        p.s = r + H < Z ? r + H : Z - 1;
        p.rw = p.r - Z;
        p.sw = p.s - Z;
        switch (body) {
        case 2: check_narrow<2, 2, MsgT, false, HC>(ed, mem, p, Xb, Pb, pbad); break;
        case 3: check_narrow<3, 2, MsgT, false, HC>(ed, mem, p, Xb, Pb, pbad); break;
        case 4: check_narrow<4, 2, MsgT, false, HC>(ed, mem, p, Xb, Pb, pbad); break;
        case 5: check_narrow<5, 2, MsgT, false, HC>(ed, mem, p, Xb, Pb, pbad); break;
        case 6: check_narrow<6, 2, MsgT, false, HC>(ed, mem, p, Xb, Pb, pbad); break;
        case 7: check_narrow<7, 2, MsgT, false, HC>(ed, mem, p, Xb, Pb, pbad); break;
        case 8: check_narrow<8, 2, MsgT, false, HC>(ed, mem, p, Xb, Pb, pbad); break;
        default:
            if constexpr (DMAX > 8) {
                if (body == 12)
                    check_12<2, MsgT, false, HC>(dc, ed, mem, p, Xb, Pb, pbad);
                else if constexpr (DMAX > 12) {
                    if (body == 16)
                        check_wide<2, 2, MsgT, false, HC>(dc, ed, mem, p, Xb, Pb, pbad);
                    else if (body == 24)
                        check_wide<3, 2, MsgT, false, HC>(dc, ed, mem, p, Xb, Pb, pbad);
                    else
                        check_wide<4, 2, MsgT, false, HC>(dc, ed, mem, p, Xb, Pb, pbad);
                }
            }
        }
        if (on) {
            i += di;
            r += dr;
            if (r >= H) {
                r -= H;
                i++;
            }
        }
    }
}

// The same of the columns, Q positions (pairs or quads) each; at(r): the thread's place at position r.
template <typename VAR, typename AT>
__device__ __forceinline__ void cl_cols_spread(const uint8_t *cend, const int4 *__restrict__ ctab,
                                               const int4 *__restrict__ tab, const int32_t *__restrict__ cols, int n_cols,
                                               int Z, int Q, int tid, int nth, AT at)
{
    int i = tid / Q, r = tid - i * Q;
    const int di = nth / Q, dr = nth - di * Q;
    for (; __any_sync(kFullWarp, i < n_cols);) {
        const bool ok = i < n_cols;
        const int ic = ok ? i : n_cols - 1, jw = cols[ic];
        const int dv = 1 + (ic >= cend[0]) + (ic >= cend[1]) + (ic >= cend[2]) + (ic >= cend[3]);  // 5: above 4
        const int top = (int)__reduce_max_sync(kFullWarp, ok ? (unsigned)dv : 0u);
        const int4 o = ctab[ic];
        const VAR p = at(r, ok);
        float2 s[VAR::NV];
        p.channel((jw & 255) * Z, s);
        auto add = [&](bool c, int addr) {  // (a lane without a message there reads its first once more)
            float2 m[VAR::NV];
#pragma unroll
            for (int v = 0; v < VAR::NV; v++) m[v] = s[v];
            p.add(m, c ? addr : o.x);
#pragma unroll
            for (int v = 0; v < VAR::NV; v++) s[v] = pick(c, m[v], s[v]);
        };
        p.add(s, o.x);
        if (top > 1) add(dv > 1, o.y);
        if (top > 2) add(dv > 2, o.z);
        if (top > 3) add(dv == 4, o.w);
        if (top > 4) {
            int k = dv == 5 ? o.w & 255 : 0;
            const int4 *m = tab + (dv == 5 ? o.w >> 8 : 0);
            for (; __any_sync(kFullWarp, k > 0); k -= 4, m++) {
                const int4 e = k > 0 ? *m : o;
                add(k > 0, e.x);
                add(k > 1, e.y);
                add(k > 2, e.z);
                add(k > 3, e.w);
            }
        }
        p.put((jw >> 8) * Z, s);
        i += di;
        r += dr;
        if (r >= Q) {
            r -= Q;
            i++;
        }
    }
}

// Shared memory ahead of the posterior array (flags, codeword, tables; see the kernel).
__host__ __device__ inline size_t cl_tables_bytes(int nnz)
{
    return (((size_t)16 + 4 * (MB_MAX + 1 + NB_MAX + 1) + 15) & ~(size_t)15) + (size_t)32 * nnz;
}

// threads per CTA: higher check degrees keep more values live per thread
template <int DMAX>
constexpr int cl_threads() { return DMAX <= 12 ? 768 : 512; }

template <int DMAX, typename MsgT, bool HC, bool SPREAD>
__global__ void __cluster_dims__(CLUSTER_CTAS, 1, 1) __launch_bounds__(cl_threads<DMAX>(), 1)
    k_flood_cluster(const CodeDev *__restrict__ cd, const __grid_constant__ ClusterArgs a)
{
    constexpr uint32_t kSign = 0x80000000u;
    constexpr int SR = (int)sizeof(MsgT);
    extern __shared__ __align__(16) unsigned char smem[];
    const int q = (int)(blockIdx.x % CLUSTER_CTAS);  // the rank in the cluster (one-dimensional grid)
    const int tid = threadIdx.x, nth = blockDim.x;
    const int Z = a.Z, H = a.H, N = a.N;
    const float Xb = a.X * kSLog2e, Pb = s_phi_b2(a.X);  // the clamp [phi(X), X] in base-2 units

    // bookkeeping: [0] bad flags (2, alternating by round; a check of either CTA sets both
    // CTAs' flag), [2] the codeword being decoded (int64 at 8: request << 32 | request-local
    // index, -1 when the work is done)
    int32_t *flags = reinterpret_cast<int32_t *>(smem);
    int64_t *cwp = reinterpret_cast<int64_t *>(smem + 8);
    // tables: the owned rows' edge descriptors (.x = shared::cluster address of the posterior of
    // position s of column j, .y = offset of the message of position s, .z = Z - s), the owned
    // columns' message addresses (position 0; four, or three and in .w the element and number
    // of the others << 8), then per row its first descriptor << 8 | degree and per column its
    // place << 8 | number
    int4 *tab = reinterpret_cast<int4 *>(smem + 16), *ctab = tab + a.n_edge[q];
    int32_t *rows = reinterpret_cast<int32_t *>(tab + a.n_tab[q]);
    const int n_rows = a.row_split[q + 1] - a.row_split[q], n_cols = a.ncols[q];
    int32_t *cols = rows + n_rows;
    float *app = reinterpret_cast<float *>(smem + a.off_app);
    // R starts at the same offset in every CTA (after the largest posterior share), so that
    // mapping an address into another CTA of the cluster finds that CTA's messages
    MsgT *R = reinterpret_cast<MsgT *>(smem + a.off_r);
    const int blk0 = cd->rowptr[a.row_split[q]], blk1 = cd->rowptr[a.row_split[q + 1]];
    for (int i = tid; i < n_rows; i += nth) {
        const int l = a.row_list[q][i], b0 = cd->rowptr[l], dc = cd->rowptr[l + 1] - b0, e0 = a.row_e0[q][i];
        rows[i] = (e0 << 8) | dc;
        for (int k = 0; k < dc; k++) {
            const int e = cd->ent[b0 + k], j = e >> 16, s = e & 0xffff;
            tab[e0 + k] = make_int4((int)(cl_map(app, a.col_owner[j]) + 4 * (a.col_slot[j] * Z + s)),
                                    a.off_r + SR * ((b0 + k - blk0) * Z + s), Z - s, 0);
        }
    }
    for (int i = tid; i < n_cols; i += nth) {
        const int j = a.col_list[q][i], i0 = cd->colptr[j], dv = cd->colptr[j + 1] - i0;
        cols[i] = (a.col_slot[j] << 8) | j;
        auto addr = [&](int k) -> int {
            if (k >= dv) return 0;
            const int b = cd->colent[i0 + k] >> 16;
            int l = 0;
            while (l < cd->mb - 1 && b >= cd->rowptr[l + 1]) l++;
            const int qo = cl_owner(a.row_split, l);
            return (int)(cl_map(R, qo) + SR * ((b - cd->rowptr[a.row_split[qo]]) * Z));
        };
        int x = a.col_x0[q][i];
        ctab[i] = make_int4(addr(0), addr(1), addr(2), dv > 4 ? (x << 8) | (dv - 3) : addr(3));
        for (int k = 3; dv > 4 && k < dv; k += 4) tab[x++] = make_int4(addr(k), addr(k + 1), addr(k + 2), addr(k + 3));
    }
    const uint32_t flag_0 = cl_map(flags, 0), flag_1 = cl_map(flags, 1);
    // row groups of WT threads (a row pair never needs more threads than a CTA has)
    const int W = a.W, WT = a.WT;
    const int w0 = (int)__reduce_min_sync(0xffffffffu, (unsigned)(tid / WT));  // (a warp reduction: known to be uniform)
    const int ru = tid - w0 * WT;
    const bool works = w0 < W;
    // the variable-node phase's groups (VarQuad)
    const int WT4 = a.WT4, w4 = (int)__reduce_min_sync(0xffffffffu, (unsigned)(tid / WT4));
    const int ru4 = tid - w4 * WT4;
    const uint32_t cw0 = cl_map(cwp, 0);
    cl_sync();  // tables built in every CTA before any remote access

    for (;;) {
        // the leader (CTA 0, thread 0) takes the next codeword; every CTA reads it
        if (q == 0 && tid == 0) {
            const unsigned long long k = atomicAdd(a.next, 1ull);
            int64_t v = -1;
            if (k < (unsigned long long)a.n_items) {
                int rq = 0;
                while (rq < a.n_req - 1 && (int64_t)k >= a.reqs[rq].item0 + a.reqs[rq].n_cw) rq++;
                v = ((int64_t)rq << 32) | ((int64_t)k - a.reqs[rq].item0);
            }
            cwp[0] = v;
        }
        cl_sync();
        int64_t item;
        asm volatile("ld.shared::cluster.b64 %0, [%1];" : "=l"(item) : "r"(cw0));
        if (__any_sync(0xffffffffu, item < 0)) break;  // (a vote: known to be warp-uniform, as the loops below need)
        const ReqDev &req = a.reqs[(int)(item >> 32)];
        const int64_t cw = item & 0xffffffffll;
        if (tid == 0) flags[0] = flags[1] = 0;
        // load: APP = L (+0: no -0) for owned variables, messages 0 for owned edges
        const float *L = static_cast<const float *>(req.llr) + cw * N;
        auto load = [&](int i, int r) {
            const int jw = cols[i];
            const float v = __ldg(L + (jw & 255) * Z + r);
            if (!isfinite(v)) atomicOr(cd->status, IN_NONFINITE);
            app[(jw >> 8) * Z + r] = v + 0.0f;
        };
        if constexpr (SPREAD) {
            for (int x = tid; x < n_cols * Z; x += nth) load(x / Z, x % Z);
        } else {
            for (int r = ru; works && r < Z; r += WT)
                for (int i = w0; i < n_cols; i += W) load(i, r);
        }
        for (int i = tid; i < (blk1 - blk0) * Z; i += nth) R[i] = MsgT(0.0f);
        cl_sync();
        int t = 0;
        bool done = false;
        while (!done) {
            const int tr = t;  // this round's flag is flags[tr & 1]
            // ---------------- check-node phase over the owned checks
            uint32_t bad = 0;
            if constexpr (SPREAD) {
                uint32_t pbad[2] = {0, 0};
                cl_rows_spread<DMAX, MsgT, HC>(tab, rows, n_rows, ClusterMem<MsgT>{reinterpret_cast<char *>(smem)}, Z, H,
                                               tid, nth, Xb, Pb, pbad);
                bad = pbad[0] | pbad[1];
            } else if (works) {
                PairPlace p;
                p.own = ru < H;
                p.r = p.own ? ru : H - 1;
                p.own2 = p.own && p.r + H < Z;
                p.s = p.r + H < Z ? p.r + H : Z - 1;
                p.rw = p.r - Z;
                p.sw = p.s - Z;
                uint32_t pbad[2] = {0, 0};
                cl_rows<0, DMAX, MsgT, HC>(a.rend[q][w0], tab, rows, ClusterMem<MsgT>{reinterpret_cast<char *>(smem)}, p,
                                           Xb, Pb, pbad, a.rstart[q][w0]);
                bad = pbad[0] | pbad[1];
            }
            if (__any_sync(0xffffffffu, (bad & kSign) != 0) && (tid & 31) == 0) {
                cl_st(flag_0 + 4 * (tr & 1), 1);
                cl_st(flag_1 + 4 * (tr & 1), 1);
            }
            cl_sync();
            // ---------------- decision (the same in every CTA)
            const bool conv = tr >= 1 && a.early_exit && flags[tr & 1] == 0;
            if (!__any_sync(0xffffffffu, conv)) {
                // ---------------- variable-node phase over the owned variables
                if constexpr (SPREAD) {
                    if (Z % 4 == 0) {
                        const bool wide = a.wide_L;
                        cl_cols_spread<VarQuad<MsgT>>(a.cend[q][0], ctab, tab, cols, n_cols, Z, Z / 4, tid, nth,
                                                      [&](int r, bool ok) {
                            return VarQuad<MsgT>{L + 4 * r, (uint32_t)(4 * SR * r), app + 4 * r, ok, wide};
                        });
                    } else {
                        cl_cols_spread<VarPair<MsgT>>(a.cend[q][0], ctab, tab, cols, n_cols, Z, H, tid, nth,
                                                      [&](int r, bool ok) {
                            const int s = r + H < Z ? r + H : Z - 1;
                            return VarPair<MsgT>{L + r,   L + s,   (uint32_t)(SR * r), (uint32_t)(SR * s),
                                                 app + r, app + s, ok,                 ok && r + H < Z};
                        });
                    }
                } else if (a.W4 > 0) {
                    const int xc = 4 * ru4 < Z ? 4 * ru4 : Z - 4;
                    const VarQuad<MsgT> v{L + xc, (uint32_t)(SR * xc), app + xc, 4 * ru4 < Z, a.wide_L != 0};
                    if (w4 < a.W4) cl_cols<1>(a.cend[q][w4], ctab, tab, cols, v, Z, a.cstart[q][w4]);
                } else if (works) {
                    const int rc = ru < H ? ru : H - 1, sc = rc + H < Z ? rc + H : Z - 1;
                    const VarPair<MsgT> v{L + rc,   L + sc,   (uint32_t)(SR * rc), (uint32_t)(SR * sc),
                                          app + rc, app + sc, ru < H,              ru < H && rc + H < Z};
                    cl_cols<1>(a.cend[q][w0], ctab, tab, cols, v, Z, a.cstart[q][w0]);
                }
                t++;
            }
            done = __any_sync(0xffffffffu, conv || t >= a.max_iter);
            // the other flag was last read before this round's first barrier: clear it for the
            // next round, which writes it after the barrier below
            if (tid == 0) flags[(tr + 1) & 1] = 0;
            cl_sync();
        }
        // output: each CTA writes its variables
        uint8_t *Bo = req.bits + cw * N;
        float *Ao = req.app ? req.app + cw * N : nullptr;
        auto store = [&](int i, int r) {
            const int jw = cols[i], n = (jw & 255) * Z + r;
            const float v = app[(jw >> 8) * Z + r];
            Bo[n] = v < 0.0f ? 1 : 0;
            if (Ao) Ao[n] = v;
        };
        if constexpr (SPREAD) {
            for (int x = tid; x < n_cols * Z; x += nth) store(x / Z, x % Z);
        } else {
            for (int r = ru; works && r < Z; r += WT)
                for (int i = w0; i < n_cols; i += W) store(i, r);
        }
        if (q == 0 && tid == 0) req.iters[cw] = t;
    }
    cl_sync();  // no CTA leaves while another may still read its shared memory
}

// ------------------------------------------------------------------ host side

// Split the block rows between the cluster's CTAs in contiguous ranges of about equal block
// counts, then give each block column to the CTA that owns most of its blocks' rows (its
// posteriors are then read locally by most of its checks), moving the least attached columns
// while a CTA would need more shared memory than the largest allowed.  Returns the per-CTA
// shared memory (the same layout in every CTA), or 0 if no assignment fits.
static size_t cl_plan(const CodeDev &h, int msg, ClusterArgs &a, size_t limit)
{
    a.row_split[0] = 0;
    for (int q = 1; q < CLUSTER_CTAS; q++) {
        const int want = (int)((int64_t)h.nnz * q / CLUSTER_CTAS);
        int l = a.row_split[q - 1] + 1;
        while (l < h.mb && h.rowptr[l] < want) l++;
        a.row_split[q] = l < h.mb ? l : h.mb - 1;
    }
    a.row_split[CLUSTER_CTAS] = h.mb;
    const size_t msz = msg == LDPC_MSG_F16 ? sizeof(__half) : sizeof(float);
    size_t nr = 0;
    for (int q = 0; q < CLUSTER_CTAS; q++) {
        const size_t nm = (size_t)(h.rowptr[a.row_split[q + 1]] - h.rowptr[a.row_split[q]]) * h.Z;
        nr = nm > nr ? nm : nr;
    }
    // affinity of column j to CTA q: its blocks in q's rows
    int aff[NB_MAX][CLUSTER_CTAS] = {};
    for (int j = 0; j < h.nb; j++)
        for (int i = h.colptr[j]; i < h.colptr[j + 1]; i++) {
            const int b = h.colent[i] >> 16;
            int l = 0;
            while (l < h.mb - 1 && b >= h.rowptr[l + 1]) l++;
            aff[j][cl_owner(a.row_split, l)]++;
        }
    int cnt[CLUSTER_CTAS] = {};
    for (int j = 0; j < h.nb; j++) {
        int best = 0;
        for (int q = 1; q < CLUSTER_CTAS; q++)
            if (aff[j][q] > aff[j][best] || (aff[j][q] == aff[j][best] && cnt[q] < cnt[best])) best = q;
        a.col_owner[j] = best;
        cnt[best]++;
    }
    // the posterior share of a CTA may not exceed what its shared memory has left
    const size_t fixed = cl_tables_bytes(h.nnz) + nr * msz;
    const int cap = limit > fixed ? (int)((limit - fixed) / (4 * (size_t)h.Z)) : 0;
    for (int q = 0; q < CLUSTER_CTAS; q++) {
        while (cnt[q] > cap) {
            // move q's column with the least attachment to q to the CTA with the most room
            int jm = -1;
            for (int j = 0; j < h.nb; j++)
                if (a.col_owner[j] == q && (jm < 0 || aff[j][q] < aff[jm][q])) jm = j;
            int to = -1;
            for (int k = 0; k < CLUSTER_CTAS; k++)
                if (k != q && cnt[k] < cap && (to < 0 || cnt[k] < cnt[to])) to = k;
            if (jm < 0 || to < 0) return 0;
            a.col_owner[jm] = to;
            cnt[q]--;
            cnt[to]++;
        }
    }
    for (int q = 0; q < CLUSTER_CTAS; q++) a.ncols[q] = 0;
    for (int j = 0; j < h.nb; j++) a.col_slot[j] = a.ncols[a.col_owner[j]]++;
    int nmax = 0;
    for (int q = 0; q < CLUSTER_CTAS; q++) nmax = a.ncols[q] > nmax ? a.ncols[q] : nmax;
    // groups of whole warps: W for two rows per thread, W4 for four positions (Z a multiple of 4;
    // else the columns go to the row groups too)
    const int nth = h.dc_max <= 12 ? cl_threads<12>() : cl_threads<32>();
    a.Z = h.Z;
    a.H = (h.Z + 1) / 2;
    static_assert(Z_MAX / 2 <= cl_threads<32>(), "a row pair's threads");
    a.WT = (a.H + 31) & ~31;
    a.W = nth / a.WT;
    a.WT4 = a.Z % 4 ? 32 : (a.Z / 4 + 31) & ~31;
    a.W4 = a.Z % 4 ? 0 : nth / a.WT4;
    // end to end over the threads where that leaves so few turns of the rows (about two thirds of the
    // time) and the columns that it pays for the votes.  (GB300, FP16, us per launch, groups of whole
    // warps / end to end: 512 codewords of a 64 x 128 code of 1024 blocks, Z = 130 2167 / 1643, Z = 136
    // 2024 / 1486; 1024 of a 34 x 68 code, Z = 260 2065 / 1664; FP32, 64 x 128, Z = 68 1184 / 954, but 30 x 90, rows of 8, Z = 278, 2334 / 2737.)
    const int Q = a.Z % 4 ? a.H : a.Z / 4, Wc = a.W4 ? a.W4 : a.W;
    double whole[2] = {}, spread[2] = {};  // turns of rows and columns, of the slower CTA
    for (int q = 0; q < CLUSTER_CTAS; q++) {
        const int n[2] = {a.row_split[q + 1] - a.row_split[q], a.ncols[q]}, w[2] = {a.W, Wc}, p[2] = {a.H, Q};
        for (int i = 0; i < 2; i++) {
            whole[i] = fmax(whole[i], (n[i] + w[i] - 1) / w[i]);
            spread[i] = fmax(spread[i], (n[i] * p[i] + nth - 1) / nth);
        }
    }
    const double gain = 0.65 * spread[0] / whole[0] + 0.35 * spread[1] / whole[1];
    a.spread = gain * (1.0 + 4.3 * h.mb / h.nnz) < 1.0;  // (rows of 9.5 edges take 1.3 to 1.45 times as long)
    if (a.spread) a.W = a.W4 = 1;  // one list of each
    // the CTAs' lists, and the size of their tables.  A phase ends at a cluster barrier, so its
    // rows (columns) go to the groups by weight, heaviest first to the least loaded group
    size_t tables = cl_tables_bytes(h.nnz);
    for (int q = 0; q < CLUSTER_CTAS; q++) {
        int ne = 0, nr = 0, nc = 0;
        uint8_t order[MB_MAX > NB_MAX ? MB_MAX : NB_MAX], group[sizeof order];
        // the items of degree deg(i) (0: not this CTA's) in ascending degree, each with its group
        auto deal = [&](int n, auto deg, int dmax, int overhead, int W) {
            int load[CL_GROUPS] = {}, m = 0;
            for (int d = 1; d <= dmax; d++)
                for (int i = 0; i < n; i++)
                    if (deg(i) == d) order[m++] = (uint8_t)i;
            for (int k = m - 1; k >= 0; k--) {
                int w = 0;
                for (int g = 1; g < W; g++)
                    if (load[g] < load[w]) w = g;
                group[k] = (uint8_t)w;
                load[w] += deg(order[k]) + overhead;
            }
            return m;
        };
        auto rdeg = [&](int l) {
            return l >= a.row_split[q] && l < a.row_split[q + 1] ? h.rowptr[l + 1] - h.rowptr[l] : 0;
        };
        auto cdeg = [&](int j) { return a.col_owner[j] == q ? h.colptr[j + 1] - h.colptr[j] : 0; };
        int m = deal(h.mb, rdeg, h.dc_max, 1, a.W);
        for (int w = 0; w < a.W; w++) {
            int c = 0;
            a.rstart[q][w] = (uint8_t)nr;
            for (int k = 0; k < m; k++) {
                if (group[k] != w) continue;
                const int d = rdeg(order[k]);
                while (d > cl_class_degree(c)) a.rend[q][w][c++] = (uint8_t)nr;
                a.row_e0[q][nr] = (uint16_t)ne;
                a.row_list[q][nr++] = order[k];
                ne += d;
            }
            while (c < CL_CLASSES) a.rend[q][w][c++] = (uint8_t)nr;
        }
        int nx = ne + a.ncols[q];
        const int Wv = a.W4 ? a.W4 : a.W;
        m = deal(h.nb, cdeg, h.mb, 3, Wv);
        for (int w = 0; w < Wv; w++) {
            int c = 1;
            a.cstart[q][w] = (uint8_t)nc;
            for (int k = 0; k < m; k++) {
                if (group[k] != w) continue;
                const int d = cdeg(order[k]);
                while (c < 5 && d > c) a.cend[q][w][c++ - 1] = (uint8_t)nc;
                a.col_x0[q][nc] = (uint16_t)nx;
                a.col_list[q][nc++] = order[k];
                if (d > 4) nx += d / 4;
            }
            while (c <= 5) a.cend[q][w][c++ - 1] = (uint8_t)nc;
        }
        a.n_edge[q] = ne;
        a.n_tab[q] = nx;
        const size_t need = ((size_t)16 + (size_t)nx * 16 + (size_t)(nr + nc) * 4 + 15) & ~(size_t)15;
        tables = need > tables ? need : tables;
    }
    a.off_app = (int)tables;
    a.off_r = (int)(tables + (((size_t)nmax * h.Z * 4 + 15) & ~(size_t)15));
    return (size_t)a.off_r + nr * msz;
}

static size_t cl_limit()
{
    int dev = 0, lim = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return lim > 0 ? (size_t)lim : 227 * 1024;
}

struct ClusterPlan {
    ClusterArgs a;  // all but the requests and parameters of a call
    size_t smem;
};

// (Planned once: forming it anew took 9 us of the host, three times per call.)
ClusterPlan *cluster_plan_create(const CodeDev &h, int msg)
{
    if (h.dc_max > 32 || h.mb < CLUSTER_CTAS || h.nb < CLUSTER_CTAS) return nullptr;
    ClusterPlan *q = new (std::nothrow) ClusterPlan;
    if (!q) return nullptr;
    memset(q, 0, sizeof *q);
    q->smem = cl_plan(h, msg, q->a, cl_limit());
    if (q->smem == 0 || q->smem > cl_limit()) {
        delete q;
        return nullptr;
    }
    return q;
}

void cluster_plan_free(ClusterPlan *plan) { delete plan; }

template <int DMAX, typename MsgT, bool HC, bool SPREAD>
static cudaError_t launch_cluster(ClusterArgs &a, size_t smem, int64_t n_cw, const CodeDev *d, cudaStream_t s)
{
    cudaError_t e = ensure_smem<k_flood_cluster<DMAX, MsgT, HC, SPREAD>>(smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CLUSTER_CTAS, 1, 1);
    cfg.blockDim = dim3(cl_threads<DMAX>(), 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    // clusters that fit the device at once, queried once per device and shared-memory size
    static int cached[64];
    static size_t cached_smem[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    int clusters = __atomic_load_n(&cached[dev], __ATOMIC_RELAXED);
    if (clusters < 1 || __atomic_load_n(&cached_smem[dev], __ATOMIC_RELAXED) != smem) {
        e = cudaOccupancyMaxActiveClusters(&clusters, k_flood_cluster<DMAX, MsgT, HC, SPREAD>, &cfg);
        if (e != cudaSuccess || clusters < 1) {
            cudaGetLastError();
            int nsm = 2;
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
            clusters = nsm / CLUSTER_CTAS;
        }
        __atomic_store_n(&cached_smem[dev], smem, __ATOMIC_RELAXED);
        __atomic_store_n(&cached[dev], clusters, __ATOMIC_RELAXED);
    }
    if ((int64_t)clusters > n_cw) clusters = (int)n_cw;
    a.wide_L = a.N % 4 == 0;
    for (int i = 0; i < a.n_req; i++)
        if (reinterpret_cast<uintptr_t>(a.reqs[i].llr) & 15) a.wide_L = 0;
    LaunchScope ls(F_SLOTS, s);
    k_flood_cluster<DMAX, MsgT, HC, SPREAD><<<(unsigned)(clusters * CLUSTER_CTAS), cl_threads<DMAX>(), smem, s>>>(d, a);
    return cudaGetLastError();
}

template <typename MsgT, bool HC, bool SPREAD>
static cudaError_t launch_cluster_d(int dmax, ClusterArgs &a, size_t smem, int64_t n_cw, const CodeDev *d,
                                    cudaStream_t s)
{
    if (dmax <= 8) return launch_cluster<8, MsgT, HC, SPREAD>(a, smem, n_cw, d, s);
    if (dmax <= 12) return launch_cluster<12, MsgT, HC, SPREAD>(a, smem, n_cw, d, s);
    return launch_cluster<32, MsgT, HC, SPREAD>(a, smem, n_cw, d, s);
}

template <typename MsgT, bool HC>
static cudaError_t launch_cluster_f(int dmax, ClusterArgs &a, size_t smem, int64_t n_cw, const CodeDev *d,
                                    cudaStream_t s)
{
    return a.spread ? launch_cluster_d<MsgT, HC, true>(dmax, a, smem, n_cw, d, s)
                    : launch_cluster_d<MsgT, HC, false>(dmax, a, smem, n_cw, d, s);
}

cudaError_t flood_cluster_decode(const ClusterPlan &plan, const CodeDev &h, const CodeDev *d,
                                 const ldpc_decode_params &p, const HostReq *reqs, int n, void *counter,
                                 cudaStream_t s)
{
    if (n < 1 || n > MULTI_MAX_REQS) return cudaErrorInvalidValue;
    ClusterArgs a = plan.a;
    const size_t smem = plan.smem;
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
    a.N = h.N;
    a.next = static_cast<unsigned long long *>(counter);
    a.max_iter = p.max_iter;
    a.early_exit = p.early_exit;
    a.X = p.phi_clamp;
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    const bool hc = p.phi_clamp < FLOOD_CLAMP_X;
    if (p.msg == LDPC_MSG_F16)
        return hc ? launch_cluster_f<__half, true>(h.dc_max, a, smem, items, d, s)
                  : launch_cluster_f<__half, false>(h.dc_max, a, smem, items, d, s);
    return hc ? launch_cluster_f<float, true>(h.dc_max, a, smem, items, d, s)
              : launch_cluster_f<float, false>(h.dc_max, a, smem, items, d, s);
}

}  // namespace ldpc
