// Host-only program around the flooding slot decoder's launch sizing (no device is used): reads
// codes and launches from standard input, prints what flood_plan made of each launch.
//   code:   C mb nb Z, then mb * nb shifts (-1: no block)
//   launch: L f16 n, then n pairs (code, codewords)
// Output per launch: whether every code is served alone, the status, bytes of shared memory, threads,
// CTAs, codewords per thread, the form, then per code its width, thread slots, row
// groups, threads and thread slots of a barrier group, and where its layout ends.
#include <stdio.h>

#include <vector>

#include "flood_slots.cu"

namespace ldpc {
template <typename M, bool H>
cudaError_t flood_slots_launch(const FloodPlan &, cudaStream_t) { return cudaErrorUnknown; }
template <typename M, bool H>
cudaError_t flood_packed_launch(const FloodPlan &, cudaStream_t) { return cudaErrorUnknown; }
template cudaError_t flood_slots_launch<float, false>(const FloodPlan &, cudaStream_t);
template cudaError_t flood_packed_launch<float, false>(const FloodPlan &, cudaStream_t);
template cudaError_t flood_slots_launch<float, true>(const FloodPlan &, cudaStream_t);
template cudaError_t flood_packed_launch<float, true>(const FloodPlan &, cudaStream_t);
template cudaError_t flood_slots_launch<__half, false>(const FloodPlan &, cudaStream_t);
template cudaError_t flood_packed_launch<__half, false>(const FloodPlan &, cudaStream_t);
template cudaError_t flood_slots_launch<__half, true>(const FloodPlan &, cudaStream_t);
template cudaError_t flood_packed_launch<__half, true>(const FloodPlan &, cudaStream_t);
}  // namespace ldpc

using namespace ldpc;

static ldpc_code *read_code()
{
    ldpc_code *c = new ldpc_code();
    CodeDev &h = c->host;
    if (scanf("%d %d %d", &h.mb, &h.nb, &h.Z) != 3) return nullptr;
    std::vector<int> base(h.mb * h.nb);
    for (int &s : base)
        if (scanf("%d", &s) != 1) return nullptr;
    for (int l = 0; l < h.mb; l++) {
        h.rowptr[l] = h.nnz;
        for (int j = 0; j < h.nb; j++)
            if (base[l * h.nb + j] >= 0) h.ent[h.nnz++] = (j << 16) | base[l * h.nb + j];
        if (h.nnz - h.rowptr[l] > h.dc_max) h.dc_max = h.nnz - h.rowptr[l];
    }
    h.rowptr[h.mb] = h.nnz;
    int k = 0;
    for (int j = 0; j < h.nb; j++) {
        h.colptr[j] = k;
        for (int b = 0; b < h.nnz; b++)
            if ((h.ent[b] >> 16) == j) h.colent[k++] = (b << 16) | (h.ent[b] & 0xffff);
    }
    h.colptr[h.nb] = k;
    h.N = h.nb * h.Z;
    h.E = h.nnz * h.Z;
    h.n_ftab = flood_table_size(h);
    std::vector<int4> tab(h.n_ftab);
    flood_build_table(h, LDPC_MSG_F32, 1, tab.data());  // (sets the degree classes)
    return c;
}

int main()
{
    const size_t limit = 227 * 1024;
    std::vector<ldpc_code *> codes;
    char what;
    while (scanf(" %c", &what) == 1) {
        if (what == 'C') {
            codes.push_back(read_code());
            if (!codes.back()) return 1;
            continue;
        }
        int f16, n;
        if (scanf("%d %d", &f16, &n) != 2) return 1;
        std::vector<HostReq> reqs(n);
        bool ok = true;  // every code is served alone
        for (HostReq &q : reqs) {
            int c;
            long long cw;
            if (scanf("%d %lld", &c, &cw) != 2) return 1;
            q = HostReq();
            q.code = codes[c];
            q.n_cw = cw;
            ok &= slots_supported(codes[c]->host, f16 ? LDPC_MSG_F16 : LDPC_MSG_F32) != 0;
        }
        ldpc_decode_params p = {};
        p.msg = f16 ? LDPC_MSG_F16 : LDPC_MSG_F32;
        p.phi_clamp = 80.0f;
        static FloodPlan q;
        unsigned long long counters[MULTI_MAX_GROUPS];
        const cudaError_t e = flood_plan(reqs.data(), n, p, counters, limit, 152, q);
        printf("%d %d %zu %d %d %d %d", (int)ok, (int)e, q.smem, q.threads, q.ctas, q.V, (int)q.form);
        for (int g = 0; e == cudaSuccess && g < q.a.n_groups; g++) {
            const FloodGroup &d = q.a.groups[g];
            const size_t E = (size_t)d.nnz * d.Z;
            const size_t end_a = (size_t)(d.G - 1) * d.strA + 4 * (size_t)q.V * d.N;
            const size_t end_r = d.offR + (size_t)(d.G - 1) * d.strR + (f16 ? 2 : 4) * q.V * E;
            printf(" %d %d %d %d %d %zu", d.Z, d.G, d.W, d.TPG, d.K, d.slots0 + (end_a > end_r ? end_a : end_r));
        }
        printf("\n");
    }
    return 0;
}
