// Launch descriptor of the flooding slot decoder, shared by its host side (flood_slots.cu) and
// its kernel (flood_slots_kernel.cuh).
#pragma once

#include "ldpc_internal.h"

namespace ldpc {

// Degree classes of the block rows: exact bodies for degrees 2..8, then up to 12, 16, 24, 32.
constexpr int FLOOD_CLASSES = 11;
__host__ __device__ constexpr int flood_class_degree(int c)
{
    return c < 7 ? c + 2 : c == 7 ? 12 : c == 8 ? 16 : c == 9 ? 24 : 32;
}

// One code of a launch: the requests' codewords are the items of its work sequence.
struct FloodGroup {
    int64_t n_items;
    int req_begin, req_end;
    int N, Z, mb, nb, nnz;
    int G;           // thread slots (V codewords each) per CTA
    int W, TPG;      // row groups a thread slot is spread over; threads of a barrier group
    int K;           // thread slots of a barrier group (1 unless they lie end to end in a warp)
    int strA, strR;  // bytes from one thread slot's posteriors / messages to the next one's
    int offR;        // first thread slot's messages, bytes after the first one's posteriors
    int book0, slots0;  // its bookkeeping and first slot, bytes from the start of shared memory
    const int4 *tab; // the code's tables on the device (see below), n_tab elements
    int n_tab, t_col, t_row;
    uint8_t rend[FLOOD_CLASSES], cend[5];  // end of each degree class in the row and column lists
    unsigned int *status;
    float cumw;      // cumulative share of the launch's work (initial CTA placement)
};

struct FloodReq {
    const float *llr;
    uint8_t *bits;
    int32_t *iters;
    float *app;
    int64_t item0;  // index of its first codeword in its group's work sequence
};

// Tables of a code, for each element size of a thread's posterior and message (V codewords,
// message type); built on the host when the code is created, copied to shared memory when a
// CTA takes the code up.  Elements, in this order:
//   edge descriptor of block b = (row l, column j, shift s): .x = byte offset of the posterior
//     j*Z + s and .y of the message b*Z + s from a thread's bases (position 0 of its slot; FP32
//     messages: .y from the posterior base too), .z = Z - s; check row r reaches variable
//     position (r + s) mod Z, so its offsets are these from its own bases (position r), less
//     one block when r >= .z
//   block columns in ascending degree (from t_col): message offsets b*Z of its blocks in row
//     order, up to four; above degree 4 three, and in .w (index of the others' elements << 8 |
//     their number).  Messages are stored at the variable's position inside the block, so the
//     variable-node phase needs no wrap
//   32-bit words (from t_row): per block row in ascending degree the index of its first edge
//     descriptor << 8 | its degree; per block column in ascending degree its first variable
struct FloodArgs {
    unsigned long long *next;  // [n_groups] work counters, zero at launch; null: one group, all codewords resident
    int n_groups;
    int max_iter, early_exit;
    float X;
    int tab0;  // a code's tables, bytes from the start of shared memory (the same for all: see flood_slots.cu)
    FloodGroup groups[MULTI_MAX_GROUPS];
    FloodReq reqs[MULTI_MAX_REQS];
};
static_assert(sizeof(FloodArgs) <= 32764, "kernel parameters");

// Bookkeeping of one slot in shared memory.
struct FloodBook {
    int64_t cw;      // its next codeword (request-local, -1: none)
    int32_t req;     // and the request
    int32_t bad[2];  // unsatisfied check seen, by round parity
    int32_t pad;
};

// How rows lie in a warp: whole warps to a thread slot's rows (flood_slots_kernel.cuh), the rows of K
// thread slots end to end, or those and the row groups end to end (flood_packed_kernel.cuh).
enum FloodForm { FLOOD_WHOLE, FLOOD_PACKED, FLOOD_SPREAD };

// A launch: its parameters and the instance they are for (rows of degree <= 8, or up to 32; V codewords
// per thread).
struct FloodPlan {
    FloodArgs a;
    int dmax, V, threads, ctas;
    FloodForm form;
    size_t smem;
};

constexpr int FLOOD_TAB0 = 16;  // a code's tables, bytes from the start of shared memory

// Named barriers thread slots can have (barrier 0 is the CTA's).
constexpr int FLOOD_BARRIERS = 15;

// Threads per CTA of an instance (rows of degree <= 8, or up to 32; message type).
__host__ __device__ constexpr int flood_threads_max(int dmax, int V, bool f16)
{
    return V == 2 && (dmax <= 8 || f16) ? 768 : 640;
}

// Size a launch for n requests (a.next: the counters, or null where none are needed and none are
// given); no call to the device.
cudaError_t flood_plan(const HostReq *reqs, int n, const ldpc_decode_params &p, void *counters, size_t limit, int nsm,
                       FloodPlan &out);

// Launch a plan.
template <typename MsgT, bool HC>
cudaError_t flood_slots_launch(const FloodPlan &q, cudaStream_t s);

template <typename MsgT, bool HC>
cudaError_t flood_packed_launch(const FloodPlan &q, cudaStream_t s);

}  // namespace ldpc
