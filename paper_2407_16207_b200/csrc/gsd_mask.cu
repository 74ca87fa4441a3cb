// gsd_build_mask: ancestor bitmask of a draft DAG from its parent lists in CSR form, i.e. what
// "a token may only attend to its ancestor nodes" (tree attention, Sec. 4.1) means for the
// merged token graph (Sec. 5.3): bit j of row n is set iff j == n or n can be reached from j.
//
// Grid (W, B): a CTA owns one word column of one sequence, i.e. the bits of 32 would-be ancestors
// for all N nodes, and a thread owns one node.  row[v] |= OR over parents p of row[p] is relaxed
// level-synchronously until nothing changes (at most longest-path + 1 rounds; parents precede
// children, so one round settles one more level).  Words only ever gain bits, so the in-place
// update needs no second copy.
//
// The work is tiny and the time is the chain of rounds, so a round has to be short: the row
// pointers and the parent indices come in one trip to memory, a node's first kRegParents parents
// sit in registers, and a round is a handful of shared-memory reads, at most one write and a
// barrier.  Columns do not depend on one another, so they go to different CTAs.  B200, ncu: 8
// sequences of N 256, depth 16: 35.2 -> 7.0 us; 32 of N 512, depth 18: 89.7 -> 10.8 us;
// one of N 16: 7.3 -> 4.3 us (before: one CTA per sequence over all N x W words, parent lists
// read from global memory in every round).
#include "gsd_internal.cuh"

namespace gsd {
namespace {

constexpr int kRegParents = 4;
constexpr int kEdgeCache = 4 * GSD_MAX_NODES;     // parent indices of one sequence kept in shared memory

// (Plain pointers: the kernel is resident while its predecessor may still write the graph, so the inputs must
// not be declared as data that nobody writes, which would let their loads go ahead of the wait.)
__global__ void __launch_bounds__(GSD_MAX_NODES)
build_mask_kernel(const int32_t* parent_ptr, const int32_t* parent_idx, uint32_t* mask, int b0, int N, int W, int Ecap,
                  int32_t* status) {
    __shared__ uint32_t s_rows[GSD_MAX_NODES];
    __shared__ int s_edge[kEdgeCache];
    volatile uint32_t* rows = s_rows;
    let_successor_start();
    const int w = blockIdx.x, b = b0 + blockIdx.y, v = threadIdx.x;
    const int32_t* pp = parent_ptr + (size_t)b * (N + 1);
    const int32_t* pi = parent_idx + (size_t)b * Ecap;
    const bool mine = v < N;
    // (the row of parent indices holds Ecap entries whatever the pointers say)
    const int cached = min(Ecap, kEdgeCache);
    int e0 = 0, e1 = 0;
    wait_for_predecessor();
    if (mine) {
        e0 = pp[v];
        e1 = pp[v + 1];
    }
    for (int e = v; e < cached; e += blockDim.x) s_edge[e] = pi[e];
    uint32_t acc = mine && w == (v >> 5) ? (1u << (v & 31)) : 0u;
    if (mine) rows[v] = acc;
    __syncthreads();
    unsigned flags = 0;
    if (e0 < 0 || e1 > Ecap || e0 > e1) {
        flags |= GSD_DEV_BAD_CSR;
        e0 = e1 = 0;
    }
    auto parent = [&](int e) -> int {       // a parent that may be followed, or -1
        const int p = e < cached ? s_edge[e] : pi[e];
        if (p >= 0 && p < v) return p;
        flags |= GSD_DEV_BAD_CSR;
        return -1;
    };
    int par[kRegParents];
#pragma unroll
    for (int k = 0; k < kRegParents; ++k) {
        // (an absent parent is the node itself, whose word is part of the result anyway)
        const int p = e0 + k < e1 ? parent(e0 + k) : -1;
        par[k] = p >= 0 ? p : (mine ? v : 0);
    }
    for (int round = 0; round < N; ++round) {
        int changed = 0;
        if (mine) {
            uint32_t got = acc;
#pragma unroll
            for (int k = 0; k < kRegParents; ++k) got |= rows[par[k]];
            for (int e = e0 + kRegParents; e < e1; ++e) {
                const int p = parent(e);
                if (p >= 0) got |= rows[p];
            }
            if (got != acc) {
                acc = got;
                rows[v] = got;
                changed = 1;
            }
        }
        if (!__syncthreads_or(changed)) break;
    }
    if (mine) mask[((size_t)b * N + v) * W + w] = acc;
    if (flags && status) atomicOr((unsigned*)status, flags);
}

}  // namespace
}  // namespace gsd

extern "C" int gsd_build_mask(const int32_t* parent_ptr, const int32_t* parent_idx,
                              uint32_t* ancestor_mask, int32_t B, int32_t N, int32_t Ecap,
                              int32_t* status, void* stream) {
    using namespace gsd;
    if (!parent_ptr || !parent_idx || !ancestor_mask) return GSD_ERR_NULL_POINTER;
    if (B < 1 || B > 65535 * 32 || N < 1 || N > GSD_MAX_NODES || Ecap < 1) return GSD_ERR_BAD_SHAPE;
    const int W = (N + 31) / 32;
    const int threads = (N + 31) / 32 * 32;                 // one per node
    for (int b0 = 0; b0 < B; b0 += 65535) {                 // (grid.y holds 65535 sequences)
        const int nb = B - b0 < 65535 ? B - b0 : 65535;
        GSD_CUDA_TRY(launch_dependent(build_mask_kernel, dim3(W, nb), dim3(threads), 0, (cudaStream_t)stream, parent_ptr, parent_idx,
                                      ancestor_mask, b0, N, W, Ecap, status));
    }
    return GSD_OK;
}
