// Longest accepted root path through the draft DAG (Sec. 4.1 longest-path selection; Sec. 3
// rejection cascade), shared by the deterministic and the non-deterministic verification.
// One CTA of kPathThreads threads per sequence.  The caller supplies the test of one step
// parent -> v; this file does the rest: parent lists on chip, the accepted steps, level-synchronous
// relaxation of best[v] = 1 + max over accepted steps into v, choice of the end node (longest, then
// lowest index), walk back (lowest predecessor that carries length - 1), emission of the path's node
// ids and drafted tokens.  The token the target model contributes at the end is the caller's.
//
// The pass runs on one SM while the rest of the device may already be idle, so it is laid out for
// short chains: tokens, row pointers and the parent indices are fetched in one trip; a node belongs
// to one thread, which tests the steps into it once and keeps the accepted ones, the first in a register
// - most nodes have one or none - so that a round of the relaxation is a read of shared memory and
// a barrier; every node picks its predecessor in parallel, after which the walk back is a pointer
// chase in shared memory.  (Steps tested again in every round, with the parent lists walked in shared
// memory: 3 sequences of N 507, the relaxation alone 4.3 us, now 1.3.  One warp doing the relaxation with votes
// instead of barriers, the accepted steps in its registers: 1 to 2 us slower than eight warps, an
// instruction of a lone warp takes as long as a barrier.)
#pragma once
#include "gsd_internal.cuh"

namespace gsd {

constexpr int kPathThreads = 256;
constexpr int kPathNodeSlots = (GSD_MAX_NODES + kPathThreads - 1) / kPathThreads;
constexpr int kPathEdgeCache = 3 * GSD_MAX_NODES;   // parent edges of one sequence kept in shared memory
static_assert(kPathEdgeCache % kPathThreads == 0, "the edge prefetch is dealt out in whole rounds");

struct PathIo {
    const int32_t* tok;     // [N] drafted tokens of the sequence
    const int32_t* pptr;    // [N+1]
    const int32_t* pidx;    // [Ecap]
    int32_t* out_tok;       // [Tcap]
    int32_t* out_nodes;     // [Tcap] or nullptr
    int32_t* out_len;       // one entry
    int32_t* status;        // device status word or nullptr
    int N, V, Ecap, Tcap;
};

struct PathResult {
    int edges;           // m: the accepted path has m + 1 nodes
    int end;             // its last node
    bool end_has_child;  // some node lists `end` as a parent
};

// The test of a step p -> v comes in two halves: `edge_pre(p, t)` fetches what the test needs from
// global memory (a float; t is v's token), `step_ok(pre, p, v, t)` decides.  With kFetch the first is
// called for all steps of a node at once and what it returned is kept on chip.  Between the two
// halves the function calls `mid()` (all threads; it returns status bits) and meets at a barrier: a
// caller whose decision needs results of an earlier kernel waits for them there, AFTER the graph
// and the values of `edge_pre` have been fetched.  `flags` carries status bits the caller has already
// found; the function adds its own and publishes them.  All threads of the CTA must call it; all
// return the same result.  out_tok[edges] is left for the caller, entries past it are set to -1.
template <bool kFetch, class StepOk, class EdgePre, class Mid>
__device__ PathResult longest_accepted_path(const PathIo& io, unsigned flags, StepOk step_ok, EdgePre edge_pre, Mid mid) {
    __shared__ int s_best[GSD_MAX_NODES];         // edges of the longest accepted root path, -1: none
    __shared__ int s_tok[GSD_MAX_NODES];
    __shared__ int s_ptr[GSD_MAX_NODES + 1];
    __shared__ int s_edge[kPathEdgeCache];
    __shared__ float s_pre[kFetch ? kPathEdgeCache : 1];   // what edge_pre fetched for each step
    __shared__ short s_pred[GSD_MAX_NODES];       // a node's predecessor on its best path
    __shared__ short s_path[GSD_MAX_NODES];       // the chosen path, root first
    __shared__ unsigned char s_child[GSD_MAX_NODES];   // the node is some node's parent
    __shared__ int s_red[kPathThreads / 32];
    __shared__ unsigned s_flags;
    const int N = io.N, tid = threadIdx.x;
    if (tid == 0) s_flags = 0;
    // tokens, row pointers and (speculatively: the row holds Ecap entries whatever the pointers
    // say) the parent indices, all in one trip to memory
    // (every load is issued before the first of them is used: the loops below have constant
    // trip counts and are unrolled, so the three arrays cost one round trip, not three)
    const int n_prefetch = min(io.Ecap, kPathEdgeCache);
    int r_tok[kPathNodeSlots], r_ptr[kPathNodeSlots + 1], r_edge[kPathEdgeCache / kPathThreads];
#pragma unroll
    for (int k = 0; k < kPathNodeSlots; ++k) r_tok[k] = tid + k * kPathThreads < N ? io.tok[tid + k * kPathThreads] : 0;
#pragma unroll
    for (int k = 0; k <= kPathNodeSlots; ++k) r_ptr[k] = tid + k * kPathThreads <= N ? io.pptr[tid + k * kPathThreads] : 0;
#pragma unroll
    for (int k = 0; k < kPathEdgeCache / kPathThreads; ++k)
        r_edge[k] = tid + k * kPathThreads < n_prefetch ? io.pidx[tid + k * kPathThreads] : 0;
#pragma unroll
    for (int k = 0; k < kPathNodeSlots; ++k) {
        const int v = tid + k * kPathThreads;
        if (v < N) {
            s_tok[v] = r_tok[k];
            if (r_tok[k] < 0 || r_tok[k] >= io.V) flags |= GSD_DEV_BAD_TOKEN;
            s_best[v] = v == 0 ? 0 : -1;
            s_child[v] = 0;
        }
    }
#pragma unroll
    for (int k = 0; k <= kPathNodeSlots; ++k) {
        const int v = tid + k * kPathThreads;
        if (v <= N) {
            int e = r_ptr[k];
            if (e < 0 || e > io.Ecap) {
                flags |= GSD_DEV_BAD_CSR;
                e = e < 0 ? 0 : io.Ecap;
            }
            s_ptr[v] = e;
        }
    }
#pragma unroll
    for (int k = 0; k < kPathEdgeCache / kPathThreads; ++k)
        if (tid + k * kPathThreads < n_prefetch) s_edge[tid + k * kPathThreads] = r_edge[k];
    __syncthreads();
    // Row pointers must start at zero and never decrease.  Otherwise they are replaced by their
    // running maximum (a row whose pointer goes backwards becomes empty, the rows stay disjoint
    // and every edge below the last pointer has exactly one owner) and the status bit is set.
    {
        int bad = 0;
        for (int v = tid; v < N; v += kPathThreads) bad |= (s_ptr[v] > s_ptr[v + 1]);
        if (tid == 0 && s_ptr[0] != 0) bad = 1;
        if (__syncthreads_or(bad)) {
            flags |= GSD_DEV_BAD_CSR;
            if (tid == 0) {
                int run = 0;
                s_ptr[0] = 0;
                for (int v = 1; v <= N; ++v) {
                    run = max(run, s_ptr[v]);
                    s_ptr[v] = run;
                }
            }
            __syncthreads();
        }
    }
    // Lists that do not fit on chip stay where they are: their steps are tested again on every use.
    const bool cached = s_ptr[N] <= kPathEdgeCache;
    auto parent_at = [&](int e) -> int { return cached ? s_edge[e] : io.pidx[e]; };
    auto token_ok = [&](int t) -> bool { return t >= 0 && t < io.V; };
    if (kFetch && cached) {
        // (four steps of a node at a time)
        for (int v = tid; v < N; v += kPathThreads) {
            const int e1 = s_ptr[v + 1], t = s_tok[v];
            for (int e = s_ptr[v]; e < e1; e += 4) {
                float got[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int p = e + k < e1 ? s_edge[e + k] : -1;
                    got[k] = p >= 0 && p < v && token_ok(t) ? edge_pre(p, t) : 0.f;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (e + k < e1) s_pre[e + k] = got[k];
            }
        }
    }
    flags |= mid();
    __syncthreads();
    // The accepted steps.  A node's thread writes its accepted parents over the front of its parent list.
    auto accepted = [&](int e, int p, int v, int t) -> bool {
        return token_ok(t) && step_ok(!kFetch ? 0.f : cached ? s_pre[e] : edge_pre(p, t), p, v, t);
    };
    // Up to three of them sit in a register, ten bits each (fewer: some of them twice), -1 when there is none;
    // with more the list is walked.
    constexpr int kHeld = 3;
    int held[kPathNodeSlots], n_acc[kPathNodeSlots];       // of the thread's nodes
    bool many = false;
#pragma unroll
    for (int k = 0; k < kPathNodeSlots; ++k) {
        const int v = tid + k * kPathThreads;
        int n = 0, h = -1;
        if (v > 0 && v < N) {
            const int e0 = s_ptr[v], e1 = s_ptr[v + 1], t = s_tok[v];
            for (int e = e0; e < e1; ++e) {
                const int p = parent_at(e);
                if ((unsigned)p >= (unsigned)v) {
                    flags |= GSD_DEV_BAD_CSR;
                    continue;
                }
                s_child[p] = 1;
                if (!accepted(e, p, v, t)) continue;
                if (n < kHeld) h = n == 0 ? p * 0x100401 : n == 1 ? (h & 1023) | p * 0x100400 : (h & 0xFFFFF) | p << 20;
                if (cached) s_edge[e0 + n] = p;
                ++n;
            }
        }
        held[k] = h;
        n_acc[k] = n;
        many |= n > kHeld;
    }
    // calls f(p) for every accepted parent of the thread's k-th node, of which there is one at least
    auto each_accepted = [&](int k, auto f) {
#pragma unroll
        for (int j = 0; j < kHeld; ++j) f(held[k] >> (10 * j) & 1023);
        if (many && n_acc[k] > kHeld) {
            const int v = tid + k * kPathThreads, e0 = s_ptr[v];
            if (cached) {
                for (int e = e0 + kHeld; e < e0 + n_acc[k]; ++e) f(s_edge[e]);
            } else {
                for (int e = e0; e < s_ptr[v + 1]; ++e) {
                    const int p = io.pidx[e];
                    if (p >= 0 && p < v && accepted(e, p, v, s_tok[v])) f(p);
                }
            }
        }
    };

    // Level-synchronous relaxation: after round r every node whose longest accepted root path has at
    // most r edges is final.  Values only grow, so a node may be met before or after its parent's update of
    // the round, and it stops when nothing changed.
    volatile int* best = s_best;
    int mine[kPathNodeSlots];
#pragma unroll
    for (int k = 0; k < kPathNodeSlots; ++k) mine[k] = tid + k * kPathThreads == 0 ? 0 : -1;
    for (int round = 0; round < N; ++round) {
        int changed = 0;
#pragma unroll
        for (int k = 0; k < kPathNodeSlots; ++k) {
            if (held[k] < 0) continue;
            int from = -1;
            each_accepted(k, [&](int p) { from = max(from, best[p]); });
            if (from >= 0 && from + 1 > mine[k]) {
                mine[k] = from + 1;
                best[tid + k * kPathThreads] = mine[k];
                changed = 1;
            }
        }
        if (!__syncthreads_or(changed)) break;
    }

    // every node's predecessor: the lowest one with an accepted step that carries length - 1; and the end
    // node: longest, then lowest index
    int key = tid == 0 ? 1023 : -1;                        // (the root: length 0)
#pragma unroll
    for (int k = 0; k < kPathNodeSlots; ++k) {
        const int v = tid + k * kPathThreads;
        if (mine[k] < 1) continue;
        int pred = N;
        each_accepted(k, [&](int p) {
            if (p < pred && best[p] == mine[k] - 1) pred = p;
        });
        s_pred[v] = (short)(pred == N ? 0 : pred);
        key = max(key, (mine[k] << 10) | (1023 - v));
    }
    key = __reduce_max_sync(0xFFFFFFFFu, key);
    if ((tid & 31) == 0) s_red[tid >> 5] = key;
    if (flags) atomicOr(&s_flags, flags);
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kPathThreads / 32; ++w) key = max(key, s_red[w]);
    const int m = key >> 10, end = 1023 - (key & 1023);
    if (tid == 0) {
        unsigned fl = s_flags;
        if (m + 1 > io.Tcap) fl |= GSD_DEV_TCAP;
        int v = end;
        for (int l = m; l > 0; --l) {
            s_path[l] = (short)v;
            v = s_pred[v];
        }
        s_path[0] = (short)v;
        *io.out_len = m + 1;
        if (fl && io.status) atomicOr((unsigned*)io.status, fl);
    }
    __syncthreads();
    for (int i = tid; i <= io.Tcap; i += kPathThreads) {
        if (i <= m) {
            const int node = s_path[i];
            if (!GSD_IN_BOUNDS(node >= 0 && node < N && i < GSD_MAX_NODES, io.status)) continue;
            if (io.out_nodes && i < io.Tcap) io.out_nodes[i] = node;
            if (i >= 1) io.out_tok[i - 1] = s_tok[node];    // i - 1 < Tcap
        } else if (i < io.Tcap) {
            io.out_tok[i] = -1;
            if (io.out_nodes) io.out_nodes[i] = -1;
        }
    }
    return PathResult{m, end, s_child[end] != 0};
}

}  // namespace gsd
