// gsd_draft_expand: one growth step of the draft token graph (Sec. 4: token tree of out-degree
// k; Sec. 4.2: probability pruning and sibling pruning; Sec. 5.2: tau-redundant nodes; Sec. 5.3:
// merge edges to the first occurrence).
//
// Two launches.  Grid (F, B): the CTA of frontier row (b, fi) - a cluster of them when there are
// few rows - streams that row of draft logits once with 16-byte loads (softmax statistics and
// every thread's best), picks the row's k best, and leaves tokens and probabilities in scratch.
// The second launch (one CTA per sequence, a programmatic dependent of the first) appends the
// children (k per frontier node, in frontier order), applies the two pruning rules, looks for
// an earlier node with the same tau-gram for every new node (first occurrence = lowest id),
// and compacts the new frontier.
#include "gsd_internal.cuh"
#include "gsd_binding.h"
#include <math_constants.h>

namespace gsd {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int K = GSD_DRAFT_MAX_K;
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kNone = 0x7FFFFFFF;      // "no token": ranks behind every token
constexpr int kMaxCluster = 8;

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// a candidate ranks before another if its logit is larger, or equal with the lower token id
__device__ __forceinline__ bool before(float va, int ia, float vb, int ib) {
    return va > vb || (va == vb && ia < ib);
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

struct TopK {
    float v[K];
    int i[K];
};

// insertion into the thread's list (descending).  A thread meets its elements in ascending
// index order, so an equal value never displaces an earlier one.
__device__ __forceinline__ void offer(TopK& t, float x, int idx) {
    if (!(x > t.v[K - 1])) return;
#pragma unroll
    for (int j = K - 1; j >= 0; --j) {
        const bool up = j > 0 && x > t.v[j - 1];     // the slot above also has to move down
        if (up) {
            t.v[j] = t.v[j - 1];
            t.i[j] = t.i[j - 1];
        } else {
            t.v[j] = x;
            t.i[j] = idx;
            break;
        }
    }
}

struct DraftArgs {
    const float* logits;
    const int32_t* frontier;
    const int32_t* frontier_len;
    int32_t* tokens;
    int32_t* tree_parent;
    int32_t* merge_to;
    uint8_t* leaf;
    float* prob;
    int32_t* num_nodes;
    int32_t* new_frontier;
    int32_t* new_frontier_len;
    int32_t* wk_tok;     // [B,F,K]
    float* wk_q;         // [B,F,K]
    int32_t* status;
    int B, F, V, Ncap, k, tau;
    int cluster;         // CTAs per row of logits
    int pad;             // fill the rest of new_frontier with -1
    float theta_prob, theta_sib;
};

__device__ void grow_sequence(const DraftArgs& a, int b) {
    __shared__ int s_tok[GSD_MAX_NODES];
    __shared__ int s_par[GSD_MAX_NODES];
    __shared__ unsigned char s_leaf[GSD_MAX_NODES];
    __shared__ __align__(16) unsigned s_key[GSD_MAX_NODES];   // hash of the tau-gram that ends at a node (kNoGram: none)
    __shared__ int s_cnt[kWarps];
    constexpr int kHashBits = 10, kHashSlots = 1 << kHashBits;     // twice the largest node count
    __shared__ unsigned s_hkey[kHashSlots];
    __shared__ int s_hmin[kHashSlots];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int Ncap = a.Ncap, k = a.k;
    int32_t* tok = a.tokens + (size_t)b * Ncap;
    int32_t* par = a.tree_parent + (size_t)b * Ncap;
    int32_t* mrg = a.merge_to + (size_t)b * Ncap;
    uint8_t* leaf = a.leaf + (size_t)b * Ncap;
    float* prob = a.prob + (size_t)b * Ncap;
    unsigned flags = 0;
    int n0 = a.num_nodes[b];
    int fl = a.frontier_len[b];
    if (n0 < 1 || n0 > Ncap || fl < 0 || fl > a.F) {
        // nothing sensible can be appended: leave the graph as it is
        wait_for_predecessor();                                // (this grid never ends before the first launch)
        if (a.pad)
            for (int i = tid; i < a.F * k; i += kThreads) a.new_frontier[(size_t)b * a.F * k + i] = -1;
        if (tid == 0) {
            a.new_frontier_len[b] = 0;
            if (a.status) atomicOr((unsigned*)a.status, GSD_DEV_BAD_FRONTIER);
        }
        return;
    }
    int want = fl * k;
    if (n0 + want > Ncap) {
        want = Ncap - n0;
        flags |= GSD_DEV_DRAFT_FULL;
    }
    const int n1 = n0 + want;
    // Everything that does not need the row kernel's results comes first - this kernel is its
    // programmatic dependent and is resident while it still runs: the graph as it stands, the
    // parents of the children to come, the tau-gram hashes of the old nodes and their entries in
    // the hash table.
    constexpr int kChildSlots = (GSD_MAX_NODES + kThreads - 1) / kThreads;
    int p_child[kChildSlots];
#pragma unroll
    for (int s = 0; s < kChildSlots; ++s) {
        const int j = tid + s * kThreads;
        int p = 0;
        if (j < want) {
            p = a.frontier[(size_t)b * a.F + j / k];
            if (p < 0 || p >= n0) {
                flags |= GSD_DEV_BAD_FRONTIER;
                p = 0;
            }
        }
        p_child[s] = p;
    }
    for (int v = tid; v < n0; v += kThreads) {
        s_tok[v] = tok[v];
        s_par[v] = par[v];
    }
    constexpr unsigned kNoGram = 0xFFFFFFFFu;
    for (int t = tid; t < kHashSlots; t += kThreads) {
        s_hkey[t] = kNoGram;
        s_hmin[t] = 0x7FFFFFFF;
    }
    __syncthreads();
    // Sec. 5.2 / 5.3: a new node whose last tau tokens along its tree path equal those of an
    // earlier node is redundant; it becomes a leaf that points at the first such node.
    // Every node's tau-gram is reduced to a 32-bit hash; equal hashes are confirmed token by token.
    auto gram_key = [&](int v) -> unsigned {
        unsigned h = 2166136261u;
        int x = v, t = 0;
        for (; t < a.tau && x >= 0; ++t) {
            h = (h ^ (unsigned)s_tok[x]) * 16777619u;
            h ^= h >> 15;
            x = s_par[x];
        }
        return (t == a.tau) ? (h == kNoGram ? 0u : h) : kNoGram;
    };
    // first occurrences through a hash table in shared memory: every node with a tau-gram enters
    // its id under its hash (open addressing; the slot keeps the lowest id), so a new node finds
    // the lowest earlier node with its hash in one probe sequence instead of a scan over all
    // earlier nodes.  Equal hashes are confirmed token by token; if the lowest id under the hash
    // is a different gram (a collision of the 32-bit hash) the node falls back to the scan.
    auto enter = [&](int v) {
        const unsigned kv = gram_key(v);
        s_key[v] = kv;
        if (kv == kNoGram) return;
        unsigned slot = (kv * 2654435761u) >> (32 - kHashBits);
        for (int probe = 0; probe < kHashSlots; ++probe) {
            const unsigned prev = atomicCAS(&s_hkey[slot], kNoGram, kv);
            if (prev == kNoGram || prev == kv) {
                atomicMin(&s_hmin[slot], v);
                break;
            }
            slot = (slot + 1) & (kHashSlots - 1);
        }
    };
    for (int v = tid; v < n0; v += kThreads) enter(v);

    // the children: k per frontier node, in frontier order, best first
    wait_for_predecessor();
#pragma unroll
    for (int s = 0; s < kChildSlots; ++s) {
        const int j = tid + s * kThreads;
        if (j >= want) continue;
        const int fi = j / k, i = j % k, c = n0 + j;
        const size_t w = ((size_t)b * a.F + fi) * K;
        if (!GSD_IN_BOUNDS(c < Ncap && fi < a.F && i < K, a.status)) continue;
        const float q = a.wk_q[w + i], qmax = a.wk_q[w];
        s_tok[c] = a.wk_tok[w + i];
        s_par[c] = p_child[s];
        // Sec. 4.2: below the probability threshold, or too far below the best sibling
        s_leaf[c] = (q < a.theta_prob) || (q < a.theta_sib * qmax);
        prob[c] = q;
    }
    __syncthreads();
    for (int v = n0 + tid; v < n1; v += kThreads) enter(v);
    auto same_gram = [&](int x, int y) -> bool {
        for (int t = 0; t < a.tau; ++t) {
            if (x < 0 || y < 0 || s_tok[x] != s_tok[y]) return false;
            x = s_par[x];
            y = s_par[y];
        }
        return true;
    };
    __syncthreads();
    for (int j = tid; j < want; j += kThreads) {
        const int c = n0 + j;
        const unsigned kc = s_key[c];
        int first = -1;
        if (kc != kNoGram) {
            unsigned slot = (kc * 2654435761u) >> (32 - kHashBits);
            int lowest = c;
            for (int probe = 0; probe < kHashSlots; ++probe) {
                const unsigned k = s_hkey[slot];
                if (k == kc) { lowest = s_hmin[slot]; break; }
                if (k == kNoGram) break;                       // (cannot happen: c itself is in the table)
                slot = (slot + 1) & (kHashSlots - 1);
            }
            if (lowest < c) {
                if (same_gram(c, lowest)) {
                    first = lowest;
                } else {
                    // another gram with the same hash sits below: look at every earlier node
                    for (int e = 0; e < c && first < 0; ++e)
                        if (s_key[e] == kc && same_gram(c, e)) first = e;
                }
            }
        }
        if (first >= 0) s_leaf[c] = 1;
        tok[c] = s_tok[c];
        par[c] = s_par[c];
        mrg[c] = first;
        leaf[c] = s_leaf[c];
    }
    __syncthreads();
    // the new frontier: the new nodes that are not leaves, in id order
    int32_t* nf = a.new_frontier + (size_t)b * a.F * k;
    int base = 0;
    for (int j0 = 0; j0 < want; j0 += kThreads) {
        const int j = j0 + tid;
        const bool keep = j < want && !s_leaf[n0 + j];
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, keep);
        if (lane == 0) s_cnt[warp] = __popc(bal);
        __syncthreads();
        int off = base;
        for (int w = 0; w < warp; ++w) off += s_cnt[w];
        if (keep && GSD_IN_BOUNDS(off + __popc(bal & ((1u << lane) - 1u)) < a.F * k, a.status))
            nf[off + __popc(bal & ((1u << lane) - 1u))] = n0 + j;
        for (int w = 0; w < kWarps; ++w) base += s_cnt[w];
        __syncthreads();
    }
    if (a.pad)
        for (int i = base + tid; i < a.F * k; i += kThreads) nf[i] = -1;
    if (tid == 0) {
        a.new_frontier_len[b] = base;
        a.num_nodes[b] = n1;
    }
    if (flags && a.status) atomicOr((unsigned*)a.status, flags);
}

// Block-wide pick of the best remaining (value, index) pair, ranked by `before`; every thread
// passes its own proposal and gets the winner (and the proposing thread) back.
__device__ __forceinline__ void block_best(float& v, int& i, int& owner, float* s_rv, int* s_ri, int* s_rt) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float v2 = __shfl_xor_sync(0xFFFFFFFFu, v, o);
        const int i2 = __shfl_xor_sync(0xFFFFFFFFu, i, o), t2 = __shfl_xor_sync(0xFFFFFFFFu, owner, o);
        if (before(v2, i2, v, i)) { v = v2; i = i2; owner = t2; }
    }
    if (lane == 0) { s_rv[warp] = v; s_ri[warp] = i; s_rt[warp] = owner; }
    __syncthreads();
    v = s_rv[0]; i = s_ri[0]; owner = s_rt[0];
    for (int q = 1; q < kWarps; ++q)
        if (before(s_rv[q], s_ri[q], v, i)) { v = s_rv[q]; i = s_ri[q]; owner = s_rt[q]; }
    __syncthreads();
}

// The k best tokens of one row of logits and their probabilities, in one pass over the row.
// Every thread streams its strided share (16-byte loads, a batch in flight while one is worked
// through) and keeps the running (maximum, sum of exponentials) pair, the best (logit, token) pair
// it has met and the VALUE of its second best entry - all without a branch, so that no lane of a
// warp waits for another's rare update.  The 256 best pairs are picked over in two stages (ranked
// by logit, ties to the lower token id): every warp picks the k best of its 32 pairs, then one
// warp picks the k best of those 8 k.  That is the exact answer unless some thread's second best
// entry ranks at or before the k-th pick - then an entry that no thread offered could belong
// to the k best; the shares of such threads are looked at once more.  Only a list of more than
// 512 such entries (long runs of equal logits) takes the slow exact way: every thread keeps the K
// best pairs it meets and the block merges the 256 lists.
// What bounds it (8 x 64 rows of 32000, k 4, 66 MB): DRAM for the first 8 to 10 us, then the pick
// of the row that finishes last.
constexpr int kBatch = 4;     // 16-byte loads of a batch; the next batch is on the way while one is worked through
struct Best {
    float v1, v2;   // best and second best logit of the thread's share (v2: value only)
    int i1;         // token of the best
};
// While a row is streamed the best is kept per 16-byte group - its maximum and which group - and
// the token inside the group is looked up once at the end: 2 instructions per entry instead of 6.
// `v2` then bounds the entries outside the best group.  `where`: group number, or ~index of a
// lone entry.
__device__ __forceinline__ void offer_group(Best& t, float x, int where) {
    // a thread meets its groups in ascending order: an equal logit never displaces an earlier one
    const bool up = x > t.v1;
    t.v2 = fmaxf(t.v2, up ? t.v1 : x);
    t.i1 = up ? where : t.i1;
    t.v1 = fmaxf(t.v1, x);
}
// Monotone map of the logits (no NaN here; -0 folded onto +0) to unsigned words, in which the warp
// can take a maximum with one instruction; 0 stands for "no pair".
__device__ __forceinline__ unsigned ordered(float v) {
    const unsigned u = __float_as_uint(v == 0.f ? 0.f : v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float from_ordered(unsigned o) {
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o);
}

// One warp picks the k best of the pairs its lanes hold, kSlots each, ranked by `before`.  A round is
// two warp-wide reductions (largest logit, then lowest token among those); with shuffle trees
// the two stages of picks took most of the 4 us between the last load of a row and its result.
// done(r, v, i) is called by all lanes with the r-th pick; i == kNone: no pair above -inf is left.
template <int kSlots, class Done>
__device__ __forceinline__ void warp_pick_k(float (&cv)[kSlots], int (&ci)[kSlots], int k, Done done) {
    unsigned key[kSlots];
#pragma unroll
    for (int j = 0; j < kSlots; ++j) key[j] = ci[j] == kNone || cv[j] == -CUDART_INF_F ? 0u : ordered(cv[j]);
    for (int r = 0; r < k; ++r) {
        unsigned mine = key[0];
#pragma unroll
        for (int j = 1; j < kSlots; ++j) mine = max(mine, key[j]);
        const unsigned top = __reduce_max_sync(0xFFFFFFFFu, mine);
        int low = kNone;
#pragma unroll
        for (int j = 0; j < kSlots; ++j) low = key[j] == top ? min(low, ci[j]) : low;
        low = top == 0u ? kNone : __reduce_min_sync(0xFFFFFFFFu, low);
#pragma unroll
        for (int j = 0; j < kSlots; ++j)
            if (key[j] == top && ci[j] == low) key[j] = 0u;
        done(r, top == 0u ? -CUDART_INF_F : from_ordered(top), low);
    }
}
// The same for `count` <= 32 * kSlots pairs in shared memory; the picks go to out_v / out_i (token
// -1: none was left).
template <int kSlots>
__device__ __forceinline__ void warp_pick_k(const float* s_cv, const int* s_ci, int count, int k, float* out_v, int* out_i) {
    const int lane = threadIdx.x & 31;
    float cv[kSlots];
    int ci[kSlots];
#pragma unroll
    for (int j = 0; j < kSlots; ++j) {
        const bool in = lane + 32 * j < count;
        cv[j] = in ? s_cv[lane + 32 * j] : -CUDART_INF_F;
        ci[j] = in ? s_ci[lane + 32 * j] : kNone;
    }
    warp_pick_k<kSlots>(cv, ci, k, [&](int r, float v, int i) {
        if (lane == 0) {
            out_v[r] = v;
            out_i[r] = i == kNone ? -1 : i;
        }
    });
}

// ---- thread-block cluster: the CTAs that share a row
__device__ __forceinline__ int cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// writes `v` to the place of *dst in the leading CTA of the cluster
__device__ __forceinline__ void put_leader(void* dst, uint32_t v) {
    uint32_t at;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(dst)));
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}

// The row's CTAs (a cluster; usually one) share it in contiguous slices; each finds the k best of
// its slice and the leading one picks the row's among those.
__global__ void __launch_bounds__(kThreads, 4) draft_expand_kernel(DraftArgs a) {
    __shared__ float s_cv[2 * kThreads];
    __shared__ int s_ci[2 * kThreads];
    __shared__ float s_rv[kWarps];
    __shared__ int s_ri[kWarps], s_rt[kWarps];
    __shared__ float s_m[kWarps], s_s[kWarps];
    __shared__ int s_flagged, s_count;
    __shared__ short s_flag[kThreads];     // threads whose share has to be looked at again
    __shared__ float s_bv[K];              // the k best of the slice
    __shared__ int s_bi[K];
    __shared__ float s_pv[kMaxCluster * K], s_pm[kMaxCluster], s_ps[kMaxCluster];   // what the cluster's CTAs hand in
    __shared__ int s_pi[kMaxCluster * K];
    wait_for_predecessor();
    // the per-sequence pass may become resident as CTAs retire; it reads the graph before it waits
    if (threadIdx.x == 0) let_successor_start();
    const int C = a.cluster, slice = C > 1 ? cluster_rank() : 0;
    const int fi = (int)blockIdx.x / C, b = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int V = a.V;
    const int fl = a.frontier_len[b];
    if (fi >= fl || fl > a.F) return;      // (all CTAs of a cluster alike; such rows are not read)
    if (C > 1) cluster_arrive();           // every CTA has started before any writes to another
    const float* x = a.logits + ((size_t)b * a.F + fi) * V;
    // The CTA's slice: 16-byte groups v0 .. v1, the entries before the first 16-byte boundary (first
    // slice) and those behind the last group (last slice).  Threads meet theirs in ascending order.
    const RowSpan sp = row_span(x, V);
    const float4* x4 = reinterpret_cast<const float4*>(x + sp.head);
    const int per = (sp.nvec + C - 1) / C;
    const int v0 = min(slice * per, sp.nvec), v1 = min(v0 + per, sp.nvec);
    const int e_head = slice == 0 && tid < sp.head ? tid : -1;
    const int e_tail = slice == C - 1 && sp.head + 4 * sp.nvec + tid < V ? sp.head + 4 * sp.nvec + tid : -1;
    float m = -CUDART_INF_F, s = 0.f;        // running maximum and sum
    Best best{-CUDART_INF_F, -CUDART_INF_F, kNone};
    auto take = [&](float val, int idx) {
        offer_group(best, val, ~idx);
        if (val > m) {
            s = s * ex2((m - val) * kLog2e) + 1.f;
            m = val;
        } else if (val > -CUDART_INF_F) {
            s += ex2((val - m) * kLog2e);
        } else if (val != val) {
            s = val;    // NaN poisons the sum and is reported below
        }
    };
    {
        const float4 none = make_float4(-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F);
        auto fetch = [&](float4 (&r)[kBatch], int i) {
#pragma unroll
            for (int k = 0; k < kBatch; ++k) r[k] = i + k * kThreads < v1 ? __ldcs(x4 + i + k * kThreads) : none;
        };
        auto work = [&](float4 (&r)[kBatch], int i) {
            float g = m;
#pragma unroll
            for (int k = 0; k < kBatch; ++k) {
                const float g4 = max3(fmaxf(r[k].x, r[k].y), r[k].z, r[k].w);
                g = fmaxf(g, g4);
                offer_group(best, g4, i + k * kThreads);
            }
            float ref = g;
            if (!(fabsf(g) <= kLargeLogit)) {
                if (g == -CUDART_INF_F) {
                    // nothing finite yet: a NaN would otherwise go unnoticed (below it poisons the sum)
#pragma unroll
                    for (int k = 0; k < kBatch; ++k) {
                        const float t = (r[k].x + r[k].y) + (r[k].z + r[k].w);
                        if (t != t) s = t;
                    }
                    return;
                }
#pragma unroll
                for (int k = 0; k < kBatch; ++k) r[k] = minus(r[k], g);
                ref = 0.f;
            }
            // One rescale per batch.  The rounding of ref * log2 e (2^-21 at a logit of 12) would be a
            // factor on every term, while the probabilities at the end use v - maximum: the
            // batch's sum is brought back by what was rounded off.
            const float kk = -ref * kLog2e, off = fmaf(-ref, kLog2e, -kk);
            float acc = 0.f;
#pragma unroll
            for (int k = 0; k < kBatch; ++k)
                acc += (ex2(fmaf(r[k].x, kLog2e, kk)) + ex2(fmaf(r[k].y, kLog2e, kk))) + (ex2(fmaf(r[k].z, kLog2e, kk)) + ex2(fmaf(r[k].w, kLog2e, kk)));
            s = fmaf(s, ex2((m - g) * kLog2e), acc * ex2(off));
            m = g;
        };
        constexpr int kStep = kBatch * kThreads;
        float4 ra[kBatch], rb[kBatch];
        fetch(ra, v0 + tid);
        if (e_head >= 0) take(__ldcs(x + e_head), e_head);
        for (int i = v0 + tid; i < v1; i += 2 * kStep) {
            fetch(rb, i + kStep);                // on the way while the other batch is worked through
            work(ra, i);
            fetch(ra, i + 2 * kStep);
            if (i + kStep < v1) work(rb, i + kStep);
        }
        if (e_tail >= 0) take(__ldcs(x + e_tail), e_tail);
    }
    // the token of the best, and the best of the other entries of its group
    if (best.i1 != kNone) {
        if (best.i1 < 0) {
            best.i1 = ~best.i1;
        } else {
            const float4 r = x4[best.i1];
            const float q[4] = {r.x, r.y, r.z, r.w};
            int at = 3;
#pragma unroll
            for (int j = 2; j >= 0; --j)
                if (q[j] == best.v1) at = j;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j != at) best.v2 = fmaxf(best.v2, q[j]);
            best.i1 = sp.head + 4 * best.i1 + at;
        }
    }
    // stage 1: every warp picks the k best of its 32 pairs
    {
        float cv[1] = {best.v1};
        int ci[1] = {best.i1};
        warp_pick_k<1>(cv, ci, a.k, [&](int r, float v, int i) {
            if (lane == 0) { s_cv[warp * a.k + r] = v; s_ci[warp * a.k + r] = i; }
        });
    }
    // (maximum, sum) of the warp's entries; a NaN sum stays
    {
        float wm = m;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xFFFFFFFFu, wm, o));
        float ws = wm == -CUDART_INF_F ? s : s * ex2((m - wm) * kLog2e);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ws += __shfl_xor_sync(0xFFFFFFFFu, ws, o);
        if (lane == 0) { s_m[warp] = wm; s_s[warp] = ws; }
    }
    if (tid == 0) { s_flagged = 0; s_count = a.k; }
    __syncthreads();
    // stage 2: the k best of the 8 k picks
    if (warp == 0) warp_pick_k<kWarps * K / 32>(s_cv, s_ci, kWarps * a.k, a.k, s_bv, s_bi);
    __syncthreads();
    // An entry that no thread offered can rank at or before the k-th pick only if it is in the share
    // of a thread whose second best does (about one random row in fifty has such a thread).
    const float tv = s_bv[a.k - 1];
    const int ti = s_bi[a.k - 1] < 0 ? kNone : s_bi[a.k - 1];
    const bool again = best.v2 > -CUDART_INF_F && best.v2 >= tv;
    if (again) s_flag[atomicAdd(&s_flagged, 1)] = (short)tid;
    if (__syncthreads_or(again)) {
        // Those shares are read once more (from L2; a warp takes a share, so a row of 32000 is one
        // trip), and the k picks together with what ranks at or before the last of them and
        // had not been offered make a short list that holds the k best.  (Reading the whole row again
        // took 8 us instead of 2.5, for 15 of 512 rows, and the call waits for the last row.)
        if (tid < a.k) { s_cv[tid] = s_bv[tid]; s_ci[tid] = s_bi[tid] < 0 ? kNone : s_bi[tid]; }
        __syncthreads();
        auto consider = [&](float val, int idx) {
            if (val == -CUDART_INF_F || !(val > tv || (val == tv && idx <= ti))) return;
            for (int r = 0; r < a.k; ++r)
                if (s_bi[r] == idx) return;
            const int slot = atomicAdd(&s_count, 1);
            if (slot < 2 * kThreads) { s_cv[slot] = val; s_ci[slot] = idx; }
        };
        for (int f = warp; f < s_flagged; f += kWarps) {
            const int t = s_flag[f];
            if (lane == 0 && slice == 0 && t < sp.head) consider(x[t], t);
            if (lane == 0 && slice == C - 1 && sp.head + 4 * sp.nvec + t < V) consider(x[sp.head + 4 * sp.nvec + t], sp.head + 4 * sp.nvec + t);
            for (int i = v0 + t + lane * kThreads; i < v1; i += 32 * kThreads) {
                const float4 r = x4[i];
                const int e = sp.head + i * 4;
                consider(r.x, e); consider(r.y, e + 1); consider(r.z, e + 2); consider(r.w, e + 3);
            }
        }
        __syncthreads();
        const int count = s_count;
        if (count <= 2 * kThreads) {
            if (warp == 0) warp_pick_k<2 * kThreads / 32>(s_cv, s_ci, count, a.k, s_bv, s_bi);
        } else {
            // more than 512 entries rank before the bound (long runs of equal logits in one thread's
            // share): per-thread lists of the K best pairs, merged by the block
            TopK t;
#pragma unroll
            for (int j = 0; j < K; ++j) {
                t.v[j] = -CUDART_INF_F;
                t.i[j] = kNone;
            }
            if (e_head >= 0) offer(t, x[e_head], e_head);
            for (int i = v0 + tid; i < v1; i += kThreads) {
                const float4 r = x4[i];
                const int e = sp.head + 4 * i;
                offer(t, r.x, e); offer(t, r.y, e + 1); offer(t, r.z, e + 2); offer(t, r.w, e + 3);
            }
            if (e_tail >= 0) offer(t, x[e_tail], e_tail);
            int head = 0;
            for (int r = 0; r < a.k; ++r) {
                float v = -CUDART_INF_F;
                int i = kNone;
#pragma unroll
                for (int j = 0; j < K; ++j)
                    if (j == head) { v = t.v[j]; i = t.i[j]; }
                int owner = tid;
                block_best(v, i, owner, s_rv, s_ri, s_rt);
                if (owner == tid && i != kNone) ++head;
                if (tid == 0) {
                    s_bv[r] = v;
                    s_bi[r] = i == kNone ? -1 : i;       // fewer than k entries above -inf
                }
            }
        }
        __syncthreads();
    }
    // (maximum, sum) of `n` parts of the row
    auto sum_up = [](const float* pm, const float* ps, int n, float& rm, float& rs) {
        rm = -CUDART_INF_F;
        for (int q = 0; q < n; ++q) rm = fmaxf(rm, pm[q]);
        rs = 0.f;
        for (int q = 0; q < n; ++q) rs += rm == -CUDART_INF_F ? ps[q] : ps[q] * ex2((pm[q] - rm) * kLog2e);
    };
    float rm, rs;
    sum_up(s_m, s_s, kWarps, rm, rs);
    if (C > 1) {
        // hand the slice's result to the leading CTA, which picks the row's k best
        cluster_wait();
        if (tid < a.k) {
            put_leader(s_pv + slice * a.k + tid, __float_as_uint(s_bi[tid] < 0 ? -CUDART_INF_F : s_bv[tid]));
            put_leader(s_pi + slice * a.k + tid, (uint32_t)(s_bi[tid] < 0 ? kNone : s_bi[tid]));
        }
        if (tid == 0) {
            put_leader(s_pm + slice, __float_as_uint(rm));
            put_leader(s_ps + slice, __float_as_uint(rs));
        }
        cluster_arrive();
        cluster_wait();
        if (slice != 0) return;
        if (warp == 0) warp_pick_k<kMaxCluster * K / 32>(s_pv, s_pi, C * a.k, a.k, s_bv, s_bi);
        __syncthreads();
        sum_up(s_pm, s_ps, C, rm, rs);
    }
    if (tid < a.k) {
        const size_t w = ((size_t)b * a.F + fi) * K;
        const bool none = s_bi[tid] < 0;
        a.wk_tok[w + tid] = s_bi[tid];
        a.wk_q[w + tid] = none ? 0.f : ex2((s_bv[tid] - rm) * kLog2e) / rs;
        if ((none || !(rs > 0.f) || rm == CUDART_INF_F) && a.status) atomicOr((unsigned*)a.status, GSD_DEV_BAD_LOGITS);
    }
}

// Second launch: one CTA per sequence appends the children and updates the graph once every
// row's result of the first launch is visible.
__global__ void __launch_bounds__(kThreads) draft_grow_kernel(DraftArgs a) {
    let_successor_start();
    grow_sequence(a, blockIdx.x);        // (waits for the first launch inside, as late as it can)
}

// CTAs per row of logits: with fewer rows than half the SMs the rows are shared, down to 4096
// entries (four rounds of a CTA's loads) per CTA.  8 rows of 128256: 25.3 us in one CTA each, 16.9
// in eight.  With more rows sharing does not pay, since every slice has to find its own k best and
// the slices without an outstanding entry need the second look more often: 120 rows of 32000, k 8:
// 24.3 us in one CTA each, 26.1 in two, 27.9 in four (before the second look became cheap).
int pick_cluster(long rows, int V, int sm_count) {
    int c = 1;
    while (c < kMaxCluster && rows * c * 2 <= sm_count && V / (c * 2) >= 4096) c *= 2;
    return c;
}

}  // namespace
}  // namespace gsd

extern "C" size_t gsd_draft_expand_workspace_bytes(const gsd_draft_params* p) {
    if (!p || p->B < 1 || p->F < 1) return 0;
    return gsd::align_up((size_t)p->B * p->F * GSD_DRAFT_MAX_K * 8, 256);
}

static int draft_expand(const float* logits, const int32_t* frontier, const int32_t* frontier_len,
                        int32_t* tokens, int32_t* tree_parent, int32_t* merge_to, uint8_t* leaf,
                        float* prob, int32_t* num_nodes, int32_t* new_frontier,
                        int32_t* new_frontier_len, const gsd_draft_params* p, void* workspace,
                        size_t workspace_bytes, int32_t* status, void* stream, bool pad) {
    using namespace gsd;
    if (!p || !logits || !frontier || !frontier_len || !tokens || !tree_parent || !merge_to || !leaf ||
        !prob || !num_nodes || !new_frontier || !new_frontier_len)
        return GSD_ERR_NULL_POINTER;
    if (p->B < 1 || p->B > 65535 || p->F < 1 || p->V < 1 || p->Ncap < 1 || p->Ncap > GSD_MAX_NODES ||
        p->k < 1 || p->k > GSD_DRAFT_MAX_K || p->k > p->V || p->tau < 1 || p->tau > GSD_MAX_NODES)
        return GSD_ERR_BAD_SHAPE;
    if (((uintptr_t)logits & 3u) != 0) return GSD_ERR_MISALIGNED;
    const size_t need = gsd_draft_expand_workspace_bytes(p);
    if (!workspace || workspace_bytes < need) return GSD_ERR_WORKSPACE;
    if (((uintptr_t)workspace & 7u) != 0) return GSD_ERR_MISALIGNED;
    DeviceInfo di;
    if (device_info(&di) != 0) return GSD_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    DraftArgs a;
    a.logits = logits; a.frontier = frontier; a.frontier_len = frontier_len;
    a.tokens = tokens; a.tree_parent = tree_parent; a.merge_to = merge_to; a.leaf = leaf; a.prob = prob;
    a.num_nodes = num_nodes; a.new_frontier = new_frontier; a.new_frontier_len = new_frontier_len;
    const size_t rows = (size_t)p->B * p->F * GSD_DRAFT_MAX_K;
    a.wk_tok = (int32_t*)workspace;
    a.wk_q = (float*)((char*)workspace + rows * 4);
    a.status = status;
    a.B = p->B; a.F = p->F; a.V = p->V; a.Ncap = p->Ncap; a.k = p->k; a.tau = p->tau;
    a.theta_prob = p->theta_prob; a.theta_sib = p->theta_sib;
    a.pad = pad;
    // every scratch entry is written before it is read: nothing has to start at zero
    a.cluster = pick_cluster((long)p->B * p->F, p->V, di.sm_count);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    dependent_launch_attr(attr);
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)a.cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)p->F * (unsigned)a.cluster, (unsigned)p->B);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = a.cluster > 1 ? 2 : 1;
    GSD_CUDA_TRY(cudaLaunchKernelEx(&cfg, draft_expand_kernel, a));
    GSD_CUDA_TRY(launch_dependent(draft_grow_kernel, dim3((unsigned)p->B), dim3(kThreads), 0, st, a));
    return GSD_OK;
}

extern "C" int gsd_draft_expand(const float* logits, const int32_t* frontier, const int32_t* frontier_len,
                                int32_t* tokens, int32_t* tree_parent, int32_t* merge_to, uint8_t* leaf,
                                float* prob, int32_t* num_nodes, int32_t* new_frontier,
                                int32_t* new_frontier_len, const gsd_draft_params* p, void* workspace,
                                size_t workspace_bytes, int32_t* status, void* stream) {
    return draft_expand(logits, frontier, frontier_len, tokens, tree_parent, merge_to, leaf, prob, num_nodes, new_frontier,
                        new_frontier_len, p, workspace, workspace_bytes, status, stream, false);
}

extern "C" int gsd_binding_draft_expand(const float* logits, const int32_t* frontier, const int32_t* frontier_len,
                                        int32_t* tokens, int32_t* tree_parent, int32_t* merge_to, uint8_t* leaf,
                                        float* prob, int32_t* num_nodes, int32_t* new_frontier,
                                        int32_t* new_frontier_len, const gsd_draft_params* p, void* workspace,
                                        size_t workspace_bytes, int32_t* status, void* stream) {
    return draft_expand(logits, frontier, frontier_len, tokens, tree_parent, merge_to, leaf, prob, num_nodes, new_frontier,
                        new_frontier_len, p, workspace, workspace_bytes, status, stream, true);
}
