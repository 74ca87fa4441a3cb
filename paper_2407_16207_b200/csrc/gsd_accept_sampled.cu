// gsd_accept_sampled: non-deterministic verification of the draft token graph (Sec. 3: a
// drafted token is accepted with probability min(1, p/q), the first rejection ends the
// hypothesis and the target model regenerates that token; Sec. 6.4: the same on the graph).
// The random numbers are inputs.  A step parent -> v of the graph is accepted iff
//     u_accept[v] * draft_q[v] < softmax(logits[parent])[token of v];
// the hypothesis is the longest root path of accepted steps (ties as in gsd_accept), and the
// regenerated token is drawn by inverting a cumulative distribution in index order with
// u_sample: that of the residual max(0, P - Q) at the end node (P the target's, Q the draft
// model's distribution there) when drafted continuations of the end node were rejected, that of
// P itself when the end node is a leaf of the graph or no draft logits are given.
//
// Two launches.  Grid (slices, B*N): each CTA streams one slice of one logits row with 16-byte
// loads; each of its warps owns a contiguous eighth of the slice and keeps a running
// (maximum, sum of exponentials) pair, which it leaves in scratch.  The second launch (a cluster
// of up to eight CTAs per sequence, a programmatic dependent of the first, so it is resident when
// the stream ends): the leading CTA combines the pairs per node, tests the steps, runs the
// level-synchronous longest-path relaxation and walks back; then the regenerated token: range sums
// (for P those in scratch; for the residual one per warp of the cluster, formed on the spot from
// the two rows of the end node and exchanged through distributed shared memory) give the range of
// the crossing, a block-wide scan over that range gives the index.
#include "gsd_internal.cuh"
#include "gsd_path.cuh"
#include <math_constants.h>

namespace gsd {
namespace {

constexpr int kThreads = kPathThreads;
constexpr int kNone = 0x7FFFFFFF;
constexpr int kMaxSlices = 16;
constexpr int kWarps = kThreads / 32;   // each warp of a CTA sums a contiguous eighth of the CTA's slice
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kResidualFloor = 1e-6f;   // a residual mass at or below this is rounding noise

// (maximum, sum of 2^((x - maximum) * log2 e)) of a set of logits; the empty set is (-inf, 0).  A NaN
// among them is a NaN sum from then on, also while the maximum is still -inf.
struct Ms {
    float m, s;
};

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ Ms combine(Ms a, Ms b) {
    const float m = fmaxf(a.m, b.m);
    if (m == -CUDART_INF_F) return Ms{m, a.s + b.s};
    return Ms{m, a.s * ex2((a.m - m) * kLog2e) + b.s * ex2((b.m - m) * kLog2e)};
}

// sixteen values at once: one rescale of the running sum per group
__device__ __forceinline__ void take16(Ms& r, float4 a, float4 b, float4 c, float4 d) {
    const float m4 = fmaxf(fmaxf(fmaxf(a.x, a.y), fmaxf(a.z, a.w)), fmaxf(fmaxf(b.x, b.y), fmaxf(b.z, b.w)));
    const float m8 = fmaxf(fmaxf(fmaxf(c.x, c.y), fmaxf(c.z, c.w)), fmaxf(fmaxf(d.x, d.y), fmaxf(d.z, d.w)));
    const float m = fmaxf(r.m, fmaxf(m4, m8));
    float ref = m;
    if (!(fabsf(m) <= kLargeLogit)) {
        if (m == -CUDART_INF_F) {
            // nothing above -inf yet: the values add up to -inf, or to NaN if there is one
            const float t = (((a.x + a.y) + (a.z + a.w)) + ((b.x + b.y) + (b.z + b.w))) + (((c.x + c.y) + (c.z + c.w)) + ((d.x + d.y) + (d.z + d.w)));
            if (t != t) r.s = t;
            return;
        }
        // entries masked with a large negative number, sixteen of them together
        a = minus(a, m); b = minus(b, m); c = minus(c, m); d = minus(d, m);
        ref = 0.f;
    }
    // (the rounding of ref * log2 e is a factor on every term; the sum is brought back by it)
    const float k = -ref * kLog2e, off = fmaf(-ref, kLog2e, -k);
    float s = ex2(fmaf(a.x, kLog2e, k)) + ex2(fmaf(a.y, kLog2e, k)) + ex2(fmaf(a.z, kLog2e, k)) + ex2(fmaf(a.w, kLog2e, k));
    s += ex2(fmaf(b.x, kLog2e, k)) + ex2(fmaf(b.y, kLog2e, k)) + ex2(fmaf(b.z, kLog2e, k)) + ex2(fmaf(b.w, kLog2e, k));
    s += ex2(fmaf(c.x, kLog2e, k)) + ex2(fmaf(c.y, kLog2e, k)) + ex2(fmaf(c.z, kLog2e, k)) + ex2(fmaf(c.w, kLog2e, k));
    s += ex2(fmaf(d.x, kLog2e, k)) + ex2(fmaf(d.y, kLog2e, k)) + ex2(fmaf(d.z, kLog2e, k)) + ex2(fmaf(d.w, kLog2e, k));
    r.s = fmaf(r.s, ex2((r.m - m) * kLog2e), s * ex2(off));
    r.m = m;
}

__device__ __forceinline__ void take1(Ms& r, float x) {
    const bool nan = x != x;
    r = combine(r, Ms{nan ? -CUDART_INF_F : x, nan ? x : x == -CUDART_INF_F ? 0.f : 1.f});
}

// The row is cut into slices (one CTA each) and every slice into kWarps contiguous ranges (one
// warp each), in units of the row's 16-byte groups; the first range has the entries before the
// first 16-byte boundary too, the last one those behind the last group.  Range r = slice * kWarps + warp.
struct Range {
    int a0, a1;    // groups
    int lo, hi;    // entries
};
__device__ __forceinline__ Range range_of(RowSpan sp, int V, int slices, int r) {
    const int per = (sp.nvec + slices - 1) / slices;
    const int slice = r / kWarps, warp = r % kWarps;
    const int v0 = min(slice * per, sp.nvec), v1 = min(v0 + per, sp.nvec);
    const int wlen = (v1 - v0 + kWarps - 1) / kWarps;
    Range g;
    g.a0 = min(v0 + warp * wlen, v1);
    g.a1 = min(g.a0 + wlen, v1);
    g.lo = r == 0 ? 0 : sp.head + g.a0 * 4;
    g.hi = r == slices * kWarps - 1 ? V : sp.head + g.a1 * 4;
    return g;
}

struct SampledArgs {
    const float* logits;
    const float* dlogits;  // draft-model logits [B,N,V] or nullptr (then no residual is formed)
    const int32_t* tok;
    const int32_t* pptr;
    const int32_t* pidx;
    const float* q;
    const float* u;
    const float* us;
    int32_t* out_tok;
    int32_t* out_len;
    int32_t* out_nodes;
    float2* part;     // [B*N][slices][kWarps] (maximum, sum) of contiguous ranges of the row, in order
    int32_t* status;
    int B, N, V, Ecap, Tcap, slices;
    int cluster;      // CTAs of the second launch per sequence
};

// ---- thread-block cluster of the second launch
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ int cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}
// writes `v` to the place of *dst in CTA `rank` of the cluster
__device__ __forceinline__ void put_remote(void* dst, int rank, uint32_t v) {
    uint32_t at;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(dst)), "r"(rank));
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}

// four consecutive entries of a row; `vec`: they start on a 16-byte boundary
__device__ __forceinline__ float4 load4(const float* p, bool vec) {
    return vec ? __ldg(reinterpret_cast<const float4*>(p)) : make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}

constexpr int kMaxCluster = 8;

// What the leading CTA finds out and the others of the cluster need.
struct Outcome {
    int edges, end, end_has_child;
    float mx, sum;
};

__device__ void finish_sequence(const SampledArgs& a, int b) {
    __shared__ float s_mx[GSD_MAX_NODES];
    __shared__ float s_sum[GSD_MAX_NODES];
    __shared__ float s_uq[GSD_MAX_NODES];
    __shared__ int s_red[kThreads / 32];
    __shared__ float s_scan[kThreads / 32];
    __shared__ float s_rm[kThreads / 32];
    __shared__ float s_cm[kMaxCluster], s_cs[kMaxCluster];
    __shared__ float s_rsum[kMaxSlices * kWarps];
    __shared__ Outcome s_outcome;
    __shared__ int s_pick;
    const int C = a.cluster, rank = C > 1 ? cluster_rank() : 0;
    static_assert(kMaxCluster <= kMaxSlices, "one range sum per warp of the cluster");
    cluster_arrive();                    // (every CTA has started before any writes to another)
    const int N = a.N, V = a.V, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float* lg = a.logits + (size_t)b * N * V;
    const float* q = a.q + (size_t)b * N;
    const float* u = a.u + (size_t)b * N;
    // Softmax statistics of every node from the pairs of the first launch, and the left sides
    // of the step tests.  This is the first thing that needs the first launch's results: the path
    // routine calls it after the graph and one logit per step have been fetched, so those two
    // trips to memory are over when the first launch ends.
    auto combine_pairs = [&]() -> unsigned {
        unsigned flags = 0;
        asm volatile("griddepcontrol.wait;" ::: "memory");
        // a node's pairs are shared by up to four neighbouring threads when there are fewer nodes than
        // threads: with few rows the rows are cut into many slices, and one thread per node had 128
        // pairs to go through (2 sequences of N 40, V 128256: 3.7 us of the call)
        const int tpn = 4 * N <= kThreads ? 4 : 2 * N <= kThreads ? 2 : 1;
        const int quads = a.slices * (kWarps / 2) / tpn;               // float4s (two pairs each) of one thread
        // (a workspace has to be on an 8-byte boundary only; 8-byte loads throughout took up to 1.3 us more:
        // 4 x 100 rows of 50257, 34.8 -> 36.1)
        const bool by16 = (reinterpret_cast<uintptr_t>(a.part) & 15u) == 0;
        auto two_pairs = [&](const float4* at) -> float4 {
            if (by16) return __ldcg(at);
            const float2 lo = __ldcg(reinterpret_cast<const float2*>(at)), hi = __ldcg(reinterpret_cast<const float2*>(at) + 1);
            return make_float4(lo.x, lo.y, hi.x, hi.y);
        };
        for (int t = tid; t < (N * tpn + 31) / 32 * 32; t += kThreads) {
            const int v = min(t / tpn, N - 1);
            // the pairs were written by other CTAs: read them past L1
            Ms r{-CUDART_INF_F, 0.f};
            const float4* pp = reinterpret_cast<const float4*>(a.part + ((size_t)b * N + v) * a.slices * kWarps) + (t % tpn) * quads;
            for (int k = 0; k < quads; k += 4) {                       // eight pairs (64 bytes) per round, loaded at once
                float4 p[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) p[i] = k + i < quads ? two_pairs(pp + k + i) : make_float4(-CUDART_INF_F, 0.f, -CUDART_INF_F, 0.f);
                float m = r.m;
#pragma unroll
                for (int i = 0; i < 4; ++i) m = fmaxf(m, fmaxf(p[i].x, p[i].z));
                if (m == -CUDART_INF_F) {                              // (sums of 0 or NaN)
#pragma unroll
                    for (int i = 0; i < 4; ++i) r.s += p[i].y + p[i].w;
                    continue;
                }
                float s = r.s * ex2((r.m - m) * kLog2e);
#pragma unroll
                for (int i = 0; i < 4; ++i) s += p[i].y * ex2((p[i].x - m) * kLog2e) + p[i].w * ex2((p[i].z - m) * kLog2e);
                r = Ms{m, s};
            }
            for (int o = 1; o < tpn; o *= 2) {
                Ms other;
                other.m = __shfl_xor_sync(0xFFFFFFFFu, r.m, o);
                other.s = __shfl_xor_sync(0xFFFFFFFFu, r.s, o);
                r = combine(r, other);
            }
            if (t >= N * tpn || t % tpn != 0) continue;
            s_mx[v] = r.m;
            s_sum[v] = r.s;
            s_uq[v] = u[v] * q[v];       // the left side of the step test, fetched beside the pairs
            if (!(r.s > 0.f) || r.m == CUDART_INF_F) flags |= GSD_DEV_BAD_LOGITS;   // no finite entry, +inf or NaN
        }
        return flags;
    };
    int32_t* out_tok = a.out_tok + (size_t)b * a.Tcap;
    if (rank == 0) {
        PathIo io;
        io.tok = a.tok + (size_t)b * N;
        io.pptr = a.pptr + (size_t)b * (N + 1);
        io.pidx = a.pidx + (size_t)b * a.Ecap;
        io.out_tok = out_tok;
        io.out_nodes = a.out_nodes ? a.out_nodes + (size_t)b * a.Tcap : nullptr;
        io.out_len = a.out_len + b;
        io.status = a.status;
        io.N = N; io.V = V; io.Ecap = a.Ecap; io.Tcap = a.Tcap;
        // the test of one step: the target's probability of v's token under its parent p (one
        // logit gathered from global memory) against u q
        const PathResult res = longest_accepted_path_ex<true>(
            io, 0u,
            [&](float logit, int p, int v, int) { return s_uq[v] < ex2((logit - s_mx[p]) * kLog2e) / s_sum[p]; },
            [&](int p, int t) -> float {
                if (!GSD_IN_BOUNDS(p >= 0 && p < N && t >= 0 && t < V, a.status)) return -CUDART_INF_F;
                return lg[(size_t)p * V + t];
            },
            combine_pairs);
        if (tid == 0) s_outcome = Outcome{res.edges, res.end, res.end_has_child ? 1 : 0, s_mx[res.end], s_sum[res.end]};
        __syncthreads();
        cluster_wait();
        constexpr int kWords = sizeof(Outcome) / 4;
        if (tid >= kWords && tid < C * kWords)
            put_remote(reinterpret_cast<uint32_t*>(&s_outcome) + tid % kWords, tid / kWords, reinterpret_cast<const uint32_t*>(&s_outcome)[tid % kWords]);
    } else {
        cluster_wait();
    }
    cluster_arrive();
    cluster_wait();
    const int s_m = s_outcome.edges, s_end = s_outcome.end;
    const float mx = s_outcome.mx, p_sum = s_outcome.sum;

    // The regenerated token: weights w_j over the vocabulary at the end node, then the smallest
    // t whose cumulative weight exceeds u * (total weight).  First the contiguous range of the
    // row that holds the crossing is found from range sums, then one CTA splits that range into
    // 256 contiguous pieces, scans the piece sums, and the thread whose piece holds the crossing
    // walks it.
    const float* x = lg + (size_t)s_end * V;
    const RowSpan xs = row_span(x, V);

    // Residual of the sampling scheme: when drafted continuations of the end node were rejected
    // (it has a child in the graph) the weights are max(0, P_j - Q_j), Q the draft model's
    // distribution at that node.  Its range sums are formed here: the row is cut into one
    // contiguous range per warp of the cluster (range_of with the CTAs as slices).  The two rows
    // come from DRAM and nothing else runs any more, so the time is the chain of dependent trips:
    // with one CTA per sequence the two passes took 9 us at V 32000 and four times that at
    // 128256; eight CTAs make each pass one trip.  8 x 256 rows of 32000, whole call: 64.8 us with
    // one CTA per sequence, 61.9 with two, 59.2 with four, 59.7 with eight.
    bool residual = false;
    float q_m = 0.f, inv_sp = 0.f, inv_sq = 0.f, res_total = 0.f;
    const float* y = nullptr;
    bool same = false;                   // both rows have their 16-byte groups at the same entries
    if (a.dlogits && s_outcome.end_has_child) {
        y = a.dlogits + ((size_t)b * N + s_end) * V;
        same = row_span(y, V).head == xs.head;
        const Range g = range_of(xs, V, C, rank * kWarps + warp);
        // entries of the range outside its groups: before (first range) and behind (last range)
        const int e_head = g.lo + lane, e_tail = xs.head + g.a1 * 4 + lane;
        const bool in_head = e_head < xs.head, in_tail = e_tail < g.hi;
        constexpr int kBatch = 4;        // groups a thread has in flight (eight made short rows 0.5 to 1 us slower: more code to fetch)
        const float4 none = make_float4(-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F);
        auto group = [&](const float* row, bool vec, int i) { return i < g.a1 ? load4(row + xs.head + 4 * i, vec) : none; };
        // softmax statistics of the draft row; the target's row is brought into L2 beside it
        Ms r{-CUDART_INF_F, 0.f};
        if (in_head) take1(r, __ldg(y + e_head));
        if (in_tail) take1(r, __ldg(y + e_tail));
        for (int i = g.a0 + lane; i < g.a1; i += kBatch * 32) {
            float4 t[kBatch];
#pragma unroll
            for (int k = 0; k < kBatch; ++k) t[k] = group(y, same, i + k * 32);
#pragma unroll
            for (int k = 0; k < kBatch; ++k)
                if (i + k * 32 < g.a1) asm volatile("prefetch.global.L2 [%0];" ::"l"(x + xs.head + 4 * (i + k * 32)));
#pragma unroll
            for (int k = 0; k < kBatch; k += 4) take16(r, t[k], t[k + 1], t[k + 2], t[k + 3]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            Ms t;
            t.m = __shfl_xor_sync(0xFFFFFFFFu, r.m, o);
            t.s = __shfl_xor_sync(0xFFFFFFFFu, r.s, o);
            r = combine(r, t);
        }
        if (lane == 0) { s_rm[warp] = r.m; s_scan[warp] = r.s; }
        __syncthreads();
        if (tid < C) {
            r = Ms{-CUDART_INF_F, 0.f};
            for (int w = 0; w < kWarps; ++w) r = combine(r, Ms{s_rm[w], s_scan[w]});
            put_remote(s_cm + rank, tid, __float_as_uint(r.m));
            put_remote(s_cs + rank, tid, __float_as_uint(r.s));
        }
        cluster_arrive();
        cluster_wait();
        r = Ms{-CUDART_INF_F, 0.f};
        for (int c = 0; c < C; ++c) r = combine(r, Ms{s_cm[c], s_cs[c]});
        if (!(r.s > 0.f) || r.m == CUDART_INF_F) {
            if (rank == 0 && tid == 0 && a.status) atomicOr((unsigned*)a.status, GSD_DEV_BAD_LOGITS);
        } else {
            q_m = r.m;
            inv_sp = 1.f / p_sum;
            inv_sq = 1.f / r.s;
            auto res1 = [&](float xv, float yv) -> float {
                return fmaxf(ex2((xv - mx) * kLog2e) * inv_sp - ex2((yv - q_m) * kLog2e) * inv_sq, 0.f);
            };
            float part = 0.f;
            if (in_head) part += res1(__ldg(x + e_head), __ldg(y + e_head));
            for (int i = g.a0 + lane; i < g.a1; i += kBatch * 32) {
                float4 xv[kBatch], yv[kBatch];
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    xv[k] = group(x, true, i + k * 32);
                    yv[k] = group(y, same, i + k * 32);
                }
#pragma unroll
                for (int k = 0; k < kBatch; ++k)
                    part += (res1(xv[k].x, yv[k].x) + res1(xv[k].y, yv[k].y)) + (res1(xv[k].z, yv[k].z) + res1(xv[k].w, yv[k].w));
            }
            if (in_tail) part += res1(__ldg(x + e_tail), __ldg(y + e_tail));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xFFFFFFFFu, part, o);
            if (lane < C) put_remote(s_rsum + rank * kWarps + warp, lane, __float_as_uint(part));
            cluster_arrive();
            cluster_wait();
            for (int w = 0; w < C * kWarps; ++w) res_total += s_rsum[w];
            // a residual without mass (the two distributions agree to rounding) leaves P
            residual = res_total > kResidualFloor;
            __syncthreads();             // (P's range sums may take the place of the residual's)
        }
    }
    if (!residual && rank != 0) return;  // (no CTA of the cluster touches another one's memory any more)
    // weight of one entry from its two logits (-inf stands for "past the end": weight 0)
    auto weight = [&](float xv, float yv) -> float {
        const float e = ex2((xv - mx) * kLog2e);
        return residual ? fmaxf(e * inv_sp - ex2((yv - q_m) * kLog2e) * inv_sq, 0.f) : e;
    };
    // sixteen consecutive entries of a row, all loads issued before any is used
    auto load16 = [&](const float* row, int j, int jend, float (&v)[16]) {
        if ((reinterpret_cast<uintptr_t>(row + j) & 15u) == 0 && j + 16 <= jend) {
            const float4* r4 = reinterpret_cast<const float4*>(row + j);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 t = r4[k];
                v[4 * k] = t.x; v[4 * k + 1] = t.y; v[4 * k + 2] = t.z; v[4 * k + 3] = t.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = j + k < jend ? row[j + k] : -CUDART_INF_F;
        }
    };
    const float target = a.us[b] * (residual ? res_total : p_sum);
    // every thread walks the range sums: the first range whose inclusive prefix exceeds the
    // target, or the last one with any mass if rounding leaves none
    int rsel = -1, last_r = 0;
    float before_range = 0.f, before_last = 0.f;
    {
        const int nr = residual ? C * kWarps : a.slices * kWarps;
        if (!residual && tid < nr) {          // one range sum per thread, brought to the row's maximum
            const float2 t = __ldcg(a.part + ((size_t)b * N + s_end) * a.slices * kWarps + tid);
            s_rsum[tid] = t.x == -CUDART_INF_F ? 0.f : t.y * ex2((t.x - mx) * kLog2e);
        }
        __syncthreads();
        float run = 0.f;
        for (int r = 0; r < nr; ++r) {
            const float sr = s_rsum[r];
            if (rsel < 0 && run + sr > target) { rsel = r; before_range = run; }
            if (sr > 0.f) { last_r = r; before_last = run; }
            run += sr;
        }
    }
    const bool crossing = rsel >= 0;
    if (!crossing) { rsel = last_r; before_range = before_last; }
    // the CTA that formed a residual range goes on with it (its part of the rows is close by)
    if (residual && rank != rsel / kWarps) return;
    if (tid == 0) s_pick = kNone;
    const Range rg = range_of(xs, V, residual ? C : a.slices, rsel);
    const int r0 = rg.lo, r1 = rg.hi;
    const int per = (r1 - r0 + kThreads - 1) / kThreads;
    const int j0 = min(r0 + tid * per, r1), j1 = min(j0 + per, r1);
    float piece = 0.f;
    int last_pos = -1;
    for (int c0 = j0; c0 < j1; c0 += 16) {
        float xv[16], yv[16];
        load16(x, c0, j1, xv);
        if (residual) load16(y, c0, j1, yv);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float e = weight(xv[k], residual ? yv[k] : 0.f);
            piece += e;
            if (e > 0.f) last_pos = c0 + k;
        }
    }
    float inc = piece;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) s_scan[warp] = inc;
    __syncthreads();
    float base = before_range;
#pragma unroll
    for (int w = 0; w < kWarps; ++w)
        if (w < warp) base += s_scan[w];
    inc += base;
    // The pieces partition the cumulative axis exactly: a piece begins where the one before it
    // ends (its predecessor's inclusive value, not inc - piece, which rounding could move past a
    // target that the predecessor had not reached).  The first piece whose inclusive value exceeds
    // the target holds the crossing.
    float before = __shfl_up_sync(0xFFFFFFFFu, inc, 1);
    if (lane == 0) before = base;
    if (crossing && inc > target) atomicMin(&s_pick, tid);
    __syncthreads();
    const int first = s_pick;           // kNone: rounding left no crossing in this range
    __syncthreads();
    if (tid == first) {
        float cum = before;
        int pick = -1;
        for (int c0 = j0; c0 < j1 && pick < 0; c0 += 16) {
            float xv[16], yv[16];
            load16(x, c0, j1, xv);
            if (residual) load16(y, c0, j1, yv);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                cum += weight(xv[k], residual ? yv[k] : 0.f);
                if (pick < 0 && cum > target) pick = c0 + k;
            }
        }
        s_pick = pick;                  // -1: the serial sum stayed at or below the target
    }
    // without a crossing the draw is the last entry with any mass at or before that piece (in
    // the whole range if no piece claimed the target)
    int lp = (first == kNone || tid <= first) ? last_pos : -1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lp = max(lp, __shfl_xor_sync(0xFFFFFFFFu, lp, o));
    if (lane == 0) s_red[warp] = lp;
    __syncthreads();
    if (tid == 0) {
        int pick = first == kNone ? -1 : s_pick;
        if (pick < 0)
            for (int w = 0; w < kWarps; ++w) pick = max(pick, s_red[w]);
        if (s_m < a.Tcap && GSD_IN_BOUNDS(s_m >= 0 && pick < V, a.status)) out_tok[s_m] = pick;
    }
}

// First launch: one CTA per (slice, row) streams its part of the row and leaves the warps'
// (maximum, sum) pairs in scratch.
__global__ void __launch_bounds__(kThreads, 8) accept_sampled_kernel(SampledArgs a) {
    // the per-sequence pass (a programmatic dependent launch) may become resident as CTAs retire
    if (threadIdx.x == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int row = blockIdx.y;  // b * N + n
    const int slice = blockIdx.x;
    const float* x = a.logits + (size_t)row * a.V;
    Ms r{-CUDART_INF_F, 0.f};
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const RowSpan sp = row_span(x, a.V);
    const Range g = range_of(sp, a.V, a.slices, slice * kWarps + warp);
    {
        const float4* x4 = reinterpret_cast<const float4*>(x + sp.head);
        if (g.lo + lane < sp.head) take1(r, __ldcs(x + g.lo + lane));       // (range 0 only: lo is 0)
        const float4 none = make_float4(-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F);
        // four independent 16-byte loads in flight per thread, each a 512-byte run per warp, in the
        // last round too (an absent group counts as -inf, which has no mass)
        for (int i = g.a0 + lane; i < g.a1; i += 4 * 32) {
            float4 t[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) t[k] = i + k * 32 < g.a1 ? __ldcs(x4 + i + k * 32) : none;
            take16(r, t[0], t[1], t[2], t[3]);
        }
        if (sp.head + g.a1 * 4 + lane < g.hi) take1(r, __ldcs(x + sp.head + g.a1 * 4 + lane));   // (last range only)
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Ms t;
        t.m = __shfl_xor_sync(0xFFFFFFFFu, r.m, o);
        t.s = __shfl_xor_sync(0xFFFFFFFFu, r.s, o);
        r = combine(r, t);
    }
    if (lane == 0) a.part[((size_t)row * a.slices + slice) * kWarps + warp] = make_float2(r.m, r.s);
}

// Second launch: one cluster per sequence does the rest (statistics per node, step tests, longest
// path, regenerated token) once every pair of the first launch is visible.
__global__ void __launch_bounds__(kThreads, 1) accept_sampled_tail_kernel(SampledArgs a) {
    finish_sequence(a, (int)blockIdx.x / a.cluster);      // (waits for the first launch inside, as late as it can)
}

int pick_slices(long rows, int V, int sm_count) {
    // enough CTAs to cover the machine a few times over, slices of at least 4096 floats
    int slices = 1;
    const long want = (long)sm_count * 8;
    while (rows * slices < want && (V / (slices * 2)) >= 4096 && slices * 2 <= kMaxSlices) slices *= 2;
    return slices;
}

// CTAs of the second launch per sequence: only the two passes over the end node's rows are shared,
// so a CTA should have at least 2048 entries of them (half a round of loads), and all of them together take
// one CTA per SM at most: they are resident while the first launch still streams, and the SMs they take
// are missing there (32 x 64 rows of 32000: 62.9 us with one CTA per sequence, 64.7 with eight, 56.9 with
// the four that this allows).  Without draft logits there is no residual and no pass.
int pick_cluster(int B, int V, bool residual, int sm_count) {
    int c = 1;
    while (residual && c * 2 <= kMaxCluster && V / (c * 2) >= 2048 && (long)B * c * 2 <= sm_count) c *= 2;
    return c;
}

}  // namespace
}  // namespace gsd

extern "C" size_t gsd_accept_sampled_workspace_bytes(const gsd_accept_params* p) {
    if (!p || p->B < 1 || p->N < 1 || p->N > GSD_MAX_NODES) return 0;
    return gsd::align_up((size_t)p->B * p->N * gsd::kMaxSlices * gsd::kWarps * 8, 256);
}

extern "C" int gsd_accept_sampled(const float* logits, const int32_t* draft_tokens,
                                  const int32_t* parent_ptr, const int32_t* parent_idx,
                                  const float* draft_logits, const float* draft_q,
                                  const float* u_accept, const float* u_sample,
                                  int32_t* accepted_tokens, int32_t* accepted_len,
                                  int32_t* accepted_nodes, const gsd_accept_params* p,
                                  void* workspace, size_t workspace_bytes, int32_t* status,
                                  void* stream) {
    using namespace gsd;
    if (!p || !logits || !draft_tokens || !parent_ptr || !parent_idx || !draft_q || !u_accept ||
        !u_sample || !accepted_tokens || !accepted_len)
        return GSD_ERR_NULL_POINTER;
    if (p->B < 1 || p->N < 1 || p->N > GSD_MAX_NODES || p->V < 1 || p->Ecap < 1 || p->Tcap < 1)
        return GSD_ERR_BAD_SHAPE;
    if ((long long)p->B * p->N > (1ll << 30)) return GSD_ERR_BAD_SHAPE;
    if (((uintptr_t)logits & 3u) != 0 || ((uintptr_t)draft_logits & 3u) != 0) return GSD_ERR_MISALIGNED;
    const size_t need = gsd_accept_sampled_workspace_bytes(p);
    if (!workspace || workspace_bytes < need) return GSD_ERR_WORKSPACE;
    if (((uintptr_t)workspace & 7u) != 0) return GSD_ERR_MISALIGNED;
    DeviceInfo di;
    if (device_info(&di) != 0) return GSD_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;

    SampledArgs a;
    a.logits = logits; a.dlogits = draft_logits; a.tok = draft_tokens; a.pptr = parent_ptr; a.pidx = parent_idx;
    a.q = draft_q; a.u = u_accept; a.us = u_sample;
    a.out_tok = accepted_tokens; a.out_len = accepted_len; a.out_nodes = accepted_nodes;
    a.part = (float2*)workspace;
    a.status = status;
    a.B = p->B; a.N = p->N; a.V = p->V; a.Ecap = p->Ecap; a.Tcap = p->Tcap;
    a.slices = pick_slices((long)p->B * p->N, p->V, di.sm_count);

    // every pair is written before it is read: nothing in the scratch has to start at zero.
    // grid.y holds at most 65535 rows: larger problems go out in blocks of whole sequences.
    const int seq_per = 65535 / p->N;
    for (int b0 = 0; b0 < p->B; b0 += seq_per) {
        const int nb = (p->B - b0 < seq_per) ? p->B - b0 : seq_per;
        SampledArgs s = a;
        s.logits += (size_t)b0 * p->N * p->V; s.tok += (size_t)b0 * p->N;
        if (s.dlogits) s.dlogits += (size_t)b0 * p->N * p->V;
        s.pptr += (size_t)b0 * (p->N + 1); s.pidx += (size_t)b0 * p->Ecap;
        s.q += (size_t)b0 * p->N; s.u += (size_t)b0 * p->N; s.us += b0;
        s.out_tok += (size_t)b0 * p->Tcap; s.out_len += b0;
        if (s.out_nodes) s.out_nodes += (size_t)b0 * p->Tcap;
        s.part += (size_t)b0 * p->N * a.slices * kWarps; s.B = nb;
        const dim3 grid(a.slices, (unsigned)(nb * p->N));
        accept_sampled_kernel<<<grid, kThreads, 0, st>>>(s);
        GSD_CUDA_TRY(cudaGetLastError());
        s.cluster = pick_cluster(nb, p->V, draft_logits != nullptr, di.sm_count);
        cudaLaunchAttribute attr[2];
        dependent_launch_attr(attr);
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)s.cluster;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(nb * s.cluster));
        cfg.blockDim = dim3(kThreads);
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = s.cluster > 1 ? 2 : 1;
        GSD_CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_sampled_tail_kernel, s));
    }
    GSD_CUDA_TRY(cudaGetLastError());
    return GSD_OK;
}
