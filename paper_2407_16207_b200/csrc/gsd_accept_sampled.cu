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
// the two rows of the end node, which stay in registers, and exchanged through distributed shared memory) give the range of
// the crossing, a scan over that range by its warp (or, when it was not kept, by a CTA) gives the index.
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

// the pairs of a warp's lanes, all of them with the same result
__device__ __forceinline__ Ms warp_combine(Ms r) {
    float m = r.m;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    float s = m == -CUDART_INF_F ? r.s : r.s * ex2((r.m - m) * kLog2e);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return Ms{m, s};
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
    __shared__ float s_cm[kMaxCluster * kWarps], s_cs[kMaxCluster * kWarps];
    __shared__ float s_rsum[kMaxSlices * kWarps];
    __shared__ Outcome s_outcome;
    __shared__ int s_pick;
    const int C = a.cluster, rank = C > 1 ? cluster_rank() : 0;
    static_assert(kPathNodeSlots == 2, "two nodes a thread at most");
    static_assert(kMaxCluster <= kMaxSlices, "one range sum per warp of the cluster");
    cluster_arrive();                    // (every CTA has started before any writes to another)
    const int N = a.N, V = a.V, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float* lg = a.logits + (size_t)b * N * V;
    const float* q = a.q + (size_t)b * N;
    const float* u = a.u + (size_t)b * N;
    const float u_draw = a.us[b];
    float uq[kPathNodeSlots];            // the left sides of the step tests
#pragma unroll
    for (int k = 0; k < kPathNodeSlots; ++k) uq[k] = tid + k * kThreads < N ? u[tid + k * kThreads] * q[tid + k * kThreads] : 0.f;
    // Softmax statistics of every node from the pairs of the first launch.  This is the first thing that needs the first launch's results: the path
    // routine calls it after the graph and one logit per step have been fetched, so those two
    // trips to memory are over when the first launch ends.
    auto combine_pairs = [&]() -> unsigned {
        unsigned flags = 0;
#pragma unroll
        for (int k = 0; k < kPathNodeSlots; ++k)
            if (tid + k * kThreads < N) s_uq[tid + k * kThreads] = uq[k];
        wait_for_predecessor();
        // A node's pairs are shared by neighbouring threads when there are fewer nodes than threads (with few rows
        // the rows are cut into many slices: 1 x 11 rows of 128256, 128 pairs a node, by at most four
        // threads: 2.5 us); with more nodes than threads a thread goes through two of them at once.
        int tpn = 1;
        while (tpn < 2 * a.slices && 2 * tpn * N <= kThreads && tpn < 32) tpn *= 2;
        const int quads = a.slices * (kWarps / 2) / tpn;               // float4s (two pairs each) of one thread
        // (a workspace has to be on an 8-byte boundary only; 8-byte loads throughout took up to 1.3 us more:
        // 4 x 100 rows of 50257, 34.8 -> 36.1)
        const bool by16 = (reinterpret_cast<uintptr_t>(a.part) & 15u) == 0;
        auto two_pairs = [&](const float4* at) -> float4 {             // (written by other CTAs: read past L1)
            if (by16) return __ldcg(at);
            const float2 lo = __ldcg(reinterpret_cast<const float2*>(at)), hi = __ldcg(reinterpret_cast<const float2*>(at) + 1);
            return make_float4(lo.x, lo.y, hi.x, hi.y);
        };
        const float4* pairs = reinterpret_cast<const float4*>(a.part + (size_t)b * N * a.slices * kWarps) + tid * quads;
        const bool two = N > kThreads + tid;                           // (a second node: tpn is 1 then)
        Ms r[2] = {{-CUDART_INF_F, 0.f}, {-CUDART_INF_F, 0.f}};
        if (tid < N * tpn) {
            for (int k = 0; k < quads; k += 4) {                       // eight pairs (64 bytes) a round and node
                float4 p[2][4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 none = make_float4(-CUDART_INF_F, 0.f, -CUDART_INF_F, 0.f);
                    p[0][i] = k + i < quads ? two_pairs(pairs + k + i) : none;
                    p[1][i] = two && k + i < quads ? two_pairs(pairs + kThreads * quads + k + i) : none;
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float m = r[h].m;
#pragma unroll
                    for (int i = 0; i < 4; ++i) m = fmaxf(m, fmaxf(p[h][i].x, p[h][i].z));
                    if (m == -CUDART_INF_F) {                          // (sums of 0 or NaN)
#pragma unroll
                        for (int i = 0; i < 4; ++i) r[h].s += p[h][i].y + p[h][i].w;
                        continue;
                    }
                    float s = r[h].s * ex2((r[h].m - m) * kLog2e);
#pragma unroll
                    for (int i = 0; i < 4; ++i) s += p[h][i].y * ex2((p[h][i].x - m) * kLog2e) + p[h][i].w * ex2((p[h][i].z - m) * kLog2e);
                    r[h] = Ms{m, s};
                }
            }
        }
        for (int o = 1; o < tpn; o *= 2) {
            Ms other;
            other.m = __shfl_xor_sync(0xFFFFFFFFu, r[0].m, o);
            other.s = __shfl_xor_sync(0xFFFFFFFFu, r[0].s, o);
            r[0] = combine(r[0], other);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int v = h == 0 ? tid / tpn : tid + kThreads;
            if (v >= N || (h == 0 && tid % tpn != 0)) continue;
            s_mx[v] = r[h].m;
            s_sum[v] = r[h].s;
            if (!(r[h].s > 0.f) || r[h].m == CUDART_INF_F) flags |= GSD_DEV_BAD_LOGITS;   // no finite entry, +inf or NaN
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
        const PathResult res = longest_accepted_path<true>(
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
    // A warp's part of the rows that fits its registers (up to 32768 entries a row on eight CTAs) is read once:
    // the weights take the target row's place there, and the warp with the crossing finds the token
    // itself.  8 x 256 rows of 32000, whole call: 56.5 us with both rows read again for the weights and for
    // the token, 52.9 this way.
    constexpr int kBatch = 4;            // groups a thread has in flight (eight made short rows 0.5 to 1 us slower: more code to fetch)
    float4 xv[kBatch], yv[kBatch];
    float w_head = 0.f, w_tail = 0.f;
    bool kept = false;
    bool residual = false;
    float q_m = 0.f, inv_sp = 0.f, inv_sq = 0.f;
    const float* y = nullptr;
    bool same = false;                   // both rows have their 16-byte groups at the same entries
    if (a.dlogits && s_outcome.end_has_child) {
        y = a.dlogits + ((size_t)b * N + s_end) * V;
        same = row_span(y, V).head == xs.head;
        const Range g = range_of(xs, V, C, rank * kWarps + warp);
        // entries of the range outside its groups: before (first range) and behind (last range)
        const int e_head = g.lo + lane, e_tail = xs.head + g.a1 * 4 + lane;
        const bool in_head = e_head < xs.head, in_tail = e_tail < g.hi;
        const float4 none = make_float4(-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F);
        auto group = [&](const float* row, bool vec, int i) { return i < g.a1 ? load4(row + xs.head + 4 * i, vec) : none; };
        // Softmax statistics of the draft row.  The first batch of both rows stays in registers; of what is
        // behind it the target's row is brought into L2.
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            yv[k] = group(y, same, g.a0 + lane + k * 32);
            xv[k] = group(x, true, g.a0 + lane + k * 32);
        }
        float hx = 0.f, hy = 0.f, tx = 0.f, ty = 0.f;
        if (in_head) { hy = __ldg(y + e_head); hx = __ldg(x + e_head); }
        if (in_tail) { ty = __ldg(y + e_tail); tx = __ldg(x + e_tail); }
        Ms r{-CUDART_INF_F, 0.f};
        if (in_head) take1(r, hy);
        if (in_tail) take1(r, ty);
        take16(r, yv[0], yv[1], yv[2], yv[3]);
        for (int i = g.a0 + lane + kBatch * 32; i < g.a1; i += kBatch * 32) {
            float4 t[kBatch];
#pragma unroll
            for (int k = 0; k < kBatch; ++k) t[k] = group(y, same, i + k * 32);
#pragma unroll
            for (int k = 0; k < kBatch; ++k)
                if (i + k * 32 < g.a1) asm volatile("prefetch.global.L2 [%0];" ::"l"(x + xs.head + 4 * (i + k * 32)));
            take16(r, t[0], t[1], t[2], t[3]);
        }
        r = warp_combine(r);
        // every warp hands its pair to every CTA of the cluster, and every warp combines them all
        if (lane < C) {
            put_remote(s_cm + rank * kWarps + warp, lane, __float_as_uint(r.m));
            put_remote(s_cs + rank * kWarps + warp, lane, __float_as_uint(r.s));
        }
        cluster_arrive();
        // (the target's probabilities, while the pairs travel)
        inv_sp = 1.f / p_sum;
        auto p_of = [&](float v) { return ex2((v - mx) * kLog2e) * inv_sp; };
        auto p_of4 = [&](const float4& v) { return make_float4(p_of(v.x), p_of(v.y), p_of(v.z), p_of(v.w)); };
#pragma unroll
        for (int k = 0; k < kBatch; ++k) xv[k] = p_of4(xv[k]);
        if (in_head) hx = p_of(hx);
        if (in_tail) tx = p_of(tx);
        cluster_wait();
        r = Ms{-CUDART_INF_F, 0.f};
        for (int w = lane; w < C * kWarps; w += 32) r = combine(r, Ms{s_cm[w], s_cs[w]});
        r = warp_combine(r);
        if (!(r.s > 0.f) || r.m == CUDART_INF_F) {
            if (rank == 0 && tid == 0 && a.status) atomicOr((unsigned*)a.status, GSD_DEV_BAD_LOGITS);
        } else {
            q_m = r.m;
            inv_sq = 1.f / r.s;
            auto rest = [&](float p, float yv) { return fmaxf(p - ex2((yv - q_m) * kLog2e) * inv_sq, 0.f); };
            if (in_head) w_head = rest(hx, hy);
            if (in_tail) w_tail = rest(tx, ty);
            float part = w_head;
            auto weigh = [&](const float4& pv, const float4& yv) -> float4 {
                const float4 w = make_float4(rest(pv.x, yv.x), rest(pv.y, yv.y), rest(pv.z, yv.z), rest(pv.w, yv.w));
                part += (w.x + w.y) + (w.z + w.w);
                return w;
            };
#pragma unroll
            for (int k = 0; k < kBatch; ++k) xv[k] = weigh(xv[k], yv[k]);
            for (int i = g.a0 + lane + kBatch * 32; i < g.a1; i += kBatch * 32) {
                float4 xa[kBatch], ya[kBatch];
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    xa[k] = group(x, true, i + k * 32);
                    ya[k] = group(y, same, i + k * 32);
                }
#pragma unroll
                for (int k = 0; k < kBatch; ++k) weigh(p_of4(xa[k]), ya[k]);
            }
            part += w_tail;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xFFFFFFFFu, part, o);
            if (lane < C) put_remote(s_rsum + rank * kWarps + warp, lane, __float_as_uint(part));
            cluster_arrive();
            cluster_wait();
            kept = ((xs.nvec + C - 1) / C + kWarps - 1) / kWarps <= kBatch * 32;      // (the longest range of the cluster)
            residual = true;             // (if it has any mass, see below)
        }
    }
    // The range of the crossing, found by every warp of the cluster with the same result: the first range whose
    // inclusive prefix exceeds the target, or the last one with any mass if rounding leaves none.  Four
    // range sums a lane (walked one by one by every thread it took 1.5 us).
    static_assert(kMaxSlices * kWarps <= 128, "four range sums a lane");
    int rsel = 0;
    float before_range = 0.f, target = 0.f;
    bool crossing = false;
    auto find_range = [&](int nr, auto target_of) -> bool {
        float w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = 4 * lane + j < nr ? s_rsum[4 * lane + j] : 0.f;
        float inc = (w[0] + w[1]) + (w[2] + w[3]);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += t;
        }
        const float total = __shfl_sync(0xFFFFFFFFu, inc, 31);
        if (!target_of(total)) return false;
        float c[5];                      // the cumulative axis at the ends of the lane's ranges
        c[0] = __shfl_up_sync(0xFFFFFFFFu, inc, 1);
        if (lane == 0) c[0] = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) c[j + 1] = c[j] + w[j];
        const float end_before = __shfl_up_sync(0xFFFFFFFFu, c[4], 1);
        if (lane > 0) c[0] = end_before;     // (a lane's first range begins where the one before it ends)
        int at = kNone, last = kNone;
        float c_at = 0.f, c_last = 0.f;
#pragma unroll
        for (int j = 3; j >= 0; --j) {
            // (rounding can put the end of a range without mass past a target that nothing before it has reached)
            if (w[j] > 0.f && c[j + 1] > target) { at = 4 * lane + j; c_at = c[j]; }
            if (w[j] > 0.f && last == kNone) { last = 4 * lane + j; c_last = c[j]; }
        }
        const unsigned hit = __ballot_sync(0xFFFFFFFFu, at != kNone), mass = __ballot_sync(0xFFFFFFFFu, last != kNone);
        crossing = hit != 0u;
        if (hit | mass) {
            const int from = crossing ? __ffs(hit) - 1 : 31 - __clz(mass);
            rsel = __shfl_sync(0xFFFFFFFFu, crossing ? at : last, from);
            before_range = __shfl_sync(0xFFFFFFFFu, crossing ? c_at : c_last, from);
        }
        return true;
    };
    if (residual)                        // a residual without mass (the two distributions agree to rounding) leaves P
        residual = find_range(C * kWarps, [&](float total) { target = u_draw * total; return total > kResidualFloor; });
    if (!residual) {
        if (rank != 0) return;           // (no CTA of the cluster touches another one's memory any more)
        const int nr = a.slices * kWarps;
        __syncthreads();                 // (P's range sums take the place of the residual's)
        if (tid < nr) {                  // one range sum per thread, brought to the row's maximum
            const float2 t = __ldcg(a.part + ((size_t)b * N + s_end) * a.slices * kWarps + tid);
            s_rsum[tid] = t.x == -CUDART_INF_F ? 0.f : t.y * ex2((t.x - mx) * kLog2e);
        }
        __syncthreads();
        find_range(nr, [&](float) { target = u_draw * p_sum; return true; });
    }
    // the CTA that formed a residual range goes on with it (its part of the rows is close by)
    if (residual && rank != rsel / kWarps) return;
    if (residual && kept) {
        // The weights of the range are in this warp's registers, in runs of 128 entries, four a lane.
        if (warp != rsel % kWarps) return;
        const Range g = range_of(xs, V, C, rsel);
        float cum = before_range;
        int pick = -1, last = -1;
        bool open = crossing;            // the crossing is still ahead
        auto run = [&](const float4& w4, int e) {                  // the lane's entries e .. e + 3 of a run
            const float w[4] = {w4.x, w4.y, w4.z, w4.w};
            const float own = (w[0] + w[1]) + (w[2] + w[3]);
            float in = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float t = __shfl_up_sync(0xFFFFFFFFu, in, o);
                if (lane >= o) in += t;
            }
            in += cum;
            // (a lane's entries begin where those of the lane before end)
            float c = __shfl_up_sync(0xFFFFFFFFu, in, 1);
            if (lane == 0) c = cum;
            cum = __shfl_sync(0xFFFFFFFFu, in, 31);
            const unsigned hit = __ballot_sync(0xFFFFFFFFu, open && own > 0.f && in > target);
            const int first = hit ? __ffs(hit) - 1 : 31;
            if (open || !crossing) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    c += w[j];
                    if (hit && lane == first && w[j] > 0.f && c > target) pick = pick < 0 ? e + j : pick;
                    if (w[j] > 0.f && lane <= first) last = e + j;
                }
            }
            open = open && !hit;
        };
        if (rsel == 0 && xs.head > 0) run(make_float4(w_head, 0.f, 0.f, 0.f), lane);
#pragma unroll 1
        for (int k = 0; k < kBatch; ++k) {
            run(xv[0], xs.head + 4 * (g.a0 + lane + k * 32));
#pragma unroll
            for (int j = 0; j + 1 < kBatch; ++j) xv[j] = xv[j + 1];
        }
        if (rsel == C * kWarps - 1) run(make_float4(w_tail, 0.f, 0.f, 0.f), xs.head + g.a1 * 4 + lane);
        pick = __reduce_max_sync(0xFFFFFFFFu, pick);
        // rounding left no entry above the target: the last one with any mass up to there
        if (pick < 0) pick = __reduce_max_sync(0xFFFFFFFFu, last);
        if (lane == 0 && s_m < a.Tcap && GSD_IN_BOUNDS(s_m >= 0 && pick < V, a.status)) out_tok[s_m] = pick;
        return;
    }
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
    if (crossing && piece > 0.f && inc > target) atomicMin(&s_pick, tid);
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
                const float e = weight(xv[k], residual ? yv[k] : 0.f);
                cum += e;
                if (pick < 0 && e > 0.f && cum > target) pick = c0 + k;
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
    wait_for_predecessor();
    // the per-sequence pass may become resident as CTAs retire; it reads the graph before it waits
    if (threadIdx.x == 0) let_successor_start();
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
    r = warp_combine(r);
    if (lane == 0) a.part[((size_t)row * a.slices + slice) * kWarps + warp] = make_float2(r.m, r.s);
}

// Second launch: one cluster per sequence does the rest (statistics per node, step tests, longest
// path, regenerated token) once every pair of the first launch is visible.
__global__ void __launch_bounds__(kThreads, 1) accept_sampled_tail_kernel(SampledArgs a) {
    let_successor_start();
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
        GSD_CUDA_TRY(launch_dependent(accept_sampled_kernel, grid, dim3(kThreads), 0, st, s));
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
