// gsd_accept: greedy verification (vocabulary argmax per draft node) and the longest
// accepted root path through the draft DAG (Sec. 3 deterministic verification and the
// rejection cascade; Sec. 4.1 longest-path selection).
//
// Two launches.  Grid (splits, B*N): each CTA streams one slice of one logits row with 16-byte
// loads, reduces (value, index) pairs and leaves the best as a packed 64-bit key in scratch.  The
// second launch (one CTA per sequence, a programmatic dependent of the first) fetches the graph
// beside the stream, takes the best key of every node and runs the path pass (gsd_path.cuh).
#include "gsd_internal.cuh"
#include "gsd_path.cuh"
#include <math_constants.h>
#include <algorithm>

namespace gsd {
namespace {

constexpr int kThreads = kPathThreads;
constexpr int kNone = 0x7FFFFFFF;
constexpr int kWaveCtas = 32;           // CTAs of a call per SM: four waves of eight
constexpr int kScratchSms = 148;        // SMs for which the scratch has room (with more of them the rows get fewer slices)

struct Best {
    float v;
    int i;
};

__device__ __forceinline__ void take(Best& b, float v, int i) {
    if (v > b.v) {  // false for NaN; strict: an equal later value never replaces
        b.v = v;
        b.i = i;
    }
}

__device__ __forceinline__ Best better(Best a, Best b) {
    return (b.v > a.v || (b.v == a.v && b.i < a.i)) ? b : a;
}

// monotone map of non-NaN floats to unsigned (with -0 folded onto +0)
__device__ __forceinline__ unsigned ordered_bits(float v) {
    if (v == 0.0f) v = 0.0f;
    unsigned u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ unsigned long long pack_key(float v, int i) {
    return ((unsigned long long)ordered_bits(v) << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned)i);
}

__device__ __forceinline__ int key_index(unsigned long long key) {
    return key == 0ull ? 0 : (int)(0xFFFFFFFFu - (unsigned)(key & 0xFFFFFFFFull));
}

__device__ Best block_best(Best b, Best* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Best t;
        t.v = __shfl_xor_sync(0xFFFFFFFFu, b.v, o);
        t.i = __shfl_xor_sync(0xFFFFFFFFu, b.i, o);
        b = better(b, t);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) sh[warp] = b;
    __syncthreads();
    if (warp == 0) {
        b = lane < (kThreads / 32) ? sh[lane] : Best{-CUDART_INF_F, kNone};
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            Best t;
            t.v = __shfl_xor_sync(0xFFFFFFFFu, b.v, o);
            t.i = __shfl_xor_sync(0xFFFFFFFFu, b.i, o);
            b = better(b, t);
        }
        if (lane == 0) sh[0] = b;
    }
    __syncthreads();
    b = sh[0];
    __syncthreads();
    return b;
}

struct AcceptArgs {
    const float* logits;
    const int32_t* tok;
    const int32_t* pptr;
    const int32_t* pidx;
    int32_t* out_tok;
    int32_t* out_len;
    int32_t* out_nodes;
    unsigned long long* keys;  // [splits][B*N]
    int32_t* status;
    int B, N, V, Ecap, Tcap, splits;
};

__global__ void __launch_bounds__(kThreads) accept_kernel(AcceptArgs a) {
    __shared__ Best sh[kThreads / 32];
    wait_for_predecessor();
    // the second launch may become resident as CTAs retire; it reads the graph before it waits
    if (threadIdx.x == 0) let_successor_start();
    const int row = blockIdx.y;  // b * N + n
    const int split = blockIdx.x;
    const float* x = a.logits + (size_t)row * a.V;
    Best best{-CUDART_INF_F, kNone};
    // The slice: a run of 16-byte groups; the first slice has the entries before the first
    // 16-byte boundary too, the last one those behind the last group.  (Every thread meets its
    // entries in ascending order.)  183 rows of 50257: 16.9 us with 4-byte loads for such rows,
    // 15.4 with groups; 3200 rows: 107.5 and 99.1.
    const RowSpan sp = row_span(x, a.V);
    const int per = (sp.nvec + a.splits - 1) / a.splits;
    const int v0 = min(split * per, sp.nvec), v1 = min(v0 + per, sp.nvec);
    const bool first = split == 0, last = split == a.splits - 1;
    const int lo = first ? 0 : sp.head + v0 * 4, hi = last ? a.V : sp.head + v1 * 4;   // its entries
    if (first && (int)threadIdx.x < sp.head) take(best, __ldcs(x + threadIdx.x), threadIdx.x);
    {
        const float4* x4 = reinterpret_cast<const float4*>(x + sp.head);
        const float4 none = make_float4(-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F);
        // four independent 16-byte loads in flight per thread, in the last round too (an absent
        // group counts as -inf, which never wins)
        for (int i = v0 + (int)threadIdx.x; i < v1; i += 4 * kThreads) {
            float4 r[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) r[k] = i + k * kThreads < v1 ? __ldcs(x4 + i + k * kThreads) : none;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int e = sp.head + (i + k * kThreads) * 4;
                take(best, r[k].x, e); take(best, r[k].y, e + 1); take(best, r[k].z, e + 2); take(best, r[k].w, e + 3);
            }
        }
        if (last) {
            const int e = sp.head + sp.nvec * 4 + (int)threadIdx.x;
            if (e < a.V) take(best, __ldcs(x + e), e);
        }
    }
    best = block_best(best, sh);
    if (best.i == kNone) {
        // nothing above -inf in this slice: the lowest non-NaN entry (a -inf), if any, stands
        int first = kNone;
        for (int i = lo + threadIdx.x; i < hi; i += kThreads)
            if (x[i] == x[i]) { first = i; break; }
        Best f{first == kNone ? -CUDART_INF_F : 0.0f, first};  // the value only orders this reduction
        f = block_best(f, sh);
        best.i = f.i;
        best.v = -CUDART_INF_F;
    }
    if (threadIdx.x == 0 && GSD_IN_BOUNDS(row < a.B * a.N && (best.i == kNone || (best.i >= 0 && best.i < a.V)), a.status))
        a.keys[(size_t)split * a.B * a.N + row] = best.i == kNone ? 0ull : pack_key(best.v, best.i);
}

// Second launch: the best key of every node, then the path.  kShare: the many slices of few rows are shared by
// neighbouring threads (a form of its own: the two shifts cost the other calls 0.1 us).
constexpr int kTrip = 8;                // slices whose keys a thread has on their way at a time
template <bool kShare>
__global__ void __launch_bounds__(kThreads) accept_tail_kernel(AcceptArgs a) {
    __shared__ int s_amax[GSD_MAX_NODES];
    let_successor_start();
    const int N = a.N, b = blockIdx.x, tid = threadIdx.x;
    PathIo io;
    io.tok = a.tok + (size_t)b * N;
    io.pptr = a.pptr + (size_t)b * (N + 1);
    io.pidx = a.pidx + (size_t)b * a.Ecap;
    io.out_tok = a.out_tok + (size_t)b * a.Tcap;
    io.out_nodes = a.out_nodes ? a.out_nodes + (size_t)b * a.Tcap : nullptr;
    io.out_len = a.out_len + b;
    io.status = a.status;
    io.N = N; io.V = a.V; io.Ecap = a.Ecap; io.Tcap = a.Tcap;
    // the keys of a thread's nodes: neighbouring threads read neighbouring keys
    auto best_keys = [&]() -> unsigned {
        int log_share = 0;
        while (kShare && (kTrip << log_share) < a.splits && (2 * N << log_share) <= kThreads && log_share < 5) ++log_share;
        const int share = 1 << log_share, node = tid >> log_share, mine = tid & (share - 1);
        wait_for_predecessor();
        const size_t rows = (size_t)a.B * N;
        const unsigned long long* keys = a.keys + (size_t)b * N + node;
        unsigned long long best[kPathNodeSlots] = {};
        for (int s0 = mine; s0 < a.splits; s0 += kTrip * share) {
            unsigned long long k[kPathNodeSlots][kTrip];
#pragma unroll
            for (int j = 0; j < kTrip; ++j)
#pragma unroll
                for (int i = 0; i < kPathNodeSlots; ++i)
                    k[i][j] = s0 + j * share < a.splits && node + i * kThreads < N ? __ldcg(keys + (s0 + j * share) * rows + i * kThreads) : 0ull;
#pragma unroll
            for (int j = 0; j < kTrip; ++j)
#pragma unroll
                for (int i = 0; i < kPathNodeSlots; ++i) best[i] = max(best[i], k[i][j]);
        }
        for (int o = 1; o < share; o *= 2) best[0] = max(best[0], __shfl_xor_sync(0xFFFFFFFFu, best[0], o));
#pragma unroll
        for (int i = 0; i < kPathNodeSlots; ++i)
            if (mine == 0 && node + i * kThreads < N) s_amax[node + i * kThreads] = key_index(best[i]);
        return 0u;
    };
    // a step parent -> v is accepted iff v's token is what the target model would emit after the parent
    const PathResult res = longest_accepted_path<false>(
        io, 0u, [&](float, int p, int, int t) { return t == s_amax[p]; }, [](int, int) { return 0.f; }, best_keys);
    // the target model's own next token
    if (tid == 0 && res.edges < a.Tcap && GSD_IN_BOUNDS(res.end >= 0 && res.end < N && res.edges >= 0, a.status))
        io.out_tok[res.edges] = s_amax[res.end];
}

}  // namespace

}  // namespace gsd

extern "C" size_t gsd_accept_workspace_bytes(const gsd_accept_params* p) {
    if (!p || p->B < 1 || p->N < 1 || p->N > GSD_MAX_NODES) return 0;
    // a key per slice: as many as the rule in gsd_accept can make of this many rows (the vocabulary may be
    // given as anything here, and nothing asks for a device)
    const size_t keys = std::max((size_t)p->B * p->N, (size_t)2 * gsd::kWaveCtas * gsd::kScratchSms);
    return std::max(gsd::accept_least_workspace(p->B, p->N), gsd::align_up(keys * 8, 256));
}

extern "C" int gsd_accept(const float* logits, const int32_t* draft_tokens,
                          const int32_t* parent_ptr, const int32_t* parent_idx,
                          int32_t* accepted_tokens, int32_t* accepted_len, int32_t* accepted_nodes,
                          const gsd_accept_params* p, void* workspace, size_t workspace_bytes,
                          int32_t* status, void* stream) {
    using namespace gsd;
    if (!p || !logits || !draft_tokens || !parent_ptr || !parent_idx || !accepted_tokens ||
        !accepted_len)
        return GSD_ERR_NULL_POINTER;
    if (p->B < 1 || p->N < 1 || p->N > GSD_MAX_NODES || p->V < 1 || p->Ecap < 1 || p->Tcap < 1)
        return GSD_ERR_BAD_SHAPE;
    if ((long long)p->B * p->N > (1ll << 30)) return GSD_ERR_BAD_SHAPE;
    if (((uintptr_t)logits & 3u) != 0) return GSD_ERR_MISALIGNED;
    // (a key per row is enough: the rows then go whole)
    const size_t need = accept_least_workspace(p->B, p->N);
    if (!workspace || workspace_bytes < need) return GSD_ERR_WORKSPACE;
    if (((uintptr_t)workspace & 7u) != 0) return GSD_ERR_MISALIGNED;
    DeviceInfo di;
    if (device_info(&di) != 0) return GSD_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;

    AcceptArgs a;
    a.logits = logits; a.tok = draft_tokens; a.pptr = parent_ptr; a.pidx = parent_idx;
    a.out_tok = accepted_tokens; a.out_len = accepted_len; a.out_nodes = accepted_nodes;
    a.keys = (unsigned long long*)workspace;
    a.status = status;
    a.B = p->B; a.N = p->N; a.V = p->V; a.Ecap = p->Ecap; a.Tcap = p->Tcap;
    // Slices of at least 4096 floats and CTAs for four waves (eight CTAs are resident per SM), so
    // that the last, partly filled wave is short: in captured graphs 2048 rows of 32000 take 44.5 us in one slice
    // each (1.7 waves), 42.5 in four; 60 rows of 128256 24.8 in one, 10.6 in sixteen; 2 rows of 1048576 9.3 in 32, 5.5
    // in the 256 that come of this.
    const size_t rows = (size_t)p->B * p->N, want = (size_t)kWaveCtas * di.sm_count;
    int splits = 1;
    while (rows * splits < want && p->V / (splits * 2) >= 4096 && rows * splits * 2 * 8 <= workspace_bytes) splits *= 2;
    a.splits = splits;
    void (*tail)(AcceptArgs) = splits > kTrip && 2 * p->N <= kThreads ? accept_tail_kernel<true> : accept_tail_kernel<false>;

    // grid.y holds at most 65535 rows: larger problems go out in blocks of whole sequences
    const int seq_per = 65535 / p->N;
    for (int b0 = 0; b0 < p->B; b0 += seq_per) {
        const int nb = (p->B - b0 < seq_per) ? p->B - b0 : seq_per;
        AcceptArgs s = a;
        s.logits += (size_t)b0 * p->N * p->V; s.tok += (size_t)b0 * p->N;
        s.pptr += (size_t)b0 * (p->N + 1); s.pidx += (size_t)b0 * p->Ecap;
        s.out_tok += (size_t)b0 * p->Tcap; s.out_len += b0;
        if (s.out_nodes) s.out_nodes += (size_t)b0 * p->Tcap;
        s.keys += (size_t)b0 * p->N * splits; s.B = nb;
        GSD_CUDA_TRY(launch_dependent(accept_kernel, dim3(splits, (unsigned)(nb * p->N)), dim3(kThreads), 0, st, s));
        GSD_CUDA_TRY(launch_dependent(tail, dim3((unsigned)nb), dim3(kThreads), 0, st, s));
    }
    return GSD_OK;
}

// ---------------------------------------------------------------------------------------
// gsd_accept_static: the same computation as gsd_accept with the scratch in a fixed array
// that lives in the library image, for callers that cannot hand over device memory.
namespace gsd {
namespace {
// A key per slice of every row, for at most GSD_STATIC_MAX_ROWS rows (the size is of an earlier layout with
// more to keep per row).
// Every GPU that loads the library holds these bytes until the process exits.
static __device__ __align__(256) unsigned char g_accept_scratch[GSD_STATIC_SCRATCH_BYTES];
}  // namespace
}  // namespace gsd

extern "C" int gsd_accept_static(const float* logits, const int32_t* draft_tokens,
                                 const int32_t* parent_ptr, const int32_t* parent_idx,
                                 int32_t* accepted_tokens, int32_t* accepted_len,
                                 int32_t* accepted_nodes, const gsd_accept_params* p,
                                 int32_t* status, void* stream) {
    using namespace gsd;
    if (!p) return GSD_ERR_NULL_POINTER;
    if (p->B < 1 || p->N < 1 || p->N > GSD_MAX_NODES) return GSD_ERR_BAD_SHAPE;
    if ((long long)p->B * p->N > GSD_STATIC_MAX_ROWS) {
        set_error_text("gsd_accept_static: B*N exceeds GSD_STATIC_MAX_ROWS");
        return GSD_ERR_WORKSPACE;
    }
    const size_t need = gsd_accept_workspace_bytes(p);
    if (need == 0 || need > (size_t)GSD_STATIC_SCRATCH_BYTES) {
        set_error_text("gsd_accept_static: scratch need exceeds GSD_STATIC_SCRATCH_BYTES");
        return GSD_ERR_WORKSPACE;
    }
    // In host code the array's name is only a handle; the device address has to be asked for,
    // once per device, with that device current.
    static void* addr[64] = {};
    int dev = 0;
    GSD_CUDA_TRY(cudaGetDevice(&dev));
    void* ptr = (dev >= 0 && dev < 64) ? addr[dev] : nullptr;
    if (!ptr) {
        GSD_CUDA_TRY(cudaGetSymbolAddress((void**)&ptr, g_accept_scratch));
        if (!ptr) return GSD_ERR_CUDA;
        if (dev >= 0 && dev < 64) addr[dev] = ptr;
    }
    return gsd_accept(logits, draft_tokens, parent_ptr, parent_idx, accepted_tokens, accepted_len,
                      accepted_nodes, p, ptr, (size_t)GSD_STATIC_SCRATCH_BYTES, status, stream);
}
