// gsd_verify_attn, last pass of a call whose items were cut along the key range: combines the
// partial results of every row.
//   m = max_s m_s;  out = sum_s 2^(m_s - m) O_s / sum_s 2^(m_s - m) l_s
//
// A block takes 32 rows of a row tile and 16 of its column groups: a lane is a row, a thread has two
// column groups (8 values, 16 bytes of output).  The rows of a column group are consecutive in the
// partial results, so every load of a warp is 512 contiguous bytes.  Few registers and short code
// on purpose: the launch lasts a few microseconds, and a form with four column groups a thread and
// the next four parts on their way while four are added up took 1 us longer.
#include "gsd_internal.cuh"
#include <cuda_bf16.h>
#include <math_constants.h>

namespace gsd {
namespace {

constexpr int kThreads = 256;
constexpr int kBatch = 4;        // parts of a row on their way at a time
constexpr int kCols = kThreads / 32 * 2;     // column groups of a block
constexpr int kWalkers = 296;    // blocks that walk over the items of a one-wave plan (two per SM)

struct MergeParams {
    const float4* part_o;
    const float2* part_ml;
    __nv_bfloat16* out;
    PlanDev plan;
    int N, Hq, Hkv, G, R, D;
    int tile_rows;           // rows of a tile in the partial results (128 or 64)
    int RT;                  // of them in use
    int tiles;               // row tiles of an item
    int groups;              // blocks of 32 rows of an item that can hold a row
    int B;
    const int* bal_hdr;      // balanced plan: [0] = items to merge (known on the device only)
    const int4* bal_merge;   // balanced plan: (pair, first slot, slots) per pair to merge, else nullptr
    int bal_groups;          // balanced plan: groups of CTAs
    SeqTable seq;            // per-sequence plan (hdr == nullptr otherwise); the grid then covers every item
    const int* left;         // one-wave plan: split counts, then (left_off on) first units per sequence; longest
    int left_off;            // first: the sequences in order; else nullptr
};

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// kWalk: a one-wave plan that cannot have cut every item.  The grid is small and walks over the items
// that were cut - none at all for sequences of one length, and then the launch should cost little: 10 x
// 64/8 heads, N 32, L 2048: 42.4 us with blocks for every item, 39.8 walking (37.1 with a plan that
// cannot cut, which takes 115 instead of 28.5 when one of the sequences has 8192 and the others 500).
// Where every item may be cut, one block for each part of it is up to 0.5 us faster.
template <bool kWalk>
__global__ void __launch_bounds__(kThreads) attn_merge_kernel(MergeParams p) {
    const int lane = threadIdx.x & 31;
    const int quads = p.D / 4, parts_of_row = quads / kCols;
    // Launched as a programmatic dependent of the attention kernel: the blocks may become
    // resident while that kernel drains; what it (or the planning kernel) wrote is only visible
    // after this wait.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    unsigned cut = 0;                                              // kWalk: the sequences that were cut
    int blocks = (int)gridDim.x;
    if (kWalk) {
        cut = __ballot_sync(0xFFFFFFFFu, lane < p.B && p.left[lane] > 1);
        blocks = __popc(cut) * p.Hkv * p.plan.tiles_per_unit * p.groups * parts_of_row;
    }
    for (int blk = blockIdx.x; blk < blocks; blk += gridDim.x) {   // (once, unless kWalk)
    const int col0 = (blk % parts_of_row) * kCols + (threadIdx.x >> 5) * 2;      // first column group of the thread
    const int g = blk / parts_of_row % p.groups;
    const int k = blk / parts_of_row / p.groups;
    // the k-th item that owns slots: group a comes first when it is split at all
    int item, nsplit, slot0, slot_step = 1;
    const int split_a = p.plan.splits_a > 1 ? p.plan.items_a : 0;
    if (kWalk) {
        const int per_seq = p.Hkv * p.plan.tiles_per_unit;
        const int at = k / per_seq, i = k - at * per_seq;
        const int b = (int)__fns(cut, 0, at + 1);                  // the at-th sequence that was cut
        nsplit = p.left[b];
        item = b * per_seq + i;
        slot0 = p.left[p.left_off + b] + i;
        slot_step = per_seq;
    } else if (p.bal_merge) {
        // the list of cut items was made on the device; the grid covers the most there can be
        const int tpu = p.plan.tiles_per_unit, rt = k % tpu;
        const int listed = p.bal_hdr[0];
        const int4 rec = p.bal_merge[k / tpu];       // a (sequence, kv head) pair that was cut (read beside the count)
        if (k / tpu >= listed) return;
        item = rec.x * tpu + rt; slot0 = rt * 2 * p.bal_groups + rec.y; nsplit = rec.z;
    } else if (p.seq.hdr) {
        const int per_seq = p.Hkv * p.plan.tiles_per_unit;
        const int b = k / per_seq;
        nsplit = p.seq.nsplit[b];
        if (nsplit == 1) return;                       // the item was stored by its only unit
        item = k;
        slot0 = p.seq.slot_off[b] + (k - b * per_seq) * nsplit;
    } else if (p.plan.balanced == 3) {
        const int per_seq = p.Hkv * p.plan.tiles_per_unit;
        const int b = k / per_seq;
        nsplit = p.left[b];
        if (nsplit == 1) return;
        item = k;
        slot0 = p.left[p.left_off + b] + (k - b * per_seq);
        slot_step = per_seq;
    } else if (k < split_a) {
        item = k; nsplit = p.plan.splits_a; slot0 = k * p.plan.splits_a;
    } else {
        item = p.plan.items_a + (k - split_a); nsplit = p.plan.splits_b;
        slot0 = split_a * p.plan.splits_a + (k - split_a) * p.plan.splits_b;
    }
    const int per_tile = p.tile_rows / 32;
    const int tile = g / per_tile, r = (g - tile * per_tile) * 32 + lane;
    const int unit = item / p.plan.tiles_per_unit;
    const int row = (item % p.plan.tiles_per_unit) * p.tiles * p.RT + tile * p.RT + r;
    if (r >= p.RT || row >= p.R) {
        if (kWalk) continue;
        return;
    }
    const int b = p.plan.longest_first ? p.left[unit / p.Hkv] : unit / p.Hkv, c = unit % p.Hkv;

    const size_t first = (size_t)slot0 * p.tiles + tile;
    const float2* ml_base = p.part_ml + first * p.tile_rows + r;
    const float4* o_base = p.part_o + (first * quads + col0) * p.tile_rows + r;
    const size_t ml_stride = (size_t)slot_step * p.tiles * p.tile_rows, o_stride = ml_stride * quads;
    float2 ml[kBatch];
    float4 v[kBatch][2];
    auto fetch = [&](int s0) {
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const bool in = s0 + j < nsplit;
            ml[j] = in ? ml_base[(size_t)(s0 + j) * ml_stride] : make_float2(-CUDART_INF_F, 0.f);
#pragma unroll
            for (int q = 0; q < 2; ++q)
                v[j][q] = in ? o_base[(size_t)(s0 + j) * o_stride + q * p.tile_rows] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    fetch(0);
    float m = fmaxf(fmaxf(ml[0].x, ml[1].x), fmaxf(ml[2].x, ml[3].x));
#pragma unroll 4
    for (int s = kBatch; s < nsplit; ++s) m = fmaxf(m, ml_base[(size_t)s * ml_stride].x);
    const float m_use = m == -CUDART_INF_F ? 0.f : m;
    float acc[2][4] = {};
    float l = 0.f;
#pragma unroll 1
    for (int s0 = 0; s0 < nsplit; s0 += kBatch) {
        if (s0 > 0) fetch(s0);
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const float wgt = exp2f(ml[j].x - m_use);     // 0 for an absent or empty split
            l += wgt * ml[j].y;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                acc[q][0] += wgt * v[j][q].x; acc[q][1] += wgt * v[j][q].y;
                acc[q][2] += wgt * v[j][q].z; acc[q][3] += wgt * v[j][q].w;
            }
        }
    }
    const float inv = l > 0.f ? 1.f / l : 0.f;
    __nv_bfloat16* dst = p.out + (((size_t)b * p.N + row / p.G) * p.Hq + c * p.G + row % p.G) * p.D + col0 * 4;
    uint4 o;
    o.x = pack_bf16(acc[0][0] * inv, acc[0][1] * inv);
    o.y = pack_bf16(acc[0][2] * inv, acc[0][3] * inv);
    o.z = pack_bf16(acc[1][0] * inv, acc[1][1] * inv);
    o.w = pack_bf16(acc[1][2] * inv, acc[1][3] * inv);
    *reinterpret_cast<uint4*>(dst) = o;
    if (!kWalk) return;
    }
}

}  // namespace

int launch_attn_merge(const AttnArgs& a) {
    MergeParams p;
    p.part_o = (const float4*)a.workspace;
    p.part_ml = (const float2*)((const char*)a.workspace + plan_part_o_bytes(a.plan, a.D));
    p.out = (__nv_bfloat16*)a.out;
    p.plan = a.plan.dev;
    p.N = a.N; p.Hq = a.Hq; p.Hkv = a.Hkv; p.G = a.G; p.R = a.N * a.G; p.D = a.D;
    p.tiles = a.plan.part_rows == 64 ? 1 : 2;
    p.tile_rows = a.plan.part_rows / p.tiles;
    p.RT = a.plan.rows_per_item / p.tiles;
    int split_items = (a.plan.dev.splits_a > 1 ? a.plan.dev.items_a : 0) +
                      (a.plan.dev.splits_b > 1 ? a.plan.items - a.plan.dev.items_a : 0);
    p.bal_hdr = nullptr;
    p.bal_merge = nullptr;
    p.bal_groups = 0;
    p.seq.hdr = nullptr; p.seq.nsplit = nullptr; p.seq.unit_off = nullptr; p.seq.slot_off = nullptr;
    p.left = a.plan.dev.balanced == 3 || a.plan.dev.longest_first ? plan_left_table(a.plan, a.D, a.workspace) : nullptr;
    p.left_off = (int)(align_up((size_t)a.B * sizeof(int), 256) / sizeof(int));
    p.B = a.B;
    bool walk = false;
    if (a.plan.dev.balanced == 3) {
        // (an item that is cut has at least one unit more than it would have whole, all items of a
        // sequence together)
        const int per_seq = a.Hkv * a.plan.dev.tiles_per_unit, most = (a.plan.ctas - a.plan.items) / per_seq * per_seq;
        walk = most < a.plan.items;
        split_items = walk ? most : a.plan.items;
    } else if (a.plan.dev.balanced == 2) {
        p.seq = plan_seq_table(a.plan, a.D, a.B, a.workspace);
        split_items = a.plan.items;
    } else if (a.plan.dev.balanced) {
        const BalTable t = plan_bal_table(a.plan, a.D, a.workspace);
        p.bal_hdr = t.hdr;
        p.bal_merge = t.merge;
        const int tpu = a.plan.dev.tiles_per_unit, groups = a.plan.ctas / tpu, pairs = a.plan.items / tpu;
        p.bal_groups = groups;
        split_items = (pairs < groups - 1 ? pairs : groups - 1) * tpu;   // one pair per cut at most
    }
    // blocks of 32 rows that can hold a row: all of them, or those up to the last row of a lone item
    const int per_tile = p.tile_rows / 32;
    p.groups = p.R >= a.plan.rows_per_item ? p.tiles * per_tile
               : p.R <= p.RT               ? (p.R + 31) / 32
                                           : per_tile + (p.R - p.RT + 31) / 32;
    long blocks = (long)split_items * p.groups * (p.D / 4 / kCols);
    if (blocks == 0) return GSD_OK;
    if (walk && blocks > kWalkers) blocks = kWalkers;
    cudaLaunchAttribute attr[1];
    dependent_launch_attr(attr);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = a.stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    GSD_CUDA_TRY(cudaLaunchKernelEx(&cfg, walk ? attn_merge_kernel<true> : attn_merge_kernel<false>, p));
    return GSD_OK;
}

}  // namespace gsd
