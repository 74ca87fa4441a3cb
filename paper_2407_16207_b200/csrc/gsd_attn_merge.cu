// gsd_verify_attn, last pass of a call whose items were cut along the key range: combines the
// partial results of every row.
//   m = max_s m_s;  out = sum_s 2^(m_s - m) O_s / sum_s 2^(m_s - m) l_s
//
// A block of four warps has 32 rows of a row tile and eight of their column groups (one of eight warps sixteen): a lane
// is a row, a thread has two column groups (8 values, 16 bytes of output).  The rows of a column group are consecutive in the
// partial results, so every load of a warp is 512 contiguous bytes.  For items of fewer than 64 rows of
// the mma.sync kernel a warp takes 8 rows and four column groups, one a thread, which leaves fewer lanes
// without a row (D 64, whole call: 2 x 12 heads, N 40, L 1500 15.2 us, 15.5 with 32 rows a warp; 32/8
// heads, N 8, L 4000 14.6 and 14.9; the tcgen05 kernel's few rows are up to 2% slower that way).
//
// The launch lasts a few microseconds: a few dependent trips to memory, in as few waves of blocks as possible.
// One pass: the sum is brought to a batch's maximum when that is larger (a pass over the maxima before it was two more
// trips for 18 parts).  Small blocks spread evenly, and what a block works on is the same for all its threads (two
// waves of blocks of 256 threads, every warp with a place of its own: D 64, 1 x 32/8 heads, N 8, L 4000, whole
// call 12.2 us, now 10.6; 1 x 32/8, N 37, L 3103 15.7, now 14.9).
#include "gsd_internal.cuh"
#include <cuda_bf16.h>
#include <math_constants.h>

namespace gsd {
namespace {

constexpr int kThreads = 128;
// Parts of a row on their way at a time, and blocks per SM that have to be resident: many parts are worth
// more than occupancy as long as all blocks are resident at once (the whole call in captured graphs: 8 items of 18
// parts, 256 rows, 42.2 us with four, 40.9 with eight; 32 items of 4 parts, 64 rows, 15.8 and 15.5), else it is the other
// way round (40 items of 3 to 5 parts: 24.2 with four, 26.0 with eight; limited to 64 registers, eight blocks an SM,
// calls took up to 2 us more).
constexpr int kBatchFew = 8, kBlocksFew = 3;
constexpr int kBatchMany = 4, kBlocksMany = 4;
constexpr int kWalkers = 592;    // blocks that walk over the items of a one-wave plan (four per SM)
// Blocks of eight warps (sixteen column groups), half as many of them, where four small blocks a SM would do but not
// three: the SMs that fall free first take five small blocks each and others are left with one or two.  512 small
// blocks -> 256 of these, whole call: 4 x 24/8 heads, N 40, L 1500 17.2 -> 16.8 us (16.7 with the former pass), D 64, 8 x
// 32/8, N 32, L 1500 18.9 -> 18.7, 2 x 64/8, N 32, L 4000 22.0 -> 21.6.  640 and 1280 small blocks are better small (1 x
// 40 heads, N 100, L 8000 36.4 and 37.3; 5 x 24/8, N 77, L 300-1999 25.5 and 27.1): the eight warps end together.
constexpr int kWideWarps = 8, kWideBlocks = 2, kWideUpTo = 4;

struct MergeParams {
    const float4* part_o;
    const float2* part_ml;
    __nv_bfloat16* out;
    PlanDev plan;
    int N, Hq, Hkv, G, R, D;
    int tile_rows;           // rows of a tile in the partial results (128 or 64)
    int RT;                  // of them in use
    int tiles;               // row tiles of an item
    int groups;              // runs of kRows rows of an item that can hold a row
    int work;                // blocks' worth of work
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
template <bool kWalk, int kRows, bool kFew, int kWarps = kThreads / 32>
__global__ void __launch_bounds__(kWarps * 32, kWarps == kWideWarps ? kWideBlocks : kFew ? kBlocksFew : kBlocksMany) attn_merge_kernel(MergeParams p) {
    const int lane = threadIdx.x & 31;
    constexpr int kBatch = kFew ? kBatchFew : kBatchMany;
    constexpr int kGroups = kRows == 32 ? 2 : 1;                   // column groups of a thread
    constexpr int kSpan = 32 / kRows * kGroups;                    // of a warp
    const int quads = p.D / 4, parts_of_row = quads / kSpan / kWarps;     // blocks that share a row
    // Launched as a programmatic dependent of the attention kernel: the blocks may become
    // resident while that kernel drains; what it (or the planning kernel) wrote is only visible
    // after this wait, which comes as late as the plan allows: working out a warp's place takes a
    // dozen divisions.
    auto ready = []() { wait_for_predecessor(); };
    unsigned cut = 0;                                              // kWalk: the sequences that were cut
    int work = p.work;
    if (kWalk) {
        ready();
        cut = __ballot_sync(0xFFFFFFFFu, lane < p.B && p.left[lane] > 1);
        work = __popc(cut) * p.Hkv * p.plan.tiles_per_unit * p.groups * parts_of_row;
    }
    for (int w = (int)blockIdx.x; w < work; w += (int)gridDim.x) {                 // (once, unless kWalk)
    // first column group of the thread
    const int col0 = (w % parts_of_row * kWarps + (int)(threadIdx.x >> 5)) * kSpan + lane / kRows * kGroups;
    const int g = w / parts_of_row % p.groups;
    const int k = w / parts_of_row / p.groups;
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
        ready();
        const int listed = p.bal_hdr[0];
        const int4 rec = p.bal_merge[k / tpu];       // a (sequence, kv head) pair that was cut (read beside the count)
        if (k / tpu >= listed) return;
        item = rec.x * tpu + rt; slot0 = rt * 2 * p.bal_groups + rec.y; nsplit = rec.z;
    } else if (p.seq.hdr) {
        const int per_seq = p.Hkv * p.plan.tiles_per_unit;
        const int b = k / per_seq;
        ready();
        nsplit = p.seq.nsplit[b];
        if (nsplit == 1) return;                       // the item was stored by its only unit
        item = k;
        slot0 = p.seq.slot_off[b] + (k - b * per_seq) * nsplit;
    } else if (p.plan.balanced == 3) {
        const int per_seq = p.Hkv * p.plan.tiles_per_unit;
        const int b = k / per_seq;
        ready();
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
    const int per_tile = p.tile_rows / kRows;
    const int tile = g / per_tile, r = (g - tile * per_tile) * kRows + lane % kRows;
    const int unit = item / p.plan.tiles_per_unit;
    const int row = (item % p.plan.tiles_per_unit) * p.tiles * p.RT + tile * p.RT + r;
    if (r >= p.RT || row >= p.R) {
        if (kWalk) continue;
        ready();                           // (the grid must not end before its predecessor)
        return;
    }
    const int place = unit / p.Hkv, c = unit % p.Hkv, node = row / p.G, head = c * p.G + row % p.G;
    if (!kWalk) ready();
    const int b = p.plan.longest_first ? p.left[place] : place;

    const size_t first = (size_t)slot0 * p.tiles + tile;
    const float2* ml_at = p.part_ml + first * p.tile_rows + r;
    const float4* o_at = p.part_o + (first * quads + col0) * p.tile_rows + r;
    const unsigned ml_stride = (unsigned)(slot_step * p.tiles * p.tile_rows), o_stride = ml_stride * (unsigned)quads;
    float m = -CUDART_INF_F, l = 0.f;
    float acc[kGroups][4] = {};
#pragma unroll 1
    for (int s0 = 0; s0 < nsplit; s0 += kBatch) {
        float2 ml[kBatch];
        float4 v[kBatch][kGroups];
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const bool in = s0 + j < nsplit;
            ml[j] = in ? *ml_at : make_float2(-CUDART_INF_F, 0.f);
#pragma unroll
            for (int q = 0; q < kGroups; ++q) v[j][q] = in ? o_at[q * p.tile_rows] : make_float4(0.f, 0.f, 0.f, 0.f);
            ml_at += ml_stride;
            o_at += o_stride;
        }
        // what has been added up so far is brought to the batch's maximum, if that is larger
        float top = m;
#pragma unroll
        for (int j = 0; j < kBatch; ++j) top = fmaxf(top, ml[j].x);
        const float top_use = top == -CUDART_INF_F ? 0.f : top;
        const float back = exp2f(m - top_use);
        m = top;
        l *= back;
#pragma unroll
        for (int q = 0; q < kGroups; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[q][e] *= back;
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const float wgt = exp2f(ml[j].x - top_use);   // 0 for an absent or empty split
            l += wgt * ml[j].y;
#pragma unroll
            for (int q = 0; q < kGroups; ++q) {
                acc[q][0] += wgt * v[j][q].x; acc[q][1] += wgt * v[j][q].y;
                acc[q][2] += wgt * v[j][q].z; acc[q][3] += wgt * v[j][q].w;
            }
        }
    }
    const float inv = l > 0.f ? 1.f / l : 0.f;
    __nv_bfloat16* dst = p.out + (((size_t)b * p.N + node) * p.Hq + head) * p.D + col0 * 4;
    uint32_t o[2 * kGroups];
#pragma unroll
    for (int q = 0; q < kGroups; ++q) {
        o[2 * q] = pack_bf16(acc[q][0] * inv, acc[q][1] * inv);
        o[2 * q + 1] = pack_bf16(acc[q][2] * inv, acc[q][3] * inv);
    }
    if constexpr (kGroups == 2) *reinterpret_cast<uint4*>(dst) = make_uint4(o[0], o[1], o[2], o[3]);
    else *reinterpret_cast<uint2*>(dst) = make_uint2(o[0], o[1]);
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
    // runs of rows that can hold a row: all of them, or those up to the last row of a lone item
    const int rows = p.tile_rows == 64 && p.R < 64 ? 8 : 32, span = rows == 8 ? 4 : 2;
    const int per_tile = p.tile_rows / rows;
    p.groups = p.R >= a.plan.rows_per_item ? p.tiles * per_tile
               : p.R <= p.RT               ? (p.R + rows - 1) / rows
                                           : per_tile + (p.R - p.RT + rows - 1) / rows;
    const long work = (long)split_items * p.groups * (p.D / 4 / span / (kThreads / 32));
    if (work == 0) return GSD_OK;
    p.work = (int)work;
    long blocks = work;
    if (walk && blocks > kWalkers) blocks = kWalkers;
    DeviceInfo di;
    if (device_info(&di) != 0) return GSD_ERR_CUDA;
    const bool few = blocks <= (long)kBlocksFew * di.sm_count;
    void (*kernel)(MergeParams) = nullptr;
    if (rows == 8) kernel = few ? attn_merge_kernel<false, 8, true> : attn_merge_kernel<false, 8, false>;    // (the mma.sync kernel has no one-wave plan)
    else if (walk) kernel = few ? attn_merge_kernel<true, 32, true> : attn_merge_kernel<true, 32, false>;
    else kernel = few ? attn_merge_kernel<false, 32, true> : attn_merge_kernel<false, 32, false>;
    int threads = kThreads;
    if (rows == 32 && !walk && !few && blocks <= (long)kWideUpTo * di.sm_count) {
        kernel = attn_merge_kernel<false, 32, false, kWideWarps>;
        threads = kWideWarps * 32;
        blocks = blocks * kThreads / threads;                      // (a row has two small blocks at least)
        p.work = (int)blocks;
    }
    GSD_CUDA_TRY(launch_dependent(kernel, dim3((unsigned)blocks), dim3(threads), 0, a.stream, p));
    return GSD_OK;
}

}  // namespace gsd
