// Internal declarations shared by the translation units of libgsd (not part of the ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>
#include "gsd.h"

namespace gsd {

void set_cuda_error(cudaError_t e, const char* where);
void set_error_text(const char* text);

#define GSD_CUDA_TRY(expr)                                   \
    do {                                                     \
        cudaError_t e__ = (expr);                            \
        if (e__ != cudaSuccess) {                            \
            ::gsd::set_cuda_error(e__, #expr);               \
            return GSD_ERR_CUDA;                             \
        }                                                    \
    } while (0)

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Index checks of the checking build (compiled with -DGSD_BOUNDS_CHECK into libgsd_check.so; the
// stand-in for a memory sanitizer): at the places where a kernel forms an index into global
// memory from data or from its work plan, GSD_IN_BOUNDS(condition, status) is the condition
// itself and, when it fails, ORs GSD_DEV_BOUNDS into the status word - the caller skips the
// access, nothing traps.  In the ordinary build it is the constant true and costs nothing.
#ifdef GSD_BOUNDS_CHECK
__device__ __forceinline__ bool note_out_of_bounds(int32_t* status) {
    if (status) atomicOr((unsigned*)status, GSD_DEV_BOUNDS);
    return false;
}
#define GSD_IN_BOUNDS(cond, status) ((cond) ? true : ::gsd::note_out_of_bounds(status))
#else
#define GSD_IN_BOUNDS(cond, status) (true)
#endif

struct DeviceInfo {
    int sm_count;
    int max_smem_optin;
};
// Properties of the current device (cached per device ordinal).
int device_info(DeviceInfo* out);

// ---- work plan of one gsd_verify_attn call ----
// A work item is one row tile (rows_per_item stacked rows) of one (sequence, kv head); item
// index = unit * tiles_per_unit + row tile.  The first items_a items are cut into splits_a
// key ranges, the remaining ones into splits_b; CTAs are numbered group a first.  Only items
// with more than one split own partial-result slots (one per split, numbered in CTA order).
//
// Balanced plan (tcgen05 back end only): the host cannot see the sequence lengths, so for
// batches whose lengths differ a plan made from Lmax leaves CTAs idle.  Here the key tiles of
// all (sequence, kv head) pairs are laid end to end - pair after pair, ceil(len/128) prefix
// tiles plus the draft tiles each - and group g of `ctas / tiles_per_unit` groups takes the
// g-th equal share of that line; CTA r of a group works on row-tile item r of every pair in
// the share.  A small kernel builds the table from seq_lens on the device before the
// attention kernel reads it: per group its units (pair, tile range, partial-result slot or -1
// for a whole pair), and per pair that was cut the run of slots to merge.  Slots are numbered
// along the line, so the pieces of one pair have consecutive slots; a group has at most two
// partial units (its first and last).  CTA r adds r * 2 * groups to a slot of its group.
//
// Per-sequence plan (tcgen05 back end only): a lighter form of the same idea that keeps the
// CTAs of one sequence in step.  Every item of sequence b is cut into nsplit[b] equal key
// ranges, nsplit[b] = its tile count over a common target length (rounded), chosen on the
// device so that the batch makes about `units_wanted` units; units are numbered sequence by
// sequence, range by range, item by item, and CTA k walks units k, k + grid, ...  The heads of
// a sequence then read the same cache rows at the same time, which the head-interleaved cache
// layout rewards (a row of the cache holds all kv heads of a position).
//
// One-wave plan (tcgen05 back end, the automatic choice for 2 to 32 sequences whose items do not
// fill the device):
// every item of sequence b is cut into ceil(tiles of b / T) equal key ranges, T the smallest tile
// count with which all units are resident at once, found by every CTA of the attention kernel
// from seq_lens; unit w belongs to CTA w and owns slot w.  With equal lengths this is the even
// split; with lengths from 1024 to 4096 the longest units are half as long as when every
// sequence is cut alike.
//
// Longest first (tcgen05 back end, the automatic choice with more items than the device holds):
// the items of a fixed plan are numbered with the sequences in descending order of length, and CTA
// k takes them forth and back - k, 2 grid - 1 - k, 2 grid + k, ... - so that every CTA gets long
// and short ones.  32 sequences of 200-2100, 512 items on 148 CTAs: the last CTA ended 28% after the
// mean, the call took 114.5 us; 103.4 in this order.
struct PlanDev {
    int items_a, splits_a, splits_b, tiles_per_unit;
    int balanced;       // 1: units come from the table built on the device; 2: per-sequence split counts
                        // from the device; 3: one-wave plan
    int longest_first;  // sequences in descending order of length (fixed plans only)
};
constexpr int kPlanSeqs = 384;      // sequences the attention kernel can put in order (one per thread)
struct AttnPlan {
    int kernel;         // GSD_ATTN_MMA or GSD_ATTN_TCGEN05
    int rows_per_item;  // stacked rows of an item: 64 (mma.sync back end) or two row tiles of attn_tcgen05_rows(G) (tcgen05 back end)
    int part_rows;      // rows of a partial-result slot: 64 or 2 x 128
    int items;
    int ctas;
    int slots;          // partial-result slots; 0 when nothing is split
    PlanDev dev;
    size_t ws_bytes;
};
// The table of a balanced plan, in the workspace behind the partial results.
struct BalTable {
    int* hdr;       // [0] pairs to merge, [1] tiles on the line, [2] tiles per group
    int2* cta;      // [groups]  (index of the group's first unit, number of units)
    int4* merge;    // [groups]  (pair, first slot, number of slots, -)
    int4* units;    // [pairs + groups]  (pair, first tile, end tile, slot or -1); tiles count the
                    //                   prefix tiles, then ALL draft tiles of the pair
    int* off;       // [B + 1] start of each sequence on the line
};
__host__ __device__ inline void plan_decode(const PlanDev& pl, int cta, int& item, int& split, int& nsplit, int& slot) {
    const int ctas_a = pl.items_a * pl.splits_a;
    if (cta < ctas_a) {
        item = cta / pl.splits_a;
        split = cta - item * pl.splits_a;
        nsplit = pl.splits_a;
        slot = cta;
    } else {
        const int rem = cta - ctas_a;
        const int k = rem / pl.splits_b;
        item = pl.items_a + k;
        split = rem - k * pl.splits_b;
        nsplit = pl.splits_b;
        slot = (pl.splits_a > 1 ? ctas_a : 0) + rem;
    }
}
// `by_length`: the plans that the attention kernel makes from seq_lens may be chosen.
AttnPlan attn_make_plan(const gsd_attn_params* p, int sm_count, bool by_length = true);

// ---- verify-attention back ends (they validate nothing: the API layer did) ----
struct AttnArgs {
    const void *q, *k_cache, *v_cache, *draft_k, *draft_v;
    const uint32_t* mask;
    const int32_t* seq_lens;
    void* out;
    int B, N, Hq, Hkv, D, Lmax, G, W;
    float scale_log2;   // softmax_scale * log2(e)
    AttnPlan plan;
    void* workspace;
    int32_t* status;
    cudaStream_t stream;
};

int attn_pick_kernel(const gsd_attn_params* p, int sm_count);   // GSD_ATTN_MMA or GSD_ATTN_TCGEN05
// Partial results: fp32 accumulators, then (max, sum) pairs.  A slot holds the row tiles of an item
// (one of 64 rows, or two of 128); a tile is [D / 4 column groups][rows] of float4 - the rows of a
// column group are consecutive, for the store of an accumulator (a lane per row) and for the merge
// alike - and [rows] of float2.
inline size_t plan_part_o_bytes(const AttnPlan& pl, int D) { return align_up((size_t)pl.slots * pl.part_rows * D * sizeof(float), 256); }
inline size_t plan_part_ml_bytes(const AttnPlan& pl) { return align_up((size_t)pl.slots * pl.part_rows * 2 * sizeof(float), 256); }

// The table of a per-sequence plan, in the workspace behind the partial results.
struct SeqTable {
    int* hdr;        // [0] units of work, [1] tiles of all items, [2] target tiles per unit
    int* nsplit;     // [B]     key ranges per item of the sequence
    int* unit_off;   // [B + 1] first unit of the sequence
    int* slot_off;   // [B + 1] first partial-result slot of the sequence (sequences cut in two or more only)
};
inline size_t plan_bal_bytes(const AttnPlan& pl, int B) {
    // what the attention kernel leaves for the merge pass: split counts and first units, or the order
    if (pl.dev.balanced == 3) return 2 * align_up((size_t)B * sizeof(int), 256);
    if (!pl.dev.balanced) return pl.dev.longest_first && pl.slots ? align_up((size_t)B * sizeof(int), 256) : 0;
    if (pl.dev.balanced == 2) return 256 + 3 * align_up((size_t)(B + 1) * sizeof(int), 256);
    return 256 + align_up((size_t)pl.ctas * sizeof(int2), 256) + align_up((size_t)pl.ctas * sizeof(int4), 256) +
           align_up((size_t)(pl.items + pl.ctas) * sizeof(int4), 256) + align_up((size_t)(B + 1) * sizeof(int), 256);
}
inline BalTable plan_bal_table(const AttnPlan& pl, int D, void* workspace) {
    char* at = (char*)workspace + plan_part_o_bytes(pl, D) + plan_part_ml_bytes(pl);
    BalTable t;
    t.hdr = (int*)at; at += 256;
    t.cta = (int2*)at; at += align_up((size_t)pl.ctas * sizeof(int2), 256);
    t.merge = (int4*)at; at += align_up((size_t)pl.ctas * sizeof(int4), 256);
    t.units = (int4*)at; at += align_up((size_t)(pl.items + pl.ctas) * sizeof(int4), 256);
    t.off = (int*)at;
    return t;
}

inline SeqTable plan_seq_table(const AttnPlan& pl, int D, int B, void* workspace) {
    char* at = (char*)workspace + plan_part_o_bytes(pl, D) + plan_part_ml_bytes(pl);
    const size_t row = align_up((size_t)(B + 1) * sizeof(int), 256);
    SeqTable t;
    t.hdr = (int*)at; at += 256;
    t.nsplit = (int*)at; at += row;
    t.unit_off = (int*)at; at += row;
    t.slot_off = (int*)at;
    return t;
}
// The first word of what the attention kernel leaves for the merge pass (balanced == 3, longest_first).
inline int* plan_left_table(const AttnPlan& pl, int D, void* workspace) {
    return (int*)((char*)workspace + plan_part_o_bytes(pl, D) + plan_part_ml_bytes(pl));
}
constexpr int kSeqPlanWaves = 2;              // units a per-sequence plan aims at, per resident CTA
constexpr int kSeqPlanMaxSplit = 32;

int launch_attn_plan(const AttnArgs& a);      // plans made on the device only: builds the table
int launch_attn_mma(const AttnArgs& a);
int launch_attn_tcgen05(const AttnArgs& a);
bool attn_tcgen05_supports(int D, int G);
int attn_tcgen05_rows(int G);                 // stacked rows of one row tile
int launch_attn_merge(const AttnArgs& a);
// test hook behind gsd_debug_attn_wait (process-wide; 0 restores the default limit)
void debug_attn_wait(unsigned long long limit_ns, int withhold_first_k);

// ---- rows of logits ----
// A row of fp32 logits as `head` entries (0 to 3) up to the first 16-byte boundary, `nvec` aligned
// groups of four, and a tail of 0 to 3 entries.  With a vocabulary that is no multiple of four
// (50257) every row starts at another alignment; the groups keep it on 16-byte loads.
struct RowSpan {
    int head, nvec;
};
__device__ __forceinline__ RowSpan row_span(const float* x, int V) {
    const int to_boundary = (int)((0u - (unsigned)(reinterpret_cast<uintptr_t>(x) >> 2)) & 3u);
    RowSpan r;
    r.head = min(to_boundary, V);
    r.nvec = (V - r.head) >> 2;
    return r;
}

// Sums of exponentials form (x - maximum) * log2 e as x * log2 e - maximum * log2 e in one fused
// multiply-add.  The rounding of the second product is 2^-24 of it: harmless for logits, but at a
// maximum of -1e10 or -3.4e38 (sixteen entries masked with such a number, next to one another in a
// thread's share) the factor it makes overflows.  Beyond this magnitude the difference is formed
// first.  (2^20: there the factor is still within 2^+-0.1.)
constexpr float kLargeLogit = 1048576.f;
__device__ __forceinline__ float4 minus(const float4& x, float m) { return make_float4(x.x - m, x.y - m, x.z - m, x.w - m); }

// The least scratch gsd_accept takes: a key per row (and four bytes per sequence, which it needed once).
inline size_t accept_least_workspace(int B, int N) { return align_up((size_t)B * N * 8 + (size_t)B * 4, 256); }

// ---- programmatic dependent launches ----
// A kernel launched with this attribute may start while its predecessor on the stream still runs; it
// executes griddepcontrol.wait before it first touches what that one (or anything before it) writes.
inline void dependent_launch_attr(cudaLaunchAttribute* attr) {
    attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr->val.programmaticStreamSerializationAllowed = 1;
}
// All small kernels of an iteration are launched this way, wait first and let their own successor start at
// once, so that the launches of a chain of them overlap.  Among other passes, one by one launched -> so:
// the step of 6 x 32/8 heads, D 64, N 9, L 200, V 128256 37.3 -> 29.2 us; gsd_accept, 3 x 61 rows of 50257, 14.0 ->
// 11.6; gsd_accept_sampled, 8 x 256 of 32000, 53.5 -> 50.8.  A kernel whose second half reads inputs before
// it waits (the acceptance and draft calls: the graph, while the logits are streamed) lets it start only
// after its own wait: by then everything that precedes the call is over.
template <class... P, class... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A... args) {
    cudaLaunchAttribute attr[1];
    dependent_launch_attr(attr);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
#ifdef __CUDACC__
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_successor_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

}  // namespace gsd
