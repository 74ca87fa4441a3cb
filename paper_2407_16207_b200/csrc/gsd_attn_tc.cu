// gsd_verify_attn, tcgen05 back end (sm_100a): TMA-fed, TMEM-resident flash-attention over the
// stacked (draft node x GQA head) rows, for head dimensions 64 and 128 and groups of up to 128 heads.
//
// Tree attention over the flattened token graph (Sec. 4.1) with the committed prefix in the
// KV cache (Sec. 4.2): row r = (node r / G, head r % G) of kv head c attends to cache rows
// j < seq_lens[b] and to the draft rows whose bit is set in the node's ancestor mask.
//
// A unit of work is up to two row tiles of 128 stacked rows (a group size G that does not divide
// 128: the 128 / G whole nodes that fit; three heads a group use 126 of the 128 rows) of one
// (sequence, kv head) and a
// contiguous range of 128-key tiles (prefix tiles, then the draft tiles that hold a visible
// key for any of its rows).  Warp roles:
//   warps 0-3   softmax of stream 0 (thread = row = TMEM lane)
//   warps 4-7   softmax of stream 1
//   warp  8     TMA producer (one thread): Q once, then K and V tiles into two smem rings
//   warp  9     QK^T issuer, warp 11 PV issuer (converged, one elected lane per instruction)
//   warp 10     TMEM allocation / release
// A stream is a row tile (two row tiles: both streams see every key tile) or, for a unit with
// one row tile, the even / odd key tiles of that row tile (merged in the epilogue).  A job is
// one key tile of one stream; jobs alternate between the streams.
// TMEM (512 columns) at D = 128: S (128) | P0 (64) | P1 (64) | O0 (128) | O1 (128); the layout at
// D = 64 is in Geo.  There is one score
// buffer: QK^T of job k+1 is issued as soon as the softmax of job k has pulled its score row
// into registers, i.e. it runs under that softmax; P (bf16) has a buffer per stream and
// O_i += P_i V follows when the softmax hands P over (in two halves of 64 keys).  So neither
// softmax warpgroup ever waits for a QK^T that could not start.  The two kinds of MMA are
// issued by two warps on different schedulers, each paced only by its own barriers (the
// softmax warps are almost always ready to issue, so one issuing warp gets too few slots
// to feed the tensor pipe).  The running maximum is only raised when a tile
// exceeds it by more than 2^8, or always, by the shape (kRescaleThreshold); the accumulator is
// then rescaled in place in TMEM by the row's own thread.  Every mbarrier wait is bounded: on
// expiry the kernel raises GSD_DEV_WAIT_EXPIRED, all roles leave their loops, TMEM is released.
#include "gsd_internal.cuh"
#include <cuda.h>
#include <cuda_bf16.h>
#include <math_constants.h>
#include <stdio.h>

namespace gsd {
namespace {

constexpr int BM = 128;            // rows per row tile
constexpr int BN = 128;            // keys per tile
constexpr int kMaxStages = 4;      // ring stages at most (barriers are laid out for this many)
constexpr uint32_t HALF_BYTES = 128 * 64 * 2;     // one [128 rows][64 bf16] swizzled block
constexpr int kThreads = 384;

// What depends on the head dimension.  A tile is HD / 64 swizzled blocks of 64 columns.  The
// rings hold 64 KB of K and as much of V either way: two stages of 32 KB or four of 16 KB.  TMEM
// columns (32-bit words): a bf16 P tile and an accumulator per stream, and the scores.  With
// HD = 128 that leaves room for ONE score tile, which the streams share; with HD = 64 the
// accumulators are half as wide and each stream has its own, so a stream's QK^T only waits for
// that stream's own softmax (at HD = 64 the exponentials cost twice the tensor time: the softmax
// warps must never wait).
// Where a CTA's units come from is a template argument: the first microseconds of a call are bound by
// the fetch of the kernel's own instructions, and with all the plans in one kernel a call of a few
// tiles started 1.5 us later.
enum PlanKind {
    PLAN_FIXED,     // host plan
    PLAN_ORDERED,   // host plan, longest sequences first
    PLAN_WAVE,      // one-wave plan
    PLAN_TABLE      // tables built by a planning kernel
};

template <int HD>
struct Geo {
    static constexpr int BLOCKS = HD / 64;
    static constexpr uint32_t TILE_BYTES = BLOCKS * HALF_BYTES;   // a 128 x HD bf16 tile
    static constexpr int ST = HD == 128 ? 2 : 4;                  // stages of the K ring and of the V ring
    static constexpr uint32_t STAGE_BYTES = 32 * 64;              // output rows of a softmax warp, 32 columns at a time
    static constexpr uint32_t SMEM_BYTES = (2 + 2 * ST) * TILE_BYTES + 8 * STAGE_BYTES + 1024;  // tiles, staging, alignment slack
    static constexpr bool TWO_S = HD == 64;
    static constexpr uint32_t COL_S0 = 0, COL_P0 = 128, COL_P1 = 192, COL_O0 = 256, COL_O1 = 256 + HD;
    static constexpr uint32_t COL_S1 = TWO_S ? 384 : COL_S0;
    static_assert(COL_O1 + HD <= (TWO_S ? 384 : 512), "512 TMEM columns");
};
// The running maximum of a row may lag behind by this much (log2 units) where groups divide 128 heads, D
// is 128 and there are 64 rows or more.  Elsewhere it is exact, as in the mma.sync kernel: the largest
// weights of a row are then 1 and lose nothing in bf16.  Error against 64 bits, lagging -> exact
// (mma.sync): 4 x 32/8 heads, D 64, N 128 2.31e-3 -> 2.21e-3 (2.24e-3); groups of 3, N 77 2.28e-3 ->
// 2.19e-3 (2.18e-3); of 7, N 200 2.34e-3 -> 2.27e-3 (2.27e-3).  Its price there: 32.7 -> 34.9 us, 25.7 ->
// 26.8, 54.3 -> 62.5 (mma.sync: 83.1, 50.5, 215).
constexpr float kRescaleThreshold = 8.0f;
// Units of work per CTA decoded in the prologue.  A fixed plan with more is launched in several parts;
// only the plans from tables decode further units where they are needed.
constexpr int kUnitTable = 128;
constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // default limit of every in-kernel wait

// Test hook (see gsd_debug_attn_wait): a shorter limit and, optionally, a CTA's first K tile
// withheld so that a wait really runs out.
unsigned long long g_wait_limit_ns = kWaitLimitNs;
int g_withhold_first_k = 0;

// What every bounded wait looks at, in shared memory: word 0 is raised by the first wait that
// gives up (all other waits then return within a few polls), words 2-3 hold the time limit.
struct WaitCtl {
    int abort;
    int pad;
    unsigned long long limit_ns;
};

enum Bar {
    BAR_Q_FULL = 0,
    BAR_K_FULL = 1,                          // one per stage
    BAR_K_EMPTY = BAR_K_FULL + kMaxStages,   // one per stage
    BAR_V_FULL = BAR_K_EMPTY + kMaxStages,   // one per stage
    BAR_V_EMPTY = BAR_V_FULL + kMaxStages,   // one per stage
    BAR_S_FULL = BAR_V_EMPTY + kMaxStages,   // 2: the scores of a job of stream i are in its S
    BAR_S_FREE = BAR_S_FULL + 2,      // 2: the softmax of stream i has read them out
    BAR_P_READY = BAR_S_FREE + 2,     // 2: keys 0..63 of P_i are in TMEM
    BAR_P_READY2 = BAR_P_READY + 2,   // 2: keys 64..127 of P_i are in TMEM
    BAR_P_FREE = BAR_P_READY2 + 2,    // 2: the PV of a job of stream i (and all before it) has completed
    BAR_O_DONE = BAR_P_FREE + 2,      // 2: every PV of the unit on stream i has completed
    BAR_O_FREE = BAR_O_DONE + 2,      // 2: the accumulator rows of the unit have been read out
    BAR_Q_EMPTY = BAR_O_FREE + 2,     // 1: every QK^T of the unit has completed
    BAR_ML_READY = BAR_Q_EMPTY + 1,   // 1: (max, sum) of the odd-tile stream are in shared memory
    BAR_DRAIN = BAR_ML_READY + 1,     // 2: every MMA issued by the QK^T / PV warp has completed
    BAR_COUNT = BAR_DRAIN + 2
};

struct TcParams {
    const uint32_t* mask;
    const int32_t* seq_lens;
    __nv_bfloat16* out;
    float* part_o;
    float* part_ml;
    int32_t* status;
    int out_by_32;    // `out` starts on a 32-byte boundary (16 is all that is promised)
    int B, N, Hq, Hkv, Lmax, G, W, R;
    int RT;           // stacked rows a row tile holds: the whole nodes that fit 128 rows, 128 / G * G
    float scale_log2;
    float raise_above;  // the running maximum of a row is raised when a tile exceeds it by more than this (log2 units)
    PlanDev plan;
    int work0;        // first unit of this launch
    int total_work;   // units of work of this launch
    int slots;        // partial-result slots of the plan
    const int2* bal_cta;     // balanced plan: (first unit, units) of every group of CTAs, else nullptr
    const int4* bal_units;   // balanced plan: (pair, first tile, end tile, slot or -1)
    int* left;               // what the merge pass needs of a plan made here (plan_left_table)
    int left_off;
    SeqTable seq;            // per-sequence plan: split counts and unit / slot offsets (hdr == nullptr otherwise)
    unsigned long long wait_limit_ns;
    int withhold_first_k;   // test hook: every CTA leaves out the K copy of its first key tile
};

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait.  Returns false when the wait gave up (time limit, or another role raised the
// abort flag); the caller then leaves its loop.  `ignore_abort` is for the final drain.
__device__ __forceinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                            int32_t* status, bool ignore_abort) {
    const unsigned long long t0 = global_ns();
    const unsigned long long limit = reinterpret_cast<const volatile WaitCtl*>(abort_flag)->limit_ns;
    for (unsigned it = 0;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 63u) {
            if (!ignore_abort && *abort_flag) return false;
            if (global_ns() - t0 > limit) {
                *abort_flag = 1;
                if (status) atomicOr((unsigned*)status, GSD_DEV_WAIT_EXPIRED);
                return false;
            }
        }
    }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          int32_t* status) {
    if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait_slow(bar, parity, abort_flag, status, false);
}
// the same, called by all lanes of a converged warp; the answer is made uniform
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               int32_t* status) {
    return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, abort_flag, status));
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// The MMA warp runs its loops with all 32 lanes converged and elects one lane per tcgen05
// instruction: addresses, descriptors and loop state are then warp-uniform, which costs the
// warp far fewer issue slots than a single-lane branch would (the softmax warps on the same
// scheduler are almost always ready to issue, so every extra instruction here waits its turn).
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile(
        "{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n"
        " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar) : "memory");
}
// 32 lanes x 32 consecutive fp32 columns: thread t of the warp gets lane (base + t).  v[0..31] must be
// register-resident (constant indices after unrolling).
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float* v) {
    uint32_t* r = reinterpret_cast<uint32_t*>(v);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc_st32(uint32_t taddr, const float (&v)[32]) {
    const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

// 32 bytes to a 32-byte aligned address
__device__ __forceinline__ void st_global8(void* dst, const uint32_t (&v)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// packed fp32 pairs (one instruction for two lanes of arithmetic)
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d)
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)),
          "l"(*reinterpret_cast<unsigned long long*>(&c)));
    return *reinterpret_cast<float2*>(&d);
}
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d)
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)));
    return *reinterpret_cast<float2*>(&d);
}

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// ---- shared-memory matrix descriptors (128-byte swizzle, 8-row groups 1024 bytes apart)
constexpr uint64_t kDescBase = (1ull << 46) | (2ull << 61);   // descriptor version 1, SWIZZLE_128B
// K-major operand (rows x 64 bf16 per block): leading offset unused (1), stride = 1024 B.
// MN-major operand (V: [key][64 d] blocks): leading offset = distance between the two
// 64-column blocks, stride = 1024 B between 8-key groups.
// Descriptors are handled as (low word, high word): the high word is common to both kinds, and
// a k-step only adds a small constant to the start-address field of the low word (the
// tiles sit below 256 KB, so the sum stays inside the 14-bit field).
constexpr uint32_t kDescHi = (uint32_t)((kDescBase | ((uint64_t)(1024 >> 4) << 32)) >> 32);
__device__ __forceinline__ uint32_t desc_lo_kmajor(uint32_t addr) { return ((addr & 0x3FFFFu) >> 4) | (1u << 16); }
__device__ __forceinline__ uint32_t desc_lo_mnmajor(uint32_t addr) { return ((addr & 0x3FFFFu) >> 4) | ((HALF_BYTES >> 4) << 16); }
// instruction descriptors: bf16 x bf16 -> fp32, M = 128; N = 128 keys
constexpr uint32_t kIdescQK = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
// O += P V: N = head dimension, B (= V) is MN-major
template <int HD>
constexpr uint32_t kIdescPV = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | (((uint32_t)HD >> 3) << 17) | ((128u >> 4) << 24);

// S = A B^T over the head dimension (HD / 16 k-steps of 16) as one block issued by one elected
// lane: per k-step one add per operand and the MMA, nothing else.  alo / blo are the low
// descriptor words of two K-major [128][HD] bf16 tiles (HD / 64 swizzled 64-column blocks each).
template <int HD>
__device__ __forceinline__ void tc_qk(uint32_t d_tmem, uint32_t alo, uint32_t blo) {
#define GSD_QK_STEP(OFF, P)                                                         \
    " add.u32 al, %1, " #OFF ";\n add.u32 bl, %2, " #OFF ";\n"                       \
    " mov.b64 a, {al, %3};\n mov.b64 b, {bl, %3};\n"                                \
    " @q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, " #P ";\n"
#define GSD_QK_HEAD                                                                 \
    "{\n .reg .pred q, pt, pf;\n .reg .b64 a, b;\n .reg .b32 al, bl;\n"             \
    " elect.sync _|q, 0xffffffff;\n"                                                \
    " setp.eq.u32 pt, %4, %4;\n setp.ne.u32 pf, %4, %4;\n"                          \
    GSD_QK_STEP(0, pf) GSD_QK_STEP(2, pt) GSD_QK_STEP(4, pt) GSD_QK_STEP(6, pt)
    if constexpr (HD == 128)
        asm volatile(
            GSD_QK_HEAD GSD_QK_STEP(1024, pt) GSD_QK_STEP(1026, pt) GSD_QK_STEP(1028, pt) GSD_QK_STEP(1030, pt) "}\n"
            ::"r"(d_tmem), "r"(alo), "r"(blo), "r"(kDescHi), "r"(kIdescQK) : "memory");
    else
        asm volatile(GSD_QK_HEAD "}\n" ::"r"(d_tmem), "r"(alo), "r"(blo), "r"(kDescHi), "r"(kIdescQK) : "memory");
#undef GSD_QK_HEAD
#undef GSD_QK_STEP
}
// O (+)= P V for four k-steps of 16 keys: A = 8 TMEM columns of bf16 pairs per step, B = the
// MN-major V tile (2048 bytes per 16 keys).  `accum_first` = 0 makes the first step overwrite O.
template <int HD>
__device__ __forceinline__ void tc_pv4(uint32_t d_tmem, uint32_t a_tmem, uint32_t blo, uint32_t accum_first) {
#define GSD_PV_STEP(ACOL, BOFF, P)                                                  \
    " add.u32 at, %1, " #ACOL ";\n add.u32 bl, %2, " #BOFF ";\n mov.b64 b, {bl, %3};\n" \
    " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [at], b, %4, " #P ";\n"
    asm volatile(
        "{\n .reg .pred q, pt, p0;\n .reg .b64 b;\n .reg .b32 at, bl;\n"
        " elect.sync _|q, 0xffffffff;\n"
        " setp.eq.u32 pt, %4, %4;\n setp.ne.u32 p0, %5, 0;\n"
        GSD_PV_STEP(0, 0, p0) GSD_PV_STEP(8, 128, pt) GSD_PV_STEP(16, 256, pt) GSD_PV_STEP(24, 384, pt)
        "}\n"
        ::"r"(d_tmem), "r"(a_tmem), "r"(blo), "r"(kDescHi), "r"(kIdescPV<HD>), "r"(accum_first) : "memory");
#undef GSD_PV_STEP
}


struct TileInfo {
    int kind;     // 0 full prefix tile, 1 ragged prefix tile, 2 draft tile
    int key0;     // first key (prefix position or draft node) of the tile; negative for a ragged tile of a prefix below 128
    int nvalid;   // prefix: visible keys in the tile (the last nvalid of a ragged tile)
};

__device__ __forceinline__ TileInfo tile_info(int t, int nPT, int L, unsigned live) {
    TileInfo ti;
    if (t < nPT) {
        ti.key0 = t * BN;
        ti.nvalid = min(BN, L - ti.key0);
        ti.kind = ti.nvalid == BN ? 0 : 1;
        // The ragged last tile is loaded as the LAST 128 rows of the prefix (rows before position
        // 0 are filled with zeros by the copy engine): it then holds no row past the sequence
        // end, whose contents could be anything, and its first 128 - nvalid keys, which the tile
        // before it has covered already, are masked like invisible draft keys.
        if (ti.kind == 1) ti.key0 = L - BN;
    } else {
        int k = t - nPT, d = 0;
        for (;; ++d) {   // the k-th set bit of `live`
            if ((live >> d) & 1u) {
                if (k == 0) break;
                --k;
            }
        }
        ti.key0 = d * BN;
        ti.nvalid = BN;
        ti.kind = 2;
    }
    return ti;
}

__device__ __forceinline__ int visible_len(const TcParams& p, int b) {
    const int L = p.seq_lens[b];
    return L < 0 ? 0 : (L > p.Lmax ? p.Lmax : L);
}

// The order of the sequences made by the CTA itself (longest first), in shared memory.
struct Order {
    const int* len;      // [B] visible lengths
    const int* seq;      // [B] sequences in order
};

// One-wave plan: what it says about unit w.  Made by one warp, a lane per sequence, without a barrier:
// all of it lies between the launch and the first copy.
struct WaveUnit {
    int units;                     // of the whole call
    int b, L, nsplit, r;           // unit w: sequence, its length and key ranges per item, unit inside the sequence
};
__device__ __forceinline__ WaveUnit wave_unit(const TcParams& p, int w, int lane, bool leave) {
    const unsigned all = 0xFFFFFFFFu;
    const bool in = lane < p.B;
    const int nd = (p.N + BN - 1) / BN, per_seq = p.Hkv * p.plan.tiles_per_unit, resident = (int)gridDim.x;
    const int L = in ? visible_len(p, lane) : 0;
    const int t = in ? (L + BN - 1) / BN + nd : 0;
    const int total = __reduce_add_sync(all, t), longest = __reduce_max_sync(all, t);
    // lane k tries the k-th candidate for the tiles of a unit, from the lower bound on (at least four
    // tiles, at most 32 parts an item); the longest sequence whole always fits, as there are no more
    // items than CTAs
    const int bound = max(max((total * per_seq + resident - 1) / resident, (longest + 31) / 32), 4);
    const int T = bound + lane * max(1, bound / 16);
    int units = 0;
    for (int j = 0; j < p.B; ++j) units += (__shfl_sync(all, t, j) + T - 1) / T;
    const int best = min(longest, (int)__reduce_min_sync(all, units * per_seq <= resident ? T : 0x7FFFFFFF));
    const int n = in ? (t + best - 1) / best : 0;
    int end = n;                                            // units up to and with this sequence, per item
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int before = __shfl_up_sync(all, end, o);
        if (lane >= o) end += before;
    }
    WaveUnit u;
    u.units = __shfl_sync(all, end, 31) * per_seq;
    if (leave && in) {                                      // for the merge pass
        p.left[lane] = n;
        p.left[p.left_off + lane] = (end - n) * per_seq;
    }
    u.b = min(__popc(__ballot_sync(all, in && end * per_seq <= w)), p.B - 1);
    u.L = __shfl_sync(all, L, u.b);
    u.nsplit = __shfl_sync(all, n, u.b);
    u.r = w - __shfl_sync(all, end - n, u.b) * per_seq;
    return u;
}

// What a role needs to know about one unit of work (a row pair of one (sequence, kv head) and
// a key range).  Every warp derives it on its own from the work index, so the roles never
// have to meet at a CTA-wide barrier between units.
struct UnitInfo {
    int b, c, row0, split, nsplit, slot;
    int L, nPT, t_begin, ntiles;
    unsigned live;   // draft tiles (128 nodes each) holding a visible key for any row of the unit
    bool two;        // the second row tile exists
};

// `w` is the work index of a fixed plan, or the index of the group's unit in the table of a balanced one.
// `wu` is set for a one-wave plan only.
// unit_base: all but the mask - which draft tiles are live - so t_begin and ntiles count every draft tile.
template <int PLAN>
__device__ __forceinline__ UnitInfo unit_base(const TcParams& p, const Order& order, int w, const WaveUnit& wu) {
    UnitInfo u;
    int item;
    const bool bal = PLAN == PLAN_TABLE && p.bal_units != nullptr;
    if (bal) {
        // the unit of this CTA's group, for the row-tile item this CTA has in every pair
        const int tpu = p.plan.tiles_per_unit, rt = (int)blockIdx.x % tpu;
        const int4 rec = p.bal_units[w];
        item = rec.x * tpu + rt; u.t_begin = rec.y; u.ntiles = rec.z - rec.y;
        u.slot = rec.w >= 0 ? rt * 2 * ((int)gridDim.x / tpu) + rec.w : -1;
        u.split = 0;
        u.nsplit = rec.w >= 0 ? 2 : 1;     // only "one piece or several" matters below
    } else if (PLAN == PLAN_WAVE) {
        const int per_seq = p.Hkv * p.plan.tiles_per_unit;
        u.nsplit = wu.nsplit;
        u.split = wu.r / per_seq;
        item = wu.b * per_seq + wu.r - u.split * per_seq;
        u.slot = w;
    } else if (PLAN == PLAN_TABLE) {
        // unit w of the per-sequence plan: the last sequence whose first unit is <= w, then
        // (key range, item) inside it
        int lo = 0, hi = p.B - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (p.seq.unit_off[mid] <= w) lo = mid; else hi = mid - 1;
        }
        const int per_seq = p.Hkv * p.plan.tiles_per_unit;
        const int r = w - p.seq.unit_off[lo];
        u.nsplit = p.seq.nsplit[lo];
        u.split = r / per_seq;
        const int i = r - u.split * per_seq;
        item = lo * per_seq + i;
        u.slot = u.nsplit > 1 ? p.seq.slot_off[lo] + i * u.nsplit + u.split : 0;
    } else {
        plan_decode(p.plan, w, item, u.split, u.nsplit, u.slot);
    }
    const int unit = item / p.plan.tiles_per_unit;
    u.row0 = (item % p.plan.tiles_per_unit) * (2 * p.RT);
    u.b = PLAN == PLAN_ORDERED ? order.seq[unit / p.Hkv] : unit / p.Hkv;
    u.c = unit % p.Hkv;
    u.two = u.row0 + p.RT < p.R;
    if (!GSD_IN_BOUNDS(u.b >= 0 && u.b < p.B && u.c < p.Hkv && u.row0 < p.R, p.status)) {
        u.b = 0; u.c = 0; u.row0 = 0; u.two = false;      // checking build only: a unit outside the problem
    }
    const int L = PLAN == PLAN_WAVE ? wu.L : PLAN == PLAN_ORDERED ? order.len[u.b] : visible_len(p, u.b);
    u.L = L;
    u.nPT = (L + BN - 1) / BN;
    u.live = 0;
    if (!bal) {
        const int T = u.nPT + (p.N + BN - 1) / BN;
        const int per = (T + u.nsplit - 1) / u.nsplit;
        u.t_begin = min(u.split * per, T);
        u.ntiles = min(u.t_begin + per, T) - u.t_begin;
    }
    return u;
}

// The draft tiles that hold a visible key for any row of the unit: the OR of the mask rows of its
// nodes, which are consecutive in memory; four or eight loads of a lane are on their way at a time.
__device__ __forceinline__ unsigned unit_live(const TcParams& p, const UnitInfo& u, int lane) {
    const int n_lo = u.row0 / p.G;
    const int n_hi = (min(u.row0 + 2 * p.RT, p.R) - 1) / p.G + 1;
    const uint32_t* words = p.mask + ((size_t)u.b * p.N + n_lo) * p.W;
    const uint32_t tail = (p.N & 31) ? (1u << (p.N & 31)) - 1u : 0xFFFFFFFFu;   // valid bits of a row's last word
    unsigned live = 0;
    if ((p.W & 3) == 0 && (reinterpret_cast<uintptr_t>(p.mask) & 15u) == 0) {
        // four words = one draft tile of a row per 16-byte load
        const int nt = p.W >> 2, total = (n_hi - n_lo) * nt;
        const uint4* quads = reinterpret_cast<const uint4*>(words);
#pragma unroll 1
        for (int base = lane; base < total; base += 8 * 32) {
            uint4 q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) q[k] = base + 32 * k < total ? quads[base + 32 * k] : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int t = (base + 32 * k) % nt;
                if (t == nt - 1) q[k].w &= tail;
                if (q[k].x | q[k].y | q[k].z | q[k].w) live |= 1u << t;
            }
        }
    } else {
        const int total = (n_hi - n_lo) * p.W;
#pragma unroll 1
        for (int base = lane; base < total; base += 4 * 32) {
            uint32_t q[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) q[k] = base + 32 * k < total ? words[base + 32 * k] : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int wi = (base + 32 * k) % p.W;
                if (wi == p.W - 1) q[k] &= tail;
                if (q[k]) live |= 1u << (wi >> 2);
            }
        }
    }
    return __reduce_or_sync(0xFFFFFFFFu, live);
}

// The same for many mask words, a slice of them: part `part` of `parts`, eight 16-byte loads of a lane on their way
// whatever the width of a row.
__device__ __forceinline__ unsigned unit_live_slice(const TcParams& p, const UnitInfo& u, int part, int parts, int lane) {
    const int n_lo = u.row0 / p.G;
    const int n_hi = (min(u.row0 + 2 * p.RT, p.R) - 1) / p.G + 1;
    const int total = (n_hi - n_lo) * p.W, lo = total * part / parts, hi = total * (part + 1) / parts;
    const uint32_t* words = p.mask + ((size_t)u.b * p.N + n_lo) * p.W;
    const uint32_t tail = (p.N & 31) ? (1u << (p.N & 31)) - 1u : 0xFFFFFFFFu;   // valid bits of a row's last word
    unsigned live = 0;
    auto note = [&](uint32_t v, int col) {
        if (col == p.W - 1) v &= tail;
        if (v) live |= 1u << (col >> 2);
    };
    // (words before the first 16-byte boundary and behind the last one go one by one)
    const int to_boundary = (int)((0u - (unsigned)(reinterpret_cast<uintptr_t>(words + lo) >> 2)) & 3u);
    const int q0 = min(lo + to_boundary, hi), nq = (hi - q0) >> 2, rest = q0 + 4 * nq;
    const uint32_t v_head = lo + lane < q0 ? words[lo + lane] : 0u, v_tail = rest + lane < hi ? words[rest + lane] : 0u;
    const uint4* quads = reinterpret_cast<const uint4*>(words + q0);
#pragma unroll 1
    for (int base = lane; base < nq; base += 8 * 32) {
        uint4 q[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) q[k] = base + 32 * k < nq ? quads[base + 32 * k] : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (!(q[k].x | q[k].y | q[k].z | q[k].w)) continue;
            const uint32_t v[4] = {q[k].x, q[k].y, q[k].z, q[k].w};
            int col = (q0 + 4 * (base + 32 * k)) % p.W;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                note(v[j], col);
                col = col + 1 == p.W ? 0 : col + 1;
            }
        }
    }
    note(v_head, (lo + lane) % p.W);
    note(v_tail, (rest + lane) % p.W);
    return __reduce_or_sync(0xFFFFFFFFu, live);
}

// Of the draft tiles only the live ones are numbered.
__device__ __forceinline__ void unit_use_live(UnitInfo& u, unsigned live) {
    u.live = live;
    auto live_index = [&](int t) { return t <= u.nPT ? t : u.nPT + __popc(live & ((1u << (t - u.nPT)) - 1u)); };
    const int t0 = live_index(u.t_begin), t1 = live_index(u.t_begin + u.ntiles);
    u.t_begin = t0;
    u.ntiles = t1 - t0;
}

// The whole unit.
template <int PLAN>
__device__ __forceinline__ UnitInfo unit_info(const TcParams& p, const Order& order, int w, int lane, const WaveUnit& wu = WaveUnit{}) {
    UnitInfo u = unit_base<PLAN>(p, order, w, wu);
    unit_use_live(u, unit_live(p, u, lane));
    return u;
}

// The sequences in descending order of length (called by the whole CTA); false: they are all alike.
__device__ __forceinline__ bool order_by_length(const TcParams& p, int* s_len, int* s_seq) {
    const int tid = threadIdx.x, B = p.B;
    const int mine = tid < B ? visible_len(p, tid) : 0;
    if (tid < B) s_len[tid] = mine;
    __syncthreads();
    int rank = 0;
    if (tid < B) {
        for (int j = 0; j < B; ++j) rank += s_len[j] > mine || (s_len[j] == mine && j < tid);
        s_seq[rank] = tid;
    }
    return __syncthreads_or(tid < B && mine != s_len[0]) != 0;
}

// Persistent kernel: CTA k walks the work indices k, k + gridDim.x, ...  Barrier phases are
// counted across units, so the producer and the QK^T issuer run ahead into the next unit
// (Q, the first K/V tiles and the first QK^T) while the softmax warps still read out the
// accumulators of the previous one.
template <int HD, int PLAN, bool LONG_MASK>
__global__ void __launch_bounds__(kThreads, 1)
attn_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
               const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_dk,
               const __grid_constant__ CUtensorMap tm_dv, const TcParams p) {
    using T = Geo<HD>;
    constexpr uint32_t TILE_BYTES = T::TILE_BYTES;
    constexpr int ST = T::ST;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long s_bars[BAR_COUNT];
    __shared__ uint32_t s_tmem_base;
    __shared__ __align__(8) WaitCtl s_wait;
    __shared__ float2 s_ml1[BM];      // (max, sum) of the odd-tile stream, one per row; who may write when: see there
    __shared__ int s_len[kPlanSeqs], s_seq[kPlanSeqs];     // longest first: lengths, order of the sequences
    __shared__ int s_wave_units;                           // one-wave plan: units of the call
    __shared__ UnitInfo s_units[kUnitTable];   // the CTA's first units of work, decoded once up front
    __shared__ unsigned s_live[kThreads / 32]; // live draft tiles in the slices of their mask rows

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int N = p.N, G = p.G, R = p.R, RT = p.RT;

    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sQ = smem_base;                                   // 2 tiles
    const uint32_t sK = smem_base + 2 * TILE_BYTES;                  // ST tiles
    const uint32_t sV = sK + ST * TILE_BYTES;                        // ST tiles
    const uint32_t sStage = sV + ST * TILE_BYTES;                    // a block per softmax warp
    const uint32_t bar0 = smem_u32(s_bars);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    volatile int* abort_flag = &s_wait.abort;

    if (warp == 8 && lane == 0) {
        // The merge pass, if there is one, may be made resident as CTAs retire.  Other successors may not, here
        // and in the merge pass: the CTAs of a next call that settle where SMs fall free cost it more than
        // its start gains (32 x 64/8 heads, N 57, L 200-2100: 109 us a call, 117 so; the step of 3 x 40 heads, N
        // 363, L 228: 142 and 162 - one of 1 x 8/1, N 27, L 97: 10.3 and 9.8).
        if (p.slots > 0) let_successor_start();
        // the first copy through a tensor map would otherwise fetch it from memory first
        prefetch_map(&tm_q); prefetch_map(&tm_k); prefetch_map(&tm_v); prefetch_map(&tm_dk); prefetch_map(&tm_dv);
        s_wait.abort = 0;
        s_wait.limit_ns = p.wait_limit_ns;
        mbar_init(bar(BAR_Q_FULL), 1);
        mbar_init(bar(BAR_Q_EMPTY), 1);
        mbar_init(bar(BAR_ML_READY), 4);
        for (int s = 0; s < ST; ++s) {
            mbar_init(bar(BAR_K_FULL + s), 1); mbar_init(bar(BAR_K_EMPTY + s), 1);
            mbar_init(bar(BAR_V_FULL + s), 1); mbar_init(bar(BAR_V_EMPTY + s), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(BAR_S_FULL + i), 1);
            mbar_init(bar(BAR_S_FREE + i), 4);     // one arrival per softmax warp
            mbar_init(bar(BAR_P_READY + i), 4);
            mbar_init(bar(BAR_P_READY2 + i), 4);
            mbar_init(bar(BAR_P_FREE + i), 1);
            mbar_init(bar(BAR_O_DONE + i), 1);
            mbar_init(bar(BAR_O_FREE + i), 4);
            mbar_init(bar(BAR_DRAIN + i), 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 10) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (RT < BM) {
        // a group size that does not divide 128: the copies of Q never write the last rows of a
        // tile, whose scores and output rows nobody uses; zeros there keep them finite
        const int words = (BM - RT) * 32;                  // 128-byte rows of one block
        for (int t = tid; t < 2 * T::BLOCKS * words; t += kThreads) {
            const int blk = t / words, w = t - blk * words;
            *reinterpret_cast<uint32_t*>(smem_raw + (sQ - smem_u32(smem_raw)) + blk * HALF_BYTES + RT * 128 + w * 4) = 0u;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    // This kernel is launched as a programmatic dependent of whatever precedes it on the stream:
    // everything above may run beside the end of that, nothing below may.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const Order order{s_len, s_seq};
    bool forth_and_back = false;
    if (PLAN == PLAN_ORDERED) {
        forth_and_back = order_by_length(p, s_len, s_seq);
        if (blockIdx.x == 0 && p.left && tid < p.B) p.left[tid] = s_seq[tid];
    }
    // The CTA's units: work indices blockIdx.x, blockIdx.x + gridDim.x, ... of a fixed plan (every
    // other round backwards when the lengths differ and the longest come first), or a run of the table that the planning
    // kernel has written.
    int n_my;
    if (PLAN == PLAN_TABLE && p.bal_cta) {
        n_my = p.bal_cta[blockIdx.x / p.plan.tiles_per_unit].y;
    } else if (PLAN == PLAN_TABLE) {
        const int units = p.seq.hdr[0];
        n_my = units > (int)blockIdx.x ? (units - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    } else if (PLAN == PLAN_WAVE) {
        n_my = 0;                          // (set below: one unit or none)
    } else if (forth_and_back) {
        const int rounds = p.total_work / (int)gridDim.x, rest = p.total_work - rounds * (int)gridDim.x;
        n_my = rounds + (((rounds & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x) < rest ? 1 : 0);
    } else {
        n_my = p.total_work > (int)blockIdx.x ? (p.total_work - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    }
    // (recomputed where it is needed rather than kept in a register through the key loops)
    auto unit_index = [&](int it) -> int {
        if (PLAN == PLAN_TABLE && p.bal_cta) return p.bal_cta[blockIdx.x / p.plan.tiles_per_unit].x + it;
        const bool back = forth_and_back && (it & 1);
        return p.work0 + it * (int)gridDim.x + (back ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x);
    };
    // The copies of one key tile (into ring slot n % ST, the n-th of the CTA).
    auto load_k = [&](const UnitInfo& u, int idx, int n) {
        const TileInfo ti = tile_info(u.t_begin + idx, u.nPT, u.L, u.live);
        mbar_expect_tx(bar(BAR_K_FULL + n % ST), TILE_BYTES);
        if (p.withhold_first_k && n == 0) return;        // (test hook: the bytes announced above never arrive)
        for (int h = 0; h < T::BLOCKS; ++h)
            tma_load_4d(sK + (n % ST) * TILE_BYTES + h * HALF_BYTES, ti.kind == 2 ? &tm_dk : &tm_k, bar(BAR_K_FULL + n % ST), h * 64, u.c, ti.key0, u.b);
    };
    auto load_v = [&](const UnitInfo& u, int idx, int n) {
        const TileInfo ti = tile_info(u.t_begin + idx, u.nPT, u.L, u.live);
        mbar_expect_tx(bar(BAR_V_FULL + n % ST), TILE_BYTES);
        for (int h = 0; h < T::BLOCKS; ++h)
            tma_load_4d(sV + (n % ST) * TILE_BYTES + h * HALF_BYTES, ti.kind == 2 ? &tm_dv : &tm_v, bar(BAR_V_FULL + n % ST), h * 64, u.c, ti.key0, u.b);
    };
    auto load_q = [&](const UnitInfo& u) {
        const int ntile_rows = u.two ? 2 : 1;
        mbar_expect_tx(bar(BAR_Q_FULL), (uint32_t)(ntile_rows * T::BLOCKS * RT) * 128u);
        for (int i = 0; i < ntile_rows; ++i)
            for (int h = 0; h < T::BLOCKS; ++h)
                tma_load_4d(sQ + i * TILE_BYTES + h * HALF_BYTES, &tm_q, bar(BAR_Q_FULL), h * 64, u.c * G, (u.row0 + i * RT) / G, u.b);
    };
    // Decoding a unit costs a trip to global memory or two (sequence length, mask rows).  The warps
    // decode the CTA's first units here, all at once, so that no role pays that latency between
    // units.  The producer warp does not wait for the mask: it issues the copies of Q and of the
    // first prefix tiles - as many as the empty rings hold - as soon as it knows the length.
    int pre = 0;             // producer: key tiles of unit 0 already on their way
    if (warp == 8) {
        WaveUnit wu{};
        if (PLAN == PLAN_WAVE) {
            wu = wave_unit(p, blockIdx.x, lane, false);
            n_my = (int)blockIdx.x < wu.units ? 1 : 0;
        }
        if (n_my > 0 && lane == 0) {
            const UnitInfo u = unit_base<PLAN>(p, order, unit_index(0), wu);
            pre = max(0, min(ST, min(u.nPT - u.t_begin, u.ntiles)));
            if (pre > 0) load_q(u);
            for (int n = 0; n < pre; ++n) { load_k(u, n, n); load_v(u, n, n); }
        }
        pre = __shfl_sync(0xFFFFFFFFu, pre, 0);
    } else if (LONG_MASK) {
        // Mask rows of many words (256 nodes, one head a group: up to 16 KB a unit): few units are shared by the
        // warps, a slice each, and put together behind a barrier (one warp a unit with four words of a lane on
        // their way took 13 us at N 338: 2 x 32 heads, N 407, L 4081 88.6 -> 83 us; D 64, 2 x 12 heads, N 346, L
        // 3900 38.2 -> 35.2).
        constexpr int kDecoders = kThreads / 32 - 1;
        WaveUnit wu{};
        int n = n_my;
        if (PLAN == PLAN_WAVE) {
            wu = wave_unit(p, blockIdx.x, lane, blockIdx.x == 0 && warp == 0);
            if (warp == 0 && lane == 0) s_wave_units = wu.units;
            n = (int)blockIdx.x < wu.units ? 1 : 0;
        }
        const int slices = max(1, kDecoders / max(n, 1)), me = warp < 8 ? warp : warp - 1;
        for (int t = me; t < min(n, kUnitTable) * slices; t += kDecoders) {
            const int k = t / slices, part = t - k * slices;
            UnitInfo u = unit_base<PLAN>(p, order, PLAN == PLAN_WAVE ? (int)blockIdx.x : unit_index(k), wu);
            const unsigned live = unit_live_slice(p, u, part, slices, lane);
            if (lane == 0) {
                if (slices > 1) s_live[t] = live;
                else unit_use_live(u, live);
                if (part == 0) s_units[k] = u;
            }
        }
        if (slices > 1) {
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kDecoders) : "memory");
            if (lane == 0 && me < n) {
                unsigned live = 0;
                for (int k = 0; k < slices; ++k) live |= s_live[me * slices + k];
                unit_use_live(s_units[me], live);
            }
        }
    } else if (PLAN == PLAN_WAVE) {
        if (warp == 0) {
            const WaveUnit wu = wave_unit(p, blockIdx.x, lane, blockIdx.x == 0);
            if (lane == 0) s_wave_units = wu.units;
            if ((int)blockIdx.x < wu.units) {
                const UnitInfo u = unit_info<PLAN>(p, order, blockIdx.x, lane, wu);
                if (lane == 0) s_units[0] = u;
            }
        }
    } else {
        for (int k = warp < 8 ? warp : warp - 1; k < kUnitTable; k += kThreads / 32 - 1) {
            if (k < n_my) {
                const UnitInfo u = unit_info<PLAN>(p, order, unit_index(k), lane);
                if (lane == 0) s_units[k] = u;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem_base;
    if (PLAN == PLAN_WAVE) {
        n_my = (int)blockIdx.x < s_wave_units ? 1 : 0;
        asm volatile("" : "+r"(n_my));      // (knowing that the unit loops run once at most, the compiler spills in the key loop)
    }
    auto unit_of = [&](int it) -> UnitInfo {
        return PLAN != PLAN_TABLE || it < kUnitTable ? s_units[it] : unit_info<PLAN>(p, order, unit_index(it), lane);
    };

    if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 96;");
    if (warp == 8) {
        // ------------------------------------------------------------ TMA producer
        // Units with one row tile, where loads are the bound: K copies run one tile ahead of the V
        // copies.  K t + 1 only waits for the QK^T of tile t - 1, and its time to land passes while V t
        // waits for the PV of tile t - 2 (4 x 40 heads, N 128, L 1024-4096: 58.4 us in step with the
        // V copies, 55.4 one ahead).  Units with two keep the copies in step, in a loop of
        // their own: the tensor pipe is the bound there, and the choice between the two kinds of copy at
        // every step cost 2% of the cycles of the key loop (32 x 64/8 heads, N 128, L 8192: 1566 -> 1539
        // thousand; 8 x 64/8, N 512, L 2048: 494 -> 485).
        int kc = pre, vc = pre;         // K and V tiles loaded so far (ring positions)
        int au = 0;                     // non-empty units so far
        bool ok = true, q_pending = pre > 0;
        for (int it = 0; it < n_my && ok; ++it) {
            const UnitInfo u = unit_of(it);
            if (u.ntiles == 0) continue;
            if (lane == 0) {
                const bool begun = it == 0 && pre > 0;
                if (!begun) {
                    // Q of the previous unit is free once its last QK^T has completed
                    ok = mbar_wait(bar(BAR_Q_EMPTY), (au & 1) ^ 1, abort_flag, p.status);
                    if (ok) {
                        load_q(u);
                        q_pending = true;
                    }
                }
                int kn = begun ? pre : 0, vn = kn;      // next tile of the unit
                if (u.two) {
                    for (; vn < u.ntiles && ok; ++vn) {
                        if (!(ok = mbar_wait(bar(BAR_K_EMPTY + kc % ST), (uint32_t)((kc / ST) & 1) ^ 1u, abort_flag, p.status))) break;
                        load_k(u, vn, kc);
                        ++kc;
                        if (!(ok = mbar_wait(bar(BAR_V_EMPTY + vc % ST), (uint32_t)((vc / ST) & 1) ^ 1u, abort_flag, p.status))) break;
                        load_v(u, vn, vc);
                        ++vc;
                    }
                } else {
                    while (ok && vn < u.ntiles) {
                        if (kn < u.ntiles && kn <= vn + 1) {
                            if (!(ok = mbar_wait(bar(BAR_K_EMPTY + kc % ST), (uint32_t)((kc / ST) & 1) ^ 1u, abort_flag, p.status))) break;
                            load_k(u, kn, kc);
                            ++kn;
                            ++kc;
                        } else {
                            if (!(ok = mbar_wait(bar(BAR_V_EMPTY + vc % ST), (uint32_t)((vc / ST) & 1) ^ 1u, abort_flag, p.status))) break;
                            load_v(u, vn, vc);
                            ++vn;
                            ++vc;
                        }
                    }
                }
                if (!ok) {
                    // gave up: let the copies already in flight land before the CTA retires
                    if (q_pending) mbar_wait_slow(bar(BAR_Q_FULL), au & 1, abort_flag, nullptr, true);
                    for (int t = max(0, kc - ST); t < kc; ++t)
                        mbar_wait_slow(bar(BAR_K_FULL + t % ST), (t / ST) & 1, abort_flag, nullptr, true);
                    for (int t = max(0, vc - ST); t < vc; ++t)
                        mbar_wait_slow(bar(BAR_V_FULL + t % ST), (t / ST) & 1, abort_flag, nullptr, true);
                }
            }
            ok = __shfl_sync(0xFFFFFFFFu, (int)ok, 0) != 0;
            kc = __shfl_sync(0xFFFFFFFFu, kc, 0);
            vc = __shfl_sync(0xFFFFFFFFu, vc, 0);
            ++au;
        }
    } else if (warp == 9) {
        // ------------------------------------------------------------ QK^T issuer (all lanes converged)
        // S = Q K^T job by job.  Nothing orders these MMAs against the PV MMAs of warp 11 in the
        // tensor pipe, and nothing has to: they touch different TMEM columns, and every
        // hand-over (S to the softmax, P to the PV, S back) goes through an mbarrier.
        int kvc = 0;              // key tiles of earlier units (ring position of this unit's first tile)
        int au = 0;               // non-empty units so far
        int jq0 = 0, jq1 = 0;     // jobs issued per stream so far (phase of S_FULL / S_FREE)
        int s_owner = -1;         // stream whose scores were last written to S
        bool ok = true;
        auto wait = [&](int b, uint32_t par) -> bool { return mbar_wait_warp(bar(b), par, abort_flag, p.status); };
        const uint32_t qlo0 = desc_lo_kmajor(sQ), qlo1 = desc_lo_kmajor(sQ + TILE_BYTES);
        const uint32_t klo0 = desc_lo_kmajor(sK);       // (stage st: + st * TILE_BYTES / 16)
        for (int it = 0; it < n_my && ok; ++it) {
            const UnitInfo u = unit_of(it);
            if (u.ntiles == 0) continue;
            const bool two = u.two;
            const int njobs = two ? 2 * u.ntiles : u.ntiles;
            ok = wait(BAR_Q_FULL, au & 1);
            for (int k = 0; k < njobs && ok; ++k) {
                const int i = k & 1;
                const int r = kvc + (two ? (k >> 1) : k), st = r % ST;
                if (!two || i == 0) {
                    if (!(ok = wait(BAR_K_FULL + st, (r / ST) & 1))) break;
                }
                if (T::TWO_S) {
                    // the scores of the stream's previous job must have left its S
                    if ((i ? jq1 : jq0) > 0 && !(ok = wait(BAR_S_FREE + i, (uint32_t)((i ? jq1 : jq0) - 1) & 1u))) break;
                } else if (s_owner >= 0) {
                    // the previous job's scores must have left S
                    if (!(ok = wait(BAR_S_FREE + s_owner, (uint32_t)((s_owner ? jq1 : jq0) - 1) & 1u))) break;
                }
                tc_fence_after();
                tc_qk<HD>(tmem + (i ? T::COL_S1 : T::COL_S0), (two && i) ? qlo1 : qlo0, klo0 + (uint32_t)st * (TILE_BYTES >> 4));
                tc_commit(bar(BAR_S_FULL + i));
                if (!two || i == 1) tc_commit(bar(BAR_K_EMPTY + st));
                if (k == njobs - 1) tc_commit(bar(BAR_Q_EMPTY));   // every QK^T of the unit is issued
                s_owner = i;
                if (i) ++jq1; else ++jq0;
            }
            kvc += u.ntiles;
            ++au;
        }
        // after an abort nothing this warp issued may still be running when TMEM is given back
        // (at a regular end the epilogues have waited for every MMA already)
        if (!ok) {
            tc_commit(bar(BAR_DRAIN + 0));
            mbar_wait_slow(bar(BAR_DRAIN + 0), 0, abort_flag, nullptr, true);
        }
    } else if (warp == 11) {
        // ------------------------------------------------------------ PV issuer (all lanes converged)
        // O_i += P_i V job by job: 8 k-steps of 16 keys, P (bf16 pairs) read from TMEM.  The
        // softmax hands P over in two halves of 64 keys, so the first four k-steps run while
        // the second half of the exponentials is still being computed.
        int kvc = 0;
        int au = 0, au1 = 0;      // non-empty units so far; those of them in which stream 1 had jobs
        int jp0 = 0, jp1 = 0;     // jobs issued per stream so far (phase of P_READY / P_FREE)
        bool ok = true;
        auto wait = [&](int b, uint32_t par) -> bool { return mbar_wait_warp(bar(b), par, abort_flag, p.status); };
        const uint32_t vlo0 = desc_lo_mnmajor(sV);      // (stage st: + st * TILE_BYTES / 16)
        for (int it = 0; it < n_my && ok; ++it) {
            const UnitInfo u = unit_of(it);
            if (u.ntiles == 0) continue;
            const bool two = u.two;
            const int njobs = two ? 2 * u.ntiles : u.ntiles;
            const int n1 = two ? u.ntiles : u.ntiles / 2;      // jobs of stream 1
            for (int k = 0; k < njobs && ok; ++k) {
                const int i = k & 1;
                const int r = kvc + (two ? (k >> 1) : k), st = r % ST;
                const bool first = k < 2;                      // first job of its stream in this unit
                const uint32_t par = (uint32_t)(i ? jp1 : jp0) & 1u;
                const uint32_t vlo = vlo0 + (uint32_t)st * (TILE_BYTES >> 4);
                const uint32_t tP = tmem + (i ? T::COL_P1 : T::COL_P0), tO = tmem + (i ? T::COL_O1 : T::COL_O0);
                if (!two || i == 0) {
                    if (!(ok = wait(BAR_V_FULL + st, (r / ST) & 1))) break;
                }
                if (!(ok = wait(BAR_P_READY + i, par))) break;
                if (first && (i ? au1 : au) > 0) {
                    // the accumulator still belongs to the previous unit until its rows were read out
                    if (!(ok = wait(BAR_O_FREE + i, (uint32_t)((i ? au1 : au) - 1) & 1u))) break;
                }
                tc_fence_after();
                tc_pv4<HD>(tO, tP, vlo, first ? 0u : 1u);
                if (!(ok = wait(BAR_P_READY2 + i, par))) break;
                tc_fence_after();
                tc_pv4<HD>(tO, tP + 32, vlo + 4 * 128, 1u);
                tc_commit(bar(BAR_P_FREE + i));
                if (!two || i == 1) tc_commit(bar(BAR_V_EMPTY + st));
                if (k + 2 >= njobs) tc_commit(bar(BAR_O_DONE + i));   // the stream's last job of the unit
                if (i) ++jp1; else ++jp0;
            }
            kvc += u.ntiles;
            ++au;
            if (n1 > 0) ++au1;
        }
        if (!ok) {
            tc_commit(bar(BAR_DRAIN + 1));
            mbar_wait_slow(bar(BAR_DRAIN + 1), 0, abort_flag, nullptr, true);
        }
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
        // ------------------------------------------------------------ softmax + epilogue
        const int i = warp >> 2;                         // stream of this warpgroup
        const int rloc = (warp & 3) * 32 + lane;         // row inside the tile = TMEM lane
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + lane_addr + (i ? T::COL_S1 : T::COL_S0);
        const uint32_t tP = tmem + lane_addr + (i ? T::COL_P1 : T::COL_P0);
        const uint32_t tO = tmem + lane_addr + (i ? T::COL_O1 : T::COL_O0);
        int kvc = 0;      // key tiles of all non-empty units so far (ring position of the V tiles)
        int tcnt = 0;     // jobs this stream has processed so far (barrier phase)
        int auc = 0;      // non-empty units this stream has finished so far (barrier phase)
        int auc1 = 0;     // units in which stream 1 had jobs (phase of its barriers as seen by warpgroup 0)
        int mlc = 0;      // single-row-tile units whose odd-tile stream had tiles
        bool ok = true;
        for (int it = 0; it < n_my && ok; ++it) {
            const UnitInfo u = unit_of(it);
            const int ntiles = u.ntiles;
            // with one row tile only, the two warpgroups take the even / odd key tiles of the
            // same rows and warpgroup 0 merges the two partial results in the epilogue
            const bool alt = !u.two;
            const int my_n = alt ? (i == 0 ? (ntiles + 1) / 2 : ntiles / 2) : ntiles;
            const int n1 = alt ? ntiles / 2 : ntiles;           // tiles of stream 1 in this unit
            const int b = u.b, c = u.c;
            const int row = u.row0 + (alt ? 0 : i * RT) + rloc;
            const bool rvalid = rloc < RT && row < R;
            if (warp == 0 && lane == 0) {
                const int Lraw = p.seq_lens[b];
                if ((Lraw < 0 || Lraw > p.Lmax) && p.status) atomicOr((unsigned*)p.status, GSD_DEV_BAD_SEQ_LEN);
            }
            float m_ref = -CUDART_INF_F, l_run = 0.f;
            const uint32_t* mrow = p.mask + ((size_t)b * N + (rvalid ? row / G : 0)) * p.W;
            for (int cnt = 0; cnt < my_n; ++cnt) {
                const int idx = alt ? 2 * cnt + i : cnt;
                const TileInfo ti = tile_info(u.t_begin + idx, u.nPT, u.L, u.live);
                // visibility words of this row for the 128 keys of the tile
                uint32_t mw[4];
                if (ti.kind == 0) {
                    mw[0] = mw[1] = mw[2] = mw[3] = 0xFFFFFFFFu;
                } else if (ti.kind == 1) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int from = (BN - ti.nvalid) - 32 * k;      // first visible key of the word
                        mw[k] = from <= 0 ? 0xFFFFFFFFu : (from >= 32 ? 0u : ~((1u << from) - 1u));
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int wi = (ti.key0 >> 5) + k;
                        uint32_t word = (rvalid && wi < p.W) ? mrow[wi] : 0u;
                        const int rem = N - 32 * wi;
                        if (rem < 32) word &= rem <= 0 ? 0u : ((1u << rem) - 1u);
                        mw[k] = word;
                    }
                }
                const uint32_t par = (uint32_t)((tcnt + cnt) & 1);
                ok = mbar_wait(bar(BAR_S_FULL + i), par, abort_flag, p.status);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                tc_fence_after();

                // the whole score row of this thread: 128 fp32 registers
                float sc[BN];
#pragma unroll
                for (int ch = 0; ch < 4; ++ch) tc_ld32(tS + ch * 32, sc + ch * 32);
                tc_wait_ld();
                tc_fence_before();
                if (lane == 0) mbar_arrive(bar(BAR_S_FREE + i));   // the next job's QK^T may overwrite S
                if (ti.kind != 0) {
#pragma unroll
                    for (int e = 0; e < BN; ++e) sc[e] = ((mw[e >> 5] >> (e & 31)) & 1u) ? sc[e] : -CUDART_INF_F;
                }
                float mx4[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
                for (int e = 0; e < BN; e += 8) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) mx4[k] = max3(mx4[k], sc[e + 2 * k], sc[e + 2 * k + 1]);
                }
                const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
                const float m_tile = mx * p.scale_log2;     // scale > 0 keeps the order
                float m_new = m_ref, alpha = 1.f;
                bool need = false;
                if (m_ref == -CUDART_INF_F) {
                    m_new = m_tile;                         // nothing accumulated for this row yet
                } else if (m_tile > m_ref + p.raise_above) {
                    m_new = m_tile;
                    alpha = fast_exp2(m_ref - m_new);
                    need = true;
                }
                // Once the PV of this stream's previous job has completed, the accumulator of this row is
                // final for all earlier tiles and can be rescaled in place.  Where that is common (D = 64)
                // it is done where P_i's release is waited for anyway (head dimension 64, 4 x 32/8 heads:
                // 36.1 us here, 35.4 there; at 128 the registers that live on cost more than the wait).
                constexpr bool kRaiseLate = HD == 64;
                const bool raise = __any_sync(0xFFFFFFFFu, need);
                auto rescale = [&]() {
#pragma unroll 1
                    for (int ch = 0; ch < HD / 32; ++ch) {
                        float v[32];
                        tc_ld32(tO + ch * 32, v);
                        tc_wait_ld();
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] *= alpha;
                        tc_st32(tO + ch * 32, v);
                    }
                    l_run *= alpha;
                };
                if (!kRaiseLate && raise) {
                    ok = mbar_wait(bar(BAR_P_FREE + i), (uint32_t)((tcnt + cnt - 1) & 1), abort_flag, p.status);
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) break;
                    tc_fence_after();
                    rescale();
                }
                m_ref = m_new;
                const float m_use = m_ref == -CUDART_INF_F ? 0.f : m_ref;

                // P = 2^(s*scale - m) as bf16 pairs into the 64 columns of P_i; a masked score is
                // -inf and comes out as exactly 0
                const float2 scale2 = make_float2(p.scale_log2, p.scale_log2);
                const float2 negm2 = make_float2(-m_use, -m_use);
                float2 sum2[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};   // four chains
                uint32_t pk[4][16];
                auto exp_chunk = [&](int ch) {
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const float2 t = ffma2(make_float2(sc[ch * 32 + 2 * e], sc[ch * 32 + 2 * e + 1]), scale2, negm2);
                        const float2 pe = make_float2(fast_exp2(t.x), fast_exp2(t.y));
                        sum2[e & 3] = fadd2(sum2[e & 3], pe);
                        pk[ch][e] = pack_bf16(pe.x, pe.y);
                    }
                };
                // The TMEM stores of one half are in flight while the next chunk's exponentials are
                // computed; the hand-off of a half follows once its stores have landed.
                exp_chunk(0);
                exp_chunk(1);
                if (tcnt + cnt > 0) {
                    // P_i is still being read until the PV of this stream's previous job has completed
                    ok = mbar_wait(bar(BAR_P_FREE + i), (uint32_t)((tcnt + cnt - 1) & 1), abort_flag, p.status);
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) break;
                    tc_fence_after();
                    if (kRaiseLate && raise) rescale();
                }
                tc_st16(tP + 0, pk[0]);
                tc_st16(tP + 16, pk[1]);
                exp_chunk(2);
                tc_wait_st();              // keys 0..63 are in place (and any rescale of O is done)
                tc_fence_before();
                if (lane == 0) mbar_arrive(bar(BAR_P_READY + i));
                exp_chunk(3);
                tc_st16(tP + 32, pk[2]);
                tc_st16(tP + 48, pk[3]);
                l_run += ((sum2[0].x + sum2[0].y) + (sum2[1].x + sum2[1].y)) + ((sum2[2].x + sum2[2].y) + (sum2[3].x + sum2[3].y));
                tc_wait_st();
                tc_fence_before();
                if (lane == 0) mbar_arrive(bar(BAR_P_READY2 + i));
            }
            if (!ok) break;
            if (alt && i == 1) {
                // odd-tile stream: publish (max, sum); warpgroup 0 reads the accumulator itself
                if (my_n > 0) {
                    // The pair of the stream's previous unit has to have been read (warpgroup 0 says so
                    // with O_FREE) before this one takes its place.  With one S for both streams that is
                    // so already: this unit's scores of stream 1 were only formed after warpgroup 0 had
                    // given S back in this unit.  With an S per stream nothing else holds this warpgroup
                    // back when a unit has a single odd tile.  Both sides count the units in which stream
                    // 1 had tiles, and O_FREE cannot go on by a further phase before the pair is published.
                    if (T::TWO_S && auc > 0) {
                        ok = mbar_wait(bar(BAR_O_FREE + 1), (uint32_t)(auc - 1) & 1u, abort_flag, p.status);
                        ok = __all_sync(0xFFFFFFFFu, ok);
                        if (!ok) break;
                    }
                    s_ml1[rloc] = make_float2(m_ref, l_run);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(BAR_ML_READY));
                    ++mlc;
                    ++auc;
                }
                kvc += ntiles;
                tcnt += my_n;
                continue;
            }
            // ---- epilogue: pull the accumulator row into registers, give TMEM back, then store
            // every wait of the epilogue first ...
            if (ntiles > 0) {
                ok = mbar_wait(bar(BAR_O_DONE + i), (uint32_t)(auc & 1), abort_flag, p.status);
                if (ok && alt && n1 > 0) {
                    ok = mbar_wait(bar(BAR_O_DONE + 1), (uint32_t)(auc1 & 1), abort_flag, p.status);
                    if (ok) ok = mbar_wait(bar(BAR_ML_READY), (uint32_t)(mlc & 1), abort_flag, p.status);
                }
                ok = __all_sync(0xFFFFFFFFu, ok);
            }
            if (!ok) break;
            float acc[HD];
            if (ntiles > 0) {
                tc_fence_after();
#pragma unroll
                for (int ch = 0; ch < HD / 32; ++ch) tc_ld32(tO + ch * 32, acc + ch * 32);
                tc_wait_ld();
                if (alt && n1 > 0) {
                    // merge the odd-tile stream: O = w0 O0 + w1 O1, l = w0 l0 + w1 l1 at the common maximum
                    const float2 ml1 = s_ml1[rloc];
                    const float m = fmaxf(m_ref, ml1.x);
                    const float m_use = m == -CUDART_INF_F ? 0.f : m;
                    const float w0 = fast_exp2(m_ref - m_use), w1 = fast_exp2(ml1.x - m_use);
                    const uint32_t tO1 = tmem + lane_addr + T::COL_O1;
#pragma unroll
                    for (int ch = 0; ch < HD / 32; ++ch) {
                        float v[32];
                        tc_ld32(tO1 + ch * 32, v);
                        tc_wait_ld();
#pragma unroll
                        for (int e = 0; e < 32; ++e) acc[ch * 32 + e] = w0 * acc[ch * 32 + e] + w1 * v[e];
                    }
                    l_run = w0 * l_run + w1 * ml1.y;
                    m_ref = m;
                    tc_fence_before();
                    __syncwarp();                       // (every lane has read its pair)
                    if (lane == 0) mbar_arrive(bar(BAR_O_FREE + 1));
                    ++mlc;
                }
                tc_fence_before();
                if (lane == 0) mbar_arrive(bar(BAR_O_FREE + i));
            } else {
#pragma unroll
                for (int e = 0; e < HD; ++e) acc[e] = 0.f;
            }
            if (u.nsplit == 1 && u.two) {
                // Normalise, round to bf16 and store the rows of a tensor-bound unit.  A lane has a row, and
                // stored as it is a store instruction touches 32 lines: about 2000 cycles of a unit,
                // during which the warp issues nothing else.  So the warp turns 32 columns of its rows
                // round in shared memory (16-byte pieces, swizzled by the row so that neither side
                // conflicts), and each of its stores writes 64 bytes of eight rows.  32 x 64/8 heads,
                // N 57, L 200-2100: 100.4 -> 96.2 us; 8 x 64/8, N 256, L 4096: 240.4 -> 239.1.  No
                // barrier: a warp's rows are its own.
                unsigned char* stage = smem_raw + (sStage - smem_u32(smem_raw)) + warp * T::STAGE_BYTES;
                const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
                const bool mine = rvalid && GSD_IN_BOUNDS(b < p.B && c < p.Hkv && row < R, p.status);
                const int at = mine ? (row / G) * p.Hq + row % G : -1;      // heads from the sequence's first row
                __nv_bfloat16* base = p.out + ((size_t)b * N * p.Hq + c * G) * HD + (lane & 3) * 8;
                int to[4];                                                   // of the four rows this lane stores a piece of
#pragma unroll
                for (int j = 0; j < 4; ++j) to[j] = __shfl_sync(0xFFFFFFFFu, at, 8 * j + (lane >> 2));
#pragma unroll
                for (int ch = 0; ch < HD / 32; ++ch) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        uint32_t v[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) v[e] = pack_bf16(acc[ch * 32 + k * 8 + 2 * e] * inv, acc[ch * 32 + k * 8 + 2 * e + 1] * inv);
                        *reinterpret_cast<uint4*>(stage + lane * 64 + ((k ^ ((lane >> 1) & 3)) << 4)) = make_uint4(v[0], v[1], v[2], v[3]);
                    }
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int r = 8 * j + (lane >> 2);
                        const uint4 v = *reinterpret_cast<const uint4*>(stage + r * 64 + (((lane & 3) ^ ((r >> 1) & 3)) << 4));
                        if (to[j] >= 0) *reinterpret_cast<uint4*>(base + (size_t)to[j] * HD + ch * 32) = v;
                    }
                    __syncwarp();                                            // (the pieces have been read)
                }
            } else if (u.nsplit == 1) {
                // Units with one row tile, where the loads are the bound, store straight from registers;
                // every store of a lane fills a 32-byte sector.  (Turned round like the above 8 x 32 heads,
                // N 8, L 64 took 15.4 us instead of 14.8.  Staged in shared memory and stored by TMA it took
                // two barriers and a wait per 64 columns: 4 x 40 heads 55.0 us instead of 54.4, D 64 37.1
                // instead of 36.6.)
                if (rvalid && GSD_IN_BOUNDS(b < p.B && c < p.Hkv && row < R, p.status)) {
                    const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
                    __nv_bfloat16* dst = p.out + (((size_t)b * N + row / G) * p.Hq + c * G + row % G) * HD;
#pragma unroll
                    for (int k = 0; k < HD / 16; ++k) {
                        uint32_t v[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) v[e] = pack_bf16(acc[k * 16 + 2 * e] * inv, acc[k * 16 + 2 * e + 1] * inv);
                        if (p.out_by_32) {
                            st_global8(dst + k * 16, v);
                        } else {
                            reinterpret_cast<uint4*>(dst)[2 * k] = make_uint4(v[0], v[1], v[2], v[3]);
                            reinterpret_cast<uint4*>(dst)[2 * k + 1] = make_uint4(v[4], v[5], v[6], v[7]);
                        }
                    }
                }
            } else if (rvalid) {
                // a partial result: float4 columns of the row tile, so that the 32 rows of a warp
                // are consecutive in memory (stored row by row, 32 rows per store instruction, the
                // store took about 1 us longer)
                const size_t tile = (size_t)u.slot * 2 + (alt ? 0 : i);
                if (GSD_IN_BOUNDS(u.slot >= 0 && u.slot < p.slots, p.status)) {
                    float4* dst = reinterpret_cast<float4*>(p.part_o) + tile * (HD / 4) * BM + rloc;
#pragma unroll
                    for (int k = 0; k < HD / 4; ++k) dst[k * BM] = make_float4(acc[4 * k], acc[4 * k + 1], acc[4 * k + 2], acc[4 * k + 3]);
                    *reinterpret_cast<float2*>(p.part_ml + (tile * BM + rloc) * 2) = make_float2(m_ref, l_run);
                }
            }
            kvc += ntiles;
            tcnt += my_n;
            if (ntiles > 0) ++auc;
            if (n1 > 0) ++auc1;
        }
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (warp == 10) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// ------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres);
        if (e != cudaSuccess || qres != cudaDriverEntryPointSuccess || !ptr) {
            if (e != cudaSuccess) set_cuda_error(e, "cudaGetDriverEntryPoint(cuTensorMapEncodeTiled)");
            else set_error_text("cuTensorMapEncodeTiled is not available in this driver");
            return nullptr;
        }
        fn = (EncodeTiledFn)ptr;
    }
    return fn;
}

// [d3][d2][d1][D] bf16 tensor; box = 64 columns x box1 x box2 x 1, 128-byte swizzle, zero fill
int make_map(CUtensorMap* m, const void* base, uint64_t HD, uint64_t d1, uint64_t d2, uint64_t d3, uint32_t box1, uint32_t box2) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return GSD_ERR_CUDA;
    const cuuint64_t dims[4] = {(cuuint64_t)HD, d1, d2, d3};
    const cuuint64_t strides[3] = {(cuuint64_t)HD * 2, (cuuint64_t)HD * 2 * d1, (cuuint64_t)HD * 2 * d1 * d2};
    const cuuint32_t box[4] = {64, box1, box2, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        char msg[96];
        snprintf(msg, sizeof msg, "cuTensorMapEncodeTiled failed with CUresult %d", (int)r);
        set_error_text(msg);
        return GSD_ERR_CUDA;
    }
    return GSD_OK;
}

}  // namespace

template <int HD, int PLAN, bool LONG_MASK>
static int launch_tc(const AttnArgs& a) {
    const int nodes = BM / a.G;           // whole nodes of a row tile
    CUtensorMap tq, tk, tv, tdk, tdv;
    int rc;
    if ((rc = make_map(&tq, a.q, HD, a.Hq, a.N, a.B, a.G, nodes)) != GSD_OK) return rc;
    if ((rc = make_map(&tk, a.k_cache, HD, a.Hkv, a.Lmax, a.B, 1, BN)) != GSD_OK) return rc;
    if ((rc = make_map(&tv, a.v_cache, HD, a.Hkv, a.Lmax, a.B, 1, BN)) != GSD_OK) return rc;
    if ((rc = make_map(&tdk, a.draft_k, HD, a.Hkv, a.N, a.B, 1, BN)) != GSD_OK) return rc;
    if ((rc = make_map(&tdv, a.draft_v, HD, a.Hkv, a.N, a.B, 1, BN)) != GSD_OK) return rc;
    TcParams p;
    p.mask = a.mask; p.seq_lens = a.seq_lens; p.out = (__nv_bfloat16*)a.out; p.status = a.status;
    p.out_by_32 = ((uintptr_t)a.out & 31u) == 0;
    p.B = a.B; p.N = a.N; p.Hq = a.Hq; p.Hkv = a.Hkv; p.Lmax = a.Lmax; p.G = a.G; p.W = a.W;
    p.R = a.N * a.G; p.RT = nodes * a.G; p.scale_log2 = a.scale_log2; p.plan = a.plan.dev;
    p.raise_above = HD == 128 && BM % a.G == 0 && a.N * a.G >= 64 ? kRescaleThreshold : 0.f;
    p.part_o = (float*)a.workspace;
    p.part_ml = (float*)((char*)a.workspace + plan_part_o_bytes(a.plan, a.D));
    {
        // the opt-in for large dynamic shared memory is per kernel and device and sticks: do it once
        static bool done[64] = {};
        int dev = 0;
        GSD_CUDA_TRY(cudaGetDevice(&dev));
        if (dev < 0 || dev >= 64 || !done[dev]) {
            GSD_CUDA_TRY(cudaFuncSetAttribute(attn_tc_kernel<HD, PLAN, LONG_MASK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Geo<HD>::SMEM_BYTES));
            if (dev >= 0 && dev < 64) done[dev] = true;
        }
    }
    p.work0 = 0;
    p.total_work = a.plan.ctas;
    p.slots = a.plan.slots;
    p.wait_limit_ns = g_wait_limit_ns;
    p.withhold_first_k = g_withhold_first_k;
    DeviceInfo di;
    if (device_info(&di) != 0) return GSD_ERR_CUDA;
    p.bal_cta = nullptr;
    p.bal_units = nullptr;
    p.left = a.plan.slots && (a.plan.dev.balanced == 3 || a.plan.dev.longest_first) ? plan_left_table(a.plan, a.D, a.workspace) : nullptr;
    p.left_off = (int)(align_up((size_t)a.B * sizeof(int), 256) / sizeof(int));
    p.seq.hdr = nullptr; p.seq.nsplit = nullptr; p.seq.unit_off = nullptr; p.seq.slot_off = nullptr;
    if (a.plan.dev.balanced == 2) {
        p.seq = plan_seq_table(a.plan, a.D, a.B, a.workspace);
    } else if (a.plan.dev.balanced == 1) {
        const BalTable t = plan_bal_table(a.plan, a.D, a.workspace);
        p.bal_cta = t.cta;
        p.bal_units = t.units;
    }
    // Persistent CTAs.  A short call sets itself up beside the end of its predecessor on the stream, which
    // saves 1 to 2 us where that is other work (beside / behind: 4 x 40 heads, N 128, L 1024-4096, 36 key
    // tiles a CTA, 51.0 / 52.5 us; the step of 8 x 64/8 heads, N 256, L 4096, 118 tiles, 340 / 342).  A
    // long one, which has nothing to gain, is launched the ordinary way: CTAs placed where and when SMs
    // fall free ran up to 1% slower (32 x 64/8 heads, L 8192, N 512, 1882 tiles, power-limited: 4155 / 4103
    // once, 4091 / 4085 another time).  256 tiles are about 400 us.
    const long long tiles = (long long)a.plan.items * ((a.Lmax + BN - 1) / BN + (a.N + BN - 1) / BN);
    const bool beside = a.plan.dev.balanced || tiles < 256ll * di.sm_count;
    cudaLaunchAttribute attr[1];
    dependent_launch_attr(attr);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.plan.dev.balanced || a.plan.ctas < di.sm_count ? a.plan.ctas : di.sm_count));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Geo<HD>::SMEM_BYTES;
    cfg.stream = a.stream;
    cfg.attrs = attr;
    cfg.numAttrs = beside ? 1 : 0;
    const int part = PLAN == PLAN_FIXED || PLAN == PLAN_ORDERED ? (int)cfg.gridDim.x * kUnitTable : a.plan.ctas;
    for (p.work0 = 0; p.work0 < a.plan.ctas; p.work0 += part) {
        p.total_work = a.plan.ctas - p.work0 < part ? a.plan.ctas - p.work0 : part;
        GSD_CUDA_TRY(cudaLaunchKernelEx(&cfg, attn_tc_kernel<HD, PLAN, LONG_MASK>, tq, tk, tv, tdk, tdv, p));
    }
    return GSD_OK;
}

int attn_tcgen05_rows(int G) { return G <= BM ? BM / G * G : BM; }

bool attn_tcgen05_supports(int D, int G) { return (D == 128 || D == 64) && G >= 1 && G <= BM; }

template <bool LONG_MASK>
static int launch_plan(const AttnArgs& a) {
    switch (a.plan.dev.balanced == 3 ? PLAN_WAVE : a.plan.dev.balanced ? PLAN_TABLE : a.plan.dev.longest_first ? PLAN_ORDERED : PLAN_FIXED) {
        case PLAN_WAVE: return a.D == 128 ? launch_tc<128, PLAN_WAVE, LONG_MASK>(a) : launch_tc<64, PLAN_WAVE, LONG_MASK>(a);
        case PLAN_ORDERED: return a.D == 128 ? launch_tc<128, PLAN_ORDERED, LONG_MASK>(a) : launch_tc<64, PLAN_ORDERED, LONG_MASK>(a);
        case PLAN_TABLE: return launch_tc<128, PLAN_TABLE, LONG_MASK>(a);     // (D = 128 only)
        default: return a.D == 128 ? launch_tc<128, PLAN_FIXED, LONG_MASK>(a) : launch_tc<64, PLAN_FIXED, LONG_MASK>(a);
    }
}

// The mask words of a unit are more than a warp fetches in one round of 16-byte loads (one head a group: N above
// 170, two: above 256, three: above 384, four and more: never).  A kernel of its own: the code for slices in the
// others' prologue cost calls of a few tiles up to 4%; with up to 1024 words it is a wash (D 64, 4 x 32/8 heads, N 428,
// L 20322, 896 words: 586 us, 592 so).
static bool long_mask(const AttnArgs& a) {
    const int nodes = 2 * (BM / a.G);
    return (nodes < a.N ? nodes : a.N) * a.W > 8 * 32 * 4;
}

int launch_attn_tcgen05(const AttnArgs& a) {
    if (!attn_tcgen05_supports(a.D, a.G)) {
        set_error_text("tcgen05 back end needs a head dimension of 64 or 128 and a group size of at most 128");
        return GSD_ERR_UNSUPPORTED;
    }
    return long_mask(a) ? launch_plan<true>(a) : launch_plan<false>(a);
}

void debug_attn_wait(unsigned long long limit_ns, int withhold_first_k) {
    g_wait_limit_ns = limit_ns ? limit_ns : kWaitLimitNs;
    g_withhold_first_k = withhold_first_k;
}

}  // namespace gsd
