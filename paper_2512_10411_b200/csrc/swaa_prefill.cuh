// Prefill attention for sm_100a: tcgen05 MMAs accumulating in tensor memory, TMA-staged operands,
// online softmax with one thread per query row.
//
// Mask policy (Sec. 1, 3.1.2, 3.2.1; App. A): a query at position i of its sequence sees key j iff
//     j <= i  and  ( is_full  or  j > i - window  or  j < n_sink ).
// Only keys near a visible one are visited (the band and the sinks), so the work is O(L * window) as App. A states; the
// element predicate is evaluated only on tiles that are not entirely visible.
//
// One thread block processes one 128-row query tile for TWO query heads of the same GQA group
// ("sides" A and B).  Both sides need exactly the same K/V tiles and the same masks, so each K/V tile
// is staged in shared memory once and feeds four MMAs.  (Short sequences are packed instead: see WorkItem.)  Roles:
//   warps 0-3   softmax of side A   (thread = query row; lane quadrant = TMEM lane quadrant)
//   warps 4-7   softmax of side B
//   warp  8     TMA producer: Q tiles once, then the K and V tile rings
//   warp  9     MMA issuer and TMEM allocation
//   warp 10     work scheduler (takes over the indices of blocks that have not started)
// Tensor memory (512 columns x 128 lanes of 32 bit): S_A | S_B | O_A | O_B.  The bf16 probabilities
// P overwrite the first 64 columns of their own S and are consumed from TMEM as the A operand of
// O += P V.  V tiles are used as the MN-major B operand exactly as TMA lands them.
// Per key tile n the issuer runs  PV_A(n) QK_A(n+1) PV_B(n) QK_B(n+1), so the softmax of one side
// overlaps the MMAs of the other.  The exponentials are taken against a reference per row that is raised
// (and O rescaled) only when a tile's scores outgrow it by far; the final division by the row sum makes the result
// independent of that choice.
//
// What bounds it.  A side is a chain softmax -> P V -> Q K^T, and two sides are in flight: per 128 x 128 tile of both 3260 cycles
// against 2050 of products and 1970 of softmax (32k tokens, Hq = 32, Hkv = 8, D = 128, full causal); with a window of 2048 the
// tensor pipe is active 59 % of the cycles.  Against the kernel that had one issuing lane, a maximum pass on every tile, sink
// tiles of their own and a fixed assignment of items (3710 cycles): 8320 -> 7580 us; the same prompt with the window 1187 -> 1087;
// eight ragged prompts of 146k tokens, Hq = 64, window 4096: 17600 -> 16090 us; a serving step of 4 prompt chunks and 24 generated
// tokens in pages: 1134 -> 504 us.
//
// Every wait is bounded: a wait that runs out records SWAA_ERR_TIMEOUT, all roles leave their loops,
// the block waits (bounded) for its outstanding copies, frees its tensor memory and returns.
#pragma once

#include <cuda.h>

#include "swaa_internal.cuh"
#include "swaa_ptx.cuh"

namespace swaa {

constexpr int kPrefillBM = 128;
constexpr int kPrefillBN = 128;
constexpr int kPrefillThreads = 384;  // 8 softmax warps + 4 auxiliary warps (producer, issuer, scheduler, 1 idle)
constexpr int kPrefillSmallBox = 16;                        // rows of the small TMA boxes over K and V
constexpr int kWorkInts = 24;                               // words of a work descriptor
constexpr float kRescaleThreshold = 8.0f;                   // log2 units
constexpr float kGrowLimit = 32768.f;                       // 2^15: row sum of a tile above which the reference is looked at
constexpr float kLeadLimit = 1073741824.f;                  // 2^30: row sum so far that the reference is raised by
constexpr float kArgLimit = 110.f;                          // argument of an exponential, and log2 of the row sum of a tile,
constexpr float kSumLimit = 1.298074214633707e33f;          // above which the item is run again

struct PrefillParams {
    const __nv_bfloat16* q;  // token_kernel only
    __nv_bfloat16* out;
    float* lse;             // nullable, [Hq, T]
    const int32_t* cu_seqlens;    // queries (and keys, when cu_seqlens_k is null)
    const int32_t* cu_seqlens_k;  // nullable: keys of a chunked prefill, len_k >= len_q per sequence
    int B, T, max_seqlen, Hq, Hkv, G;
    int Tk, max_seqlen_k;         // packed key tokens and longest key sequence (chunked prefill only)
    // paged keys/values (kMode 2): cu_seqlens_k holds the key LENGTHS [B]; entry j of sequence b lives in page
    // block_table[b * max_blocks + j / page_size] at row j % page_size
    const int32_t* block_table;
    int max_blocks, page_size, num_pages;
    int heads;              // query heads per unpacked item: two, one per side, or one
    int units_per_kv;       // ceil(G / heads)
    int n_units;            // Hkv * units_per_kv
    int tiles_ub;           // upper bound on the number of query tiles over all sequences
    int pack_tokens;        // 128 / G: a sequence of at most this many queries is one item per kv head (see WorkItem)
    int window, n_sink, is_full;
    const uint8_t* is_full_seq;   // nullable (chunked / paged): mask policy per sequence, replaces is_full
    // context-parallel prefill (kMode 3): the local keys of sequence b start at position key_pos0[b]; the keys at
    // positions 0 .. sink_rows-1 of every sequence come from a separate buffer [B, sink_rows, Hkv, D]
    const int32_t* key_pos0;
    int sink_rows;
    float sl2;              // softmax scale * log2(e)
    float scale;
    // Chunked / paged: sequences of at most this many queries are left to token_kernel, which is launched behind this kernel
    // and may start as soon as all blocks of this one have (-1: there are none).
    int token_len;
    int sms;
    // token_kernel: tickets, (max, sum) and unnormalised O of the rows of split items (null: none are split), see there
    unsigned long long* split_tickets;
    float2* split_ml;
    float* split_o;
    unsigned long long stamp;     // 48-bit number unique to this call (never 0)
};

// Tensor maps of one call; an instance reads those that it needs.
struct PrefillMaps {
    CUtensorMap q;                 // [128 rows] x 1 head
    CUtensorMap q_packed;          // [128 / G tokens] x G heads
    CUtensorMap k, v;              // one key tile
    CUtensorMap k_small, v_small;  // kPrefillSmallBox keys
    CUtensorMap out;               // [32 rows] x 1 head
    CUtensorMap sink_k, sink_v;    // context-parallel
};

// ------------------------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// D[tmem] (+)= A * B with A in shared memory (ss) or tensor memory (ts) and B in shared memory.  The shared-memory descriptors
// are given as (low word, shared high word): the low word holds the start address and the leading-dimension offset, so
// stepping through a tile is one 32-bit add per operand.
__device__ __forceinline__ void mma_ss_lh(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_ts_lh(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\tsetp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Packed pairs of fp32 in one 64-bit register (two lanes per FMA/ADD instruction on sm_100).
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// Asks the hardware for the index of a block of this grid that has not started yet (and will then never start): the
// answer, 16 bytes, lands in shared memory.
__device__ __forceinline__ void next_block_request(uint32_t dst, uint32_t bar) {
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(dst),
                 "r"(bar)
                 : "memory");
}
// Block index of the answer, -1 when none was left.
__device__ __forceinline__ int next_block_answer(uint32_t src) {
    uint32_t ok, x;
    asm volatile(
        "{\n\t.reg .b128 r;\n\t.reg .pred p;\n\t.reg .b32 y, z, w;\n\t"
        "ld.shared.b128 r, [%2];\n\t"
        "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t"
        "mov.u32 %1, 0;\n\t"
        "@p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%1, y, z, w}, r;\n\t}"
        : "=r"(ok), "=r"(x)
        : "r"(src)
        : "memory");
    return ok ? (int)x : -1;
}

// True in one lane of the (converged) warp.  An issuing warp runs its loop with all lanes and lets the elected
// lane issue: control flow and descriptors then stay in uniform registers.  Measured with completed barriers: two
// looks and two commits per 13-instruction step cost 470 cycles in a loop run by one lane alone, 100 this way.
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\tselp.u32 %0, 1, 0, e;\n\t}" : "=r"(r));
    return r != 0;
}
// Bounded wait of a whole warp, one decision for all lanes.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag)) != 0;
}

// 2^x for a pair of arguments on the FMA and integer pipes instead of the special-function unit:
// x = n + f with n = round(x), f in [-1/2, 1/2]; 2^f by a cubic with constant term exactly 1 (minimax fit of
// the other three coefficients: relative error 1.0e-4, far below the bf16 rounding of P), so that 2^0 = 1
// exactly as on the special-function unit and a row of equal scores sums to its key count; n is added into
// the exponent field.  The argument is first raised to -127, where the result is exactly 0 (f = 0, the cubic gives
// 1.0 and the exponent field cancels), so masked scores (-inf) and anything below 2^-127 give exact zeros as
// ex2.approx.ftz does, at the price of one max per element instead of a compare and a select.
__device__ __forceinline__ void exp2_poly_x2(float x0, float x1, float& r0, float& r1) {
    const float kMagic = 12582912.f;  // 1.5 * 2^23: adding it leaves round(x) in the low mantissa bits
    x0 = fmaxf(x0, -127.f);
    x1 = fmaxf(x1, -127.f);
    const uint64_t xx = pack_f32x2(x0, x1);
    uint64_t t, fl, f, q;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(xx), "l"(pack_f32x2(kMagic, kMagic)));
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(fl) : "l"(t), "l"(pack_f32x2(kMagic, kMagic)));
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(f) : "l"(xx), "l"(fl));
    q = fma_f32x2(f, pack_f32x2(0.055009059607982635f, 0.055009059607982635f),
                  pack_f32x2(0.2422109693288803f, 0.2422109693288803f));
    q = fma_f32x2(q, f, pack_f32x2(0.6932829022407532f, 0.6932829022407532f));
    q = fma_f32x2(q, f, pack_f32x2(1.0f, 1.0f));
    float t0, t1, q0, q1;
    unpack_f32x2(t, t0, t1);
    unpack_f32x2(q, q0, q1);
    r0 = __uint_as_float(__float_as_uint(q0) + (__float_as_uint(t0) << 23));
    r1 = __uint_as_float(__float_as_uint(q1) + (__float_as_uint(t1) << 23));
}

// Bit c (0..15) set: column pair c of every 32-column chunk of a score tile takes the polynomial path.
// Three in sixteen: none, 1/8, 3/16 and 1/4 of the exponentials give 7743, 7727, 7624 and 7667 us on a full causal 32k
// prompt (Hq = 32, Hkv = 8, D = 128) and 1106, 1113, 1102 and 1100 us on the same prompt with a 2048-key window.
constexpr uint32_t kPolyPairMask = 0x8420u;

#define SWAA_R8(r, o) "=r"(r[o + 0]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), "=r"(r[o + 6]), "=r"(r[o + 7])
#define SWAA_I8(r, o) "r"(r[o + 0]), "r"(r[o + 1]), "r"(r[o + 2]), "r"(r[o + 3]), "r"(r[o + 4]), "r"(r[o + 5]), "r"(r[o + 6]), "r"(r[o + 7])

// 32 lanes x 32 consecutive columns: thread `lane` of the warp receives columns c .. c+31 of TMEM
// lane (quadrant base + lane).  These and the waits for them are .aligned: all lanes have to arrive together, so a branch that
// only some lanes take (a lane that arrives on a barrier, rows that do not exist) is closed with a __syncwarp first.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,"
        "%29,%30,%31}, [%32];"
        : SWAA_R8(r, 0), SWAA_R8(r, 8), SWAA_R8(r, 16), SWAA_R8(r, 24)
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,"
        "%29,%30,%31};" ::SWAA_I8(r, 0),
        SWAA_I8(r, 8), SWAA_I8(r, 16), SWAA_I8(r, 24), "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};" ::
            SWAA_I8(r, 0),
        SWAA_I8(r, 8), "r"(taddr)
        : "memory");
}

// Keeps the uses of 64 registers that asynchronous tensor-memory loads fill behind the wait for those loads.
__device__ __forceinline__ void pin64(uint32_t* r) {
#pragma unroll
    for (int i = 0; i < 64; ++i) asm volatile("" : "+r"(r[i]));
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : SWAA_R8(r, 0), SWAA_R8(r, 8)
        : "r"(taddr)
        : "memory");
}

// Shared-memory matrix descriptors for tiles stored as 128-byte rows with the 128-byte swizzle (what
// TMA writes for a [rows][64 bf16] box).  14-bit fields hold byte values >> 4.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version of this architecture
    d |= (uint64_t)2 << 61;  // 128-byte swizzle
    return d;
}

// kind::f16 instruction descriptor: bf16 x bf16 -> f32, M x N, A K-major, B K- or MN-major.
__host__ __device__ constexpr uint32_t make_idesc(int M, int N, int b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)b_mn_major << 16) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

template <int D>
struct PrefillSmem {
    static constexpr int kTileBytes = 128 * D * 2;  // one 128-row tile of Q, K or V
    static constexpr int kPanelBytes = 128 * 128;   // one [128 rows][64 ch] panel
    static constexpr int kPanels = D / 64;
    static constexpr int kStages = D == 128 ? 2 : 4;
    // Q of side A, then tile-sized slots one after another: Q of side B, kStages of K, kStages of V, the output staging
    // (8 x 4 KiB, one per softmax warp).  A packed item has one Q tile and no staged output, so all of the slots are
    // its ring of K and V tiles.
    static constexpr int kOffQ = 0;
    static constexpr int kOffSlots = kTileBytes;
    static constexpr int kSlotK = 1, kSlotV = 1 + kStages, kSlotStage = 1 + 2 * kStages;
    static constexpr int kStageBytes = 8 * 4096;
    static constexpr int kSlots = kSlotStage + kStageBytes / kTileBytes;
    static constexpr int kOffStage = kOffSlots + kSlotStage * kTileBytes;
    static constexpr int kOffMerge = kOffStage + kStageBytes;  // packed items: (max, sum) of side B's rows
    static constexpr int kOffBar = kOffMerge + 128 * 8;
    // barriers: Q full/empty; full/empty/V-tile-cleared (paged keys only) per slot; per side S full / P ready / O done /
    // O free; work descriptor full/empty per slot, next-block answer, hand-over of packed items per row quadrant,
    // staging free per work slot, final
    static constexpr int kNumBars = 2 + 3 * kSlots + 2 * 4 + 5 + 4 + 3;
    static constexpr int kOffMisc = (kOffBar + kNumBars * 8 + 15) / 16 * 16;  // next-block answer, tmem slot, flags, work descriptors
    static constexpr int kBytes = kOffMisc + 32 + 2 * kWorkInts * 4;
    static constexpr int kDynamicBytes = kBytes + 1024;          // room to align the base to 1024 B
    static_assert(kDynamicBytes <= 232448, "shared memory per block");
};

// One unit of work.  Usual form: a 128-row query tile of one sequence for one pair of query heads (one per side), or for a
// single query head, both sides on its rows, when the call has too few tiles for the SMs (see the launch).
// Packed form, for sequences whose queries times the group size fit in 128 rows (very short prompts; generated tokens where
// token_kernel does not take them): the rows are (query, head of the group) for ALL heads of one kv head, so K and V are read once per kv head
// and no row is padding that another head could use; the two sides then take alternate key tiles and merge at the end.
//
// Key columns of an item: the keys are enumerated as one list [band keys lo .. i1, rounded up
// to 16 | the sink keys before them] and cut into tiles of BN columns: a few sink keys share the last band tile or make
// a narrow tile of their own, and a tile that is not full runs fewer MMA steps.  lo is the first key of the window rounded
// down to 16 keys, so that the columns are whole groups of 16 keys counted from the start of the sequence: a sequence
// whose length is a multiple of 16 reads no key of the next one (a column that is not visible still counts as 0 * V in the
// P V product, and V may hold NaN there).  In pages lo is rounded down to a tile, so that a tile of band keys lies in one page.  A context-parallel item has n_rem whole tiles from the sink buffer in front.
// The scheduler writes the descriptor to shared memory; the other roles read the fields from there as they need them.
struct WorkItem {
    int valid, seq_start, seq_len;
    int q0;       // first query of the tile, counted inside the sequence's queries
    int hk, hA;   // kv head, (side A's, first) query head
    int packed;   // both sides work on one tile of rows; heads of a row group: rows = (query, head of the group), 1: queries of one head
    int hasB;     // side B has a query head of its own (unpacked items)
    int shared;   // packed item of several tiles: the sides take alternate key tiles and merge
    int full;     // this item runs full causal attention (per sequence in a mixed batch)
    int k_start;  // first packed key token of the sequence (= seq_start for self attention; sequence index when paged)
    int k_off;    // index of the sequence's first query among its (local) keys: len_k - len_q (0 for self attention)
    int i0, i1;   // first and last query position, counted among the (local) keys
    int lo, nb16, nv;  // key list: first band key, band columns, all columns
    int n_rem, nt;     // tiles from the sink buffer, all tiles
    int n_sink;   // sink keys among the local keys (context-parallel: n_sink - key_pos0, clamped; else n_sink)
    int s_rem;    // context-parallel: sink keys that come from the separate sink buffer, min(n_sink, key_pos0)
    int b;        // context-parallel: sequence index (row of the sink buffer)
    int n_rows;   // rows in use
    int careful;  // second run of an item whose scores left the exponent range of the first (see the softmax role)

    // fills the rest from seq_len, q0, packed, full, k_off, n_sink, s_rem and the unit: head pair (or head), or kv head when packed
    template <int BN, bool kPaged, bool kCp, bool kLseOnly>
    __host__ __device__ __forceinline__ void complete(const PrefillParams& p, int unit) {
        if (packed) {
            hk = unit;
            hA = unit * p.G;
            hasB = 0;
            n_rows = seq_len * p.G;
            i0 = k_off;
            i1 = k_off + seq_len - 1;
            packed = p.G;
        } else {
            hk = unit / p.units_per_kv;
            hA = hk * p.G + p.heads * (unit - hk * p.units_per_kv);
            hasB = p.heads == 2 && (hA + 1) < (hk + 1) * p.G ? 1 : 0;
            if (!kLseOnly && p.heads == 1) packed = 1;  // one tile of rows, both sides on it as in a packed item
            n_rows = min(kPrefillBM, seq_len - q0);
            i0 = q0 + k_off;
            i1 = i0 + n_rows - 1;
        }
        const int first = i0 - p.window + 1;
        lo = (full || first <= 0) ? 0 : (kPaged ? first / BN * BN : first / 16 * 16);
        nb16 = (i1 + 1 - lo + 15) / 16 * 16;
        const int ns = full ? 0 : min(n_sink, lo);
        nv = ns > 0 ? nb16 + ns : i1 + 1 - lo;
        n_rem = kCp ? (s_rem + BN - 1) / BN : 0;
        nt = n_rem + (nv + BN - 1) / BN;
        shared = packed && nt > 1 ? 1 : 0;
    }
};
static_assert(sizeof(WorkItem) == kWorkInts * 4, "words of a work descriptor");

// Tile t (t >= n_rem): column c holds band key jb + c for c < cb, else sink key js + c; the first 16 * nk columns are used.
template <int BN>
struct TileGeom {
    int cb, jb, js, left, nk;  // left: columns of the list from this tile on
    __host__ __device__ __forceinline__ TileGeom(const volatile WorkItem& g, int t) {
        const int v0 = (t - g.n_rem) * BN, nb16 = g.nb16;
        cb = max(0, min(BN, nb16 - v0));
        jb = g.lo + v0;
        js = v0 - nb16;
        left = g.nv - v0;
        nk = min(BN / 16, (left + 15) / 16);
    }
    __host__ __device__ __forceinline__ int key(int c) const { return c < cb ? jb + c : js + c; }
    __device__ __forceinline__ bool joins_sinks() const { return cb < 16 * nk; }
    // Columns of the tile that the query at index i (among the local keys) sees: band keys (c < cb) not after it (c <= dc) that
    // lie in its window (c >= wl) or among the sinks (c < sk), and the sink keys that follow the band (s0 <= c < s1), which
    // every query sees.  A remote tile (from the sink buffer) holds positions before every local key: its keys below s_rem.
    struct Seen {
        int dc, wl, sk, s0, s1;
    };
    __host__ __device__ __forceinline__ Seen seen(const volatile WorkItem& g, int t, bool remote, int i, int window) const {
        const bool full = g.full != 0;
        Seen s;
        s.dc = remote ? -1 : min(i - jb, cb - 1);
        s.wl = full ? 0 : i - jb - window + 1;
        s.sk = full ? 0 : g.n_sink - jb;
        s.s0 = remote ? 0 : cb;
        s.s1 = remote ? g.s_rem - t * BN : left;
        return s;
    }
    // rows [bad0, bad1) of the tile lie past the last of len_k keys (none: bad0 >= bad1)
    __device__ __forceinline__ int bad0(int len_k) const { return cb > 0 ? len_k - jb : BN; }
    __device__ __forceinline__ int bad1() const { return min(cb, 16 * nk); }
};

// Whether some query of item w does not see some column of its tile t, number n.  Text and not a function: as a function the
// kernel comes out 11 % slower at head size 64 (12.6k tokens, full attention, 32 heads: 919 us against 816; at head size 128
// the two are within 1 %).
#define SWAA_TILE_NEEDS_MASK(t, w, n, remote, window, BN)                                \
    ((remote) ? (w).s_rem - (n) * (BN) < (BN)                                            \
              : ((t).cb < (BN) ? ((t).cb > 0 || (t).left < (BN))                         \
                               : ((t).jb + (BN) - 1 > (w).i0 || (!(w).full && (t).jb <= (w).i1 - (window)))))

// A flag of a piece of code: known when it is compiled, or read when it runs.
template <bool kValue>
struct ConstFlag {
    static constexpr bool known = true, value = kValue;
};
struct RuntimeFlag {
    static constexpr bool known = false, value = false;
};

// kMode 0: self attention.  1: chunked prefill, the queries are the last len_q tokens of a longer key sequence
// (separate packing of the keys).  2: the same with keys and values in pages addressed through a block table.
// 3: context-parallel prefill, mode 1 with the local keys starting at position key_pos0[b] of their sequence and the
// sink keys before that position read from a separate buffer (sink_k, sink_v) as leading key tiles of the item.
// The self-attention instance compiles the offsets away.
// kLseOnly: only the log-sum-exp of every row is wanted (the lazy-ratio probe): no V tiles are fetched, no P V product
// is issued, P is not formed and nothing is written to `out`; the barrier protocol stays the same, with "P ready"
// meaning "S has been read"; items are never packed.
template <int D, int kMode, bool kLseOnly = false>
__global__ void __launch_bounds__(kPrefillThreads, 1)
prefill_kernel(const __grid_constant__ PrefillMaps tm, const PrefillParams p) {
    using L = PrefillSmem<D>;
    constexpr bool kChunked = kMode >= 1, kPaged = kMode == 2, kCp = kMode == 3;
    constexpr int BM = kPrefillBM, BN = kPrefillBN;
    constexpr int ST = L::kStages;
    constexpr int NK = BN / 16;        // 16-key steps of a tile
    // A packed item's ring spans all slots where the keys of a short sequence can be many (generated tokens).  In the
    // self-attention instance they cannot, and the loops are shorter without the second order of slots.
    constexpr bool kDeepRing = kChunked && !kLseOnly;
    using Tile = TileGeom<BN>;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t sQ = smem_base + L::kOffQ, sSlots = smem_base + L::kOffSlots;
    const uint32_t sStage = smem_base + L::kOffStage;
    const uint32_t bars = smem_base + L::kOffBar;
    auto bar = [&](int i) -> uint32_t { return bars + 8u * (uint32_t)i; };
    // barrier indices
    constexpr int NS = L::kSlots;
    constexpr int BAR_QF = 0, BAR_QE = 1, BAR_F = 2, BAR_E = BAR_F + NS;  // slot full, slot empty
    // paged only, one per slot: the rows of the V tile in that slot past the last key have been cleared.
    // Completed once per cleared tile; the issuer keeps the slot's phase bit.  The producer cannot
    // clear a slot twice before the issuer has waited for the first clear: reusing the slot needs the
    // issuer's empty commit, which follows that wait.
    constexpr int BAR_VC = BAR_E + NS;
    // per side: S full; P ready; O done, O free
    constexpr int BAR_SF = BAR_VC + NS, BAR_PR = BAR_SF + 2, BAR_OD = BAR_PR + 2, BAR_OF = BAR_OD + 2;
    // work descriptor full / empty per slot, next-block answer, hand-over of packed items (per row quadrant), staging free
    // for the ring of a packed item (per work slot), final
    constexpr int BAR_WF = BAR_OF + 2, BAR_WE = BAR_WF + 2, BAR_NB = BAR_WE + 2, BAR_MG = BAR_NB + 1, BAR_SG = BAR_MG + 4;
    constexpr int BAR_FIN = BAR_SG + 2;
    static_assert(BAR_FIN + 1 == L::kNumBars, "barrier count");
    const uint32_t s_answer = smem_base + L::kOffMisc;  // 16 bytes
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_gen + L::kOffMisc + 16);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* s_again = reinterpret_cast<volatile int*>(tmem_slot + 2);  // per slot: the item is to be run again
    volatile WorkItem* work_slots = reinterpret_cast<volatile WorkItem*>(tmem_slot + 4);  // two
    float2* s_merge = reinterpret_cast<float2*>(smem_gen + L::kOffMerge);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const bool full_all = p.is_full != 0;

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        s_again[0] = s_again[1] = 0;
        for (int i = 0; i < L::kNumBars; ++i) {
            uint32_t count = 1u;
            if ((i >= BAR_PR && i < BAR_OD) || i == BAR_OF || i == BAR_OF + 1) count = 4u;  // a lane of each softmax warp of the side
            if (i == BAR_WE || i == BAR_WE + 1) count = 10u;   // producer, issuer, eight softmax warps
            if (i == BAR_SG || i == BAR_SG + 1) count = 8u;    // a lane of each softmax warp
            mbar_init(bar(i), count);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 8 && elect_one()) {
        prefetch_map(&tm.q);
        if (p.pack_tokens > 0) prefetch_map(&tm.q_packed);
        prefetch_map(&tm.k);
        prefetch_map(&tm.v);
    }
    if (warp == 9) {  // TMEM: all 512 columns (S_A, S_B, O_A, O_B)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    grid_wait();  // nothing above touches global memory
    if ((kMode == 1 || kMode == 2) && p.token_len >= 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // Consumers of the work descriptors: item `it` is in slot it & 1; they read it in place and release it at their end of
    // the item.
    auto wait_work = [&](int it) -> bool { return warp_wait(bar(BAR_WF + (it & 1)), (uint32_t)(it >> 1) & 1u, abort_flag); };
    auto release_work = [&](int it) {
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(BAR_WE + (it & 1)));
        __syncwarp();
    };
    auto uniform = [](int x) -> int { return __shfl_sync(0xffffffffu, x, 0); };

    // Register budget per scheduler partition: two softmax warps at 216 + one auxiliary warp at 72.
    if (warp >= 8) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
      if (warp == 10) {
        // ====================================================================== work scheduler
        // The grid has one block per item (an upper bound); as many as fit start, and each takes over the indices of
        // blocks that have not started, so items go to whichever SM is free.  Items are ordered heavy-first, so that the
        // short ones fill the end: by the key tiles that they visit, over 32 sequences at a time (the last ones of the batch
        // first), and last tile of a sequence first.  Lane l looks after sequence base_b - l.  Sequences one after another, the heaviest
        // first, had left SMs with long items of the last sequence when the others were done: 3366 and 3292 tokens, full attention,
        // 28 heads of 128: 200 -> 186 us; five of 149 to 3766, 16 heads: 172 -> 155; eight of 641 to 3009: 159 -> 148.  A block waits
        // for the look for its first item, mostly for instructions that are not in its cache yet: the loops are not unrolled, and
        // calls whose items all start at once pass the search over.
        int base_b = p.B - 1;       // sequence of lane 0
        int base_w = 0;             // index of the first item of this group of 32 sequences
        int f_s = 0, f_len = 0, f_ks = 0, f_off = 0, f_full = full_all ? 1 : 0, f_sink = p.n_sink, f_srem = 0;
        int f_packed = 0, f_tiles = 0, f_units = 0, f_top = 0;  // of the lane's sequence: query tiles, items per tile, most key tiles of an item
        int group_items = 0, group_top = 0;                     // of the 32 sequences: items, most key tiles of an item
        auto load_group = [&]() {
            const int b = base_b - lane;
            f_tiles = f_units = f_top = 0;
            if (b >= 0) {
                const int s0 = p.cu_seqlens[b], e0 = p.cu_seqlens[b + 1];
                int len = e0 - s0;
                bool bad = len < 0 || len > p.max_seqlen || s0 < 0 || e0 > p.T;
                f_ks = s0;
                f_off = 0;
                if (kPaged) {  // keys in pages: cu_seqlens_k holds the key lengths
                    const int lk = p.cu_seqlens_k[b];
                    bad = bad || lk < len || lk > p.max_seqlen_k;
                    f_ks = b;
                    f_off = lk - len;
                } else if (kChunked) {  // chunked prefill: the queries are the last `len` tokens
                    const int ks = p.cu_seqlens_k[b], ke = p.cu_seqlens_k[b + 1];
                    bad = bad || ke - ks < len || ke - ks > p.max_seqlen_k || ks < 0 || ke > p.Tk;
                    f_ks = ks;
                    f_off = ke - ks - len;
                    if (kCp) {
                        // the local keys start at position p0: the sink keys before it come from the sink buffer,
                        // and the window of the first query must not reach below p0 (halo of window - 1 keys)
                        const int p0 = p.key_pos0[b];
                        bad = bad || p0 < 0 || (p0 > 0 && f_off < p.window - 1) || (p0 > 0 && p.n_sink > p.sink_rows);
                        f_srem = p0 < p.n_sink ? max(p0, 0) : p.n_sink;
                        f_sink = p.n_sink - f_srem;
                    }
                }
                if (bad) {
                    record_device_error(SWAA_ERR_BAD_SEQLENS);
                    len = 0;
                }
                if (kChunked && p.is_full_seq != nullptr) f_full = p.is_full_seq[b] != 0 ? 1 : 0;
                f_s = s0;
                f_len = len;
                f_packed = !kLseOnly && len <= p.pack_tokens ? 1 : 0;
                if (len > 0 && !(kChunked && !kCp && len <= p.token_len)) {
                    f_tiles = f_packed ? 1 : (len + BM - 1) / BM;
                    f_units = f_packed ? p.Hkv : p.n_units;
                    f_top = (f_off + len + BM - 1) / BM;
                    if (!f_full) f_top = (int)min((long long)f_top, ((long long)p.window + p.n_sink + BM) / BM + 1);
                }
            }
            group_items = __reduce_add_sync(0xffffffffu, f_tiles * f_units);
            group_top = __reduce_max_sync(0xffffffffu, f_top);
        };
        // query tiles of the lane's sequence (the last ones) whose items visit at least `level` key tiles, nearly: an order, no more
        auto tiles_from = [&](int level) -> int {
            if (level > f_top) return 0;
            const int x = (level - 1) * BM - f_off;
            return x <= 0 ? f_tiles : max(0, f_tiles - x / BM);
        };
        load_group();
        const bool at_once = p.B <= 32 && group_items <= p.sms;  // every item starts at once: any order will do
        int w = (int)blockIdx.x, it = 0;
        auto slot_words = [&](int slot) -> volatile int* { return reinterpret_cast<volatile int*>(work_slots + slot); };
        // publishes the descriptor that lies in slot it & 1 as a second run of the item of slot o
        auto run_again = [&](int o) {
            if (lane == 0) {
                work_slots[it & 1].careful = 1;
                s_again[o] = 0;
                mbar_arrive(bar(BAR_WF + (it & 1)));
            }
            __syncwarp();
            ++it;
        };
        // waits until slot it & 1 may be written; an item there that is to be run again is published first
        auto free_slot = [&]() -> bool {
            while (true) {
                if (!warp_wait(bar(BAR_WE + (it & 1)), ((uint32_t)(it >> 1) & 1u) ^ 1u, abort_flag)) return false;
                if (!uniform(s_again[it & 1])) return true;
                run_again(it & 1);
            }
        };
        uint32_t nb_phase = 0;
        bool ok = true;
        while (w >= 0) {
            if (w < base_w) {  // an index before this group of sequences: start over
                base_b = p.B - 1;
                base_w = 0;
                load_group();
            }
            bool valid;  // an index past the last item is passed over (the grid is an upper bound)
            while (true) {
                valid = w < base_w + group_items;
                if (valid || base_b < 32) break;
                base_w += group_items;
                base_b -= 32;
                load_group();
            }
            if (valid) {
                int local = w - base_w, last = f_tiles - 1;  // among the items of a lane's tiles up to the last one
                bool mine = lane == 0;
                if (p.B > 1) {
                    int own = f_tiles * f_units, above = 0;
                    if (!at_once) {
                        int lo = 1, hi = group_top + 1;  // the item's level: items from lo on are more than `local`, from hi on they are not
                        while (hi - lo > 1) {            // above: items from hi on
                            const int mid = (lo + hi) / 2, n = __reduce_add_sync(0xffffffffu, f_units * tiles_from(mid));
                            if (n > local) {
                                lo = mid;
                            } else {
                                hi = mid;
                                above = n;
                            }
                        }
                        last -= tiles_from(hi);
                        own = f_units * (last + 1 - (f_tiles - tiles_from(lo)));
                    }
                    int before = own;
#pragma unroll 1
                    for (int o = 1; o < 32; o <<= 1) {
                        const int x = __shfl_up_sync(0xffffffffu, before, o);
                        if (lane >= o) before += x;
                    }
                    local -= above + before - own;
                    mine = local >= 0 && local < own;
                }
                ok = free_slot();
                if (!ok) break;
                if (mine) {  // one lane
                    WorkItem d;
                    d.valid = 1;
                    d.seq_start = f_s;
                    d.seq_len = f_len;
                    const int back = (int)((unsigned)local / (unsigned)f_units);
                    d.q0 = f_packed ? 0 : (last - back) * BM;
                    d.packed = f_packed;
                    d.full = f_full;
                    d.k_start = f_ks;
                    d.k_off = f_off;
                    d.n_sink = f_sink;
                    d.s_rem = f_srem;
                    d.b = base_b - lane;
                    d.careful = 0;
                    d.complete<BN, kPaged, kCp, kLseOnly>(p, local - back * f_units);
                    volatile int* to = slot_words(it & 1);
                    const int* from = reinterpret_cast<const int*>(&d);
#pragma unroll
                    for (int i = 0; i < kWorkInts; ++i) to[i] = from[i];
                    mbar_arrive(bar(BAR_WF + (it & 1)));
                }
                __syncwarp();
                ++it;
            }
            if (lane == 0) {
                fence_proxy_async_smem();  // the previous answer has been read
                mbar_arrive_expect_tx(bar(BAR_NB), 16u);
                next_block_request(s_answer, bar(BAR_NB));
            }
            ok = warp_wait(bar(BAR_NB), nb_phase, abort_flag);
            if (!ok) {  // another role gave up: the answer has to land before the block's memory is released
                const uint64_t t0 = global_timer_ns();
                while (!mbar_try_wait(bar(BAR_NB), nb_phase) && global_timer_ns() - t0 < kWaitLimitNs) {
                }
                break;
            }
            nb_phase ^= 1u;
            w = uniform(next_block_answer(s_answer));
        }
        if (lane == 0 && (p.cu_seqlens[0] != 0 || p.cu_seqlens[p.B] != p.T)) record_device_error(SWAA_ERR_BAD_SEQLENS);
        // the last items have to be done before the end is published, lest one is to be run again
        while (ok) {
            ok = free_slot();
            if (!ok || it == 0) break;
            const int o = (it - 1) & 1;
            ok = warp_wait(bar(BAR_WE + o), (uint32_t)((it - 1) >> 1) & 1u, abort_flag);
            if (!ok || !uniform(s_again[o])) break;
            if (lane < kWorkInts) slot_words(it & 1)[lane] = slot_words(o)[lane];
            __syncwarp();
            run_again(o);
        }
        if (ok && lane == 0) {
            work_slots[it & 1].valid = 0;
            mbar_arrive(bar(BAR_WF + (it & 1)));
        }
        __syncwarp();
      } else if (warp == 8) {
        // =========================================================================== TMA producer
        // The whole warp walks the items and waits; one elected lane starts the copies.
        const bool el = elect_one();
        uint32_t phases = 0;             // bit: parity of the slot's next use
        int sk = 0, sv = 0, sx = 0;      // next stage of the K and V rings, next slot of a packed item's ring
        uint32_t sg_phase = 0;           // bit: parity of the work slot's next packed item
        bool ok = true;
        int items = 0;
        for (int it = 0; ok; ++it) {
            ok = wait_work(it);
            if (!ok) break;
            const volatile WorkItem& w = work_slots[it & 1];
            if (!uniform(w.valid)) break;
            const bool packed = !kLseOnly && uniform(w.packed) != 0, hasB = uniform(w.hasB) != 0;
            const int nt = uniform(w.nt), n_rem = kCp ? uniform(w.n_rem) : 0;
            const int len_k = uniform(w.k_off + w.seq_len), hk = uniform(w.hk), k_start = uniform(w.k_start);
            // Q tiles of both sides (the previous item's last Q K^T must have retired); packed: one tile serves both
            auto slot_free = [&](int slot) -> bool { return warp_wait(bar(BAR_E + slot), ((phases >> slot) & 1u) ^ 1u, abort_flag); };
            ok = warp_wait(bar(BAR_QE), ((uint32_t)items & 1u) ^ 1u, abort_flag) && (!kDeepRing || packed || slot_free(0));
            if (!ok) break;
            if (el) {
                const int hA = w.hA, tq = w.seq_start + w.q0;
                if (packed && w.packed > 1) {  // rows = (query, head of the group)
                    mbar_arrive_expect_tx(bar(BAR_QF), (uint32_t)(p.pack_tokens * p.G * 128 * L::kPanels));
#pragma unroll
                    for (int pn = 0; pn < L::kPanels; ++pn)
                        tma_load_3d(sQ + pn * L::kPanelBytes, &tm.q_packed, pn * 64, hA, tq, bar(BAR_QF));
                } else {
                    mbar_arrive_expect_tx(bar(BAR_QF), (hasB ? 2u : 1u) * (uint32_t)L::kTileBytes);
#pragma unroll
                    for (int pn = 0; pn < L::kPanels; ++pn) {
                        tma_load_3d(sQ + pn * L::kPanelBytes, &tm.q, pn * 64, hA, tq, bar(BAR_QF));
                        if (hasB)
                            tma_load_3d(sQ + L::kTileBytes + pn * L::kPanelBytes, &tm.q, pn * 64, hA + 1, tq, bar(BAR_QF));
                    }
                }
            }
            ++items;
            // page of a key, out of range (the copy delivers zeros) when the table is wrong
            auto page_of = [&](int key) -> int {
                const int page = p.block_table[(size_t)k_start * p.max_blocks + key / p.page_size];
                if (page >= 0 && page < p.num_pages) return page;
                record_device_error(SWAA_ERR_BAD_SEQLENS);
                return p.num_pages;
            };
            // K or V tile n into a slot.  A tile of band keys comes in one box per panel, one that joins sink keys in pieces of
            // 16 keys.
            auto load_tile = [&](int n, int slot, const CUtensorMap* map, const CUtensorMap* map_small,
                                 const CUtensorMap* map_sink) -> bool {
                const bool remote = kCp && n < n_rem;
                const Tile t(w, n);
                const bool whole = remote || !t.joins_sinks();
                const uint32_t dst = sSlots + (uint32_t)(slot * L::kTileBytes), full_bar = bar(BAR_F + slot);
                int page0 = 0, row0 = 0;  // of the first key, looked up ahead of the wait for the slot
                if (kPaged) {
                    const int key = t.key(0);
                    page0 = page_of(key);
                    row0 = key % p.page_size;
                }
                if (!slot_free(slot)) return false;
                if (el) {
                    mbar_arrive_expect_tx(full_bar, whole ? (uint32_t)L::kTileBytes : (uint32_t)(t.nk * 16 * 128 * L::kPanels));
                    if (whole) {
#pragma unroll
                        for (int pn = 0; pn < L::kPanels; ++pn) {
                            const uint32_t d = dst + (uint32_t)(pn * L::kPanelBytes);
                            if (remote) tma_load_4d(d, map_sink, pn * 64, hk, n * BN, w.b, full_bar);
                            else if (kPaged) tma_load_4d(d, map, pn * 64, hk, row0, page0, full_bar);
                            else tma_load_3d(d, map, pn * 64, hk, k_start + t.jb, full_bar);
                        }
                    } else {
                        for (int x = 0; x < t.nk; ++x) {
                            const int key = t.key(16 * x);
                            const int page = kPaged ? page_of(key) : 0;
#pragma unroll
                            for (int pn = 0; pn < L::kPanels; ++pn) {
                                const uint32_t d = dst + (uint32_t)(pn * L::kPanelBytes + x * 2048);
                                if (kPaged) tma_load_4d(d, map_small, pn * 64, hk, key % p.page_size, page, full_bar);
                                else tma_load_3d(d, map_small, pn * 64, hk, k_start + key, full_bar);
                            }
                        }
                    }
                }
                phases ^= 1u << slot;
                return true;
            };
            auto load_k = [&](int n, int slot) -> bool { return load_tile(n, slot, &tm.k, &tm.k_small, &tm.sink_k); };
            auto load_v = [&](int n, int slot) -> bool {
                if (kLseOnly) return true;
                if (!load_tile(n, slot, &tm.v, &tm.v_small, &tm.sink_v)) return false;
                if (kPaged) {
                    // The rows of a page past the sequence's last key may hold anything (also NaN, and 0 * NaN is
                    // NaN in the PV product): clear those that the P V product reads before the issuer may use the
                    // tile.  Only the last band tile of a sequence that does not end on a 16-key boundary is concerned.
                    const Tile t(w, n);
                    const int r0 = t.bad0(len_k), r1 = t.bad1();
                    if (r0 < r1) {
                        if (!warp_wait(bar(BAR_F + slot), ((phases >> slot) & 1u) ^ 1u, abort_flag)) return false;
                        const uint32_t dV = sSlots + (uint32_t)(slot * L::kTileBytes);
                        for (int c = lane; c < (r1 - r0) * 8; c += 32)
#pragma unroll
                            for (int pn = 0; pn < L::kPanels; ++pn)
                                st_shared_v4(dV + pn * L::kPanelBytes + (r0 + (c >> 3)) * 128 + (c & 7) * 16, 0u, 0u, 0u, 0u);
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (el) mbar_arrive(bar(BAR_VC + slot));
                    }
                }
                return true;
            };
            if (!(kDeepRing && packed)) {
                for (int n = 0; n < nt && ok; ++n) {
                    ok = load_k(n, L::kSlotK + sk);
                    sk = sk + 1 == ST ? 0 : sk + 1;
                    ok = ok && load_v(n, L::kSlotV + sv);
                    sv = sv + 1 == ST ? 0 : sv + 1;
                }
            } else {
                // One ring over all slots, in the order in which the issuer uses the tiles: K(0) K(1) V(0) K(2) V(1) K(3) ...
                // A generated token at a long context runs at the pace of memory, and how far the copies run ahead sets it: with
                // the two K and two V slots of the usual items one token at 32768 keys takes 421 us, 16 of them 499 us, a
                // serving step of 4 chunks and 24 generated tokens 805 us; with all six slots 363, 430 and 595 us.
                // Every softmax warp says once per packed item that it has no store from the staging under way.  The warps of a
                // side without work run ahead into the next item, so the barrier goes with the work slot: a slot takes another
                // item only when all roles have released this one, that is after all of its eight arrivals and this wait.
                bool staging = false;  // the output staging is known to be free
                auto wait_staging = [&]() {
                    if (!staging) ok = ok && warp_wait(bar(BAR_SG + (it & 1)), (sg_phase >> (it & 1)) & 1u, abort_flag);
                    staging = true;
                };
                auto next_slot = [&]() -> int {
                    const int slot = sx;
                    sx = sx + 1 == NS ? 0 : sx + 1;
                    if (slot >= L::kSlotStage) wait_staging();
                    return slot;
                };
                for (int n = -2; n < nt && ok; ++n) {
                    if (n >= 0) {
                        const int slot = next_slot();
                        ok = ok && load_v(n, slot);
                    }
                    if (ok && n + 2 < nt) {
                        const int slot = next_slot();
                        ok = ok && load_k(n + 2, slot);
                    }
                }
                wait_staging();
                sg_phase ^= 1u << (it & 1);
            }
            if (!ok) break;
            release_work(it);
        }
        if (!ok) {
            // give outstanding copies a bounded chance to land before the block's memory is released
            const uint64_t t0 = global_timer_ns();
            bool landed = false;
            while (!landed && global_timer_ns() - t0 < kWaitLimitNs) {
                landed = items == 0 || mbar_try_wait(bar(BAR_QF), (uint32_t)(items - 1) & 1u);
                for (int slot = 0; slot < NS; ++slot) landed = landed && mbar_try_wait(bar(BAR_F + slot), ((phases >> slot) & 1u) ^ 1u);
            }
        }
        __syncwarp();
      } else if (warp == 9) {
        // ============================================================================ MMA issuer
        // The warp runs the loop as a whole, one elected lane issues and commits (see elect_one).
        const bool el = elect_one();
        // Descriptor words are built once: per operand tile a low word (address, leading-dimension offset)
        // and one shared high word (stride 1024 B, descriptor version, 128-byte swizzle).
        const uint32_t desc_hi = (uint32_t)(smem_desc_sw128(0, 0, 1024) >> 32);
        const uint32_t q_lo = (uint32_t)smem_desc_sw128(sQ, 16, 1024);
        const uint32_t k_lo = (uint32_t)smem_desc_sw128(sSlots, 16, 1024);
        const uint32_t v_lo = (uint32_t)smem_desc_sw128(sSlots, L::kPanelBytes, 1024);
        constexpr uint32_t kStep = (uint32_t)L::kTileBytes >> 4;
        constexpr uint32_t kIdescQK = make_idesc(BM, BN, 0), kIdescPV = make_idesc(BM, D, 1);
        // Q K^T of a side over the first 16 * nk keys of a tile; q_tile: 0, or the side
        auto issue_qk = [&](int side, int q_tile, int slot, int nk) {
            const uint32_t qa = q_lo + (uint32_t)q_tile * kStep, kb = k_lo + (uint32_t)slot * kStep;
            const uint32_t idesc = nk == NK ? kIdescQK : (make_idesc(BM, 0, 0) | ((uint32_t)(2 * nk) << 17));
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
                const uint32_t off = ((uint32_t)(kk >> 2) * L::kPanelBytes + (uint32_t)(kk & 3) * 32u) >> 4;
                mma_ss_lh(tmem_base + 128u * (uint32_t)side, qa + off, kb + off, desc_hi, idesc, kk > 0 ? 1u : 0u);
            }
        };
        auto issue_pv = [&](int side, int slot, bool acc, int nk) {
            const uint32_t vb = v_lo + (uint32_t)slot * kStep, a = tmem_base + 128u * (uint32_t)side;
            const uint32_t d = tmem_base + 256u + (uint32_t)(D * side);
#pragma unroll
            for (int kk = 0; kk < NK; ++kk) {
                // P: 16 keys = 8 TMEM columns of packed bf16 pairs.  V: 16 key rows of 128 bytes.
                if (kk < nk)
                    mma_ts_lh(d, a + (uint32_t)kk * 8u, vb + (((uint32_t)kk * 2048u) >> 4), desc_hi, kIdescPV, (acc || kk > 0) ? 1u : 0u);
            }
        };
        uint32_t phases = 0;           // bit: parity of the slot's next use
        int sk = 0, sv = 0, sx = 0;    // next stage of the K and V rings, next slot of a packed item's ring
        int gs[2] = {0, 0};            // tiles processed per side (phase of P ready)
        int items_side[2] = {0, 0};    // items each side took part in (phase of O free)
        int items = 0;
        uint32_t vc_phase = 0;         // paged only: bit: phase of the slot's V-tile-cleared barrier
        bool ok = true;
        auto slot_full = [&](int slot) -> bool {
            const uint32_t parity = (phases >> slot) & 1u;
            phases ^= 1u << slot;
            return warp_wait(bar(BAR_F + slot), parity, abort_flag);
        };
        for (int it = 0; ok; ++it) {
            ok = wait_work(it);
            if (!ok) break;
            const volatile WorkItem& w = work_slots[it & 1];
            if (!uniform(w.valid)) break;
            const bool is_packed = !kLseOnly && uniform(w.packed) != 0, hasB = uniform(w.hasB) != 0;
            const int nt = uniform(w.nt), n_rem = kCp ? uniform(w.n_rem) : 0;
            // Only the last tile can be narrow, and only the last band tile can have rows past the last key: the loop below reads
            // nothing of the descriptor.
            const int nk_last = uniform((kCp && n_rem == nt) ? NK : Tile(w, nt - 1).nk);
            int vc_tile = -1;
            if (kPaged) {
                const int n = n_rem + (w.nb16 - 1) / BN;
                const Tile t(w, n);
                vc_tile = uniform(t.bad0(w.k_off + w.seq_len) < t.bad1() ? n : -1);
            }
            const bool shared = is_packed && nt > 1;
            ok = warp_wait(bar(BAR_QF), (uint32_t)items & 1u, abort_flag);
            auto run_item = [&](auto packed_tag) {
                const bool packed = decltype(packed_tag)::known ? decltype(packed_tag)::value : is_packed;
                const bool late_k = kDeepRing && packed;
                auto steps_of = [&](int n) -> int { return n == nt - 1 ? nk_last : NK; };
                const int ahead = packed ? 2 : 1;  // Q K^T runs this many tiles ahead of P V
                auto k_slot = [&]() -> int {
                    int slot;
                    if (late_k) {
                        slot = sx;
                        sx = sx + 1 == NS ? 0 : sx + 1;
                    } else {
                        slot = L::kSlotK + sk;
                        sk = sk + 1 == ST ? 0 : sk + 1;
                    }
                    return slot;
                };
                auto v_slot = [&]() -> int {
                    if (late_k) return k_slot();
                    const int slot = L::kSlotV + sv;
                    sv = sv + 1 == ST ? 0 : sv + 1;
                    return slot;
                };
                // the first scores of each side
                for (int n = 0; n < min(ahead, nt) && ok; ++n) {
                    const int nk = steps_of(n), ks = k_slot();
                    ok = slot_full(ks);
                    if (!ok) break;
                    tc_fence_after();
                    if (el) {
                        issue_qk(n, 0, ks, nk);
                        tc_commit(bar(BAR_SF + n));
                        if (hasB) {
                            issue_qk(1, 1, ks, nk);
                            tc_commit(bar(BAR_SF + 1));
                        }
                        tc_commit(bar(BAR_E + ks));
                        if (n == nt - 1) tc_commit(bar(BAR_QE));  // Q is no longer needed by this item
                    }
                }
                for (int n = 0; n < nt && ok; ++n) {
                    const int nk = steps_of(n);
                    const bool has_next = n + ahead < nt;
                    const int nk_next = has_next ? steps_of(n + ahead) : 0;
                    const int vs = kLseOnly ? 0 : v_slot(), ks = has_next ? k_slot() : 0;
                    // The tiles first (they landed long ago as a rule), then the side's P: what follows the P barrier is on
                    // the side's critical path softmax -> P V -> Q K^T -> softmax.
                    if (!kLseOnly) ok = slot_full(vs);
                    if (kPaged && ok && n == vc_tile) {  // rows past the last key, cleared by the producer
                        ok = warp_wait(bar(BAR_VC + vs), (vc_phase >> vs) & 1u, abort_flag);
                        vc_phase ^= 1u << vs;
                    }
                    if (has_next && !late_k) ok = ok && slot_full(ks);
                    if (!ok) break;
#pragma unroll
                    for (int side = 0; side < 2; ++side) {
                        if (packed ? (n & 1) != side : (side == 1 && !hasB)) continue;
                        const bool first = n < ahead;  // the side's first tile of this item
                        ok = ok && warp_wait(bar(BAR_PR + side), (uint32_t)gs[side] & 1u, abort_flag);
                        // the first P V of an item overwrites O: the previous item's epilogue must have read it
                        if (!kLseOnly && first) ok = ok && warp_wait(bar(BAR_OF + side), ((uint32_t)items_side[side] & 1u) ^ 1u, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        if (!kLseOnly && el) issue_pv(side, vs, !first, nk);
                        if (has_next && late_k) {  // packed items run at the pace of memory: free the V tile early, ask for K late
                            if (el) tc_commit(bar(BAR_E + vs));
                            ok = slot_full(ks);
                            if (!ok) break;
                            tc_fence_after();
                        }
                        if (el) {
                            // O done is only waited for by the item's epilogue: between tiles S full of the side's next tile
                            // already implies the P V before it (a commit covers every product issued before it)
                            if (!kLseOnly && !has_next) tc_commit(bar(BAR_OD + side));
                            if (has_next) {
                                issue_qk(side, packed ? 0 : side, ks, nk_next);
                                tc_commit(bar(BAR_SF + side));
                            }
                        }
                        ++gs[side];
                    }
                    if (!ok) break;
                    if (el) {
                        if (!kLseOnly && !(has_next && late_k)) tc_commit(bar(BAR_E + vs));
                        if (has_next) {
                            tc_commit(bar(BAR_E + ks));
                            if (n + ahead == nt - 1) tc_commit(bar(BAR_QE));
                        }
                    }
                }
            };
            if (!kDeepRing) run_item(RuntimeFlag{});
            else if (is_packed) run_item(ConstFlag<true>{});
            else run_item(ConstFlag<false>{});
            ++items;
            ++items_side[0];
            if (hasB || shared) ++items_side[1];
            release_work(it);
        }
        // all MMAs issued by this warp must have retired before the tensor memory is freed
        if (el) tc_commit(bar(BAR_FIN));
        warp_wait(bar(BAR_FIN), 0, abort_flag);
        __syncwarp();
      }
    } else {
        // ==================================================================== softmax + epilogue
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        const int side = warp >> 2;
        const int wq = warp & 3;
        const int row = wq * 32 + lane;
        const uint32_t lane_base = (uint32_t)(wq * 32) << 16;
        const uint32_t tS = tmem_base + lane_base + (uint32_t)side * 128u;
        const uint32_t tO = tmem_base + lane_base + 256u + (uint32_t)side * (uint32_t)D;
        // phases (bits) of: S full, O done (side A also keeps side B's), hand-over of packed items; and of the item:
        // some tile's scores outgrew the reference of a row of this warp by far
        uint32_t phases = 0;
        constexpr uint32_t kPhS = 1u, kPhO = 2u, kPhOB = 4u, kPhM = 8u, kGrown = 16u;
        bool ok = true;
        auto arrive_warp = [&](int b) {
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(b));
        };
        for (int it = 0; ok; ++it) {
            // every decision taken after a bounded wait is made for the whole warp: the warp-wide tensor-memory
            // instructions and votes below need all 32 lanes
            ok = wait_work(it);
            if (!ok) break;
            const volatile WorkItem& w = work_slots[it & 1];
            if (!uniform(w.valid)) break;
            const bool packed = !kLseOnly && uniform(w.packed) != 0;
            const bool shared = packed && uniform(w.shared) != 0;
            if (kDeepRing && packed && lane == 0) {  // the item's ring takes the staging area: earlier output stores have read it
                tma_store_wait_read();
                mbar_arrive(bar(BAR_SG + (it & 1)));
            }
            __syncwarp();
            if (side == 1 && !shared && !uniform(w.hasB)) {
                release_work(it);
                continue;
            }
            const int n_rows = uniform(w.n_rows), nt = uniform(w.nt);
            const bool row_ok = row < n_rows;
            const bool idle = wq * 32 >= n_rows;  // none of this warp's rows exists: it only keeps the barriers going
            float m_used = -INFINITY, l_sum = 0.f;
            const bool careful = uniform(w.careful) != 0;
            if (careful) {  // the first run of this item stored the same rows: its copies have to be performed before the next ones start
                if (lane == 0) tma_store_wait_all();
                __syncwarp();
            }
            bool fresh = true;   // some row of this warp has no reference yet, or one that is far behind
            for (int n = shared ? side : 0; n < nt; n += shared ? 2 : 1) {
                const bool remote = kCp && n < w.n_rem;
                const Tile t(w, n);
                const bool need_mask = SWAA_TILE_NEEDS_MASK(t, w, n, remote, p.window, BN);
                ok = warp_wait(bar(BAR_SF + side), (phases & kPhS) != 0 ? 1u : 0u, abort_flag);
                if (!ok) break;
                phases ^= kPhS;
                tc_fence_after();
                if (idle) {
                    arrive_warp(BAR_PR + side);
                    continue;
                }
                if (!kChunked && !kLseOnly && t.cb == 0 && t.left <= 32) {
                    // A few sink keys in a tile of their own, which every row sees: 32 columns instead of 128.  A block's last
                    // step before its output, so it counts in full where a block has few tiles: 1024 tokens, 4 heads of 64,
                    // window 128: 11.8 -> 10.6 us; 63 sequences at head size 64, forward and backward: 459 -> 455.  In the
                    // instances with a key list of its own the step's items are long and it measured nothing (506, 509).
                    uint32_t sn[32];
                    tmem_ld32(tS, sn);
                    tc_wait_ld();
                    float mx = -INFINITY;
#pragma unroll
                    for (int c = 0; c < 32; ++c) {
                        sn[c] = c < t.left ? sn[c] : 0xff800000u;  // -inf
                        mx = fmaxf(mx, __uint_as_float(sn[c]));
                    }
                    const float m_new = fmaxf(m_used, mx);
                    const bool need = (m_used != -INFINITY) && ((m_new - m_used) * p.sl2 > kRescaleThreshold);
                    if (__any_sync(0xffffffffu, row_ok && need)) {
                        const float alpha = (m_used == -INFINITY) ? 1.f : ex2f((m_used - m_new) * p.sl2);
#pragma unroll 1
                        for (int cc = 0; cc < D / 16; ++cc) {
                            uint32_t orr[16];
                            tmem_ld16(tO + (uint32_t)(cc * 16), orr);
                            tc_wait_ld();
#pragma unroll
                            for (int c = 0; c < 16; ++c) orr[c] = __float_as_uint(__uint_as_float(orr[c]) * alpha);
                            tmem_st16(tO + (uint32_t)(cc * 16), orr);
                        }
                        tc_wait_st();
                        l_sum *= alpha;
                        m_used = m_new;
                    } else if (m_used == -INFINITY) {
                        m_used = m_new;
                    }
                    fresh = __any_sync(0xffffffffu, row_ok && m_used == -INFINITY);
                    const float off = m_used == -INFINITY ? 0.f : m_used * p.sl2;
                    uint32_t pk[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        const float p0 = ex2f(fmaf(__uint_as_float(sn[2 * c]), p.sl2, -off));
                        const float p1 = ex2f(fmaf(__uint_as_float(sn[2 * c + 1]), p.sl2, -off));
                        l_sum += p0 + p1;
                        pk[c] = pack_bf16x2(p0, p1);
                    }
                    tmem_st16(tS, pk);
                    tc_wait_st();
                    tc_fence_before();
                    arrive_warp(BAR_PR + side);
                    continue;
                }
                uint32_t sr[BN];
                tmem_ld32(tS, sr);
                tmem_ld32(tS + 32u, sr + 32);
                tc_wait_ld();
                // the second half is fetched under the first half's exponentials (P goes to columns 0..63)
                tmem_ld32(tS + 64u, sr + 64);
                tmem_ld32(tS + 96u, sr + 96);
                // Usual tile: the exponentials are taken against the reference as it stands, without forming the tile's maximum
                // first (64 of some 600 instructions per row and tile; 3.5 % of the kernel's time at 32k tokens).  That loses
                // no precision as long as nothing leaves the exponent range: bf16 P and the fp32 sums do not mind a common
                // factor.  Masked tiles, and the tile after one whose row sum came out above 2^15 (the most that 128 scores
                // within 2^8 of the reference give), do form the maximum, and raise the reference where it is more than 2^8
                // behind.
                const bool exact = need_mask || fresh || careful;
                if (exact) {
                    tc_wait_ld();
                    pin64(sr + 64);
                    if (need_mask) {
                        // Bit b of vis <=> column 32*cc + b of this tile is visible to this row (see Seen).
                        // index of this thread's query among the (local) keys; rows past the end take the last one's
                        const int i = min(w.i0 + (packed && w.packed > 1 ? row / p.G : row), w.i1);
                        const typename Tile::Seen v = t.seen(w, n, remote, i, p.window);
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc) {
                            auto below = [&](int x) -> uint32_t {  // bits below x of this 32-column chunk
                                const int d = x - 32 * cc;
                                return d <= 0 ? 0u : (d >= 32 ? 0xffffffffu : (1u << d) - 1u);
                            };
                            const uint32_t vis = (below(v.dc + 1) & (~below(v.wl) | below(v.sk))) | (below(v.s1) & ~below(v.s0));
#pragma unroll
                            for (int b = 0; b < 32; ++b)
                                sr[cc * 32 + b] = ((vis >> b) & 1u) ? sr[cc * 32 + b] : 0xff800000u;  // -inf
                        }
                    }
                    float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
                    for (int c = 0; c < BN; c += 8) {
                        mx0 = fmax3(mx0, __uint_as_float(sr[c + 0]), __uint_as_float(sr[c + 1]));
                        mx1 = fmax3(mx1, __uint_as_float(sr[c + 2]), __uint_as_float(sr[c + 3]));
                        mx2 = fmax3(mx2, __uint_as_float(sr[c + 4]), __uint_as_float(sr[c + 5]));
                        mx3 = fmax3(mx3, __uint_as_float(sr[c + 6]), __uint_as_float(sr[c + 7]));
                    }
                    const float rmax = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3));
                    // a row whose sum has run far ahead of its reference takes the sum as the reference
                    const float lead = l_sum > kLeadLimit ? __fdividef(__log2f(l_sum), p.sl2) : 0.f;
                    const float m_new = fmaxf(m_used + lead, rmax);
                    const bool need = (m_used != -INFINITY) && ((m_new - m_used) * p.sl2 > kRescaleThreshold);
                    if (__any_sync(0xffffffffu, row_ok && need)) {
                        // raise the reference maximum of every row of this warp and rescale O accordingly; PV of the
                        // side's previous tile has completed: it was issued before the QK whose S-full barrier this warp
                        // passed
                        const float alpha = (m_used == -INFINITY) ? 1.f : ex2f((m_used - m_new) * p.sl2);
#pragma unroll
                        for (int cc = 0; cc < (kLseOnly ? 0 : D / 32); ++cc) {
                            uint32_t orr[32];
                            tmem_ld32(tO + cc * 32, orr);
                            tc_wait_ld();
#pragma unroll
                            for (int c = 0; c < 32; ++c) orr[c] = __float_as_uint(__uint_as_float(orr[c]) * alpha);
                            tmem_st32(tO + cc * 32, orr);
                        }
                        if (!kLseOnly) tc_wait_st();
                        l_sum *= alpha;
                        m_used = m_new;
                    } else if (m_used == -INFINITY) {
                        m_used = m_new;  // nothing accumulated yet for this row
                    }
                    fresh = __any_sync(0xffffffffu, row_ok && m_used == -INFINITY);
                }
                // P = 2^(s * sl2 - off) into tensor memory as bf16 pairs, and into the row sum
                const float off = m_used == -INFINITY ? 0.f : m_used * p.sl2;
                const uint64_t sl2x2 = pack_f32x2(p.sl2, p.sl2), noffx2 = pack_f32x2(-off, -off);
                uint64_t psum_a = pack_f32x2(0.f, 0.f), psum_b = pack_f32x2(0.f, 0.f);
                float hi = -INFINITY;  // largest argument of the polynomial path
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    if (cc == 2) {
                        tc_wait_ld();
                        pin64(sr + 64);
                    }
                    uint32_t pk[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        const uint64_t x = fma_f32x2(
                            pack_f32x2(__uint_as_float(sr[cc * 32 + 2 * c]), __uint_as_float(sr[cc * 32 + 2 * c + 1])),
                            sl2x2, noffx2);
                        float x0, x1;
                        unpack_f32x2(x, x0, x1);
                        float p0, p1;
                        if ((kPolyPairMask >> c) & 1u) {
                            hi = fmax3(hi, x0, x1);
                            exp2_poly_x2(x0, x1, p0, p1);  // FMA pipe: takes load off the special-function unit
                        } else {
                            p0 = ex2f(x0);
                            p1 = ex2f(x1);
                        }
                        if (c & 1) psum_b = add_f32x2(psum_b, pack_f32x2(p0, p1));
                        else psum_a = add_f32x2(psum_a, pack_f32x2(p0, p1));
                        if (!kLseOnly) pk[c] = pack_bf16x2(p0, p1);
                    }
                    if (!kLseOnly) tmem_st16(tS + (uint32_t)cc * 16u, pk);
                }
                float sum;
                {
                    float a0, a1;
                    unpack_f32x2(add_f32x2(psum_a, psum_b), a0, a1);
                    sum = a0 + a1;
                }
                l_sum += sum;
                if (!exact && __any_sync(0xffffffffu, row_ok && !(sum <= kGrowLimit && hi <= 15.f))) {
                    // Growth shows in the row sum, except in the columns of the polynomial path: those are bounded by their
                    // largest argument.  Far out of range (2^110, also: not a number) the whole item is run again, forming every
                    // tile's maximum, which takes as long again.  Up to there P and its sums are as precise as ever, and whether
                    // O stayed finite, which depends on the values too, is looked at when the item is done.  Scores of standard
                    // deviation 1, 4, 8, 16, 30 and 60 nats (32k prompt, window 2048): 925, 980, 1180, 1204, 1375 and 2300 us.
                    fresh = true;
                    phases |= kGrown;
                    if (__any_sync(0xffffffffu, row_ok && !(sum <= kSumLimit && hi <= kArgLimit))) s_again[it & 1] = 1;  // all lanes the same
                }
                if (!kLseOnly) tc_wait_st();
                tc_fence_before();
                arrive_warp(BAR_PR + side);
            }
            if (!ok) break;
            // ---- epilogue of this item: O / l -> bf16 -> global
            if (!kLseOnly) {
                ok = warp_wait(bar(BAR_OD + side), (phases & kPhO) != 0 ? 1u : 0u, abort_flag);
                if (!ok) break;
                phases ^= kPhO;
                tc_fence_after();
                if ((phases & kGrown) != 0) {  // an accumulator that left the range of fp32: the item is run again
                    phases &= ~kGrown;
                    uint32_t top = 0;  // largest magnitude (bits) of the row; no branch in which lanes could differ
#pragma unroll 1
                    for (int cc = 0; cc < D / 32; ++cc) {
                        uint32_t o[32];
                        __syncwarp();
                        tmem_ld32(tO + (uint32_t)(cc * 32), o);
                        tc_wait_ld();
#pragma unroll
                        for (int e = 0; e < 32; ++e) {
                            asm volatile("" : "+r"(o[e]));  // behind the wait
                            top = max(top, o[e] & 0x7fffffffu);
                        }
                    }
                    if (__any_sync(0xffffffffu, row_ok && top >= 0x7f800000u)) s_again[it & 1] = 1;
                    __syncwarp();
                }
            }
            const int q_off = packed && w.packed > 1 ? row / p.G : row;
            const int q_row = w.q0 + q_off;  // this thread's query, counted inside the sequence
            const int token = w.seq_start + q_row, tok0 = w.seq_start + w.q0;
            const int h = w.hA + (packed ? (w.packed > 1 ? row - q_off * p.G : 0) : side);
            const bool sideB = shared || uniform(w.hasB) != 0;
            release_work(it);
            __nv_bfloat16* orow = p.out + ((size_t)token * p.Hq + h) * D;
            // eight channels of this thread's row
            auto pack8 = [](const uint32_t* o, float inv) {
                return make_uint4(pack_bf16x2(__uint_as_float(o[0]) * inv, __uint_as_float(o[1]) * inv),
                                  pack_bf16x2(__uint_as_float(o[2]) * inv, __uint_as_float(o[3]) * inv),
                                  pack_bf16x2(__uint_as_float(o[4]) * inv, __uint_as_float(o[5]) * inv),
                                  pack_bf16x2(__uint_as_float(o[6]) * inv, __uint_as_float(o[7]) * inv));
            };
            auto o_free = [&]() {  // O may be overwritten by the next item's first P V
                tc_fence_before();
                arrive_warp(BAR_OF + side);
            };
            const uint32_t od_b = (phases & kPhOB) != 0 ? 1u : 0u;  // side A: parity of side B's O done in this item
            if (sideB) phases ^= kPhOB;
            if (idle) {
                if (!kLseOnly && !(shared && side == 1)) {
                    o_free();
                    if (shared && lane == 0) mbar_arrive(bar(BAR_OF + 1));
                }
                continue;
            }
            if (shared) {
                if (side == 1) {
                    // Side A's warp of the same rows reads both accumulators; it only lacks (max, sum).  (O done above implies
                    // that the previous hand-over has been read.)
                    s_merge[row] = make_float2(m_used, l_sum);
                    arrive_warp(BAR_MG + wq);
                    continue;
                }
                ok = warp_wait(bar(BAR_OD + 1), od_b, abort_flag) &&
                     warp_wait(bar(BAR_MG + wq), (phases & kPhM) != 0 ? 1u : 0u, abort_flag);
                if (!ok) break;
                phases ^= kPhM;
                tc_fence_after();
                const float2 other = s_merge[row];
                const float M = fmaxf(m_used, other.x);
                const float wa = m_used == -INFINITY ? 0.f : ex2f((m_used - M) * p.sl2);
                const float wb = other.x == -INFINITY ? 0.f : ex2f((other.x - M) * p.sl2);
                l_sum = wa * l_sum + wb * other.y;
                m_used = M;
                const float inv = l_sum > 0.f ? 1.f / l_sum : 0.f;
#pragma unroll 1
                for (int cc = 0; cc < D / 32; ++cc) {
                    uint32_t o[32], ob[32];
                    __syncwarp();  // behind the stores of rows that exist
                    tmem_ld32(tO + (uint32_t)(cc * 32), o);
                    tmem_ld32(tO + (uint32_t)(D + cc * 32), ob);
                    tc_wait_ld();
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        // a side without any visible key of the row has no usable O
                        const float x = wa > 0.f ? __uint_as_float(o[e]) * wa : 0.f;
                        const float y = wb > 0.f ? __uint_as_float(ob[e]) * wb : 0.f;
                        o[e] = __float_as_uint(x + y);
                    }
                    if (row_ok)
#pragma unroll
                        for (int v = 0; v < 4; ++v) *reinterpret_cast<uint4*>(orow + cc * 32 + v * 8) = pack8(o + v * 8, inv);
                }
                o_free();
                if (lane == 0) mbar_arrive(bar(BAR_OF + 1));
            } else if (!kLseOnly) {
                uint32_t orr[D];
#pragma unroll
                for (int cc = 0; cc < D / 32; ++cc) tmem_ld32(tO + cc * 32, orr + cc * 32);
                tc_wait_ld();
                o_free();
                const float inv = l_sum > 0.f ? 1.f / l_sum : 0.f;
                if (!packed && wq * 32 + 31 < n_rows) {
                    // all 32 rows of this warp are valid: stage [32 rows][64 ch] panels in shared memory in the
                    // 128-byte-swizzled layout and let TMA write them (fully coalesced, off the LSU path)
                    const uint32_t stage = sStage + (uint32_t)warp * 4096u;
#pragma unroll
                    for (int pn = 0; pn < D / 64; ++pn) {
                        if (lane == 0) tma_store_wait_read();  // the previous store has finished reading the stage
                        __syncwarp();
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const uint4 v = pack8(orr + pn * 64 + j * 8, inv);
                            st_shared_v4(stage + (uint32_t)lane * 128u + (uint32_t)((j ^ (lane & 7)) * 16), v.x, v.y, v.z, v.w);
                        }
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            tma_store_3d(&tm.out, stage, pn * 64, h, tok0 + wq * 32);
                            tma_store_commit();
                        }
                    }
                } else if (row_ok) {
                    // packed rows, or the ragged tail of a sequence: plain predicated row stores
#pragma unroll
                    for (int v = 0; v < D / 8; ++v) *reinterpret_cast<uint4*>(orow + v * 8) = pack8(orr + v * 8, inv);
                }
            }
            if (row_ok && p.lse != nullptr) {
                const float lse2 = (m_used == -INFINITY) ? -INFINITY : m_used * p.sl2 + log2f(l_sum);
                p.lse[(size_t)h * p.T + token] = lse2 * 0.6931471805599453f;
            }
        }
        if (lane == 0) tma_store_wait_read();  // outstanding output stores of this warp have read their staging
    }

    // ---- teardown: every thread arrives here (also after a failed wait); free the tensor memory
    tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

}  // namespace swaa
