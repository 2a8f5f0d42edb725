// Attention of generated tokens in a batch with prompt chunks (chunked and paged prefill, Fig. 1a): sequences with at most
// kTokenRows rows, rows = (query, head of the group).  An item is one kv head of such a sequence; K and V are read once.
//
// Eight warps take the item's key tiles in turn, four per tile with 32 keys each, on warp-level MMAs with the rows in N as the
// decode kernel does; one warp hands out the items and keeps a ring of copies full.  Key lists are cut into parts for
// several SMs where the call brings a workspace; the last part of a row to end merges them.
//
// What bounds it: memory, as soon as enough SMs are at work.  An SM takes 1100 cycles for a tile of 128 keys (64 KiB at D = 128) where
// the copies alone take 790.  As packed items of the prefill kernel, where a tile costs as much as one of 128 rows (2300 cycles,
// tcgen05 products and the waits of one issuing warp) and an SM walked a whole context: 24 generated tokens at 1k to 32k
// keys in pages 306 us, 153 this way (0.99 of the copy rate); one at 32k keys 297 and 38; a serving step of the 24 with 4 prompt chunks
// 485 and 432.  Called without a workspace, whole lists on one SM: the step 482, 405 with one (both replayed from a CUDA graph).
//
// The kernel is launched behind the prefill kernel of the same call, whose blocks let it in as soon as all of them have
// started (they have then seen the end of what comes before the call), so it fills the SMs that run out of prompt items; it
// neither reads nor writes what that kernel writes, and its blocks end only when that kernel has.
//
// Precision: fp32 scores, sums and partial results and bf16 P, as in the prefill kernel, but every exponential on the special-function
// unit and P against each warp's own running maximum.  Against float64 over 18 mixed steps (1 to 8 heads per group, head sizes 64 and
// 128, contexts 64 to 32768) 1.97e-3 to 2.13e-3 in the 2-norm, as packed items 2.07e-3 to 2.46e-3.
//
// Every wait is bounded, as in the prefill kernel.
#pragma once

#include <type_traits>

#include "swaa_prefill.cuh"

namespace swaa {

constexpr int kTokenThreads = 288;
constexpr int kTokenRows = 8;
constexpr int kTokenPackedTiles = 10;  // a few lists of up to this many key tiles stay with the prefill kernel (see the launch)
constexpr int kSplitMinTiles = 8;   // key tiles of a part, at least
constexpr int kSplitMaxParts = 32;  // parts of an item (one lane each when they are merged)

// What the warps have to know of an item.  Written to shared memory by the warp that hands out the items.
struct TokenItem {
    WorkItem w;   // key list and rows
    int valid;
    int t0, t1;   // tiles of this part
    int parts;    // parts of the item (1: not cut)
    int slot, first_slot;  // of this part, and of the item's first one (slots hold the rows of parts: see merge_parts)
};
constexpr int kTokenInts = sizeof(TokenItem) / 4;

template <int D>
struct TokenSmem {
    static constexpr int kTileBytes = 128 * D * 2;  // 128 keys of K or V, in panels of [128][64 ch]
    static constexpr int kPanelBytes = 128 * 128;
    static constexpr int kPanels = D / 64;
    static constexpr int kSlots = 6 * 128 / D;                       // a half for each group of four warps
    static constexpr int kOffPart = kSlots * kTileBytes;             // partial O of the warps, [8][kTokenRows][D]
    static constexpr int kOffMl = kOffPart + 8 * kTokenRows * D * 4;  // their (max, sum)
    static constexpr int kOffBar = kOffMl + 8 * kTokenRows * 8;
    // slot full, slot empty; partial results written, read; descriptor full, empty (two each); next-block answer
    static constexpr int kBarF = 0, kBarE = kSlots, kBarW = 2 * kSlots, kBarR = kBarW + 1, kBarWF = kBarR + 1, kBarWE = kBarWF + 2, kBarNB = kBarWE + 2;
    static constexpr int kOffAnswer = (kOffBar + (kBarNB + 1) * 8 + 15) / 16 * 16;
    static constexpr int kOffWork = kOffAnswer + 32;  // behind the answer: abort flag
    static constexpr int kBytes = kOffWork + 2 * kTokenInts * 4;
    static constexpr int kDynamicBytes = kBytes + 1024;  // room to align the base to 1024 B
    static_assert(kDynamicBytes <= 232448, "shared memory per block");
};

// Counts the parts of an item's row that are done; true for the last one.  The word holds (stamp of the call << 16 | arrivals): one
// whose stamp is not this call's is left over and starts again, so nothing has to be cleared before a call, and the last
// arrival clears it, because a call that a CUDA graph replays comes with the same stamp again.
__device__ __forceinline__ bool split_arrive(unsigned long long* t, unsigned long long stamp, int parts) {
    unsigned long long seen = *reinterpret_cast<volatile unsigned long long*>(t), now = 0;
    while ((seen >> 16) != stamp) {
        const unsigned long long prev = atomicCAS(t, seen, (stamp << 16) | 1ull);
        if (prev == seen) {
            now = (stamp << 16) | 1ull;
            break;
        }
        seen = prev;
    }
    if (now == 0) now = atomicAdd(t, 1ull) + 1ull;
    const bool last = (int)(now & 0xffffull) == parts;
    if (last) *reinterpret_cast<volatile unsigned long long*>(t) = 0ull;
    return last;
}

// Merges the parts of a row (at stride kTokenRows): lane = part for (max, sum), then lane = D / 32 channels, sixteen parts in
// flight.  (Loads past the last part are repeated and not used: conditional loads into an array cost 44 registers, which spilled.)
template <int D>
struct RowResult {
    float m, l, o[D / 32];
};
template <int D>
__device__ __forceinline__ RowResult<D> merge_parts(const float2* part_ml, const float* part_o, int parts, float sl2) {
    constexpr int kCh = D / 32, kBatch = 16;
    using Vec = typename std::conditional<kCh == 4, float4, float2>::type;
    const int lane = threadIdx.x & 31;
    RowResult<D> r;
    float2 ml = __ldcg(part_ml + min(lane, parts - 1) * kTokenRows);
    if (lane >= parts) ml = make_float2(-INFINITY, 0.f);
    float wgt = 0.f;
#pragma unroll
    for (int e = 0; e < kCh; ++e) r.o[e] = 0.f;
#pragma unroll 1
    for (int j = 0; j < parts; j += kBatch) {
        Vec u[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i)
            u[i] = __ldcg(reinterpret_cast<const Vec*>(part_o + (size_t)min(j + i, parts - 1) * kTokenRows * D) + lane);
        if (j == 0) {
            r.m = ml.x;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) r.m = fmaxf(r.m, __shfl_xor_sync(0xffffffffu, r.m, o));
            wgt = ml.x == -INFINITY ? 0.f : ex2f((ml.x - r.m) * sl2);
            r.l = wgt * ml.y;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) r.l += __shfl_xor_sync(0xffffffffu, r.l, o);
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            const float wi = __shfl_sync(0xffffffffu, wgt, (j + i) & 31);
            if (j + i < parts) {
                const float* y = reinterpret_cast<const float*>(&u[i]);
#pragma unroll
                for (int e = 0; e < kCh; ++e) r.o[e] = fmaf(wi, y[e], r.o[e]);
            }
        }
    }
    return r;
}

template <int D, bool kPaged>
__global__ void __launch_bounds__(kTokenThreads, 1)
token_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
             const __grid_constant__ CUtensorMap tm_ks, const __grid_constant__ CUtensorMap tm_vs, const PrefillParams p) {
    using L = TokenSmem<D>;
    using Tile = TileGeom<kPrefillBN>;
    constexpr int BN = kPrefillBN, kHalf = L::kSlots / 2;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    auto bar = [&](int i) -> uint32_t { return smem_base + (uint32_t)L::kOffBar + 8u * (uint32_t)i; };
    const uint32_t s_answer = smem_base + L::kOffAnswer;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_gen + L::kOffAnswer + 16);
    volatile TokenItem* items = reinterpret_cast<volatile TokenItem*>(smem_gen + L::kOffWork);
    auto uniform = [](int x) -> int { return __shfl_sync(0xffffffffu, x, 0); };
    const int warp = uniform((int)(threadIdx.x >> 5)), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        for (int i = 0; i <= L::kBarNB; ++i) {
            uint32_t count = 1u;
            if (i >= L::kBarE && i < L::kBarW) count = 4u;                                                      // of the warps that share a tile
            if (i == L::kBarW || i == L::kBarR || i == L::kBarWE || i == L::kBarWE + 1) count = 8u;  // a lane of each warp
            mbar_init(bar(i), count);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // Not grid_wait: this kernel starts when the blocks of the prefill kernel before it are all past theirs.  Without such a
    // kernel (token_len < 0) it is like any other.
    if (p.token_len < 0) grid_wait();

    if (warp == 8) {
        // ===================================================================== items and copies
        // Items: parts of a sequence next to one another, the same keys of all heads first; sequences 32 at a time, lane l
        // looks after sequence base_b - l.  The grid is an upper bound: a block takes over the indices of others that have not started.
        const bool el = elect_one();
        int base_b = p.B - 1, base_w = 0, base_slot = 0;
        int f_s = 0, f_len = 0, f_ks = 0, f_off = 0, f_full = p.is_full != 0 ? 1 : 0;  // of the lane's sequence
        int f_tiles = 0, f_parts = 0, f_items = 0, f_before = 0, f_slot = 0, group_items = 0, group_slots = 0;
        int part_tiles = 1 << 30;
        auto describe = [&](WorkItem& d, int hk) {
            d.seq_start = f_s;
            d.seq_len = f_len;
            d.q0 = 0;
            d.packed = 1;
            d.full = f_full;
            d.k_start = f_ks;
            d.k_off = f_off;
            d.n_sink = p.n_sink;
            d.s_rem = 0;
            d.complete<BN, kPaged, false, false>(p, hk);
        };
        auto load_group = [&]() {
            const int b = base_b - lane;
            f_tiles = 0;
            if (b >= 0) {
                const int s0 = p.cu_seqlens[b], e0 = p.cu_seqlens[b + 1];
                const int k0 = kPaged ? 0 : p.cu_seqlens_k[b], k1 = kPaged ? p.cu_seqlens_k[b] : p.cu_seqlens_k[b + 1];
                if (p.is_full_seq != nullptr) f_full = p.is_full_seq[b] != 0 ? 1 : 0;
                f_s = s0;
                f_len = e0 - s0;
                f_ks = kPaged ? b : k0;
                f_off = k1 - k0 - f_len;
                const bool bad = f_len < 0 || f_len > p.max_seqlen || s0 < 0 || e0 > p.T || k1 - k0 < f_len || k1 - k0 > p.max_seqlen_k ||
                                 (!kPaged && (k0 < 0 || k1 > p.Tk));
                if (bad) record_device_error(SWAA_ERR_BAD_SEQLENS);
                if (!bad && f_len > 0 && f_len * p.G <= kTokenRows) {
                    WorkItem d;
                    describe(d, 0);
                    f_tiles = d.nt;
                }
            }
        };
        auto plan_group = [&]() {
            f_parts = min(kSplitMaxParts, (f_tiles + part_tiles - 1) / part_tiles);
            f_items = f_parts * p.Hkv;
            const int slots = f_parts > 1 ? f_items : 0;
            f_before = f_slot = 0;
            for (int j = 0; j < min(32, p.B); ++j) {
                const int ij = __shfl_sync(0xffffffffu, f_items, j), sj = __shfl_sync(0xffffffffu, slots, j);
                if (j < lane) {
                    f_before += ij;
                    f_slot += sj;
                }
            }
            group_items = __reduce_add_sync(0xffffffffu, f_items);
            group_slots = __reduce_add_sync(0xffffffffu, slots);
        };
        load_group();
        if (p.split_tickets != nullptr) {
            // The key tiles of all items are cut into one to four parts per SM of at least kSplitMinTiles tiles.  (The launch allows
            // for four parts per SM more than there are items, and twice as many slots.)
            long long total = 0;
            while (true) {
                total += (long long)__reduce_add_sync(0xffffffffu, min(f_tiles, 1 << 24)) * p.Hkv;
                if (base_b < 32) break;
                base_b -= 32;
                load_group();
            }
            const long long waves = min(4ll, max(1ll, total / ((long long)kSplitMinTiles * p.sms)));
            part_tiles = (int)min(max((long long)kSplitMinTiles, (total + waves * p.sms - 1) / (waves * p.sms)), 1ll << 30);
            if (p.B > 32) {
                base_b = p.B - 1;
                load_group();
            }
        }
        plan_group();

        int next[2] = {0, 0};   // next slot of each half of the ring
        uint32_t phases = 0;    // bit: parity of the slot's next use
        uint32_t nb_phase = 0;
        bool asked = false;     // for the next index, and the answer has not been seen
        int w = (int)blockIdx.x, it = 0;
        bool ok = true;
        // page of a key, out of range (the copy delivers zeros) when the table is wrong
        auto page_of = [&](int seq, int key) -> int {
            const int page = p.block_table[(size_t)seq * p.max_blocks + key / p.page_size];
            if (page >= 0 && page < p.num_pages) return page;
            record_device_error(SWAA_ERR_BAD_SEQLENS);
            return p.num_pages;
        };
        while (w >= 0 && ok) {
            // the index of the next item is asked for ahead of this one's copies
            __syncwarp();
            if (lane == 0) {
                fence_proxy_async_smem();  // the previous answer has been read
                mbar_arrive_expect_tx(bar(L::kBarNB), 16u);
                next_block_request(s_answer, bar(L::kBarNB));
            }
            __syncwarp();
            asked = true;
            if (w < base_w) {  // an index before this group of sequences: start over
                base_b = p.B - 1;
                base_w = base_slot = 0;
                load_group();
                plan_group();
            }
            while (w >= base_w + group_items && base_b >= 32) {
                base_w += group_items;
                base_slot += group_slots;
                base_b -= 32;
                load_group();
                plan_group();
            }
            if (w < base_w + group_items) {  // (an index past the last item is passed over)
                ok = warp_wait(bar(L::kBarWE + (it & 1)), ((uint32_t)(it >> 1) & 1u) ^ 1u, abort_flag);
                if (!ok) break;
                const int local = w - base_w - f_before;
                if (local >= 0 && local < f_items) {  // one lane
                    TokenItem d;
                    const int hk = local % p.Hkv, part = local / p.Hkv;
                    describe(d.w, hk);
                    d.valid = 1;
                    d.t0 = (int)((long long)d.w.nt * part / f_parts);
                    d.t1 = (int)((long long)d.w.nt * (part + 1) / f_parts);
                    d.parts = f_parts;
                    d.first_slot = base_slot + f_slot + hk * f_parts;
                    d.slot = d.first_slot + part;
                    volatile int* to = reinterpret_cast<volatile int*>(items + (it & 1));
                    const int* from = reinterpret_cast<const int*>(&d);
#pragma unroll
                    for (int i = 0; i < kTokenInts; ++i) to[i] = from[i];
                    mbar_arrive(bar(L::kBarWF + (it & 1)));
                }
                __syncwarp();
                // ---- copies: K(0) V(0) K(1) V(1) ..., tiles to the two groups of warps in turn
                const volatile TokenItem& t = items[it & 1];
                const int t0 = t.t0, nt = t.t1 - t0, lo = t.w.lo, nb16 = t.w.nb16, hk = t.w.hk, k_start = t.w.k_start;
                int pages = 0;  // lane l: page of tile l of 32
                for (int n = 0; n < nt && ok; ++n) {
                    const int half = n & 1, key = lo + (t0 + n) * BN;
                    if (kPaged && (n & 31) == 0) {
                        if (key - lo + lane * BN < nb16 && n + lane < nt) pages = page_of(k_start, key + lane * BN);
                        __syncwarp();
                    }
                    const int page = kPaged ? __shfl_sync(0xffffffffu, pages, n & 31) : 0;
                    const int row = kPaged ? key % p.page_size : k_start + key;
                    const bool whole = key - lo + BN <= nb16 || !Tile(t.w, t0 + n).joins_sinks();  // one box per panel
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        const int slot = half * kHalf + next[half];
                        next[half] = next[half] + 1 == kHalf ? 0 : next[half] + 1;
                        ok = ok && warp_wait(bar(L::kBarE + slot), ((phases >> slot) & 1u) ^ 1u, abort_flag);
                        if (!ok) break;
                        if (el) {
                            const uint32_t full_bar = bar(L::kBarF + slot), dst = smem_base + (uint32_t)(slot * L::kTileBytes);
                            if (whole) {
                                const CUtensorMap* map = v ? &tm_v : &tm_k;
                                mbar_arrive_expect_tx(full_bar, (uint32_t)L::kTileBytes);
#pragma unroll
                                for (int pn = 0; pn < L::kPanels; ++pn) {
                                    if (kPaged) tma_load_4d(dst + pn * L::kPanelBytes, map, pn * 64, hk, row, page, full_bar);
                                    else tma_load_3d(dst + pn * L::kPanelBytes, map, pn * 64, hk, row, full_bar);
                                }
                            } else {  // joins sink keys: pieces of 16 keys
                                const CUtensorMap* map = v ? &tm_vs : &tm_ks;
                                const Tile g(t.w, t0 + n);
                                mbar_arrive_expect_tx(full_bar, (uint32_t)(g.nk * 16 * 128 * L::kPanels));
                                for (int x = 0; x < g.nk; ++x) {
                                    const int k16 = g.key(16 * x), pg = kPaged ? page_of(k_start, k16) : 0;
#pragma unroll
                                    for (int pn = 0; pn < L::kPanels; ++pn) {
                                        const uint32_t d = dst + (uint32_t)(pn * L::kPanelBytes + x * 2048);
                                        if (kPaged) tma_load_4d(d, map, pn * 64, hk, k16 % p.page_size, pg, full_bar);
                                        else tma_load_3d(d, map, pn * 64, hk, k_start + k16, full_bar);
                                    }
                                }
                            }
                        }
                        __syncwarp();
                        phases ^= 1u << slot;
                    }
                }
                if (!ok) break;
                ++it;
            }
            ok = warp_wait(bar(L::kBarNB), nb_phase, abort_flag);
            if (!ok) break;
            asked = false;
            nb_phase ^= 1u;
            w = uniform(next_block_answer(s_answer));
        }
        if (lane == 0 && (p.cu_seqlens[0] != 0 || p.cu_seqlens[p.B] != p.T)) record_device_error(SWAA_ERR_BAD_SEQLENS);
        ok = ok && warp_wait(bar(L::kBarWE + (it & 1)), ((uint32_t)(it >> 1) & 1u) ^ 1u, abort_flag);
        if (ok && lane == 0) {
            items[it & 1].valid = 0;
            mbar_arrive(bar(L::kBarWF + (it & 1)));
        }
        if (!ok) {
            // give outstanding copies, and the answer to the last request, a bounded chance to land before the block's memory is released
            const uint64_t start = global_timer_ns();
            bool done = false;
            while (!done && global_timer_ns() - start < kWaitLimitNs) {
                done = !asked || mbar_try_wait(bar(L::kBarNB), nb_phase);
                for (int slot = 0; slot < L::kSlots; ++slot) done = done && mbar_try_wait(bar(L::kBarF + slot), ((phases >> slot) & 1u) ^ 1u);
            }
        }
        __syncwarp();
    } else {
        // ============================================================================== products
        const int side = warp >> 2, wq = warp & 3;
        int t_slot = side * kHalf;  // next slot of this group's half of the ring
        uint32_t t_phases = 0;      // bit: parity of the slot's next use
        auto arrive = [&](int b) {
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(b));
        };
        // an item; false when a wait has run out
        auto item = [&](const volatile TokenItem& ti, uint32_t t_items) -> bool {
            WorkItem w;  // in registers
            w.full = uniform(ti.w.full);
            w.i0 = uniform(ti.w.i0);
            w.i1 = uniform(ti.w.i1);
            w.lo = uniform(ti.w.lo);
            w.nb16 = uniform(ti.w.nb16);
            w.nv = uniform(ti.w.nv);
            w.n_sink = uniform(ti.w.n_sink);
            w.n_rem = w.s_rem = 0;
            constexpr int NKK = D / 16, kCh = D / 32;
            using Vec = typename std::conditional<kCh == 4, float4, float2>::type;
            const int n_rows = uniform(ti.w.n_rows), G = uniform(ti.w.packed), t0 = uniform(ti.t0), t1 = uniform(ti.t1);
            const int tok = uniform(ti.w.seq_start), hA = uniform(ti.w.hA);
            const int g = lane >> 2, c = lane & 3;
            const int key0 = 32 * wq;  // first of the warp's keys in a tile
            const int krow = key0 + (lane & 15), kchk = lane >> 4;                              // ldmatrix rows: see decode_kernel
            const int vrow = key0 + (lane & 7) + 8 * (lane >> 4), vchk = (lane >> 3) & 1;
            // Q^T fragments: lane (g, c) holds channels 16kk + 2c, +1 and 16kk + 2c + 8, +9 of row g
            uint32_t qf[NKK][2];
            const uint32_t* qrow = reinterpret_cast<const uint32_t*>(p.q + ((size_t)(tok + (g < n_rows ? g / G : 0)) * p.Hq + hA + (g < n_rows ? g % G : 0)) * D);
#pragma unroll
            for (int kk = 0; kk < NKK; ++kk) {
                qf[kk][0] = g < n_rows ? qrow[kk * 8 + c] : 0u;
                qf[kk][1] = g < n_rows ? qrow[kk * 8 + c + 4] : 0u;
            }
            float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f}, oacc[NKK][4];
#pragma unroll
            for (int qb = 0; qb < NKK; ++qb) oacc[qb][0] = oacc[qb][1] = oacc[qb][2] = oacc[qb][3] = 0.f;
            // A half of the slots is this side's ring.  (Sides that shared a ring would wait for a use of a slot without having seen
            // the other side's use before it, and take that for this one's while it has not landed.)
            auto pass_slot = [&]() {
                t_phases ^= 1u << t_slot;
                t_slot = t_slot + 1 == (side + 1) * kHalf ? side * kHalf : t_slot + 1;
            };
            auto landed = [&]() -> bool { return warp_wait(bar(L::kBarF + t_slot), (t_phases >> t_slot) & 1u, abort_flag); };
            for (int n = t0 + side; n < t1; n += 2) {
                const Tile t(w, n);
                const bool need_mask = SWAA_TILE_NEEDS_MASK(t, w, n, false, p.window, BN);
                // what the first and the last row of the item see
                const typename Tile::Seen first = t.seen(w, n, false, w.i0, p.window), last = t.seen(w, n, false, w.i1, p.window);
                auto seen_by_any = [&](int col) -> bool {
                    return !need_mask || (col <= last.dc && (col >= first.wl || col < last.sk)) || (col >= last.s0 && col < last.s1);
                };
                const bool mine = !need_mask || __any_sync(0xffffffffu, seen_by_any(key0 + lane)) != 0;
                if (!landed()) return false;
                uint32_t tile = smem_base + (uint32_t)(t_slot * L::kTileBytes);
                uint32_t pb[2][2];
                if (mine) {
                    // ---- S^T = K Q^T: rows = keys (g, g + 8) of two groups of 16, columns = rows of the item (2c, 2c + 1)
                    float sa[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
                    for (int kk = 0; kk < NKK; ++kk) {
                        const int chunk = 2 * kk + kchk;
                        const uint32_t at = tile + (uint32_t)((chunk >> 3) * L::kPanelBytes + krow * 128 + (((chunk & 7) ^ (krow & 7)) << 4));
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t a0, a1, a2, a3;
                            ldmatrix_x4(at + (uint32_t)(h * 2048), a0, a1, a2, a3);
                            mma_bf16_16816(sa[h], a0, a1, a2, a3, qf[kk][0], qf[kk][1]);
                        }
                    }
                    arrive(L::kBarE + t_slot);
                    __syncwarp();
                    float alpha[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        if (need_mask) {
                            const typename Tile::Seen v = t.seen(w, n, false, min(w.i0 + (2 * c + e) / G, w.i1), p.window);
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                const int col = key0 + g + 8 * x;
                                const bool seen = (col <= v.dc && (col >= v.wl || col < v.sk)) || (col >= v.s0 && col < v.s1);
                                float& s = sa[x >> 1][2 * (x & 1) + e];
                                s = seen ? s : -INFINITY;
                            }
                        }
                        float bm = fmaxf(fmaxf(sa[0][e], sa[0][2 + e]), fmaxf(sa[1][e], sa[1][2 + e]));
                        bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 4));
                        bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 8));
                        bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 16));
                        const float m_new = fmaxf(m_run[e], bm);
                        alpha[e] = m_run[e] == m_new ? 1.f : ex2f((m_run[e] - m_new) * p.sl2);
                        m_run[e] = m_new;
                        const float off = m_new == -INFINITY ? 0.f : m_new * p.sl2;  // a row that none of the warp's keys reaches yet
                        float sum = 0.f;
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            float& s = sa[x >> 1][2 * (x & 1) + e];
                            s = ex2f(fmaf(s, p.sl2, -off));
                            sum += s;
                        }
                        l_run[e] = l_run[e] * alpha[e] + sum;
                    }
                    if (__any_sync(0xffffffffu, alpha[0] != 1.f || alpha[1] != 1.f)) {
#pragma unroll
                        for (int qb = 0; qb < NKK; ++qb) {
                            oacc[qb][0] *= alpha[0];
                            oacc[qb][1] *= alpha[1];
                            oacc[qb][2] *= alpha[0];
                            oacc[qb][3] *= alpha[1];
                        }
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        pb[h][0] = movmatrix_trans(pack_bf16x2(sa[h][0], sa[h][1]));
                        pb[h][1] = movmatrix_trans(pack_bf16x2(sa[h][2], sa[h][3]));
                    }
                } else {
                    arrive(L::kBarE + t_slot);
                    __syncwarp();
                }
                pass_slot();
                if (!landed()) return false;
                if (mine) {
                    // ---- O^T += V^T P^T: rows = channels (16qb + g, + 8), columns = rows of the item.  Rows of V that no row of the
                    // item sees may hold anything (also NaN), or were not fetched: they are cleared.
                    tile = smem_base + (uint32_t)(t_slot * L::kTileBytes);
                    uint32_t mask[2][2] = {{0xffffffffu, 0xffffffffu}, {0xffffffffu, 0xffffffffu}};
                    if (need_mask)
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int col = key0 + 2 * c + 8 * x;
                            mask[x >> 1][x & 1] = (seen_by_any(col) ? 0x0000ffffu : 0u) | (seen_by_any(col + 1) ? 0xffff0000u : 0u);
                        }
#pragma unroll
                    for (int qb = 0; qb < NKK; ++qb) {
                        const int chunk = 2 * qb + vchk;
                        const uint32_t at = tile + (uint32_t)((chunk >> 3) * L::kPanelBytes + vrow * 128 + (((chunk & 7) ^ (vrow & 7)) << 4));
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t a0, a1, a2, a3;
                            ldmatrix_x4_trans(at + (uint32_t)(h * 2048), a0, a1, a2, a3);
                            mma_bf16_16816(oacc[qb], a0 & mask[h][0], a1 & mask[h][0], a2 & mask[h][1], a3 & mask[h][1], pb[h][0], pb[h][1]);
                        }
                    }
                }
                arrive(L::kBarE + t_slot);
                __syncwarp();
                pass_slot();
            }
            // ---- the warps' partial results meet in shared memory: row r of warp i at (8 i + r) D, channels rotated by 8 per pair of
            // rows (no bank conflicts); warp r then takes row r
            if (__any_sync(0xffffffffu, m_run[0] == -INFINITY || m_run[1] == -INFINITY)) {
                // A row that sees none of the warp's keys: 0 times the values of keys that other rows see, which may not be numbers.
#pragma unroll
                for (int qb = 0; qb < NKK; ++qb)
#pragma unroll
                    for (int e = 0; e < 4; ++e) oacc[qb][e] = m_run[e & 1] == -INFINITY ? 0.f : oacc[qb][e];
            }
            if (!warp_wait(bar(L::kBarR), t_items ^ 1u, abort_flag)) return false;  // of the item before have been read
            float* part_o = reinterpret_cast<float*>(smem_gen + L::kOffPart);
            float2* part_ml = reinterpret_cast<float2*>(smem_gen + L::kOffMl);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float l = l_run[e];
                l += __shfl_xor_sync(0xffffffffu, l, 4);
                l += __shfl_xor_sync(0xffffffffu, l, 8);
                l += __shfl_xor_sync(0xffffffffu, l, 16);
                const int r = 2 * c + e;
                if (g == 0) part_ml[8 * warp + r] = make_float2(m_run[e], l);
                float* row_o = part_o + (8 * warp + r) * D;
#pragma unroll
                for (int qb = 0; qb < NKK; ++qb) {
                    row_o[(16 * qb + g + 8 * c) & (D - 1)] = oacc[qb][e];
                    row_o[(16 * qb + g + 8 + 8 * c) & (D - 1)] = oacc[qb][2 + e];
                }
            }
            arrive(L::kBarW);
            if (!warp_wait(bar(L::kBarW), t_items, abort_flag)) return false;
            const int r = warp;
            float M = -INFINITY, den = 0.f, acc[kCh];
#pragma unroll
            for (int e = 0; e < kCh; ++e) acc[e] = 0.f;
            if (r < n_rows) {
#pragma unroll
                for (int i = 0; i < 8; ++i) M = fmaxf(M, part_ml[8 * i + r].x);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float2 ml = part_ml[8 * i + r];
                    const float wgt = ml.x == -INFINITY ? 0.f : ex2f((ml.x - M) * p.sl2);
                    den = fmaf(wgt, ml.y, den);
                    const Vec v = *reinterpret_cast<const Vec*>(part_o + (8 * i + r) * D + ((lane * kCh + 8 * (r >> 1)) & (D - 1)));
                    const float* x = reinterpret_cast<const float*>(&v);
#pragma unroll
                    for (int e = 0; e < kCh; ++e) acc[e] = fmaf(wgt, x[e], acc[e]);
                }
            }
            arrive(L::kBarR);
            __syncwarp();
            if (r >= n_rows) return true;
            const int parts = uniform(ti.parts);
            if (parts > 1) {
                // this part's row to its slot; the last part to arrive merges the row
                const size_t at = (size_t)ti.slot * kTokenRows + r, at0 = (size_t)ti.first_slot * kTokenRows + r;
                Vec v;
                float* x = reinterpret_cast<float*>(&v);
#pragma unroll
                for (int e = 0; e < kCh; ++e) x[e] = acc[e];
                reinterpret_cast<Vec*>(p.split_o + at * D)[lane] = v;
                if (lane == 0) p.split_ml[at] = make_float2(M, den);
                __threadfence();
                __syncwarp();
                int done = 0;
                if (lane == 0) done = split_arrive(p.split_tickets + at0, p.stamp, parts) ? 1 : 0;
                if (!uniform(done)) return true;
                __threadfence();
                const RowResult<D> row = merge_parts<D>(p.split_ml + at0, p.split_o + at0 * D, parts, p.sl2);
                M = row.m;
                den = row.l;
#pragma unroll
                for (int e = 0; e < kCh; ++e) acc[e] = row.o[e];
            }
            const float inv = den > 0.f ? 1.f / den : 0.f;
            const int t = tok + r / G, h = hA + r % G;
            uint32_t* to = reinterpret_cast<uint32_t*>(p.out + ((size_t)t * p.Hq + h) * D + lane * kCh);
#pragma unroll
            for (int e = 0; e < kCh; e += 2) to[e / 2] = pack_bf16x2(acc[e] * inv, acc[e + 1] * inv);
            if (p.lse != nullptr && lane == 0)
                p.lse[(size_t)h * p.T + t] = M == -INFINITY ? -INFINITY : (M * p.sl2 + log2f(den)) * 0.6931471805599453f;
            return true;
        };
        for (int it = 0;; ++it) {
            if (!warp_wait(bar(L::kBarWF + (it & 1)), (uint32_t)(it >> 1) & 1u, abort_flag)) break;
            if (!uniform(items[it & 1].valid)) break;
            if (!item(items[it & 1], (uint32_t)it & 1u)) break;
            arrive(L::kBarWE + (it & 1));
            __syncwarp();
        }
    }
    // what comes behind this kernel on the stream also relies on the prefill kernel before it
    if (p.token_len >= 0) grid_wait();
}

}  // namespace swaa
