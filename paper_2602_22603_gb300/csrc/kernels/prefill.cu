// Masked prefill attention on the 5th-generation tensor cores.
//
// What it computes (Algorithm 2, BuildMask; Sec. 3.3): the last n_q tokens of
// a sequence attend causally to its tokens, with the tokens of the given spans
// (closed cursors) removed from every query's view:
//   query at position p, query head h, KV head g = floor(h / G):
//     s_j = sm_scale * q_h . k_{g,j}   for visible keys j (j <= p, j in no span)
//     o_h = sum_j softmax_j(s) v_{g,j}
//
// A query tile is 128 rows: floor(128 / G) consecutive query positions times
// the G query heads of one KV head (Sec. 2.1).  One CTA owns two consecutive
// query tiles (a, b) of the same KV head, and every K/V tile it loads serves
// both, which halves the loads per tensor-core FLOP.  Keys go 128 at a time;
// tiles whose keys are all masked are never loaded (the host lists the others
// with a visibility bitmap).  Per key tile j and query tile t:
//   S_t = Q_t K_j^T           tcgen05.mma, Q and K from shared memory, S in TMEM
//   P_t = exp2(S_t - m)       softmax warpgroup t: tcgen05.ld of S, mask, bf16 P
//                             stored back over the first half of S_t
//   O_t += P_t V_j            tcgen05.mma with A = P from TMEM and V read
//                             token-major from shared memory (MN-major B)
// The MMA issuer interleaves the two tiles (PV_a(j), S_a(j+1), PV_b(j),
// S_b(j+1)), so while one warpgroup turns S into P the tensor core works for
// the other.  P_t(j) shares TMEM with S_t: S_t(j+1) is issued after PV_t(j),
// and tcgen05.mma operations of one thread execute in issue order.  The same
// order means that when S_t(j) is ready, PV_t(j-1) is complete, so a
// warpgroup may rescale O_t then without another wait.  The running maximum
// is raised lazily: a key tile's weights are taken with the current maximum
// and accepted while every row's sum of them stays at most 2^16 (so does each
// weight; 2^8 in warps with rows that are no query); only then is a maximum
// raised and O rescaled.  K and V stream through
// one ring of shared-memory slots (K_0, V_0, K_1, ...); V_j and K_{j+1} are
// released together, after the products PV_b(j) and S_b(j+1).
//
// What bounds it: the one thread that issues the MMAs (see there), then the
// softmax chain of each tile.  32,768 queries, 40% masked, 32q/8kv, d = 128:
// 3.55 -> 3.25 ms a layer (1,320 -> 1,440 TFLOP/s
// over the visible pairs); 3,001 queries over 33,001 tokens: 1,027 -> 845 us.
//
// Short query blocks: when a CTA tile's queries all fit in tile a, tile b's
// warpgroup takes the same rows over every other key tile (dual-key mode, the
// two results merged per row at the end, loads in the order the MMAs consume
// them).
//
// Work items: the host lists (CTA tile, KV head, key range) items, longest
// first, and the grid has one CTA per item, of which an SM holds one.  A CTA
// that has issued most loads of its item asks the launch hardware for the next
// CTA not started yet (clusterlaunchcontrol.try_cancel) and takes over its
// item, so the ring, the barriers' phases and tensor memory run on from item
// to item and the next item's first keys and queries load while the last one's
// softmax, PV and output finish.  One CTA per item paid a start and a drain
// each, ~5 us; dealing the items to persistent CTAs beforehand lost 4%, since
// SMs run this kernel at speeds up to 7% apart (1.78 to 1.91 us per key tile).
// A unit split in several items (too few units for the SMs, or a last round
// that would leave most SMs idle) leaves normalised partial results that a
// second kernel merges.
//
// Calls whose queries fit in one query tile (kOne: the 8-query calls of an
// auxiliary thread, every item dual-key) run an instance without the two-tile
// path.  HBM bounds them, so, when the plan was on the device before, their
// producer loads its item's first two key tiles before the dependency wait,
// while the previous launch's last CTAs finish and are merged: 8 queries over
// 131,080 tokens, 87.0 -> 85.4 us a layer (79 at the read probe's rate).  Loading early in the two-tile instance gained nothing (the
// issuing lane bounds it) and lost 1 to 2% to the code generated around it; a
// ring one slot longer (the second query tile's space), or L2 prefetches beyond
// the ring, slow the CTAs still at work by more than they save the next ones.
//
// Warp roles (320 threads): warp 0 loads (lanes 0 and 1 issue the TMA copies,
// two loads at a time), lane 0 of warp 1 issues the MMAs and warp 1 owns the
// TMEM allocation, warps 2-5
// are the softmax warpgroup of tile a and warps 6-9 that of tile b (warp w
// reads TMEM lanes 32 (w mod 4) .. +31, one row per thread).  Every wait is
// bounded; a wait that runs out sets the error word and the CTA winds down
// after its copies and MMAs in flight have completed.
#include <type_traits>

#include "launch.hpp"
#include "ptx.cuh"
#include "tc.cuh"

namespace sq {
namespace dev {
namespace {

// Items in flight between the producer and the other roles, and the warps that
// read each (MMA warp and eight softmax warps).
constexpr int kItemSlots = 4;
constexpr int kItemReaders = 9;

template <int D, bool kOne>
struct PreCfg {
    static constexpr int kThreads = 320;
    static constexpr int kColBlocks = D / 64;                  // 64-column (128-byte) blocks
    static constexpr int kBlockBytes = kPrefillRows * 128;      // one block of a 128-row tile
    static constexpr int kQBytes = kColBlocks * kBlockBytes;    // one query tile
    static constexpr int kSlotBytes = kColBlocks * kBlockBytes;  // 128 keys of K or of V
    static constexpr int kSlots = D == 128 ? 5 : 12;
    static constexpr int kOffQ = 0;
    static constexpr int kOffRing = kOffQ + (kOne ? 1 : kPrefillQTiles) * kQBytes;
    static constexpr int kOffBar = kOffRing + kSlots * kSlotBytes;
    static constexpr int kBarQ = 0;
    static constexpr int kBarFull = 1;                  // [kSlots] tile landed (V: and ready)
    static constexpr int kBarEmpty = kBarFull + kSlots; // [kSlots] slot consumed by the MMAs
    static constexpr int kBarS = kBarEmpty + kSlots;    // [2] S_t written (and PV_t before it done)
    static constexpr int kBarP = kBarS + 2;             // [2] P_t written (128 arrivals)
    static constexpr int kBarO = kBarP + 2;             // [2] last PV_t done
    static constexpr int kBarVfix = kBarO + 2;          // V of the last key tile landed
    static constexpr int kBarQFree = kBarVfix + 1;      // the item's last QK product done
    static constexpr int kBarDone = kBarQFree + 1;      // every MMA of the CTA done
    static constexpr int kBarItem = kBarDone + 1;       // [kItemSlots] item written
    static constexpr int kBarItemFree = kBarItem + kItemSlots;  // [kItemSlots] item read by all
    static constexpr int kBarClc = kBarItemFree + kItemSlots;   // answer of the launch hardware
    static constexpr int kBarX = kBarClc + 1;           // dual-key mode: tile b's half handed over
    static constexpr int kBarXFree = kBarX + 1;         // ... and read by tile a
    static constexpr int kNumBars = kBarXFree + 1;
    static constexpr int kOffItems = (kOffBar + kNumBars * 8 + 15) & ~15;  // [kItemSlots] int4
    static constexpr int kOffClc = kOffItems + kItemSlots * 16;           // 16-byte answer
    static constexpr int kOffMisc = kOffClc + 16;
    // dual-key mode: tile b's (max, normaliser) of each row, for the merge
    static constexpr int kOffXchg = (kOffMisc + 32 + 15) & ~15;
    static constexpr int kSmemBytes = kOffXchg + kPrefillRows * 8 + 1024;  // + alignment slack
    static constexpr uint32_t kTmemCols = 512;
    static constexpr uint32_t kColS = 0;    // S_t (fp32) at 128 t; P_t (bf16 pairs) over its first 64
    static constexpr uint32_t kColO = 256;  // O_t (fp32) at 256 + 128 t
    static constexpr uint32_t kIdescQK = mma_idesc_bf16(128, kPrefillKeys, false);
    static constexpr uint32_t kIdescPV = mma_idesc_bf16(128, D, true);
    static_assert(kSmemBytes <= 232448, "shared memory");
    static_assert(kOffXchg % 16 == 0 && kOffRing % 1024 == 0 && kOffBar % 8 == 0, "alignment");
    static_assert(kPrefillQTiles == 2, "two query tiles per CTA");
};

struct Smem {
    uint32_t base;  // shared address of the 1024-aligned region
    uint8_t* ptr;
    template <int D, bool kOne>
    __device__ uint32_t bar(int i) const {
        return base + PreCfg<D, kOne>::kOffBar + 8 * i;
    }
};

// A work item as the roles see it; raw.z (its key tiles) is -1 after the last.
struct Item {
    int g, pos_lo, t0, T, part;
    bool two;   // tile b holds query rows
    bool dual;  // tile b takes every other key tile of tile a's rows
};

template <bool kOne>
__device__ __forceinline__ Item make_item(const PrefillArgs& a, int4 raw) {
    Item it;
    const int qt = raw.x / a.Hkv;
    it.g = raw.x - qt * a.Hkv;
    it.pos_lo = qt * kPrefillQTiles * a.BP;
    it.t0 = raw.y;
    it.T = raw.z;
    it.part = raw.w;
    // tile b is empty when every query of the CTA tile fits in tile a
    it.two = !kOne && it.pos_lo + a.BP < a.n_q;
    it.dual = !it.two && it.T >= 2;
    return it;
}

// Asks the launch hardware for a CTA of the grid that has not started; the
// 16-byte answer lands at `dst`, completing `bar`.
__device__ __forceinline__ void clc_request(uint32_t dst, uint32_t bar) {
    asm volatile(
        "clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], "
        "[%1];" ::"r"(dst),
        "r"(bar)
        : "memory");
}

// The answer at `src`: the index of the CTA taken over, or -1.
__device__ __forceinline__ int clc_answer(uint32_t src) {
    uint32_t ok, x;
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b128 r;\n\t"
        "ld.shared.b128 r, [%2];\n\t"
        "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t"
        "mov.u32 %1, 0;\n\t"
        "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, r;\n\t}"
        : "=r"(ok), "=r"(x)
        : "r"(src)
        : "memory");
    return ok ? (int)x : -1;
}

// The reading side of the item ring: item k of the CTA is in slot k mod
// kItemSlots until every reader has freed it.
template <int D, bool kOne>
__device__ __forceinline__ bool item_wait(const Smem& sm, uint32_t k, const volatile int* abort_flag) {
    return mbar_wait(sm.bar<D, kOne>(PreCfg<D, kOne>::kBarItem + k % kItemSlots),
                     (k / kItemSlots) & 1, abort_flag);
}
template <int D, bool kOne>
__device__ __forceinline__ int4 item_read(const Smem& sm, uint32_t k) {
    return *reinterpret_cast<const int4*>(sm.ptr + PreCfg<D, kOne>::kOffItems + k % kItemSlots * 16);
}
template <int D, bool kOne>
__device__ __forceinline__ void item_free(const Smem& sm, uint32_t k) {
    mbar_arrive(sm.bar<D, kOne>(PreCfg<D, kOne>::kBarItemFree + k % kItemSlots));
}

// Bits 0 .. x of a word (x < 0: none; x >= 31: all).
__device__ __forceinline__ uint32_t low_bits_through(int x) {
    return x >= 31 ? 0xffffffffu : (x < 0 ? 0u : ((2u << x) - 1u));
}

// Order of the K and V loads of a CTA's T key tiles, load u into ring slot
// u mod kSlots.  Normally key tile by key tile: u = 2 j is K_j, u = 2 j + 1
// is V_j.  In dual-key mode (tile a takes the even key tiles, tile b the odd
// ones) the loads follow the order in which the MMA warp consumes them, so
// that no tile waits in the ring for a later one: K_0, K_1, then V_j and
// K_{j+2} in turn, and the last two V tiles.
__device__ __forceinline__ void load_of(int u, int T, bool dual, int& j, int& kv) {
    if (!dual) {
        j = u >> 1;
        kv = u & 1;
    } else if (u < 2) {
        j = u;
        kv = 0;
    } else if (u >= 2 * T - 2) {
        j = u - T;
        kv = 1;
    } else {
        j = ((u - 2) >> 1) + ((u & 1) ? 2 : 0);
        kv = (u & 1) ? 0 : 1;
    }
}

// {first key of each half, page of box 0, page of box 1} of key tile
// tb + lane % kBatch of an item (x = key0, y = page 0, z = page 1, w = key0b).
constexpr int kBatch = 16;
__device__ __forceinline__ int4 tile_record(const PrefillArgs& a, int t0, int T, int tb, int lane) {
    int4 r = make_int4(0, -1, -1, kPrefillNoKeys);
    const int jj = tb + (lane & (kBatch - 1));
    if (jj < T) {
        const size_t t = (size_t)(t0 + jj);
        r.x = __ldg(&a.tiles[t].key0);
        r.w = __ldg(&a.tiles[t].key0b);
        r.y = __ldg(&a.tile_pages[t * a.n_pieces]);
        if (a.n_pieces > 1) r.z = __ldg(&a.tile_pages[t * a.n_pieces + 1]);
    }
    return r;
}

// A CTA's own item and its first batch of records, in the producer's lanes.
struct FirstItem {
    int4 raw, rec;
    __device__ void read(const PrefillArgs& a, int lane) {
        raw = __ldg(reinterpret_cast<const int4*>(a.items) + blockIdx.x);
        rec = tile_record(a, raw.y, raw.z, 0, lane);
    }
};

// K_0 and K_1 of a CTA's own dual-key item, before the grid-dependency wait:
// unless a page of theirs may still be being written, or one has rows past the
// sequence's end.  Returns the loads issued (2 or 0).  Two of the ring's slots
// and not all: where nothing precedes the launch, the queries, whose load waits
// for the dependency, would queue behind the ring's 20 MB (8 queries over
// 131,080 tokens: calls apart 90.4 us with four loads, 89.3 with two or none;
// layers back to back 85.4, 85.4 and 86.3).
template <int D, bool kOne>
__device__ __forceinline__ int early_loads(const CUtensorMap* pool_map, const PrefillShortArgs& a,
                                           const Smem& sm, const FirstItem& start, const Item& it,
                                           int lane) {
    using C = PreCfg<D, kOne>;
    static_assert(C::kSlots > 2, "ring");
    const int32_t unsafe = lane < a.n_unsafe ? a.unsafe[lane] : -1;
    const int j_tail = it.t0 + it.T == a.n_tiles ? it.T - 1 : it.T;
    // lanes 0 and 1 have the records of key tiles 0 and 1
    const int pg0 = start.rec.y, pg1 = start.rec.z;
    bool safe = it.dual && j_tail > 1;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int p0 = __shfl_sync(0xffffffffu, pg0, x), p1 = __shfl_sync(0xffffffffu, pg1, x);
        safe = safe && (uint32_t)p0 < (uint32_t)a.num_pages && (uint32_t)p1 < (uint32_t)a.num_pages;
        safe = safe && !(unsafe >= 0 && (unsafe == p0 || unsafe == p1));
    }
    safe = __all_sync(0xffffffffu, safe);
    __syncwarp();  // (lane 0 initialised the barriers)
    if (safe && lane < 2) {
        const uint32_t fb = sm.bar<D, kOne>(C::kBarFull + lane);
        const uint32_t dst = sm.base + C::kOffRing + lane * C::kSlotBytes;
        mbar_arrive_expect_tx(fb, C::kSlotBytes);
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int cb = 0; cb < C::kColBlocks; ++cb)
                tma_load_4d(dst + cb * C::kBlockBytes + b * 64 * 128, pool_map, fb, cb * 64,
                            it.g * a.P + ((b ? start.rec.w : start.rec.x) & (a.P - 1)), b ? pg1 : pg0,
                            a.layer);
    }
    __syncwarp();
    return safe ? 2 : 0;
}

// The producer warp, item by item: the query tiles, then the K and V tiles of
// every key tile into the ring in the order of load_of, two loads at a time:
// the whole warp waits for both slots, then lanes 0 and 1 arm their barriers
// and issue their copies together, so that the shared-memory round trips of
// the two overlap.  The queries of an item wait until the previous item's last
// QK product is done; its first two loads go out before that wait.  What a
// tile's copies need, {first key, page of box 0, page of box 1}, is held in
// registers: lane l has the record of the window's key tile j = l (mod 32),
// batches of 16 tiles alternating between the lower and the upper half-warp;
// a batch is read from global memory about ten tiles before its first use and
// moved into place a few tiles before it, an item's first batch while the item
// before it runs.  Boxes past the second (pages of fewer than 64 tokens) take
// their page from global memory.
template <int D, bool kOne>
__device__ void prefill_produce(const CUtensorMap* pool_map, const CUtensorMap* qmap,
                                const PrefillArgs& a, const Smem& sm, const FirstItem& start,
                                int u_early, volatile int* abort_flag, int lane) {
    using C = PreCfg<D, kOne>;
    const int br = a.P < 64 ? a.P : 64;  // rows of one TMA box
    const int n_pieces = a.n_pieces;      // <= 16
    auto load_rec = [&](int t0, int T, int tb) { return tile_record(a, t0, T, tb, lane); };
    int4 raw = start.raw, first = start.rec;  // the item, and its first batch of records
    uint32_t n_items = 1;     // items published (the first at start-up)
    bool asked = false;       // an answer of the launch hardware is due
    uint32_t ub = 0;          // loads issued before this item (even)
    uint32_t n_queries = 0;   // items whose queries were loaded
    uint32_t n_fix = 0;       // uses of the fix-up barrier
    uint32_t issued = u_early;
    // Slots are freed by the MMA warp's commits: one for every V tile, which
    // covers the K tile loaded right after it too, and one for each item's
    // first K tile; in dual-key mode one for every tile.  Bit i of `own`: the
    // load i + 1 before the next one has a commit of its own; bit s of `par`:
    // parity of slot s's next commit.
    uint32_t own = 0, par = 0;
    uint32_t slot0 = u_early;  // slot of the next load
    uint32_t tail_u = 0;      // the load that used the fix-up barrier last
    bool tail_open = false;   // ... and was not handed over on its slot's barrier
    bool ok = true;
    auto load_queries = [&](const Item& it) {
        if (n_queries > 0)
            ok = mbar_wait(sm.bar<D, kOne>(C::kBarQFree), (n_queries - 1) & 1, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (ok && lane == 0) {
            const int nq = it.two ? 2 : 1;  // tile b is loaded only when it holds queries
            mbar_arrive_expect_tx(sm.bar<D, kOne>(C::kBarQ), nq * C::kColBlocks * a.BP * a.G * 128);
            for (int t = 0; t < nq; ++t)
                for (int cb = 0; cb < C::kColBlocks; ++cb)
                    tma_load_3d(sm.base + C::kOffQ + t * C::kQBytes + cb * C::kBlockBytes, qmap,
                                sm.bar<D, kOne>(C::kBarQ), cb * 64, it.g * a.G, it.pos_lo + t * a.BP);
        }
        if (ok) ++n_queries;
    };
    // hands an item (or the end mark) to the other roles
    auto publish = [&](int4 r) {
        const int slot = n_items % kItemSlots;
        if (n_items >= kItemSlots)
            ok = __all_sync(0xffffffffu,
                            mbar_wait(sm.bar<D, kOne>(C::kBarItemFree + slot),
                                      (n_items / kItemSlots - 1) & 1, abort_flag));
        if (ok && lane == 0) {
            *reinterpret_cast<int4*>(sm.ptr + C::kOffItems + slot * 16) = r;
            mbar_arrive(sm.bar<D, kOne>(C::kBarItem + slot));
        }
        if (ok) ++n_items;
    };
    // The next item: requested six key tiles before an item's end, as late as
    // the answer and its records allow, so that the SMs that are ahead take the
    // items left (asking with the first loads gave them out an item early: 3,001
    // queries over 33,001 tokens 841 -> 835 us); taken in with the last loads.
    int4 next = make_int4(0, 0, -1, 0);
    auto request = [&]() {
        if (lane == 0) {
            mbar_arrive_expect_tx(sm.bar<D, kOne>(C::kBarClc), 16);
            clc_request(sm.base + C::kOffClc, sm.bar<D, kOne>(C::kBarClc));
        }
        asked = true;
    };
    auto take_next = [&](uint32_t parity) {
        ok = __all_sync(0xffffffffu, mbar_wait(sm.bar<D, kOne>(C::kBarClc), parity, abort_flag));
        if (!ok) return;
        asked = false;
        const int cta = clc_answer(sm.base + C::kOffClc);
        next = make_int4(0, 0, -1, 0);
        if (cta >= 0 && cta < a.n_items)
            next = __ldg(reinterpret_cast<const int4*>(a.items) + cta);
        first = load_rec(next.y, next.z, 0);
        // the answer's words are read before the next request overwrites them
        fence_proxy_async_smem();
        __syncwarp();
    };
    if (u_early > 0) own = 3;  // as the loop below keeps it
    while (ok && raw.z >= 0) {
        const Item it = make_item<kOne>(a, raw);
        const uint32_t clc_parity = (n_items - 1) & 1;
        int4 rec = first, pend = first;
        const int T = it.T;
        const int n_units = 2 * T;
        const int take_at = n_units - 2, ask_at = n_units > 14 ? n_units - 12 : 0;
        const bool late_queries = ub > 0;
        if (T > 0 && !late_queries) load_queries(it);
        if (u_early > ask_at) request();
        if (T == 0) {
            request();
            take_next(clc_parity);
        }
        int fill_b = 1;    // the next batch to read
        int merge_b = -1;  // the batch read into `pend`, not yet in place
        // only the sequence's last key tile has rows past its end
        const int j_tail = it.t0 + T == a.n_tiles ? T - 1 : T;
        for (int u0 = u_early; ok && u0 < n_units; u0 += 2) {  // n_units is even
            int j0, kv0, j1, kv1;
            load_of(u0, T, it.dual, j0, kv0);
            load_of(u0 + 1, T, it.dual, j1, kv1);
            const int jmax = j0 > j1 ? j0 : j1;
            if (merge_b >= 0 && jmax + 4 >= kBatch * merge_b) {
                if ((lane >> 4) == (merge_b & 1)) rec = pend;
                merge_b = -1;
            }
            if (merge_b < 0 && fill_b * kBatch < T && jmax + 10 >= kBatch * fill_b) {
                if ((lane >> 4) == (fill_b & 1)) pend = load_rec(it.t0, T, fill_b * kBatch);
                merge_b = fill_b++;
            }
            const uint32_t U0 = ub + u0;
            const uint32_t slot1 = slot0 + 1 == C::kSlots ? 0 : slot0 + 1;
            const int j = (lane & 1) ? j1 : j0, kv = (lane & 1) ? kv1 : kv0;
            const int key0 = __shfl_sync(0xffffffffu, rec.x, j & 31);
            const int pg0 = __shfl_sync(0xffffffffu, rec.y, j & 31);
            const int pg1 = __shfl_sync(0xffffffffu, rec.z, j & 31);
            const int key0b = __shfl_sync(0xffffffffu, rec.w, j & 31);
            const int slot = (lane & 1) ? slot1 : slot0;  // lanes 0 and 1 issue
            const uint32_t dst = sm.base + C::kOffRing + slot * C::kSlotBytes;
            const int head_row = (kv ? a.Hkv + it.g : it.g) * a.P;
            // every lane polls the slots' barriers in turn: warp-uniform waits,
            // so no lane waits at the vote below for two polling lanes
            if (U0 >= C::kSlots && ((own >> (C::kSlots - 1)) & 1u)) {
                ok = mbar_wait(sm.bar<D, kOne>(C::kBarEmpty + slot0), (par >> slot0) & 1u, abort_flag);
                par ^= 1u << slot0;
            }
            if (U0 + 1 >= C::kSlots && ((own >> (C::kSlots - 2)) & 1u)) {
                if (ok)
                    ok = mbar_wait(sm.bar<D, kOne>(C::kBarEmpty + slot1), (par >> slot1) & 1u, abort_flag);
                par ^= 1u << slot1;
            }
            own = own << 2 | (it.dual || j0 == 0 ? 3u : 1u);  // K_j0, V_j1 but in dual-key mode
            // both slots free, or neither load is issued
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            auto checked = [&](int32_t page) {
                if ((uint32_t)page < (uint32_t)a.num_pages) return page;
                // a page outside the pool: flagged; the box is read from page 0
                // so that the barrier's byte count still completes
                set_error(a.err, kErrBounds);
                return 0;
            };
            auto load_box = [&](uint32_t bar, int i, int key, int32_t page) {
                const int row = head_row + (key & (a.P - 1));  // P is a power of two
#pragma unroll
                for (int cb = 0; cb < C::kColBlocks; ++cb)
                    tma_load_4d(dst + cb * C::kBlockBytes + i * br * 128, pool_map, bar, cb * 64, row,
                                page, a.layer);
            };
            if (n_pieces == 2 && jmax < j_tail) {
                // two whole boxes of 64 rows, as almost every tile has
                if (lane < 2) {
                    const uint32_t fb = sm.bar<D, kOne>(C::kBarFull + slot);
                    mbar_arrive_expect_tx(fb, C::kSlotBytes);
                    load_box(fb, 0, key0, checked(pg0));
                    load_box(fb, 1, key0b, checked(pg1));
                }
            } else {
                // rows of the tile inside the sequence: the lower half's, then
                // the upper half's
                const int rows_b = key0b < a.n ? min(64, a.n - key0b) : 0;
                const int rows = rows_b > 0 ? 64 + rows_b : min(64, a.n - key0);
                const bool vfix = lane < 2 && kv == 1 && rows < kPrefillKeys;
                if (lane < 2) {
                    const int nv = (rows + br - 1) / br;  // boxes inside the sequence (a prefix)
                    const uint32_t fb = vfix ? sm.bar<D, kOne>(C::kBarVfix) : sm.bar<D, kOne>(C::kBarFull + slot);
                    mbar_arrive_expect_tx(fb, (uint32_t)nv * br * 128 * C::kColBlocks);
                    const int half = n_pieces / 2;
#pragma unroll 1
                    for (int i = 0; i < nv; ++i) {
                        const int32_t page =
                            i == 0
                                ? pg0
                                : (i == 1 ? pg1
                                          : __ldg(&a.tile_pages[(size_t)(it.t0 + j) * n_pieces + i]));
                        load_box(fb, i, i < half ? key0 + i * br : key0b + (i - half) * br,
                                 checked(page));
                    }
                }
                const uint32_t fix = __ballot_sync(0xffffffffu, vfix);
                if (fix) {
                    // V of the last key tile: its rows past the sequence's end hold
                    // stale or never-written data.  Their weights are zero, but
                    // 0 * NaN is not, so zero those rows before the MMAs read the slot.
                    const int src = __ffs(fix) - 1;
                    const int fslot = __shfl_sync(0xffffffffu, slot, src);
                    const int r0 = __shfl_sync(0xffffffffu, rows, src);  // 1 .. 127
                    tail_u = U0 + src;
                    tail_open = true;
                    issued = U0 + 2;
                    if (lane == 0) ok = mbar_wait(sm.bar<D, kOne>(C::kBarVfix), n_fix & 1, abort_flag);
                    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0);
                    if (!ok) break;
                    ++n_fix;
                    const int chunks = (kPrefillKeys - r0) * 8;
                    uint8_t* vsp = sm.ptr + C::kOffRing + fslot * C::kSlotBytes;
                    for (int cb = 0; cb < C::kColBlocks; ++cb)
                        for (int c = lane; c < chunks; c += 32)
                            *reinterpret_cast<uint4*>(vsp + cb * C::kBlockBytes +
                                                      (r0 + (c >> 3)) * 128 + (c & 7) * 16) =
                                make_uint4(0, 0, 0, 0);
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(sm.bar<D, kOne>(C::kBarFull + fslot));
                    tail_open = false;
                }
            }
            issued = U0 + 2;
            slot0 = slot1 + 1 == C::kSlots ? 0 : slot1 + 1;
            if (u0 == ask_at) request();
            if (u0 == 0 && late_queries) load_queries(it);
            if (ok && u0 == take_at) take_next(clc_parity);
        }
        ub += n_units;
        u_early = 0;
        raw = next;
        if (ok) publish(raw);  // an item, or the end mark
    }
    if (!ok && lane == 0) {
        if (!*abort_flag) set_error(a.err, kErrTimeout);
        *abort_flag = 1;
    }
    // Drain: every copy this CTA issued lands before the CTA exits (immediate
    // unless a consumer gave up early).
    if (lane == 0) {
        if (asked) mbar_wait(sm.bar<D, kOne>(C::kBarClc), (n_items - 1) & 1);
        if (n_queries > 0) mbar_wait(sm.bar<D, kOne>(C::kBarQ), (n_queries - 1) & 1);
        for (uint32_t u = issued > C::kSlots ? issued - C::kSlots : 0; u < issued; ++u) {
            if (u == tail_u && tail_open) mbar_wait(sm.bar<D, kOne>(C::kBarVfix), n_fix & 1);
            else mbar_wait(sm.bar<D, kOne>(C::kBarFull + u % C::kSlots), (u / C::kSlots) & 1);
        }
    }
}

// Descriptors of a CTA's operands: the two query tiles, and the ring's slot 0
// as a K tile (K-major) and as a V tile (MN-major).  Slot s is s *
// kSlotBytes / 16 further in the address field.
struct MmaDesc {
    uint32_t q[2], k, v;      // low words
    uint32_t k_hi, v_hi;      // high words (the queries' is the K tile's)
    uint32_t tmem;
};
template <int D, bool kOne>
__device__ __forceinline__ MmaDesc mma_desc(const Smem& sm, uint32_t tmem) {
    using C = PreCfg<D, kOne>;
    static_assert(C::kBlockBytes == 16384, "the K-major steps' block stride");
    const uint64_t q = smem_desc_sw128(sm.base + C::kOffQ, 16, 1024);
    const uint64_t k = smem_desc_sw128(sm.base + C::kOffRing, 16, 1024);
    const uint64_t v = smem_desc_sw128(sm.base + C::kOffRing, C::kBlockBytes, 1024);
    MmaDesc d;
    d.q[0] = (uint32_t)q;
    d.q[1] = (uint32_t)q + (C::kQBytes >> 4);
    d.k = (uint32_t)k;
    d.v = (uint32_t)v;
    d.k_hi = (uint32_t)(k >> 32);
    d.v_hi = (uint32_t)(v >> 32);
    d.tmem = tmem;
    return d;
}

// S_t = Q_q K^T for the K tile in `slot`, into TMEM columns 128 t (q = t
// except in dual-key mode, where both tiles use query tile 0).
template <int D, bool kOne>
__device__ __forceinline__ void issue_qk(const MmaDesc& d, int t, int q, uint32_t slot) {
    using C = PreCfg<D, kOne>;
    mma_bf16_ss_steps<D / 16>(d.tmem + C::kColS + (uint32_t)t * kPrefillKeys, d.q[q],
                              d.k + slot * (C::kSlotBytes >> 4), d.k_hi, C::kIdescQK);
}

// O_t += P_t V for the V tile in `slot`; P_t from TMEM over the first half of S_t.
template <int D, bool kOne>
__device__ __forceinline__ void issue_pv(const MmaDesc& d, int t, uint32_t slot, bool first) {
    using C = PreCfg<D, kOne>;
    static_assert(kPrefillKeys == 128, "8 steps of 16 keys");
    mma_bf16_ts_steps8(d.tmem + C::kColO + (uint32_t)t * 128,
                       d.tmem + C::kColS + (uint32_t)t * kPrefillKeys,
                       d.v + slot * (C::kSlotBytes >> 4), d.v_hi, C::kIdescPV, first ? 0u : 1u);
}

// Phases of the barriers the MMA warp waits on, running on from item to item.
struct MmaPhase {
    uint32_t ub;    // loads of the items before (K_j, V_j: load_of)
    uint32_t slot;  // ub mod kSlots
    uint32_t p;     // bit t: parity of the next P_t hand-off
    uint32_t q;     // items whose queries were used
};

// The lane that issues the MMAs is the busiest thread of the kernel: whatever
// it does between two products, the tensor core's short queue drains.  So it
// waits for P_t alone: a softmax warp of tile a hands over P only when V_j and
// K_{j+1} have landed too, and one commit after the second PV frees V_j and,
// with it, the K tile used by the QK products issued just before.  (With its
// own waits for both tiles and a commit for each slot the lane needed 3,434
// cycles per key tile for products of 2,650, and was never waiting for P.)
// In dual-key mode memory is the bound, not this lane: it waits for each tile
// by itself and frees each slot at once.
//
// Dual-key mode (every query of the CTA tile fits in tile a): both tiles
// hold tile a's queries; tile a takes key tiles 0, 2, 4, ... and tile b the
// odd ones, and the two results are merged at the end.  Key tile j's PV and
// the QK of key tile j + 2 (into the same S columns) are issued in the order
// of the loads, each as soon as its tile has landed.
template <int D, bool kOne>
__device__ bool prefill_mma_dual(const Smem& sm, const MmaDesc& d, int T, MmaPhase& ph,
                                 volatile int* abort_flag) {
    using C = PreCfg<D, kOne>;
    // the tiles are used in the order of their loads: K_0, K_1, V_0, K_2, V_1, ...
    uint32_t slot = ph.slot, full = (ph.ub / C::kSlots) & 1;
    auto landed = [&]() { return mbar_wait(sm.bar<D, kOne>(C::kBarFull + slot), full, abort_flag); };
    auto used = [&]() {
        mma_commit(sm.bar<D, kOne>(C::kBarEmpty + slot));
        if (++slot == C::kSlots) {
            slot = 0;
            full ^= 1;
        }
    };
    for (int t = 0; t < 2; ++t) {
        // S_t = Q_a K_t
        if (!landed()) return false;
        issue_qk<D, kOne>(d, t, 0, slot);
        mma_commit(sm.bar<D, kOne>(C::kBarS + t));
        used();
    }
    if (T == 2) mma_commit(sm.bar<D, kOne>(C::kBarQFree));  // the item's last QK
    for (int j = 0; j < T; ++j) {
        const int t = j & 1;
        if (!landed()) return false;
        if (!mbar_wait(sm.bar<D, kOne>(C::kBarP + t), (ph.p >> t) & 1, abort_flag)) return false;
        ph.p ^= 1u << t;
        tc_fence_after();
        issue_pv<D, kOne>(d, t, slot, j < 2);
        used();
        if (j + 2 >= T) {  // the last key tile of tile t
            mma_commit(sm.bar<D, kOne>(C::kBarO + t));
            continue;
        }
        if (!landed()) return false;
        issue_qk<D, kOne>(d, t, 0, slot);
        mma_commit(sm.bar<D, kOne>(C::kBarS + t));
        used();
        if (j + 3 == T) mma_commit(sm.bar<D, kOne>(C::kBarQFree));  // the item's last QK
    }
    ph.slot = slot;
    return true;
}

// One step of the two-tile path: O_t += P_t V_j, then S_t for the next key tile,
// for tile a and then tile b.
template <int D, bool kOne, bool kFirst, bool kMore>
__device__ __forceinline__ bool prefill_mma_step(const Smem& sm, const MmaDesc& d, uint32_t vslot,
                                                 uint32_t kslot, uint32_t pa, uint32_t pb,
                                                 const volatile int* abort_flag) {
    using C = PreCfg<D, kOne>;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        if (!mbar_wait(sm.bar<D, kOne>(C::kBarP + t), t ? pb : pa, abort_flag)) return false;
        tc_fence_after();
        issue_pv<D, kOne>(d, t, vslot, kFirst);
        if (kMore) issue_qk<D, kOne>(d, t, t, kslot);
        mma_commit(sm.bar<D, kOne>(kMore ? C::kBarS + t : C::kBarO + t));
    }
    mma_commit(sm.bar<D, kOne>(C::kBarEmpty + vslot));  // V_j, and K_{j+1} with it
    return true;
}

// `two`: tile b holds query rows (false for an item of one key tile whose rows
// all fit in tile a; tile b's products are then skipped).
template <int D, bool kOne>
__device__ bool prefill_mma_item(const Smem& sm, const MmaDesc& d, int T, bool two, MmaPhase& ph,
                                 volatile int* abort_flag) {
    using C = PreCfg<D, kOne>;
    auto after = [](uint32_t slot) { return slot + 1 == C::kSlots ? 0u : slot + 1; };
    uint32_t slot = ph.slot;
    if (!mbar_wait(sm.bar<D, kOne>(C::kBarFull + slot), (ph.ub / C::kSlots) & 1, abort_flag)) return false;
    issue_qk<D, kOne>(d, 0, 0, slot);
    mma_commit(sm.bar<D, kOne>(C::kBarS + 0));
    if (two) {
        issue_qk<D, kOne>(d, 1, 1, slot);
        mma_commit(sm.bar<D, kOne>(C::kBarS + 1));
    }
    mma_commit(sm.bar<D, kOne>(C::kBarEmpty + slot));
    uint32_t vslot = after(slot), kslot = after(vslot);
    if (kOne || !two) {
        mma_commit(sm.bar<D, kOne>(C::kBarQFree));
        if (!mbar_wait(sm.bar<D, kOne>(C::kBarP + 0), ph.p & 1, abort_flag)) return false;
        tc_fence_after();
        issue_pv<D, kOne>(d, 0, vslot, true);
        mma_commit(sm.bar<D, kOne>(C::kBarO + 0));
        mma_commit(sm.bar<D, kOne>(C::kBarEmpty + vslot));
        ph.p ^= 1u;
        ph.slot = kslot;
        return true;
    }
    uint32_t pa = ph.p & 1, pb = (ph.p >> 1) & 1;
    if (T == 1) {
        mma_commit(sm.bar<D, kOne>(C::kBarQFree));
        if (!prefill_mma_step<D, kOne, true, false>(sm, d, vslot, kslot, pa, pb, abort_flag)) return false;
    } else {
        if (!prefill_mma_step<D, kOne, true, true>(sm, d, vslot, kslot, pa, pb, abort_flag)) return false;
        for (int j = 1; j + 1 < T; ++j) {
            vslot = after(kslot);
            kslot = after(vslot);
            pa ^= 1;
            pb ^= 1;
            if (!prefill_mma_step<D, kOne, false, true>(sm, d, vslot, kslot, pa, pb, abort_flag))
                return false;
        }
        mma_commit(sm.bar<D, kOne>(C::kBarQFree));  // the item's last QK
        vslot = after(kslot);
        kslot = after(vslot);
        if (!prefill_mma_step<D, kOne, false, false>(sm, d, vslot, kslot, pa ^ 1, pb ^ 1, abort_flag))
            return false;
    }
    ph.p ^= (T & 1) ? 3u : 0u;
    ph.slot = kslot;
    return true;
}

// The MMA-issuing lane, item by item.  The next item's first S may be issued
// while the softmax warps still write out this one's O: S has columns of its
// own, and the first PV, which overwrites O, waits for a P that each softmax
// thread hands over only after it has read its O.
template <int D, bool kOne>
__device__ void prefill_mma(const PrefillArgs& a, const Smem& sm, uint32_t tmem,
                            volatile int* abort_flag) {
    using C = PreCfg<D, kOne>;
    MmaPhase ph = {0, 0, 0, 0};
    const MmaDesc d = mma_desc<D, kOne>(sm, tmem);
    bool ok = true, any = false;
    for (uint32_t k = 0;; ++k) {
        if (!(ok = item_wait<D, kOne>(sm, k, abort_flag))) break;
        const int4 raw = item_read<D, kOne>(sm, k);
        item_free<D, kOne>(sm, k);
        if (raw.z < 0) break;
        if (raw.z == 0) continue;
        const Item it = make_item<kOne>(a, raw);
        if (!(ok = mbar_wait(sm.bar<D, kOne>(C::kBarQ), ph.q & 1, abort_flag))) break;
        tc_fence_after();
        ++ph.q;
        any = true;
        ok = it.dual ? prefill_mma_dual<D, kOne>(sm, d, it.T, ph, abort_flag)
                     : prefill_mma_item<D, kOne>(sm, d, it.T, it.two, ph, abort_flag);
        if (!ok) break;
        ph.ub += 2 * it.T;
    }
    if (!ok) {
        set_error(a.err, kErrTimeout);
        *abort_flag = 1;
    }
    if (any) {
        // every MMA issued here completes before TMEM is released
        mma_commit(sm.bar<D, kOne>(C::kBarDone));
        mbar_wait(sm.bar<D, kOne>(C::kBarDone), 0);
    }
}

// Packed fp32 pair helpers (sm_100 family): d = a * b + c on two lanes at once.
__device__ __forceinline__ uint64_t f2pack(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2unpack(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t ffma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// lo += the low bf16 of w, hi += its high bf16 (mixed-precision adds: the
// bf16 operands are exact in fp32).
__device__ __forceinline__ void add_bf16x2_f32(uint32_t w, float& lo, float& hi) {
    asm("{\n\t.reg .b16 l16, h16;\n\tmov.b32 {l16, h16}, %2;\n\t"
        "add.rn.f32.bf16 %0, l16, %0;\n\tadd.rn.f32.bf16 %1, h16, %1;\n\t}"
        : "+f"(lo), "+f"(hi)
        : "r"(w));
}
// 2^x as the single PTX instruction ex2.approx.ftz (relative error about
// 2^-22).  Results below 2^-126 flush to zero: every row holds a weight of at
// least 1 (its running maximum's), so they change its sums by under 2^-119.
__device__ __forceinline__ float ex2_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Every lane of the warp polls the barrier (one instruction for the warp,
// no hand-on from a polling lane: a softmax warp sees its S ready sooner);
// returns the warp-uniform result.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, const volatile int* abort) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort));
}

// Normalises and writes one row of O_t (with tile b's part in dual-key mode) to
// the outputs, or to the item's partial result.
template <int D, bool kOne>
__device__ __forceinline__ void prefill_write(const PrefillArgs& a, const Item& it, uint32_t tl,
                                              uint32_t col_o, int t, int row, bool valid,
                                              float m_run, float l, float wa, float wb) {
    using C = PreCfg<D, kOne>;
    const bool dual = it.dual, any_keys = it.T > 0;
    const int qi = it.pos_lo + (dual ? 0 : t) * a.BP + row / a.G;
    const float inv = l > 0.f ? 1.f / l : 0.f;
    const float lse2 = l > 0.f ? m_run + __log2f(l) : -INFINITY;
    const int h = it.g * a.G + row % a.G;
    float* part_row = nullptr;
    uint8_t* out_row = nullptr;
    if (it.part >= 0) {
        const size_t pr = ((size_t)it.part * kPrefillQTiles + t) * kPrefillRows + row;
        part_row = a.part_o + pr * D;
        if (valid) a.part_ml[pr] = lse2;
    } else {
        out_row = reinterpret_cast<uint8_t*>(a.out) +
                  ((size_t)qi * a.Hq + h) * D * (a.out_f32 ? 4 : 2);
        if (valid && a.lse) a.lse[(size_t)qi * a.Hq + h] = lse2 * 0.69314718055994531f;
    }
#pragma unroll
    for (int c = 0; c < D / 32; ++c) {
        uint32_t o[32];
        if (any_keys) {
            tmem_ld32(tl + col_o + c * 32, o);
            tmem_wait_ld();
        } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = 0u;
        }
        float f[32];
        if (dual) {
            uint32_t ob[32];
            tmem_ld32(tl + C::kColO + 128 + c * 32, ob);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i)
                f[i] = (__uint_as_float(o[i]) * wa + __uint_as_float(ob[i]) * wb) * inv;
        } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) f[i] = __uint_as_float(o[i]) * inv;
        }
        if (!valid) continue;
        if (part_row || a.out_f32) {
            float4* dst = reinterpret_cast<float4*>(part_row ? part_row + c * 32
                                                             : reinterpret_cast<float*>(out_row) + c * 32);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                dst[i] = make_float4(f[4 * i], f[4 * i + 1], f[4 * i + 2], f[4 * i + 3]);
        } else {
            uint4* dst = reinterpret_cast<uint4*>(out_row + c * 64);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t w[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const __nv_bfloat162 hb = __floats2bfloat162_rn(f[8 * i + 2 * e], f[8 * i + 2 * e + 1]);
                    w[e] = *reinterpret_cast<const uint32_t*>(&hb);
                }
                dst[i] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    }
}

// What a softmax warp carries from item to item, in two words so that the
// loop over key tiles keeps its registers: the loads of the items before, and,
// as bits of `par`, the parities of the hand-offs to wait for next.  The item
// itself stays in its ring slot until the warp has written its output.
struct SoftmaxPhase {
    uint32_t ub, par;
};
constexpr uint32_t kParS = 1, kParO = 2, kParX = 4;  // S_t, O_t, dual-key exchange

// Softmax warpgroup of query tile t (one row per thread) and its epilogue,
// for one item.  False: a wait ran out.
template <int D, bool kOne>
__device__ bool prefill_softmax(const PrefillArgs& a, const Smem& sm, uint32_t tmem, int t,
                                uint32_t k, SoftmaxPhase& ph, volatile int* abort_flag, int warp,
                                int lane) {
    using C = PreCfg<D, kOne>;
    const int wq = warp & 3;
    const int row = wq * 32 + lane;
    const Item it = make_item<kOne>(a, item_read<D, kOne>(sm, k));
    const bool dual = it.dual;
    const int T_cta = it.T, t0 = it.t0;
    // dual-key mode: both tiles hold tile a's queries, tile t takes key tiles
    // t, t + 2, t + 4, ... of the CTA's range
    const int qi = it.pos_lo + (dual ? 0 : t) * a.BP + row / a.G;
    const bool valid = row < a.BP * a.G && qi < a.n_q;
    const int T = dual ? (T_cta + 1 - t) / 2 : T_cta;
    const int kstep = dual ? 2 : 1, kfirst = dual ? t : 0;
    float* xchg = reinterpret_cast<float*>(sm.ptr + C::kOffXchg);
    // A warp none of whose rows is a query only keeps the barrier count: it
    // waits for each S and signals its P without computing (its rows of P
    // and O are never read back).
    if (!__any_sync(0xffffffffu, valid)) {
        for (int j = 0; j < T; ++j) {
            if (!warp_wait(sm.bar<D, kOne>(C::kBarS + t), ph.par & kParS, abort_flag)) return false;
            ph.par ^= kParS;
            tc_fence_before();
            mbar_arrive(sm.bar<D, kOne>(C::kBarP + t));
        }
        if (T > 0) ph.par ^= kParO;
        if (dual) {
            mbar_arrive(sm.bar<D, kOne>(t == 1 ? C::kBarX : C::kBarXFree));
            // (tile b's next P waits for tile a's reads also here)
            if (t == 1 && !warp_wait(sm.bar<D, kOne>(C::kBarXFree), (ph.par & kParX) != 0, abort_flag))
                return false;
            ph.par ^= kParX;
        }
        return true;
    }
    // rows that are no query (their results are never read) mask as the last
    // one does and stay out of the warp's votes, so that a tile with some does
    // not take the masked, twice-computed path (2.33 instead of 1.77 us a tile)
    const int p_row = a.n - a.n_q + (valid ? qi : a.n_q - 1);
    const uint32_t tl = tmem + ((uint32_t)(wq * 32) << 16);
    const uint32_t col_s = C::kColS + (uint32_t)t * kPrefillKeys;
    const uint32_t col_o = C::kColO + (uint32_t)t * 128;
    const float sc = a.scale_log2;  // > 0 (the host raises a zero scale to a tiny one)
    // most that a row's weights of one tile may sum to without a look at their
    // maximum (a power of two above the running one).  A warp with rows that are
    // no query raises its maxima where a weight passes 2^8, as such warps did
    // when every tile of theirs took the path with the maximum: the largest
    // weight of a row is then more often exactly 1, and not rounded (with 2^16
    // the log-sum-exp of 3 queries over 9,892 tokens was off by 2.4e-5 instead
    // of 1.3e-5 of its size).
    const float accept = __all_sync(0xffffffffu, valid) ? 65536.f : 256.f;
    float m_run = -INFINITY, l = 0.f;
    // {first keys, flags} of the next key tile; its visibility bits are read
    // only where a tile is masked (they would hold eight registers of the loop)
    const PrefillTile* tp = a.tiles + t0 + kfirst;
    int2 nk = make_int2(0, 0);
    int nb = 0;
    if (T > 0) {
        nk = __ldg(reinterpret_cast<const int2*>(tp));
        nb = __ldg(&tp->key0b);
    }
    for (int j = 0; j < T; ++j) {
        // this tile's record; the next one is fetched while this tile is worked on
        const int2 wk = nk;
        const int wb_ = nb;
        if (j + 1 < T) {
            nk = __ldg(reinterpret_cast<const int2*>(tp + kstep));
            nb = __ldg(&tp[kstep].key0b);
        }
        if (!warp_wait(sm.bar<D, kOne>(C::kBarS + t), ph.par & kParS, abort_flag)) return false;
        ph.par ^= kParS;
        tc_fence_after();
        // Raw logits q.k (the scale is applied inside the exponent; it is > 0),
        // taken 64 columns at a time to keep registers low: one pass for the
        // row maximum, one for the weights.
        // keys key0 + c (lower half) and key0b + c (upper half) with c <= lim,
        // c <= limb are causal
        const int lim = p_row - wk.x, limb = p_row - wb_;
        const bool unmasked = (wk.y & kPrefillTileFull) && lim >= 63 && limb >= 63;
        // Weights 2^(s * scale - m) with the running maximum m, two arguments
        // at a time with a packed FMA, rounded to bf16 into wt (32 words per
        // 64 keys).  The normaliser sums the same rounded weights that the PV
        // product takes (eight fp32 chains), so the output is a convex
        // combination of the V rows whatever the rounding.
        // Nothing is stored: S stays intact until the weights are accepted.
        const uint64_t sc2 = f2pack(sc, sc);
        uint32_t wt[2][32];
        auto weights = [&](float m, float& tile_sum) {
            const float nmu = m == -INFINITY ? 0.f : -m;
            const uint64_t nmu2 = f2pack(nmu, nmu);
            float ls[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                uint32_t x[64];
                tmem_ld32(tl + col_s + 64 * hh, *reinterpret_cast<uint32_t(*)[32]>(&x[0]));
                tmem_ld32(tl + col_s + 64 * hh + 32, *reinterpret_cast<uint32_t(*)[32]>(&x[32]));
                tmem_wait_ld();
                if (!unmasked) {
#pragma unroll
                    for (int w = 0; w < 2; ++w) {
                        const int ww = 2 * hh + w;
                        const uint32_t mw =
                            __ldg(&tp->vis[ww]) & low_bits_through((ww < 2 ? lim : limb) - 32 * (ww & 1));
#pragma unroll
                        for (int c = 0; c < 32; ++c)
                            if (!((mw >> c) & 1u)) x[32 * w + c] = 0xff800000u;  // -inf
                    }
                }
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const float x0 = __uint_as_float(x[2 * i]), x1 = __uint_as_float(x[2 * i + 1]);
                    float a0, a1;
                    f2unpack(ffma2(f2pack(x0, x1), sc2, nmu2), a0, a1);
                    const __nv_bfloat162 hb = __floats2bfloat162_rn(ex2_ftz(a0), ex2_ftz(a1));
                    wt[hh][i] = *reinterpret_cast<const uint32_t*>(&hb);
                    add_bf16x2_f32(wt[hh][i], ls[2 * (i & 3)], ls[2 * (i & 3) + 1]);
                }
            }
            tile_sum = ((ls[0] + ls[1]) + (ls[2] + ls[3])) + ((ls[4] + ls[5]) + (ls[6] + ls[7]));
        };
        // The maximum is raised lazily, so most tiles keep it: take the
        // weights with the current maximum and accept them when no row's sum
        // exceeds `accept`, which bounds every weight; no maximum is needed for
        // that.  Otherwise (or when a row has seen no key yet) find the tile's
        // maximum and redo the tile with it wherever it exceeds the running
        // one by more than 2^8.
        float mt = -INFINITY, tsum = 0.f;
        bool done = false;
        if (__all_sync(0xffffffffu, m_run != -INFINITY || !valid)) {
            weights(m_run, tsum);
            done = !__any_sync(0xffffffffu, valid && tsum > accept);
        }
        if (!done) {
            // row maximum: three-input max over four independent chains
            float mx[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) mx[c] = -INFINITY;
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                uint32_t x[64];
                tmem_ld32(tl + col_s + 64 * hh, *reinterpret_cast<uint32_t(*)[32]>(&x[0]));
                tmem_ld32(tl + col_s + 64 * hh + 32, *reinterpret_cast<uint32_t(*)[32]>(&x[32]));
                tmem_wait_ld();
                if (!unmasked) {
#pragma unroll
                    for (int w = 0; w < 2; ++w) {
                        const int ww = 2 * hh + w;
                        const uint32_t mw =
                            __ldg(&tp->vis[ww]) & low_bits_through((ww < 2 ? lim : limb) - 32 * (ww & 1));
#pragma unroll
                        for (int c = 0; c < 32; ++c)
                            if (!((mw >> c) & 1u)) x[32 * w + c] = 0xff800000u;  // -inf
                    }
                }
#pragma unroll
                for (int c = 0; c < 64; c += 8) {
                    mx[0] = fmax3(mx[0], __uint_as_float(x[c]), __uint_as_float(x[c + 1]));
                    mx[1] = fmax3(mx[1], __uint_as_float(x[c + 2]), __uint_as_float(x[c + 3]));
                    mx[2] = fmax3(mx[2], __uint_as_float(x[c + 4]), __uint_as_float(x[c + 5]));
                    mx[3] = fmax3(mx[3], __uint_as_float(x[c + 6]), __uint_as_float(x[c + 7]));
                }
            }
            mt = fmaxf(fmax3(mx[0], mx[1], mx[2]), mx[3]) * sc;
        }
        if (done) {
            l += tsum;
        } else {
            const bool need = valid && mt > m_run + 8.f;
            float alpha = 1.f;
            if (need) {
                alpha = exp2f(m_run - mt);
                m_run = mt;
                l *= alpha;
            }
            if (j > 0 && __any_sync(0xffffffffu, need)) {
                // O_t holds the products up to key tile j - 1 (complete: S_t(j)
                // was issued after them): rescale it in place
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t o[32];
                    tmem_ld32(tl + col_o + c * 32, o);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                    tmem_st32(tl + col_o + c * 32, o);
                }
            }
            weights(m_run, tsum);
            l += tsum;
        }
        // P_t over the first half of S_t: keys 64 hh .. +63 to columns 32 hh .. +31.
        // One warp also sees that the tiles of the products that follow have
        // landed (long ago, as a rule): V_j, and the K tile of the next S.
        bool landed = true;
        uint32_t fv = 0, fk = 0, pv = 0, pk = 0;
        if (wq == 0 && t == 0 && !dual) {
            const uint32_t uv = ph.ub + 2 * j + 1, uk = uv + 1;
            fv = sm.bar<D, kOne>(C::kBarFull + uv % C::kSlots);
            pv = (uv / C::kSlots) & 1;
            fk = j + 1 < T ? sm.bar<D, kOne>(C::kBarFull + uk % C::kSlots) : fv;
            pk = j + 1 < T ? (uk / C::kSlots) & 1 : pv;
            landed = mbar_try_wait(fv, pv) & mbar_try_wait(fk, pk);
        }
        tmem_st32(tl + col_s, wt[0]);
        tmem_st32(tl + col_s + 32, wt[1]);
        tmem_wait_st();
        if (!__all_sync(0xffffffffu, landed)) {
            if (!warp_wait(fv, pv, abort_flag) || !warp_wait(fk, pk, abort_flag)) return false;
        }
        tc_fence_before();
        mbar_arrive(sm.bar<D, kOne>(C::kBarP + t));
        tp += kstep;
    }
    if (T > 0) {
        if (!warp_wait(sm.bar<D, kOne>(C::kBarO + t), (ph.par & kParO) != 0, abort_flag)) return false;
        ph.par ^= kParO;
    }
    // dual-key mode: tile b hands its (max, normaliser) to tile a, which
    // merges the two partial results of each row (weights 2^(m_t - max)) and
    // reads O_b, complete by tile b's wait above
    float wa = 1.f, wb = 0.f;
    tc_fence_after();
    if (dual && t == 1) {
        xchg[2 * row] = m_run;
        xchg[2 * row + 1] = l;
        tc_fence_before();
        mbar_arrive(sm.bar<D, kOne>(C::kBarX));
        // tile b's next P (and with it the products that overwrite O_b) waits
        // until tile a has read O_b
        if (!warp_wait(sm.bar<D, kOne>(C::kBarXFree), (ph.par & kParX) != 0, abort_flag)) return false;
        ph.par ^= kParX;
        tc_fence_after();
        return true;
    }
    if (dual) {
        if (!warp_wait(sm.bar<D, kOne>(C::kBarX), (ph.par & kParX) != 0, abort_flag)) return false;
        ph.par ^= kParX;
        tc_fence_after();
        const float mb = xchg[2 * row], lb = xchg[2 * row + 1];
        const float M = fmaxf(m_run, mb);
        wa = m_run == -INFINITY ? 0.f : exp2f(m_run - M);
        wb = mb == -INFINITY ? 0.f : exp2f(mb - M);
        l = l * wa + lb * wb;
        m_run = M;
    }
    // the item again, from its slot
    const int4 raw = item_read<D, kOne>(sm, k);
    prefill_write<D, kOne>(a, make_item<kOne>(a, raw), tl, col_o, t, row, valid, m_run, l, wa, wb);
    if (dual) {
        tc_fence_before();
        mbar_arrive(sm.bar<D, kOne>(C::kBarXFree));
    }
    return true;
}

template <int D, typename Args>
__global__ void __launch_bounds__(320, 1)
    sq_prefill_kernel(const __grid_constant__ CUtensorMap pool_map,
                      const __grid_constant__ CUtensorMap qmap, const Args a) {
    constexpr bool kOne = std::is_same<Args, PrefillShortArgs>::value;
    using C = PreCfg<D, kOne>;
    extern __shared__ uint8_t smem_raw[];
    Smem sm;
    sm.ptr = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                        ~static_cast<uintptr_t>(1023));
    sm.base = smem_addr(sm.ptr);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm.ptr + C::kOffMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm.ptr + C::kOffMisc + 4);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the split-merging kernel that follows may be scheduled from here on
    grid_launch_dependents();
    if (threadIdx.x == 0) {
        mbar_init(sm.bar<D, kOne>(C::kBarQ), 1);
        for (int s = 0; s < C::kSlots; ++s) {
            mbar_init(sm.bar<D, kOne>(C::kBarFull + s), 1);
            mbar_init(sm.bar<D, kOne>(C::kBarEmpty + s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(sm.bar<D, kOne>(C::kBarS + b), 1);
            mbar_init(sm.bar<D, kOne>(C::kBarP + b), 128);
            mbar_init(sm.bar<D, kOne>(C::kBarO + b), 1);
        }
        mbar_init(sm.bar<D, kOne>(C::kBarVfix), 1);
        mbar_init(sm.bar<D, kOne>(C::kBarQFree), 1);
        mbar_init(sm.bar<D, kOne>(C::kBarDone), 1);
        for (int s = 0; s < kItemSlots; ++s) {
            mbar_init(sm.bar<D, kOne>(C::kBarItem + s), 1);
            mbar_init(sm.bar<D, kOne>(C::kBarItemFree + s), kItemReaders);
        }
        mbar_init(sm.bar<D, kOne>(C::kBarClc), 1);
        mbar_init(sm.bar<D, kOne>(C::kBarX), 128);
        mbar_init(sm.bar<D, kOne>(C::kBarXFree), 128);
        fence_mbar_init();
        *abort_flag = 0;
    }
    if (warp == 1) {
        tmem_alloc(smem_addr(tmem_slot), C::kTmemCols);
        tmem_relinquish();
    }
    FirstItem start;
    int u_early = 0;
    if (warp == 0) {
        if (lane == 0) {
            prefetch_tmap(&pool_map);
            prefetch_tmap(&qmap);
        }
        if (a.plan_ready) start.read(a, lane);
        if constexpr (kOne) {
            if (a.kv_early) {
                const Item it = make_item<kOne>(a, start.raw);
                u_early = early_loads<D, kOne>(&pool_map, a, sm, start, it, lane);
            }
        }
    }
    // Launched as a programmatic dependent: the set-up above overlapped the
    // preceding kernel's tail; the queries and the pool, and a plan that was
    // not on the device before that kernel, are read only from here on (but for
    // the first K/V tiles of early_loads).
    grid_dependency_wait();
    if (warp == 0) {
        if (!a.plan_ready) start.read(a, lane);
        if (lane == 0) {  // the thread that initialised the barriers
            *reinterpret_cast<int4*>(sm.ptr + C::kOffItems) = start.raw;
            mbar_arrive(sm.bar<D, kOne>(C::kBarItem));
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (warp == 0) {
        prefill_produce<D, kOne>(&pool_map, &qmap, a, sm, start, u_early, abort_flag, lane);
    } else if (warp == 1) {
        if (lane == 0) prefill_mma<D, kOne>(a, sm, tmem, abort_flag);
        __syncwarp();
    } else {
        const int t = (warp - 2) >> 2;
        SoftmaxPhase ph = {0, 0};
        bool ok;
        for (uint32_t k = 0;; ++k) {
            ok = __all_sync(0xffffffffu, item_wait<D, kOne>(sm, k, abort_flag));
            if (!ok) break;
            const int4 raw = item_read<D, kOne>(sm, k);
            if (raw.z < 0) break;
            const Item it = make_item<kOne>(a, raw);
            if (t == 0 || it.two || it.dual) {
                ok = prefill_softmax<D, kOne>(a, sm, tmem, t, k, ph, abort_flag, warp, lane);
                if (!ok) break;
            }
            ph.ub += 2 * raw.z;
            __syncwarp();
            if (lane == 0) item_free<D, kOne>(sm, k);
        }
        if (!ok && lane == 0) {
            if (!*abort_flag) set_error(a.err, kErrTimeout);
            *abort_flag = 1;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, C::kTmemCols);
    }
}

// Merges the key-range splits of each query row: weights 2^(lse_s - max).
// One warp per (split unit, row, 32 V columns); the lanes take the splits' log-
// sum-exps (up to 64 splits).  The partial outputs of the first U splits are
// loaded together with them, so a row of up to U splits costs one round trip;
// an empty split's partial (never written) is read but selected away.  The
// kernel lets the next one be scheduled at once: a next layer's prefill CTAs
// take the SMs as this layer's leave.
//
// What bounds it: the loads in flight.  Many rows of few splits (a split last
// round: 10,240 rows of 7) want many warps, each with a whole row in few
// registers (V = D / 32, U = 8); few rows of many splits (an 8-query call: 256
// rows of 19) one round trip, spread over the SMs (V = 2, U = 24).  With the
// second form for both, a turn with four layers of the former took 2,500 us
// instead of 2,484; with the first for both, an 8-query call needs three round
// trips for its 19 splits.
constexpr int kCombineThreads = 128;
constexpr int kCombineFew = 8;  // splits up to which the first form is used
template <int D, int V, int U>  // V: output elements per lane, U: splits per batch of loads
__global__ void __launch_bounds__(kCombineThreads, U > kCombineFew ? 6 : 8)
    sq_prefill_combine_kernel(const PrefillCombineArgs a) {
    constexpr int kParts = D / (32 * V);
    grid_launch_dependents();
    const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    constexpr int kRowsPerUnit = kPrefillQTiles * kPrefillRows;
    const int m = gw / (a.rows * kParts);
    if (m >= a.n_merges) return;
    const int tr = (gw / kParts) % a.rows, col = (gw % kParts) * 32 * V + lane * V;
    // the plan was uploaded before the prefill kernel started
    const PrefillMerge mg = a.merges[m];
    const int n_split = mg.n;
    const int t = tr / kPrefillRows, row = tr % kPrefillRows;
    const int qt = mg.unit / a.Hkv, g = mg.unit % a.Hkv;
    const int qi = (qt * kPrefillQTiles + t) * a.BP + row / a.G;
    // programmatic dependent of the prefill kernel: wait for its partials
    grid_dependency_wait();
    if (row >= a.BP * a.G || qi >= a.n_q) return;
    const int h = g * a.G + row % a.G;
    // partial row of split s: part0 + s * kRowsPerUnit
    const size_t part0 = ((size_t)mg.part0 * kPrefillQTiles + t) * kPrefillRows + row;
    const float ml0 = lane < n_split ? a.part_ml[part0 + (size_t)lane * kRowsPerUnit] : -INFINITY;
    const float ml1 =
        lane + 32 < n_split ? a.part_ml[part0 + (size_t)(lane + 32) * kRowsPerUnit] : -INFINITY;
    float vals[U][V];
    auto load = [&](int s0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int s = s0 + u;  // the same in every lane
            const float* po = a.part_o + (part0 + (size_t)s * kRowsPerUnit) * D + col;
#pragma unroll
            for (int e = 0; e < V; ++e) vals[u][e] = 0.f;
            if (s >= n_split) continue;
            if constexpr (V == 4) {
                const float4 v = *reinterpret_cast<const float4*>(po);
                vals[u][0] = v.x; vals[u][1] = v.y; vals[u][2] = v.z; vals[u][3] = v.w;
            } else {
                const float2 v = *reinterpret_cast<const float2*>(po);
                vals[u][0] = v.x; vals[u][1] = v.y;
            }
        }
    };
    load(0);
    float M = fmaxf(ml0, ml1);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
    float w0 = 0.f, w1 = 0.f;
    if (M != -INFINITY) {
        if (ml0 != -INFINITY) w0 = exp2f(ml0 - M);
        if (ml1 != -INFINITY) w1 = exp2f(ml1 - M);
    }
    float W = w0 + w1;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) W += __shfl_xor_sync(0xffffffffu, W, off);
    float acc[V] = {};
    for (int s0 = 0; W > 0.f && s0 < n_split; s0 += U) {
        if (s0 > 0) load(s0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int s = s0 + u;
            const float ws = __shfl_sync(0xffffffffu, s < 32 ? w0 : w1, s & 31);
            if (s < n_split && ws > 0.f) {
#pragma unroll
                for (int e = 0; e < V; ++e) acc[e] += ws * vals[u][e];
            }
        }
    }
    const float inv = W > 0.f ? 1.f / W : 0.f;
    const size_t o = ((size_t)qi * a.Hq + h) * D + col;
    if (a.out_f32) {
        float* out = reinterpret_cast<float*>(a.out) + o;
        if constexpr (V == 4)
            *reinterpret_cast<float4*>(out) =
                make_float4(acc[0] * inv, acc[1] * inv, acc[2] * inv, acc[3] * inv);
        else
            *reinterpret_cast<float2*>(out) = make_float2(acc[0] * inv, acc[1] * inv);
    } else {
        __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(a.out) + o;
        if constexpr (V == 4) {
            uint2 u;
            u.x = pack_bf16x2(acc[0] * inv, acc[1] * inv);
            u.y = pack_bf16x2(acc[2] * inv, acc[3] * inv);
            *reinterpret_cast<uint2*>(out) = u;
        } else {
            *reinterpret_cast<uint32_t*>(out) = pack_bf16x2(acc[0] * inv, acc[1] * inv);
        }
    }
    if (lane == 0 && col == 0 && a.lse)
        a.lse[(size_t)qi * a.Hq + h] = W > 0.f ? (M + __log2f(W)) * 0.69314718055994531f : -INFINITY;
}

}  // namespace
}  // namespace dev

template <int D>
static cudaError_t prepare() {
    cudaError_t e = cudaFuncSetAttribute(dev::sq_prefill_kernel<D, PrefillArgs>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         dev::PreCfg<D, false>::kSmemBytes);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(dev::sq_prefill_kernel<D, PrefillShortArgs>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             dev::PreCfg<D, true>::kSmemBytes);
    if (e != cudaSuccess) return e;
    // the same split of L1 and shared memory as the prefill kernel's: they take
    // turns on every SM
    e = cudaFuncSetAttribute(dev::sq_prefill_combine_kernel<D, 2, 24>,
                             cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(dev::sq_prefill_combine_kernel<D, D / 32, dev::kCombineFew>,
                                cudaFuncAttributePreferredSharedMemoryCarveout,
                                cudaSharedmemCarveoutMaxShared);
}

int prefill_smem_bytes(int D) {
    return D == 128 ? dev::PreCfg<128, false>::kSmemBytes : dev::PreCfg<64, false>::kSmemBytes;
}

cudaError_t prefill_prepare(int D) { return D == 128 ? prepare<128>() : prepare<64>(); }

cudaError_t launch_prefill(const CUtensorMap& pool_map, const CUtensorMap& qmap,
                           const PrefillShortArgs& a, int D, cudaStream_t st) {
    const unsigned grid = (unsigned)a.n_items;
    if (grid == 0) return cudaSuccess;
    // a programmatic dependent of whatever precedes it: its barrier and tensor
    // memory set-up overlaps that work's tail.  Before its wait it reads only a
    // plan that was on the device already (plan_ready), and, in the short
    // instance, keys and values that no running work writes (kv_early).
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    auto launch = [&](auto cfg_of, auto kernel, const auto& args) {
        using C = decltype(cfg_of);
        cfg.blockDim = dim3(C::kThreads);
        cfg.dynamicSmemBytes = C::kSmemBytes;
        return cudaLaunchKernelEx(&cfg, kernel, pool_map, qmap, args);
    };
    const PrefillArgs& base = a;
    const bool one = a.n_q <= a.BP;  // every query in tile a of the only CTA tile
    if (D == 128)
        return one ? launch(dev::PreCfg<128, true>{}, dev::sq_prefill_kernel<128, PrefillShortArgs>, a)
                   : launch(dev::PreCfg<128, false>{}, dev::sq_prefill_kernel<128, PrefillArgs>, base);
    return one ? launch(dev::PreCfg<64, true>{}, dev::sq_prefill_kernel<64, PrefillShortArgs>, a)
               : launch(dev::PreCfg<64, false>{}, dev::sq_prefill_kernel<64, PrefillArgs>, base);
}

cudaError_t launch_prefill_combine(const PrefillCombineArgs& a, int D, cudaStream_t st) {
    const bool few = a.max_splits <= dev::kCombineFew;
    const int64_t warps = (int64_t)a.n_merges * a.rows * (few ? 1 : D / 64);
    const int per = dev::kCombineThreads / 32;
    const unsigned grid = (unsigned)((warps + per - 1) / per);
    if (grid == 0) return cudaSuccess;
    // scheduled while the prefill kernel's last CTAs run; waits for them
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(dev::kCombineThreads);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    constexpr int kF = dev::kCombineFew;
    if (D == 128)
        return few ? cudaLaunchKernelEx(&cfg, dev::sq_prefill_combine_kernel<128, 4, kF>, a)
                   : cudaLaunchKernelEx(&cfg, dev::sq_prefill_combine_kernel<128, 2, 24>, a);
    return few ? cudaLaunchKernelEx(&cfg, dev::sq_prefill_combine_kernel<64, 2, kF>, a)
               : cudaLaunchKernelEx(&cfg, dev::sq_prefill_combine_kernel<64, 2, 24>, a);
}

}  // namespace sq
