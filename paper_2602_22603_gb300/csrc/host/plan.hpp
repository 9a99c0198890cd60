// Plain-old-data work descriptions the host planners write and the kernels
// read.  Shared by host code (C++) and device code (CUDA); no CUDA types.
#pragma once
#include <stdint.h>

#if defined(__CUDACC__)
#define SQ_HOST_DEVICE __host__ __device__
#else
#define SQ_HOST_DEVICE
#endif

namespace sq {

// Rows of one tensor-core tile: the query rows a decode work item serves
// (Sec. 2.1: a KV head is shared by G query heads; with several sequences
// sharing the same pages, their query groups stack up to this many rows).
constexpr int kRowsPerTile = 16;
// Tokens of K/V one pipeline stage of the decode kernel holds.
constexpr int kStageTokens = 64;
// Consumer warps of the decode kernel: two groups that take alternate stages,
// four warps each, kStageTokens / 4 tokens of a stage per warp.
constexpr int kDecodeGroups = 2;
constexpr int kDecodeConsumerWarps = 4 * kDecodeGroups;
// Fixed cost of starting a work unit, in stages: its query reload and its
// item-end merge.  The planner balances stages plus this cost per unit, so a
// CTA that gets many short units (e.g. the few-token tails of several forks)
// is not the one every other CTA waits for.  A stage passes in 0.7 us; a unit's
// start and end hide behind the stages of its neighbours unless it is a stage
// or two long.  Measured, us per pass for costs (2, 2) (4, 4) (4, 8) (6, 6):
// 36 short sequences x 8 layers 379 376 376 383; four agents with forks and
// their one-stage tails x 8 layers 384 377 371 372; an agent turn 2,624 2,549
// 2,514 2,513; one 32k sequence x 32 layers 809 805 805 802.
constexpr int kShortUnitStages = 2;
constexpr int kDecodeUnitCost = 4;
constexpr int kDecodeShortUnitCost = 8;

// The arrival word of a (sequence, KV head) run of n entries: one claim (1) for
// each, and one release (kArriveRelease) for each but the last to claim, which
// merges the run.
constexpr uint32_t kArriveRelease = 0x10000u;
// Whether a word counts the releases of all the other entries.
SQ_HOST_DEVICE constexpr bool arrive_complete(uint32_t word, uint32_t n) {
    return word >> 16 == n - 1;
}
// What the merger adds when it leaves: it takes back every claim and release of
// the run, also the releases that come after it (its wait for them is bounded),
// so that the word is zero when the call is done.
SQ_HOST_DEVICE constexpr uint32_t arrive_settle(uint32_t n) {
    return 0u - (n + (n - 1) * kArriveRelease);
}

// A run of logical pages read once for a group of sequences that hold the
// same physical pages there (a main thread and its forks, Sec. 3.4).
struct DecodeSeg {
    int32_t page_off;                 // into DecodePlan page_ids
    int32_t n_pages;                  // pages in the run
    int32_t n_tok;                    // tokens to read (max over the group)
    int32_t n_grp;                    // sequences in the group
    int32_t grp_seq[kRowsPerTile];    // call-local sequence indices
    int32_t grp_lim[kRowsPerTile];    // valid tokens of each, from the run start
    int32_t q0;                       // page index of the run's first page in its members
    int32_t tail;                     // bit j: the run holds member j's last page (the
                                      // others' limit is the whole run)
};

// A contiguous range of stages of one (segment, KV head) — one partial result
// per group member.  Member j's G rows go to partial entry ent[j]; the entries
// of one (sequence, KV head) are contiguous, so that its merge reads them
// without an index.  A member whose (sequence, KV head) has this one entry
// only (bit j of `sole`) gets its normalised output written directly.
struct DecodeItem {
    int32_t seg;
    int32_t head;
    int32_t s0, s1;                   // stages [s0, s1)
    int32_t sole;                     // bit j: member j's run is this item alone
    int32_t ent[kRowsPerTile];        // partial entry of each group member (n_grp used)
};

// Eviction compaction, planned once per eviction and shared by every
// (layer, K/V, head) plane: destination tiles (contiguous rows of one page, in
// increasing logical order) and, per tile, the contiguous source pieces that
// fill it.  A tile without pieces writes zeros (the unused slots of a page
// that a ragged eviction leaves partial).
struct EvictTile {
    int32_t dst_page;
    int32_t dst_slot;     // first destination slot in the page
    int32_t n_rows;       // rows written (<= tile capacity)
    int32_t piece_begin;  // pieces [piece_begin, next tile's piece_begin); none: zero rows
};

struct EvictPiece {
    int32_t src_page;
    int32_t src_slot;
    int32_t n_rows;
    int32_t dst_row;      // row offset inside the tile
};

// Masked prefill attention (Algorithm 2, BuildMask).  A query tile holds
// kPrefillRows rows: floor(kPrefillRows / G) consecutive query positions times
// the G query heads of one KV head (Sec. 2.1), so one K/V tile serves them all.
// Keys are taken kPrefillKeys at a time, aligned to kPrefillKeys.
constexpr int kPrefillRows = 128;
constexpr int kPrefillKeys = 128;
// Query tiles one CTA owns; they share every K/V tile it loads.
constexpr int kPrefillQTiles = 2;
constexpr int32_t kPrefillTileFull = 1;  // every key of the tile exists and is visible

// One key tile that holds at least one visible key of the sequence: two
// halves of 64 keys, each 64 consecutive positions starting at a multiple of
// 64 (key0, key0b).  With pages of >= 64 tokens the halves are the visible
// 64-key boxes of the sequence taken two by two, so a box that a span covers
// entirely is skipped even when its neighbour is not; with smaller pages the
// tile is 128 aligned keys (key0b = key0 + 64).  A missing second half has
// key0b = kPrefillNoKeys (past any sequence).
constexpr int32_t kPrefillNoKeys = 0x7fffffc0;
struct PrefillTile {
    int32_t key0;      // first key of the lower half
    int32_t flags;     // kPrefillTileFull or 0
    uint32_t vis[4];   // bit c of word w: key (w < 2 ? key0 : key0b) + 32 (w % 2) + c
                       // exists and lies in no span
    int32_t key0b;     // first key of the upper half
    int32_t pad;
};

// One work item of the prefill kernel: key tiles [t0, t0 + n_tiles) of one
// query unit (the two query tiles of CTA tile unit / Hkv at KV head
// unit % Hkv).  A unit of several items leaves normalised partial results in
// entry `part` (-1: its only item, written to the outputs).
struct PrefillItem {
    int32_t unit;
    int32_t t0;
    int32_t n_tiles;
    int32_t part;
};

// A unit whose items' partial results [part0, part0 + n) are merged.
struct PrefillMerge {
    int32_t unit;
    int32_t part0;
    int32_t n;
    int32_t pad;
};
// Partial results one unit may have at most (a lane of the merge takes two).
constexpr int32_t kPrefillMaxSplit = 64;
// Bytes of one partial result (normalised outputs and log-sum-exps of the rows
// of a unit, fp32), and of all that a plan may have: they are held for the
// cache's life.  The limit is 1,016 partial results at d = 128.  By the planner's
// model of the time, over 600 shapes drawn from 4k to 256k tokens and 8 to 16k
// queries, it costs 11 of them up to 1.7% (unlimited, one wanted 2,272, 300 MB);
// half of it would cost 49 of them up to 22%, such as 120 units whose five key
// ranges each fill four rounds.
constexpr int64_t prefill_part_bytes(int32_t D) {
    return (int64_t)kPrefillQTiles * kPrefillRows * (D + 1) * (int64_t)sizeof(float);
}
constexpr int64_t kPrefillPartLimit = int64_t(128) << 20;

// Byte offsets of the arrays of a decode plan inside one upload buffer.
// Byte offsets of the serialised decode plan.  `arrive` holds one 32-bit
// arrival count per (sequence, KV head), zero in the serialised plan; the
// kernel counts on it and leaves it at zero again.
// `page_fill` is -1 when the plan carries no page fills.
struct DecodePlanLayout {
    int64_t segs, items, cta_begin, page_ids, comb_off, arrive, page_fill, total;
    int32_t n_segs, n_items, n_ctas, n_page_ids, n_comb_keys, n_comb_ent;
};

}  // namespace sq
