// Split-K flash-decoding over the paged bf16 KV pool, with the log-sum-exp
// merge of its partial results in the same kernel.
//
// What is computed (Sec. 1 and Sec. 3.4: for every generated token,
// attention reads the whole KV cache of the context; Sec. 2.1: in
// grouped-query attention a K/V head serves G query heads): for sequence i,
// query head h and KV head g = h / G,
//     out[i][h] = sum_t softmax_t(sm_scale * q[i][h] . K_g[t]) V_g[t].
//
// Work decomposition (host planner, core.cpp): every run of pages that a
// group of sequences holds in common (a main thread and its forked auxiliary
// threads, Sec. 3.4) is one segment; a (segment, KV head) pair is a list of
// 64-token stages; the stages of all pairs are dealt evenly to persistent
// CTAs, one per SM.
//
// A CTA has two consumer groups of four warps, each with a producer warp and a
// TMA + mbarrier ring of its own (2 x 96 KiB in flight per SM); the groups take
// alternate stages.  A consumer warp owns 16 tokens of a stage and keeps an
// online-softmax partial (max, sum, unnormalised output) for up to 16 query
// rows - the G heads of every sequence in the segment's group, so a shared page
// is read from HBM once for all of them.  At an item's end the consumers leave
// their rows in shared memory and go on; two closing warps add them, write the
// item's partial and merge what it completes.
//
// What bounds it: HBM in long calls (the read probe's rate at 128k); in short
// ones the chain after the last stage (add, partial, arrival, merge: 5 us from
// the slowest CTA's last stage to the next call's start) and the SMs' unequal
// shares of HBM (2 us between most and the slowest).  Two CTAs per SM with the
// same ring space, each closing its items itself, left twice the entries per
// run and stalled at every item's end.  Per call at 32q/8kv, d = 128, so and
// now: one sequence of 32,768 tokens 27.5 and 24.6 us, 36 sequences of 250 ..
// 6,000 tokens 51.4 and 46.4 us, four agents and their forks at 20,000 ..
// 60,000 tokens with partial pages 54.6 and 45.6 us; eight of 131,072 and their
// forks 600 us either way.  Prefetching stages past the ring into L2 while the
// previous call ends gains nothing: 6 instead of 4 stages 795 -> 810 us for 32
// layers of the 32k sequence.
//
// Merge: an item leaves one partial (max, sum, unnormalised output) per group
// member, in that (sequence, KV head)'s contiguous run of entries; a member
// whose run is this one item gets its normalised output directly.  After an
// item a CTA counts its arrival on each of the item's runs; the CTA that brings
// a count to the number of entries merges that run (max of the maxima, weights
// 2^(m - M)) and writes the normalised output.  Counts are zero in every
// uploaded plan and the merger resets its count, so every call starts from
// zero.
//
// Start-up: the kernel is a programmatic dependent of whatever precedes it.
// When the plan was already on the device (a reused plan), every role reads its
// first items before the dependency wait, and stages in pages that no running
// work writes are loaded before it.
//
// Page fills: after a ragged eviction a page may hold fewer rows than it has
// slots (its rows first, then zeros or rows once appended).  Stages are in
// slot space (page index x P + slot); the plan then carries every page's
// fill, and the rows past a page's fill get no weight.
//
// Tensor cores: S = Q K^T and O += P V are m16n8k16 bf16 mma.sync with fp32
// accumulation; rows = query rows (<= 16), columns = tokens / head dims.  The
// contraction is tiny (G x d per token) and the kernel is HBM-bound, so the
// warp-level mma is the right size: the point is to keep HBM busy.
#include <math.h>

#include "launch.hpp"
#include "ptx.cuh"

namespace sq {
namespace {

using namespace dev;

template <int D>
struct DecCfg {
    static constexpr int kColBlocks = D / 64;                    // 128-byte column blocks
    static constexpr int kBlockBytes = kStageTokens * 128;       // one column block of a tile
    static constexpr int kTileBytes = kColBlocks * kBlockBytes;  // K (or V) of one stage
    static constexpr int kStageBytes = 2 * kTileBytes;
    static constexpr int kStages = (D == 128) ? 3 : 6;           // per group: 96 KiB in flight
    static constexpr int kConsumers = kDecodeConsumerWarps * 32;
    static constexpr int kRingBytes = kDecodeGroups * kStages * kStageBytes;
    // warps: consumers, a producer per group, two that close items
    static constexpr int kClosers = 64;
    static constexpr int kThreads = kConsumers + kDecodeGroups * 32 + kClosers;
    static constexpr int kOffBars = kRingBytes;
    // barriers: per group full [kStages], empty [kStages]; then the three of the
    // items' ends; then the abort flag
    static constexpr int kBarOut = kDecodeGroups * 2 * kStages;  // a pass's rows are written
    static constexpr int kBarOutFree = kBarOut + 1;              // ... and read
    static constexpr int kBarRuns = kBarOut + 2;                 // the last item's runs are listed
    static constexpr int kOffRed = kOffBars + 256;
    // item ends: per-warp row max / sum, eight rows of every warp's output, and
    // the runs an item completed
    static constexpr int kPassRows = 8;
    static constexpr int kOffRuns = kOffRed + 2 * kDecodeConsumerWarps * kRowsPerTile * 4;
    static constexpr int kOffOut = kOffRuns + 256;
    static constexpr int kOutBytes = kDecodeConsumerWarps * kPassRows * D * 4;
    static constexpr int kSmemBytes = kOffOut + kOutBytes + 1024;  // + alignment slack
    static constexpr int kNT = D / 8;   // 8-wide output column tiles
    static constexpr int kKS = D / 16;  // 16-deep contraction steps
    static_assert(kSmemBytes <= 232448 && kOffOut % 16 == 0, "shared memory");
    static_assert((kBarRuns + 1) * 8 + 4 <= 256, "mbarriers");
};

__device__ __forceinline__ uint32_t ld_u32(const __nv_bfloat16* p) {
    return *reinterpret_cast<const uint32_t*>(p);
}

// Sum of the two bf16 halves of a packed pair, in fp32.
__device__ __forceinline__ float bf16x2_sum(uint32_t v) {
    return __uint_as_float(v << 16) + __uint_as_float(v & 0xffff0000u);
}

// ---- producers: one warp per group issues the TMA loads of its stages --------
// The groups take alternate stages of the CTA, each through a ring of its own.
// The warp walks its stages in order; the page of the next stage is read while
// the current one waits for its slot.  Whole-page stages (P >= 64) are issued by
// lane 0; with smaller pages each lane issues one box (page, column block, K or
// V).
template <int D>
struct Producer {
    using C = DecCfg<D>;
    const CUtensorMap* tmap;
    const DecodeArgs& a;
    uint8_t* ring;      // the group's slots
    uint64_t* bars;     // the group's barriers: full [kStages], empty [kStages]
    volatile int* abort_flag;
    int group, lane;
    // this lane's box within a stage of small pages
    int box_page, box_cb, box_kv;
    // the current stage: stage s of item it (it0 .. it1), and its lane's page
    int it, it1, s, s1, head, page_off, n_pages;
    int32_t pid;      // -1: no box for this lane
    int slot;
    uint32_t phase;   // parity of the slot's use
    uint32_t issued, issued_phase;  // per-slot bits of the last issue
    bool first;       // the CTA's first stage has not gone out yet

    __device__ void init() {
        box_cb = lane % C::kColBlocks;
        box_kv = (lane / C::kColBlocks) % 2;
        box_page = a.P < kStageTokens ? lane / (2 * C::kColBlocks) : 0;
        it = a.cta_begin[blockIdx.x];
        it1 = a.cta_begin[blockIdx.x + 1];
        slot = 0;
        phase = 0;
        issued = issued_phase = 0;
        first = group == 0;
        if (it < it1) {
            open_item();
            s += group;
            settle();
        }
    }
    __device__ bool more() const { return it < it1; }
    __device__ void open_item() {
        const DecodeItem* item = a.items + it;
        const DecodeSeg* seg = a.segs + item->seg;
        s = item->s0;
        s1 = item->s1;
        head = item->head;
        page_off = seg->page_off;
        n_pages = seg->n_pages;
    }
    // Carries a stage past the item's end into the items that follow.
    __device__ void settle() {
        while (s >= s1) {
            const int over = s - s1;
            if (++it == it1) return;
            open_item();
            s += over;
        }
        const int pi = s * kStageTokens / a.P + box_page;
        const int per = a.P < kStageTokens ? kStageTokens / a.P : 1;
        pid = box_page < per && pi < n_pages ? a.page_ids[page_off + pi] : -1;
    }
    __device__ int row(int kv) const {
        const int row0 = a.P > kStageTokens ? (s * kStageTokens) & (a.P - 1) : 0;
        return (kv ? a.Hkv + head : head) * a.P + row0;
    }
    __device__ void advance() {
        first = false;
        if (++slot == C::kStages) {
            slot = 0;
            phase ^= 1;
        }
        s += kDecodeGroups;
        settle();
    }
    // Issues the current stage into its (free) slot.
    __device__ void issue() {
        const uint32_t full = smem_addr(&bars[slot]);
        const uint32_t dst = smem_addr(ring) + slot * C::kStageBytes;
        if (a.P >= kStageTokens) {
            if (lane == 0) {
                if ((uint32_t)pid < (uint32_t)a.num_pages) {
                    mbar_arrive_expect_tx(full, C::kStageBytes);
                    const int rk = row(0), rv = row(1);
#pragma unroll
                    for (int cb = 0; cb < C::kColBlocks; ++cb) {
                        tma_load_4d(dst + cb * C::kBlockBytes, tmap, full, cb * 64, rk, pid, a.layer);
                        tma_load_4d(dst + cb * C::kBlockBytes + C::kTileBytes, tmap, full, cb * 64, rv,
                                    pid, a.layer);
                    }
                } else {
                    set_error(a.err, kErrBounds);
                    mbar_arrive(full);
                }
            }
        } else {
            const bool valid = pid >= 0 && pid < a.num_pages;
            if (pid < -1 || pid >= a.num_pages) set_error(a.err, kErrBounds);
            const uint32_t n = __popc(__ballot_sync(0xffffffffu, valid));
            if (lane == 0) {
                if (n) mbar_arrive_expect_tx(full, n * a.P * 128u);
                else mbar_arrive(full);
            }
            __syncwarp();
            if (valid)
                tma_load_4d(dst + box_kv * C::kTileBytes + box_cb * C::kBlockBytes +
                                box_page * a.P * 128,
                            tmap, full, box_cb * 64, row(box_kv), pid, a.layer);
        }
        issued |= 1u << slot;
        issued_phase = (issued_phase & ~(1u << slot)) | (phase << slot);
    }
    // Before the grid-dependency wait (a plan that was on the device): stages in
    // pages that no running work writes are loaded, up to the ring's depth, and
    // the first few of the others prefetched into L2.
    __device__ void early() {
        if ((int)blockIdx.x == a.debug_drop_cta) return;
        int n = 0;
        if (a.kv_early && a.P >= kStageTokens) {
            for (; n < C::kStages && more(); ++n) {
                bool unsafe = false;
                for (int u = lane; u < a.n_unsafe; u += 32) unsafe |= a.unsafe[u] == pid;
                if (__any_sync(0xffffffffu, unsafe)) break;
                issue();
                advance();
            }
        }
        // (the walk goes on from here after the wait: look ahead on a copy)
        Producer ahead = *this;
        for (; n < kPrefetchStages && ahead.more(); ++n) {
            if (ahead.pid >= 0 && ahead.pid < a.num_pages && (a.P < kStageTokens || lane < 2 * C::kColBlocks))
                tma_prefetch_l2_4d(tmap, box_cb * 64, ahead.row(box_kv), ahead.pid, a.layer);
            ahead.advance();
        }
    }
    static constexpr int kPrefetchStages = 4;
    __device__ void run() {
        bool ok = true;
        while (more()) {
            const uint32_t empty = smem_addr(&bars[C::kStages + slot]);
            ok = __all_sync(0xffffffffu, mbar_wait(empty, phase ^ 1, abort_flag));
            if (!ok) break;
            // test hook: leave this stage unsignalled (the consumers' bounded wait
            // runs out; nothing is in flight for it)
            if (!(first && (int)blockIdx.x == a.debug_drop_cta)) issue();
            advance();
        }
        if (!ok && lane == 0) {
            if (!*abort_flag) set_error(a.err, kErrTimeout);
            *abort_flag = 1;
            // Leave only after every copy already issued has landed (bounded).
            for (int sl = 0; sl < C::kStages; ++sl)
                if ((issued >> sl) & 1u)
                    mbar_wait(smem_addr(&bars[sl]), (issued_phase >> sl) & 1u);
        }
        __syncwarp();
    }
};

// ---- consumers: two groups of four warps, 16 tokens of a stage per warp ------
// The groups take alternate stages of the CTA.  Every consumer warp runs every
// item and reaches every named barrier of every item, also after a wait ran
// out (it then skips the work only), so the barriers never miss a participant.

// What a consumer lane needs of an item before its first stage; read one item
// ahead.  (The token count and the members' limits are not among it: an append
// may rewrite them in a plan that is on the device, so they are read after the
// dependency wait.)
struct ItemHead {
    int seg, head, s0, s1, n_grp, seq0, seq1;
    __device__ void read(const DecodeArgs& a, int it, int j0, int j1) {
        const DecodeItem* item = a.items + it;
        seg = item->seg;
        head = item->head;
        s0 = item->s0;
        s1 = item->s1;
        const DecodeSeg* sg = a.segs + seg;
        n_grp = sg->n_grp;
        seq0 = sg->grp_seq[j0];  // (entries past n_grp are zero)
        seq1 = sg->grp_seq[j1];
    }
};

// One fp32 row of the item-end merge: eight-float blocks XORed with the row, so
// that the eight rows of a warp's store hit different banks.
template <int D>
__device__ __forceinline__ int out_pos(int row, int col) {
    return row * D + ((((col >> 3) ^ row) & (D / 8 - 1)) << 3) + (col & 7);
}

// Four consecutive output elements from element `at`: v * inv.
__device__ __forceinline__ void write_out(const DecodeArgs& a, size_t at, const float4& v, float inv) {
    if (a.out_f32) {
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(a.out) + at) =
            make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
    } else {
        uint2 u;
        u.x = pack_bf16x2(v.x * inv, v.y * inv);
        u.y = pack_bf16x2(v.z * inv, v.w * inv);
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(a.out) + at) = u;
    }
}

// Adds the consumer warps' rows rb .. rb + 7 of an item (weights 2^(m_w - M),
// warps in order) and writes its partials or outputs: `n` threads, `v0` = which.
template <int D>
__device__ __forceinline__ void close_rows(const DecodeArgs& a, const DecodeItem* item,
                                           const DecodeSeg* seg, int head, int sole, int rows, int rb,
                                           const uint8_t* smem, int v0, int n) {
    using C = DecCfg<D>;
    constexpr int kVec = D / 4;  // float4 per output row
    const int G = a.G;
    const float* red_m = reinterpret_cast<const float*>(smem + C::kOffRed);
    const float* red_l = red_m + kDecodeConsumerWarps * kRowsPerTile;
    const float* red_o = reinterpret_cast<const float*>(smem + C::kOffOut);
    const int n_out = min(rows - rb, (int)C::kPassRows) * kVec;
    for (int v = v0; v < n_out; v += n) {
        const int pr = v / kVec, c4 = v % kVec, r = rb + pr, j = r / G;
        // a member whose run is this item alone gets its normalised output
        const bool alone = (sole >> j) & 1;
        const int to = alone ? seg->grp_seq[j] : item->ent[j];
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < kDecodeConsumerWarps; ++w) M = fmaxf(M, red_m[w * kRowsPerTile + r]);
        const float Ms = M == -INFINITY ? 0.f : M;
        float L = 0.f;
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < kDecodeConsumerWarps; ++w) {
            const float f = exp2f(red_m[w * kRowsPerTile + r] - Ms);
            L += red_l[w * kRowsPerTile + r] * f;
            const float4 x =
                *reinterpret_cast<const float4*>(red_o + w * C::kPassRows * D + out_pos<D>(pr, c4 * 4));
            sum.x += x.x * f; sum.y += x.y * f; sum.z += x.z * f; sum.w += x.w * f;
        }
        if (alone) {
            write_out(a, ((size_t)to * a.Hq + head * G + r % G) * D + c4 * 4, sum, 1.f / L);
        } else {
            const size_t pe = (size_t)to * G + r % G;
            *reinterpret_cast<float4*>(a.part_o + pe * D + c4 * 4) = sum;
            if (c4 == 0)
                *reinterpret_cast<float4*>(a.part_ml + pe * 4) = make_float4(M, L, 0.f, 0.f);
        }
    }
}

template <int D>
__device__ void consume(const DecodeArgs& a, int it0, int it1, ItemHead next, uint8_t* smem,
                        uint64_t* all_bars, volatile int* abort_flag, int warp, int lane) {
    using C = DecCfg<D>;
    const int gid = lane >> 2, tig = lane & 3;
    const int r0 = gid, r1 = gid + 8;
    const int mi = lane >> 3, rr = lane & 7;
    const int group = warp >> 2, w4 = warp & 3;
    const int G = a.G;
    const int j0 = r0 / G, j1 = r1 / G;
    uint64_t* bars = all_bars + group * 2 * C::kStages;
    float* red_m = reinterpret_cast<float*>(smem + C::kOffRed);     // [8][16]
    float* red_l = red_m + kDecodeConsumerWarps * kRowsPerTile;     // [8][16]
    float* red_o = reinterpret_cast<float*>(smem + C::kOffOut);     // [8][8][D], out_pos
    uint32_t n_pass = 0;  // item-end passes so far
    uint8_t* ring = smem + group * C::kStages * C::kStageBytes;  // the group's slots
    int slot = 0;
    uint32_t phase = 0;
    int skip = group;   // stages to the group's next one
    bool dead = false;  // warp-uniform: a wait ran out or the CTA aborted
    for (int it = it0; it < it1; ++it) {
        const ItemHead item = next;
        const DecodeSeg* seg = a.segs + item.seg;
        const int n_grp = item.n_grp;
        const bool v0 = j0 < n_grp, v1 = j1 < n_grp;
        const int lim0 = v0 ? seg->grp_lim[j0] : 0;
        const int lim1 = v1 ? seg->grp_lim[j1] : 0;
        const int n_tok = seg->n_tok;

        uint32_t qa[C::kKS][4];
        {
            const __nv_bfloat16* q0 =
                a.q + ((size_t)(v0 ? item.seq0 : 0) * a.Hq + item.head * G + r0 % G) * D;
            const __nv_bfloat16* q1 =
                a.q + ((size_t)(v1 ? item.seq1 : 0) * a.Hq + item.head * G + r1 % G) * D;
#pragma unroll
            for (int kk = 0; kk < C::kKS; ++kk) {
                const int c = kk * 16 + tig * 2;
                qa[kk][0] = v0 ? ld_u32(q0 + c) : 0u;
                qa[kk][1] = v1 ? ld_u32(q1 + c) : 0u;
                qa[kk][2] = v0 ? ld_u32(q0 + c + 8) : 0u;
                qa[kk][3] = v1 ? ld_u32(q1 + c + 8) : 0u;
            }
        }
        if (it + 1 < it1) next.read(a, it + 1, j0, j1);
        float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
        float o[C::kNT][4];
#pragma unroll
        for (int nd = 0; nd < C::kNT; ++nd) o[nd][0] = o[nd][1] = o[nd][2] = o[nd][3] = 0.f;

        int s = item.s0 + skip;
        for (; s < item.s1; s += kDecodeGroups) {
            const uint32_t full = smem_addr(&bars[slot]);
            const uint32_t empty = smem_addr(&bars[C::kStages + slot]);
            // Pages a ragged eviction left partial: bit r of vm says whether
            // row r of this warp's 16 holds a row of its page (read before
            // the wait, off the critical path).  The unused slots hold zeros
            // or rows once appended, so only their scores are masked.
            uint32_t vm = 0xffffu;
            if (a.page_fill) {
                // P is a power of two >= 8 and the 16 rows start at a multiple
                // of 16: one page holds them all (P >= 16), or two (P = 8)
                const int P = a.P;
                const int t0 = s * kStageTokens + w4 * 16;  // segment slot position
                const int pq = t0 >> (__ffs(P) - 1);
                const int f0 = pq < seg->n_pages ? __ldg(&a.page_fill[seg->page_off + pq]) : 0;
                if (P >= 16) {
                    const int v = min(max(f0 - (t0 & (P - 1)), 0), 16);
                    vm = (uint32_t)((1u << v) - 1u);   // v = 16 gives 0xffff
                } else {
                    const int f1 =
                        pq + 1 < seg->n_pages ? __ldg(&a.page_fill[seg->page_off + pq + 1]) : 0;
                    vm = ((1u << min(f0, 8)) - 1u) | (((1u << min(f1, 8)) - 1u) << 8);
                }
            }
            if (!dead) {
                const bool ok = mbar_wait(full, phase, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) {
                    if (lane == 0 && !*abort_flag) set_error(a.err, kErrTimeout);
                    *abort_flag = 1;
                    dead = true;
                }
            }
            if (!dead) {
                const uint32_t kb = smem_addr(ring + slot * C::kStageBytes);
                const uint32_t vb = kb + C::kTileBytes;
                const int tbase = s * kStageTokens + w4 * 16;  // segment-relative

                // S = Q K^T over this warp's 16 tokens (two n8 tiles)
                float sc[2][4];
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
                {
                    const int t = w4 * 16 + (mi >> 1) * 8 + rr;
                    const uint32_t row = kb + t * 128;
                    const int sw = t & 7;
#pragma unroll
                    for (int kk = 0; kk < C::kKS; ++kk) {
                        const int d0 = kk * 16 + (mi & 1) * 8;
                        uint32_t b0, b1, b2, b3;
                        ldsm_x4(row + (d0 >> 6) * C::kBlockBytes + ((((d0 & 63) >> 3) ^ sw) << 4), b0,
                                b1, b2, b3);
                        mma_bf16(sc[0], qa[kk], b0, b1);
                        mma_bf16(sc[1], qa[kk], b2, b3);
                    }
                }

                // masking, scaling, online softmax (log2 domain)
                float x[2][4];
                float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int tk = tbase + nt * 8 + tig * 2 + e;
                        const bool rv = (vm >> (nt * 8 + tig * 2 + e)) & 1u;
                        x[nt][e] = tk < lim0 && rv ? sc[nt][e] * a.scale_log2 : -INFINITY;
                        x[nt][2 + e] = tk < lim1 && rv ? sc[nt][2 + e] * a.scale_log2 : -INFINITY;
                        mx0 = fmaxf(mx0, x[nt][e]);
                        mx1 = fmaxf(mx1, x[nt][2 + e]);
                    }
                mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
                mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
                mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
                mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
                const float mn0 = fmaxf(m0, mx0), mn1 = fmaxf(m1, mx1);
                const float ms0 = mn0 == -INFINITY ? 0.f : mn0;
                const float ms1 = mn1 == -INFINITY ? 0.f : mn1;
                const float al0 = exp2f(m0 - ms0), al1 = exp2f(m1 - ms1);
                m0 = mn0;
                m1 = mn1;
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        x[nt][e] = exp2f(x[nt][e] - ms0);
                        x[nt][2 + e] = exp2f(x[nt][2 + e] - ms1);
                    }
                // P in bf16 for the PV product; the normaliser sums the same
                // rounded weights, so the output is an exact convex combination
                uint32_t pa[4];
                pa[0] = pack_bf16x2(x[0][0], x[0][1]);
                pa[1] = pack_bf16x2(x[0][2], x[0][3]);
                pa[2] = pack_bf16x2(x[1][0], x[1][1]);
                pa[3] = pack_bf16x2(x[1][2], x[1][3]);
                const float ps0 = bf16x2_sum(pa[0]) + bf16x2_sum(pa[2]);
                const float ps1 = bf16x2_sum(pa[1]) + bf16x2_sum(pa[3]);
                l0 = l0 * al0 + ps0;
                l1 = l1 * al1 + ps1;
#pragma unroll
                for (int nd = 0; nd < C::kNT; ++nd) {
                    o[nd][0] *= al0;
                    o[nd][1] *= al0;
                    o[nd][2] *= al1;
                    o[nd][3] *= al1;
                }

                // Rows past the last valid token hold stale or never-written
                // shared memory: zero this warp's such V rows so 0 * V stays 0.
                const bool tail = tbase + 16 > n_tok;
                if (tail) {
                    const int first = max(0, n_tok - tbase);
                    const int per_row = C::kColBlocks * 8;  // 16-byte chunks per row
                    const int total = (16 - first) * per_row;
                    uint8_t* vgen = ring + slot * C::kStageBytes + C::kTileBytes;
                    for (int idx = lane; idx < total; idx += 32) {
                        const int row = w4 * 16 + first + idx / per_row;
                        const int rem = idx % per_row;
                        *reinterpret_cast<uint4*>(vgen + (rem >> 3) * C::kBlockBytes + row * 128 +
                                                  (rem & 7) * 16) = make_uint4(0, 0, 0, 0);
                    }
                    __syncwarp();
                }

                // O += P V (V^T fragments through ldmatrix.trans)
                {
                    const int t = w4 * 16 + (mi & 1) * 8 + rr;
                    const uint32_t row = vb + t * 128;
                    const int sw = t & 7;
#pragma unroll
                    for (int nd2 = 0; nd2 < C::kKS; ++nd2) {
                        const int d0 = nd2 * 16 + (mi >> 1) * 8;
                        uint32_t b0, b1, b2, b3;
                        ldsm_x4_trans(row + (d0 >> 6) * C::kBlockBytes + ((((d0 & 63) >> 3) ^ sw) << 4),
                                      b0, b1, b2, b3);
                        mma_bf16(o[2 * nd2], pa, b0, b1);
                        mma_bf16(o[2 * nd2 + 1], pa, b2, b3);
                    }
                }
                if (tail) fence_proxy_async_smem();  // generic writes before the next TMA fill
                __syncwarp();
                if (lane == 0) mbar_arrive(empty);
            }
            if (++slot == C::kStages) {
                slot = 0;
                phase ^= 1;
            }
        }
        skip = s - item.s1;

        // Leave the item's rows to the closing warps, eight at a time, and go on
        // with the next item: nothing here waits for the other consumers.
        l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
        l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
        l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
        l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
        const int rows = n_grp * G;
        const bool last = it + 1 == it1;
        for (int rb = 0; rb < rows; rb += C::kPassRows, ++n_pass) {
            // the previous pass's rows have been read
            if (!dead && n_pass > 0 && !(last && rb > 0)) {
                const bool ok =
                    mbar_wait(smem_addr(&all_bars[C::kBarOutFree]), (n_pass - 1) & 1, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) {
                    if (lane == 0 && !*abort_flag) set_error(a.err, kErrTimeout);
                    *abort_flag = 1;
                    dead = true;
                }
            }
            if (dead && !last) continue;
            const int r = rb + gid;  // this lane's row of the pass: r0, then r1
            if (tig == 0) {
                red_m[warp * kRowsPerTile + r] = rb ? m1 : m0;
                red_l[warp * kRowsPerTile + r] = rb ? l1 : l0;
            }
            if (r < rows) {
                float* wo = red_o + warp * C::kPassRows * D;
#pragma unroll
                for (int nd = 0; nd < C::kNT; ++nd)
                    *reinterpret_cast<float2*>(wo + out_pos<D>(gid, nd * 8 + tig * 2)) =
                        rb ? make_float2(o[nd][2], o[nd][3]) : make_float2(o[nd][0], o[nd][1]);
            }
            if (last) {
                // nothing is left to stream: the consumers add the rows themselves
                // (every warp gets here, also after a wait ran out)
                const int sole = a.items[it].sole;
                named_bar_sync(1, C::kConsumers);
                close_rows<D>(a, a.items + it, seg, item.head, sole, rows, rb, smem, threadIdx.x,
                              C::kConsumers);
                if (rb + C::kPassRows < rows) {
                    named_bar_sync(1, C::kConsumers);
                    continue;
                }
            }
            __syncwarp();
            if (lane == 0 && !dead) mbar_arrive(smem_addr(&all_bars[C::kBarOut]));
        }
    }
}

// ---- item ends: arrivals and the merge of finished (sequence, KV head) runs ---
// Two warps close the items while the consumers stream the next ones: they add
// the consumer warps' rows (weights 2^(m_w - M), warps in order), write the
// item's partials or outputs, arrive on the runs it belongs to and merge those
// it completes.  (With the consumers doing this between items, a batch of 36
// short sequences, ~3 items per CTA, stalled at every end: 51.4 us per call
// against 46.9.)  Of a CTA's last item the consumers add and write the rows
// themselves and merge the runs it completes, since nothing is left to stream;
// the closing warps only arrive.  That shortens the chain after the last stage,
// which a call cannot hide: one sequence of 32,768 tokens 25.1 -> 24.6 us per
// call, the 36 short ones 46.9 -> 46.4.
//
// The arrival word of a run holds two counts.  Its low half counts the items
// that finished (an acquire add, the claim); the claim that brings it to the
// run's length makes its CTA the merger.  Every other CTA then publishes its
// partial with a release add to the high half, and the merger, instead of
// releasing its own partial first (a GPU-scope fence on its critical path),
// reads whether the high half counts the other entries: in the claim's own
// answer, as a rule (the last one to finish), else in acquire loads until it
// does (their claims came first, so their releases are under way: the wait
// depends on nothing this CTA still has to do); its own partial it reads back
// within the CTA.  The merger then takes all of the run's claims and releases off
// the word, also the releases still due when its own wait ran out (a store of
// zero would leave those to the next call, which could then merge too early).
// Every CTA claims once per (item, group member), also after a wait ran out, so
// every call leaves every word at zero, and a plan upload writes zeros; the word
// therefore always starts a call at zero.  A run holds at most 65,535 entries
// (the planner's limit), so the low half never carries.

// GPU-scope atomics of the arrival protocol.
__device__ __forceinline__ unsigned atom_add_acquire_gpu(unsigned* p, unsigned v) {
    unsigned old;
    asm volatile("atom.acquire.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ void red_add_release_gpu(unsigned* p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// (max, sum, weighted output) of one output float4.
struct MergeAcc {
    float M, L;
    float4 o;
    __device__ void clear() {
        M = -INFINITY;
        L = 0.f;
        o = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __device__ void rescale(float to) {  // to >= M
        const float sc = exp2f(M - (to == -INFINITY ? 0.f : to));
        L *= sc;
        o.x *= sc; o.y *= sc; o.z *= sc; o.w *= sc;
        M = to;
    }
    __device__ void add(float w, float l, const float4& v) {
        L += w * l;
        o.x += w * v.x; o.y += w * v.y; o.z += w * v.z; o.w += w * v.w;
    }
};

// One run completed by an item: its (sequence, KV head), entries [e0, e0 + n).
struct RunRef {
    int key, e0, n;
};

// A run's entries are added in two shares (the even and the odd ones), each in
// order, whoever merges it: the result does not depend on which CTA, or which
// of its warps, completes the run.  The entries come straight from L2, kBatch
// at a time.
template <int D, int kBatch>
__device__ __forceinline__ MergeAcc merge_batches(const DecodeArgs& a, const RunRef& run, int row,
                                                  int c4, int share) {
    const int G = a.G;
    const float* po = a.part_o + ((size_t)run.e0 * G + row) * D + c4 * 4;
    const float* pm = a.part_ml + ((size_t)run.e0 * G + row) * 4;
    MergeAcc acc;
    acc.clear();
    for (int e = share; e < run.n; e += 2 * kBatch) {
        float2 ml[kBatch];
        float4 o[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int x = e + 2 * u;
            if (x < run.n) {
                ml[u] = __ldcg(reinterpret_cast<const float2*>(pm + (size_t)x * G * 4));
                o[u] = __ldcg(reinterpret_cast<const float4*>(po + (size_t)x * G * D));
            } else {
                ml[u] = make_float2(-INFINITY, 0.f);
                o[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        float bm = acc.M;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) bm = fmaxf(bm, ml[u].x);
        acc.rescale(bm);
        const float bs = bm == -INFINITY ? 0.f : bm;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) acc.add(exp2f(ml[u].x - bs), ml[u].y, o[u]);
    }
    return acc;
}

// Long runs (one sequence spread over the GPU: ~19 entries per run) want every
// load in one round trip; short ones little besides their few entries.
template <int D>
__device__ __forceinline__ MergeAcc merge_share(const DecodeArgs& a, const RunRef& run, int row,
                                                int c4, int share) {
    return run.n <= 8 ? merge_batches<D, 4>(a, run, row, c4, share)
                      : merge_batches<D, 12>(a, run, row, c4, share);
}

// Adds the second share to the first and writes the normalised output.
template <int D>
__device__ __forceinline__ void merge_finish(const DecodeArgs& a, const RunRef& run, int row, int c4,
                                             MergeAcc x, const MergeAcc& y) {
    const float bm = fmaxf(x.M, y.M);
    x.rescale(bm);
    x.add(exp2f(y.M - (bm == -INFINITY ? 0.f : bm)), y.L, y.o);
    const int i = run.key / a.Hkv, h = (run.key % a.Hkv) * a.G + row;
    write_out(a, ((size_t)i * a.Hq + h) * D + c4 * 4, x.o, 1.f / x.L);
}

// The closing warps (et: thread 0 .. 63 of them).
template <int D>
__device__ void close_items(const DecodeArgs& a, int it0, int it1, uint8_t* smem, uint64_t* bars,
                            volatile int* abort_flag, int et) {
    using C = DecCfg<D>;
    constexpr int kVec = D / 4;  // float4 per output row
    const int G = a.G, lane = et & 31;
    int* n_runs = reinterpret_cast<int*>(smem + C::kOffRuns);
    RunRef* runs = reinterpret_cast<RunRef*>(n_runs + 4);
    uint32_t n_pass = 0;
    bool dead = false;  // warp-uniform
    for (int it = it0; it < it1; ++it) {
        // read while the item is streamed
        const DecodeItem* item = a.items + it;
        const DecodeSeg* seg = a.segs + item->seg;
        const int head = item->head, sole = item->sole, n_grp = seg->n_grp;
        const int rows = n_grp * G;
        // the arrival of this lane's group member (first warp)
        int key = -1;
        RunRef mine{-1, 0, 0};
        if (et < n_grp && !((sole >> et) & 1)) {
            key = seg->grp_seq[et] * a.Hkv + head;
            mine.key = key;
            mine.e0 = a.comb_off[key];
            mine.n = a.comb_off[key + 1] - mine.e0;
        }
        for (int rb = 0; rb < rows; rb += C::kPassRows, ++n_pass) {
            if (!dead) {
                const bool ok = mbar_wait(smem_addr(&bars[C::kBarOut]), n_pass & 1, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) {
                    if (lane == 0 && !*abort_flag) set_error(a.err, kErrTimeout);
                    *abort_flag = 1;
                    dead = true;
                }
            }
            if (dead) continue;
            if (it + 1 == it1) break;  // the consumers have added and written its rows
            close_rows<D>(a, item, seg, head, sole, rows, rb, smem, et, C::kClosers);
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&bars[C::kBarOutFree]));
        }
        // both warps' partials are written (and the list of the item before read)
        named_bar_sync(3, C::kClosers);
        if (et < 32) {
            bool merger = false;
            if (key >= 0) {
                const unsigned old = atom_add_acquire_gpu(a.arrive + key, 1u);
                merger = (old & 0xffffu) + 1u == (unsigned)mine.n;
                if (!merger) {
                    red_add_release_gpu(a.arrive + key, kArriveRelease);
                } else if (!arrive_complete(old, mine.n)) {
                    const uint64_t t0 = globaltimer_ns();
                    for (uint32_t spin = 1;; ++spin) {
                        if (arrive_complete(ld_acquire_gpu(a.arrive + key), mine.n)) break;
                        if ((spin & 31) == 0 && globaltimer_ns() - t0 > kWaitLimitNs) {
                            set_error(a.err, kErrTimeout);
                            break;
                        }
                    }
                }
                if (merger) atomicAdd(a.arrive + key, arrive_settle(mine.n));
            }
            const unsigned mask = __ballot_sync(0xffffffffu, merger);
            if (merger) runs[__popc(mask & ((1u << lane) - 1u))] = mine;
            if (lane == 0) *n_runs = __popc(mask);
            __syncwarp();
        }
        if (it + 1 == it1) {
            if (et == 0) mbar_arrive(smem_addr(&bars[C::kBarRuns]));
            break;
        }
        named_bar_sync(3, C::kClosers);
        const int n = *reinterpret_cast<volatile int*>(n_runs);
        for (int q = 0; q < n; ++q) {
            const RunRef run = runs[q];
            for (int x = et; x < G * kVec; x += C::kClosers) {
                const int row = x / kVec, c4 = x % kVec;
                const MergeAcc s0 = merge_share<D>(a, run, row, c4, 0);
                merge_finish<D>(a, run, row, c4, s0, merge_share<D>(a, run, row, c4, 1));
            }
        }
    }
}

// The runs of the CTA's last item, by the consumers: a thread per share of an
// output, the second shares through shared memory.
template <int D>
__device__ void merge_last_runs(const DecodeArgs& a, uint8_t* smem, uint64_t* bars,
                                volatile int* abort_flag, int lane) {
    using C = DecCfg<D>;
    constexpr int kT = C::kConsumers, kVec = D / 4;
    const int tid = threadIdx.x;
    const int outs = a.G * kVec;  // of one run, <= 512
    const int* n_runs = reinterpret_cast<const int*>(smem + C::kOffRuns);
    volatile int* failed = const_cast<volatile int*>(n_runs + 1);
    const RunRef* runs = reinterpret_cast<const RunRef*>(n_runs + 4);
    const bool ok = mbar_wait(smem_addr(&bars[C::kBarRuns]), 0, abort_flag);
    if (!ok) {
        if (!*abort_flag) set_error(a.err, kErrTimeout);
        *abort_flag = 1;
        *failed = 1;
    }
    named_bar_sync(1, kT);  // from here on every consumer sees the same
    const int n = *failed ? 0 : *reinterpret_cast<const volatile int*>(n_runs);
    // (the item-end rows have been read: their buffer takes the shares)
    float4* x_o = reinterpret_cast<float4*>(smem + C::kOffOut);
    float2* x_ml = reinterpret_cast<float2*>(x_o + kT);
    static_assert(kT * 24 <= C::kOutBytes, "shares");
    // kT / 2 outputs at a time
    for (int b = 0; b < n * outs; b += kT / 2) {
        const int x = b + tid % (kT / 2), share = tid / (kT / 2);
        const bool on = x < n * outs;
        MergeAcc acc;
        RunRef run{};
        int row = 0, c4 = 0;
        if (on) {
            run = runs[x / outs];
            row = x % outs / kVec;
            c4 = x % kVec;
            acc = merge_share<D>(a, run, row, c4, share);
            if (share) {
                x_o[tid] = acc.o;
                x_ml[tid] = make_float2(acc.M, acc.L);
            }
        }
        named_bar_sync(1, kT);
        if (on && !share) {
            MergeAcc other;
            const float2 ml = x_ml[tid + kT / 2];
            other.M = ml.x;
            other.L = ml.y;
            other.o = x_o[tid + kT / 2];
            merge_finish<D>(a, run, row, c4, acc, other);
        }
        named_bar_sync(1, kT);
    }
}

template <int D>
__global__ void __launch_bounds__(DecCfg<D>::kThreads, 1)
    sq_decode_splitk_kernel(const __grid_constant__ CUtensorMap tmap,
                            const __grid_constant__ DecodeArgs a) {
    using C = DecCfg<D>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kOffBars);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + C::kBarRuns + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        // per group: full [kStages], empty [kStages]
        for (int s = 0; s < kDecodeGroups * 2 * C::kStages; ++s)
            mbar_init(smem_addr(&bars[s]),
                      s / C::kStages % 2 ? kDecodeConsumerWarps / kDecodeGroups : 1);
        mbar_init(smem_addr(&bars[C::kBarOut]), kDecodeConsumerWarps);
        mbar_init(smem_addr(&bars[C::kBarOutFree]), C::kClosers / 32);
        mbar_init(smem_addr(&bars[C::kBarRuns]), 1);
        reinterpret_cast<int*>(smem + C::kOffRuns)[1] = 0;
        *abort_flag = 0;
        fence_mbar_init();
    }
    const int group = warp - kDecodeConsumerWarps;
    if (group >= 0 && group < kDecodeGroups) {
        if (threadIdx.x == C::kConsumers) prefetch_tmap(&tmap);
        Producer<D> pr{&tmap, a, smem + group * C::kStages * C::kStageBytes,
                       bars + group * 2 * C::kStages, abort_flag, group, lane};
        // A reused plan is read before the wait.  Pages no in-flight work writes
        // (the host checked every library write to them is complete; the kernels
        // before this one write no other pool memory) are loaded before it too:
        // the first stages stream in while the previous kernel finishes.
        if (a.plan_ready) pr.init();
        named_bar_sync(2, C::kThreads);  // (the barriers are initialised)
        if (a.plan_ready) pr.early();
        grid_dependency_wait();
        grid_launch_dependents();  // the next kernel may be scheduled as CTAs retire
        if (!a.plan_ready) pr.init();
        pr.run();
        return;
    }
    const bool closer = group >= kDecodeGroups;
    const int j0 = (lane >> 2) / a.G, j1 = ((lane >> 2) + 8) / a.G;
    int it0 = 0, it1 = 0;
    ItemHead head{};
    auto read_plan = [&]() {
        it0 = a.cta_begin[blockIdx.x];
        it1 = a.cta_begin[blockIdx.x + 1];
        if (it0 < it1 && !closer) head.read(a, it0, j0, j1);
    };
    if (a.plan_ready) read_plan();
    named_bar_sync(2, C::kThreads);
    // Launched as a programmatic dependent: the set-up above overlapped the
    // previous kernel's tail; nothing else it may have written is read before here.
    grid_dependency_wait();
    grid_launch_dependents();
    if (!a.plan_ready) read_plan();
    if (it0 == it1) return;
    if (closer) {
        close_items<D>(a, it0, it1, smem, bars, abort_flag,
                       threadIdx.x - C::kConsumers - kDecodeGroups * 32);
        return;
    }
    consume<D>(a, it0, it1, head, smem, bars, abort_flag, warp, lane);
    merge_last_runs<D>(a, smem, bars, abort_flag, lane);
}

}  // namespace

int64_t decode_partial_bytes(int32_t n_ent, int32_t G, int32_t D) {
    return (int64_t)n_ent * G * (D + 4) * (int64_t)sizeof(float);
}

template <int D>
static cudaError_t prepare_one() {
    cudaError_t e = cudaFuncSetAttribute(sq_decode_splitk_kernel<D>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         DecCfg<D>::kSmemBytes);
    if (e != cudaSuccess) return e;
    // the largest shared-memory carveout
    return cudaFuncSetAttribute(sq_decode_splitk_kernel<D>,
                                cudaFuncAttributePreferredSharedMemoryCarveout,
                                cudaSharedmemCarveoutMaxShared);
}

cudaError_t decode_prepare(int D) { return D == 128 ? prepare_one<128>() : prepare_one<64>(); }

int decode_ctas_per_sm(int D) {
    int n = 0;
    cudaError_t e;
    if (D == 128)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, sq_decode_splitk_kernel<128>,
                                                          DecCfg<128>::kThreads,
                                                          DecCfg<128>::kSmemBytes);
    else
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, sq_decode_splitk_kernel<64>,
                                                          DecCfg<64>::kThreads,
                                                          DecCfg<64>::kSmemBytes);
    if (e != cudaSuccess || n < 1) return 1;
    return n;
}

// The kernel is launched as a programmatic dependent of whatever precedes it
// on the stream: it waits (griddepcontrol.wait) before it reads anything the
// preceding work may write, so its launch and set-up overlap that work's tail.
static cudaLaunchAttribute pdl_attr() {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    return at;
}

cudaError_t launch_decode(const CUtensorMap& tmap, const DecodeArgs& a, int n_ctas, int D,
                          cudaStream_t st) {
    cudaLaunchAttribute at = pdl_attr();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_ctas);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (D == 128) {
        cfg.blockDim = dim3(DecCfg<128>::kThreads);
        cfg.dynamicSmemBytes = DecCfg<128>::kSmemBytes;
        return cudaLaunchKernelEx(&cfg, sq_decode_splitk_kernel<128>, tmap, a);
    }
    cfg.blockDim = dim3(DecCfg<64>::kThreads);
    cfg.dynamicSmemBytes = DecCfg<64>::kSmemBytes;
    return cudaLaunchKernelEx(&cfg, sq_decode_splitk_kernel<64>, tmap, a);
}

}  // namespace sq
