// K/V row movement in the paged pool: append, copy-on-write of a partial
// page, and in-place span-eviction compaction.
//
// Pool layout: [L][num_pages][2 (K, V)][Hkv][P][D] bf16, so the rows of one
// (layer, page, K/V, head) are P*D contiguous elements and one token row is
// D*2 bytes.  Appends move 16-byte vectors, evictions whole runs of rows.
#include <algorithm>
#include <type_traits>

#include "launch.hpp"
#include "ptx.cuh"

namespace sq {
namespace {

using namespace dev;

__device__ __forceinline__ int64_t row_offset(int64_t num_pages, int Hkv, int P, int D, int layer,
                                              int page, int kv, int head, int slot) {
    return (((((int64_t)layer * num_pages + page) * 2 + kv) * Hkv + head) * P + slot) * (int64_t)D;
}

// The new lengths of the appended sequences, into the cached decode plans
// that stay valid (block 0; read by later kernels of the stream).
__device__ __forceinline__ void write_lens(const AppendLens& l) {
    if (blockIdx.x == 0 && threadIdx.x < l.n) *l.ptr[threadIdx.x] = l.val[threadIdx.x];
}

// ---- append (Algorithm 1: C <- C + R, C <- C + O) and copy-on-write ----------
//
// Bound by memory: every row is read once and written once.  For one layer and
// one of K, V the appended tokens are contiguous in the caller's buffer, so a
// block takes kAppendVecs 16-byte vectors of it (whole tokens: 16 of them at
// 8 x 128), issues all its loads, then scatters them: a head's row is D * 2
// contiguous bytes of the pool.  The indices of a thread's next vector follow
// from the last one by adds; dividing them out again for every vector (64-bit,
// four divisions) had held the kernel at 4.1 TB/s: 24,000 tokens x 32 layers at
// 8 x 128 (6.3 GB moved) took 1,531 us in seven appends, now 930 (6.8 TB/s).
//
// Copy-on-write: the blocks after the append's copy the rows that a sequence
// keeps of a shared last page to its fresh page, one plane each, in no order
// with the appended rows.  A sequence's copy reads slots below its fill and its
// row goes to the slot at it.  Of two sequences of a batch that hold one page
// with different fills, the shorter may write in place to a row that the longer
// copies: the host ends the launch before such a write (append_launch_end), so
// the two parts of a launch never touch the same row.
constexpr int kAppendThreads = 256;
constexpr int kAppendUnroll = 8;  // vectors a thread has in flight
constexpr int kAppendVecs = kAppendThreads * kAppendUnroll;

// Streaming 16-byte load (read once).
__device__ __forceinline__ uint4 ld_once(const void* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

__host__ __device__ inline int append_chunk_tokens(int Hkv, int D) {
    const int t = kAppendVecs / (Hkv * (D / 8));
    return t > 1 ? t : 1;
}

// Tokens [t0, t0 + n) of the block's chunk: `src` their first vector (n x Hkv
// rows, contiguous), `plane0` the pool offset of (layer, page 0, K or V, head
// 0, slot 0).  place(t, page, slot) gives token t's place; false: out of range.
template <typename Place>
__device__ __forceinline__ void append_rows(__nv_bfloat16* pool, const __nv_bfloat16* src,
                                            int64_t plane0, int64_t page_elems, int n, int Hkv,
                                            int P, int D, int* err, Place place) {
    const int lv = D == 128 ? 4 : 3;  // log2 of the vectors per row
    const int nvec = (n * Hkv) << lv;
    const int vc = threadIdx.x & ((1 << lv) - 1);
    const int row = threadIdx.x >> lv;
    const int step = kAppendThreads >> lv;  // rows between a thread's vectors
    const int dt = step / Hkv, dh = step - dt * Hkv;
    int t = row / Hkv, head = row - t * Hkv;
    for (int base = threadIdx.x; base < nvec; base += kAppendVecs) {
        uint4 v[kAppendUnroll];
#pragma unroll
        for (int u = 0; u < kAppendUnroll; ++u) {
            const int i = base + u * kAppendThreads;
            if (i < nvec) v[u] = ld_once(src + (int64_t)i * 8);
        }
#pragma unroll
        for (int u = 0; u < kAppendUnroll; ++u) {
            if (base + u * kAppendThreads < nvec) {
                int page, slot;
                if (place(t, page, slot)) {
                    *reinterpret_cast<uint4*>(pool + plane0 + page * page_elems +
                                              (int64_t)(head * P + slot) * D + vc * 8) = v[u];
                } else {
                    set_error(err, kErrBounds);
                }
            }
            t += dt;
            head += dh;
            if (head >= Hkv) {
                head -= Hkv;
                ++t;
            }
        }
    }
}

// Block b of the copy-on-write blocks: plane b % planes of copy b / planes.
__device__ __forceinline__ void cow_rows(__nv_bfloat16* pool, int64_t num_pages, int L, int Hkv,
                                         int P, int D, const CowCopy* copies, int b, int* err) {
    const int planes = L * 2 * Hkv;
    const CowCopy c = copies[b / planes];
    const int plane = b % planes;
    const int head = plane % Hkv, kv = (plane / Hkv) % 2, layer = plane / (2 * Hkv);
    if ((uint64_t)c.src_page >= (uint64_t)num_pages || (uint64_t)c.dst_page >= (uint64_t)num_pages ||
        c.rows < 0 || c.rows > P) {
        if (threadIdx.x == 0) set_error(err, kErrBounds);
        return;
    }
    const uint4* from = reinterpret_cast<const uint4*>(
        pool + row_offset(num_pages, Hkv, P, D, layer, c.src_page, kv, head, 0));
    uint4* to = reinterpret_cast<uint4*>(
        pool + row_offset(num_pages, Hkv, P, D, layer, c.dst_page, kv, head, 0));
    const int nvec = c.rows * (D / 8);
    for (int i = threadIdx.x; i < nvec; i += kAppendThreads) to[i] = from[i];
}

__global__ void __launch_bounds__(kAppendThreads)
    sq_append_kv_kernel(const __grid_constant__ AppendArgs a) {
    // a programmatic dependent of whatever precedes it: only its launch overlaps
    grid_dependency_wait();
    grid_launch_dependents();
    write_lens(a.lens);
    if (blockIdx.x >= (unsigned)a.n_blocks) {
        cow_rows(a.pool, a.num_pages, a.L, a.Hkv, a.P, a.D, &a.cow, blockIdx.x - a.n_blocks, a.err);
        return;
    }
    const int chunk = append_chunk_tokens(a.Hkv, a.D);
    const int n_chunks = (a.n_tok + chunk - 1) / chunk;
    const int c = blockIdx.x % n_chunks, lk = blockIdx.x / n_chunks;
    const int kv = lk & 1, layer = lk >> 1;
    const int t0 = c * chunk, n = min(chunk, a.n_tok - t0);
    const int64_t page_elems = (int64_t)2 * a.Hkv * a.P * a.D;
    const int lp = __ffs(a.P) - 1;
    append_rows(a.pool,
                (kv ? a.v : a.k) + ((int64_t)layer * a.n_total + a.tok_begin + t0) * a.Hkv * a.D,
                ((int64_t)layer * a.num_pages * 2 + kv) * a.Hkv * a.P * a.D, page_elems, n, a.Hkv,
                a.P, a.D, a.err, [&](int t, int& page, int& slot) {
                    const int pos = a.pos0 + t0 + t;
                    const int pi = (pos >> lp) - a.page_index0;
                    slot = pos & (a.P - 1);
                    if (pi < 0 || pi >= a.n_pages) return false;
                    page = a.pages[pi];
                    return (uint64_t)page < (uint64_t)a.num_pages;
                });
}

// One new token for each of a batch of sequences.
__global__ void __launch_bounds__(kAppendThreads)
    sq_append_kv_batch_kernel(const __grid_constant__ AppendBatchArgs a) {
    grid_dependency_wait();
    grid_launch_dependents();
    write_lens(a.lens);
    if (blockIdx.x >= (unsigned)a.n_blocks) {
        cow_rows(a.pool, a.num_pages, a.L, a.Hkv, a.P, a.D, a.cow, blockIdx.x - a.n_blocks, a.err);
        return;
    }
    const int chunk = append_chunk_tokens(a.Hkv, a.D);
    const int n_chunks = (a.n + chunk - 1) / chunk;
    const int c = blockIdx.x % n_chunks, lk = blockIdx.x / n_chunks;
    const int kv = lk & 1, layer = lk >> 1;
    const int t0 = c * chunk, n = min(chunk, a.n - t0);
    const int64_t page_elems = (int64_t)2 * a.Hkv * a.P * a.D;
    append_rows(a.pool,
                (kv ? a.v : a.k) + ((int64_t)layer * a.n_total + a.row0 + t0) * a.Hkv * a.D,
                ((int64_t)layer * a.num_pages * 2 + kv) * a.Hkv * a.P * a.D, page_elems, n, a.Hkv,
                a.P, a.D, a.err, [&](int t, int& page, int& slot) {
                    page = a.page[t0 + t];
                    slot = a.slot[t0 + t];
                    return (uint64_t)page < (uint64_t)a.num_pages && slot >= 0 && slot < a.P;
                });
}

// ---- span eviction: in-place compaction ---------------------------------------
//
// Algorithm 1, C.clear_kv(Delta_ids): the j-th kept row moves to position j.
// Since the kept positions increase, the source of destination row j is at
// position >= j.  The host splits the rows that change into destination
// tiles (contiguous rows of one page, increasing logical order) and each tile
// into contiguous source pieces; the list is the same for every
// (layer, K/V, head) plane.  One CTA owns one plane; one thread drives it
// with 1-D bulk copies (TMA):
//   * bulk loads of tile t's pieces land in a shared-memory slot, tracked by
//     an mbarrier (expect-tx);
//   * after the barrier completes, one bulk store writes the tile back;
//   * the slot is refilled (tile t + S - 1) once that store has read it.
// All sources of tile t sit at positions >= its first destination row, so
// (a) every source a store of tile t could overwrite belongs to tile t or an
// earlier tile, whose loads have all completed before the store is issued,
// and (b) the loads issued ahead for later tiles read positions past every
// row written so far.  Copy-on-write destination pages are fresh pages that
// hold no source row.  No inter-CTA wait is needed.
//
// A ragged eviction's windows share no page, so the tile list is cut at
// window starts into chunks that separate CTAs of one plane run in parallel;
// each chunk keeps the in-order rule above.  A tile without pieces writes
// zeros: the unused slots of a page that a ragged eviction leaves partial.  Its store reads a zero tile that the
// CTA's warp clears once; it writes only past the rows its window kept, and
// later tiles read only later windows' pages.
//
// What bounds it: latency.  A CTA moves a few tiles, and every record it reads
// from memory is a round trip ahead of its first load.  A plan of up to
// kEvictInline records therefore comes with the launch's arguments (read from
// the constant bank, with no upload before the launch): 25 spans of a context
// of 98,304 tokens, 8 layers of 8 heads, d = 128: 29.7 -> 24.8 us, the call with
// its fork and release 39.8 -> 33.8 us (the 115 MB moved allow 17).  Longer
// plans than fit the 4 KB of arguments are read from memory: their CTAs move
// many tiles each, which hides the records' latency.
template <int S, typename Args>  // ring slots; EvictArgs or EvictInlineArgs
__global__ void __launch_bounds__(32)
    sq_evict_compact_kernel(const __grid_constant__ Args a) {
    constexpr bool kInline = std::is_same<Args, EvictInlineArgs>::value;
    auto tile_at = [&](int g) {
        int4 r;
        if constexpr (kInline) r = a.rec[g];
        else r = __ldg(reinterpret_cast<const int4*>(a.tiles) + g);
        return EvictTile{r.x, r.y, r.z, r.w};
    };
    auto piece_at = [&](int k) {
        int4 r;
        if constexpr (kInline) r = a.rec[a.n_tiles + k];
        else r = __ldg(reinterpret_cast<const int4*>(a.pieces) + k);
        return EvictPiece{r.x, r.y, r.z, r.w};
    };
    auto chunk_at = [&](int c) {
        if constexpr (kInline) return a.inline_chunk[c];
        else return __ldg(&a.chunk[c]);
    };
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    const uint32_t row_bytes = (uint32_t)a.D * 2u;
    const uint32_t tile_bytes = (uint32_t)a.tile_rows * row_bytes;
    uint8_t* zero = smem + S * tile_bytes;   // the zero tile (a.zero_tiles only)
    if (a.zero_tiles) {
        for (uint32_t i = threadIdx.x * 16u; i < tile_bytes; i += blockDim.x * 16u)
            *reinterpret_cast<uint4*>(zero + i) = make_uint4(0, 0, 0, 0);
        fence_proxy_async_smem();  // the bulk stores read it through the async proxy
        __syncwarp();
    }
    if (threadIdx.x != 0) return;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (S + (a.zero_tiles ? 1 : 0)) * tile_bytes);
    // CTA = (chunk of independent windows, plane); tiles [tb, te) of the list
    const int planes = a.L * 2 * a.Hkv;
    const int plane = blockIdx.x % planes;
    const int ch = blockIdx.x / planes;
    const int tb = a.n_chunks > 1 ? chunk_at(ch) : 0;
    const int te = a.n_chunks > 1 ? chunk_at(ch + 1) : a.n_tiles;
    if (tb < 0 || te > a.n_tiles || tb > te) {
        set_error(a.err, kErrBounds);
        return;
    }
    const int head = plane % a.Hkv;
    const int kv = (plane / a.Hkv) % 2;
    const int layer = plane / (2 * a.Hkv);
    uint8_t* base = reinterpret_cast<uint8_t*>(a.pool) +
                    row_offset(a.num_pages, a.Hkv, a.P, a.D, layer, 0, kv, head, 0) * 2;
    const int64_t page_stride = (int64_t)2 * a.Hkv * a.P * row_bytes;  // bytes between pages
    for (int s = 0; s < S; ++s) mbar_init(smem_addr(&full[s]), 1);
    fence_mbar_init();

    auto issue_loads = [&](int t) {   // t: index in the chunk
        const int slot = t % S;
        const int g = tb + t;
        const uint32_t bar = smem_addr(&full[slot]);
        const uint32_t dst0 = smem_addr(smem + slot * tile_bytes);
        const int pb = tile_at(g).piece_begin;
        const int pe = g + 1 < a.n_tiles ? tile_at(g + 1).piece_begin : a.n_pieces;
        uint32_t bytes = 0;
        for (int k = pb; k < pe; ++k) {
            const EvictPiece pc = piece_at(k);
            if ((uint64_t)pc.src_page >= (uint64_t)a.num_pages || pc.src_slot < 0 ||
                pc.n_rows <= 0 || pc.src_slot + pc.n_rows > a.P || pc.dst_row < 0 ||
                pc.dst_row + pc.n_rows > a.tile_rows)
                continue;
            bytes += (uint32_t)pc.n_rows * row_bytes;
        }
        if (bytes == 0) {
            mbar_arrive(bar);
        } else {
            mbar_arrive_expect_tx(bar, bytes);
        }
        for (int k = pb; k < pe; ++k) {
            const EvictPiece pc = piece_at(k);
            if ((uint64_t)pc.src_page >= (uint64_t)a.num_pages || pc.src_slot < 0 ||
                pc.n_rows <= 0 || pc.src_slot + pc.n_rows > a.P || pc.dst_row < 0 ||
                pc.dst_row + pc.n_rows > a.tile_rows) {
                set_error(a.err, kErrBounds);
                continue;
            }
            bulk_load(dst0 + (uint32_t)pc.dst_row * row_bytes,
                      base + pc.src_page * page_stride + (int64_t)pc.src_slot * row_bytes,
                      (uint32_t)pc.n_rows * row_bytes, bar);
        }
    };

    const int T = te - tb;
    for (int t = 0; t < S - 1 && t < T; ++t) issue_loads(t);
    int t = 0;
    for (; t < T; ++t) {
        const int slot = t % S;
        if (!mbar_wait(smem_addr(&full[slot]), (uint32_t)(t / S) & 1u)) {
            set_error(a.err, kErrTimeout);
            break;
        }
        fence_proxy_async_smem();
        const int g = tb + t;
        const EvictTile tl = tile_at(g);
        const int pe = g + 1 < a.n_tiles ? tile_at(g + 1).piece_begin : a.n_pieces;
        const bool zeros = tl.piece_begin == pe;  // no pieces: a tile of zeros
        if ((uint64_t)tl.dst_page < (uint64_t)a.num_pages && tl.dst_slot >= 0 && tl.n_rows > 0 &&
            tl.n_rows <= a.tile_rows && tl.dst_slot + tl.n_rows <= a.P && (!zeros || a.zero_tiles)) {
            bulk_store(base + tl.dst_page * page_stride + (int64_t)tl.dst_slot * row_bytes,
                       smem_addr(zeros ? zero : smem + slot * tile_bytes),
                       (uint32_t)tl.n_rows * row_bytes);
        } else {
            set_error(a.err, kErrBounds);
        }
        bulk_commit();
        const int tn = t + S - 1;
        if (tn < T) {
            bulk_wait_read<1>();  // the store of tile t - 1 has read its slot
            issue_loads(tn);
        }
    }
    if (t < T) {
        // timed out: let the loads already issued land (bounded) before leaving
        for (int u = t + 1; u < T && u < t + S - 1; ++u)
            mbar_wait(smem_addr(&full[u % S]), (uint32_t)(u / S) & 1u);
    }
    bulk_wait<0>();
}

}  // namespace

// Blocks of an append: one per chunk of tokens, layer and K or V.
static int64_t append_blocks(int L, int Hkv, int D, int n) {
    const int chunk = append_chunk_tokens(Hkv, D);
    return (int64_t)L * 2 * ((n + chunk - 1) / chunk);
}

template <typename Args>
static cudaError_t launch_append_kernel(void (*kernel)(Args), Args& a, int n, int n_cow,
                                        cudaStream_t st) {
    const int64_t rows = append_blocks(a.L, a.Hkv, a.D, n);
    const int64_t blocks = rows + (int64_t)n_cow * a.L * 2 * a.Hkv;
    if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
    a.n_blocks = (int32_t)rows;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kAppendThreads);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

cudaError_t launch_append(AppendArgs& a, cudaStream_t st) {
    if (a.n_tok <= 0) return cudaSuccess;
    return launch_append_kernel(sq_append_kv_kernel, a, a.n_tok, a.cow.rows > 0 ? 1 : 0, st);
}

cudaError_t launch_append_batch(AppendBatchArgs& a, cudaStream_t st) {
    if (a.n <= 0) return cudaSuccess;
    return launch_append_kernel(sq_append_kv_batch_kernel, a, a.n, a.n_cow, st);
}

int evict_smem_bytes(int tile_rows, int D, int stages, bool zero_tiles) {
    return (stages + (zero_tiles ? 1 : 0)) * tile_rows * D * 2 + stages * 8 + 128;
}

// The ring depths built: 3, 4 and 6 slots (the host's choices).
template <typename Args, typename F>
static cudaError_t with_evict_kernel(int stages, F f) {
    switch (stages) {
        case 3: return f(sq_evict_compact_kernel<3, Args>);
        case 4: return f(sq_evict_compact_kernel<4, Args>);
        case 6: return f(sq_evict_compact_kernel<6, Args>);
        default: return cudaErrorInvalidValue;
    }
}

int evict_ctas_per_sm(int tile_rows, int D, int stages) {
    int n = 0;
    const cudaError_t e = with_evict_kernel<EvictArgs>(stages, [&](auto kernel) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, 32,
                                                             evict_smem_bytes(tile_rows, D, stages));
    });
    return e != cudaSuccess || n < 1 ? 1 : n;
}

cudaError_t evict_prepare() {
    for (int stages : {3, 4, 6}) {
        auto raise = [&](auto kernel) {
            return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        evict_smem_bytes(kStageTokens, 128, stages, true));
        };
        cudaError_t e = with_evict_kernel<EvictArgs>(stages, raise);
        if (e == cudaSuccess) e = with_evict_kernel<EvictInlineArgs>(stages, raise);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename Args>
static cudaError_t launch_evict_kernel(const Args& a, cudaStream_t st) {
    const int blocks = a.L * 2 * a.Hkv * std::max(a.n_chunks, 1);
    if (blocks == 0 || a.n_tiles == 0) return cudaSuccess;
    const int smem = evict_smem_bytes(a.tile_rows, a.D, a.stages, a.zero_tiles != 0);
    const cudaError_t e = with_evict_kernel<Args>(a.stages, [&](auto kernel) {
        kernel<<<blocks, 32, smem, st>>>(a);
        return cudaSuccess;
    });
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_evict(const EvictArgs& a, cudaStream_t st) { return launch_evict_kernel(a, st); }

cudaError_t launch_evict_inline(const EvictInlineArgs& a, cudaStream_t st) {
    return launch_evict_kernel(a, st);
}

}  // namespace sq
