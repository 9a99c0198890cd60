// A stand-in for the CUDA runtime and the kernels' launchers, so that CPU tests
// can drive the library's C API (sq_api.cpp) itself: device memory is host
// memory, the two append launches move their rows (a launch's parts in an order
// the test picks, since a launch gives them none), the attention launches only
// note which buffers they use, and any call can be made to fail.
//
// Streams are not run but ordered: every operation carries the operations known
// to precede it (its stream's earlier ones, and those behind events waited for),
// and two uses of one allocation, at least one of them a write, of which neither
// precedes the other count as a race.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <vector>

#include "../paper_2602_22603_gb300/csrc/kernels/launch.hpp"
#include "../paper_2602_22603_gb300/csrc/kernels/noalloc.hpp"

using namespace sq;

namespace {

typedef std::map<void*, uint64_t> Clock;  // stream -> its operations known to be earlier

void merge(Clock& a, const Clock& b) {
    for (const auto& x : b) a[x.first] = std::max(a[x.first], x.second);
}

struct Use {
    void* stream;
    uint64_t seq;
    bool write;
};
struct Block {
    size_t bytes;
    std::vector<Use> uses;
};

std::map<void*, Clock> g_streams;
std::map<void*, Clock> g_events;
Clock g_host;  // operations the host has waited for
std::map<char*, Block> g_blocks;
int64_t g_races = 0, g_count[8];
int g_fail = -1;
size_t g_malloc_limit = ~size_t(0);
int g_copies_last = 0;

// The clock of a new operation on a stream (its own entry: its sequence number).
Clock& tick(void* st) {
    Clock& c = g_streams[st];
    merge(c, g_host);
    ++c[st];
    return c;
}

void use(void* st, const Clock& c, const void* p, bool write) {
    auto it = g_blocks.upper_bound((char*)p);
    if (!p || it == g_blocks.begin()) return;
    --it;
    if ((char*)p >= it->first + it->second.bytes) return;
    for (const Use& u : it->second.uses) {
        auto known = c.find(u.stream);
        if ((u.write || write) && (known == c.end() || known->second < u.seq)) ++g_races;
    }
    it->second.uses.push_back({st, c.at(st), write});
}

bool fails(int kind) {
    ++g_count[kind];
    if (g_fail != kind) return false;
    g_fail = -1;
    return true;
}

int64_t row_at(int64_t num_pages, int Hkv, int P, int D, int layer, int page, int kv, int head,
               int slot) {
    return (((((int64_t)layer * num_pages + page) * 2 + kv) * Hkv + head) * P + slot) * (int64_t)D;
}

template <typename A>
void copy_rows(const A& a, const CowCopy& c) {
    for (int l = 0; l < a.L; ++l)
        for (int kv = 0; kv < 2; ++kv)
            for (int h = 0; h < a.Hkv; ++h)
                std::memcpy(a.pool + row_at(a.num_pages, a.Hkv, a.P, a.D, l, c.dst_page, kv, h, 0),
                            a.pool + row_at(a.num_pages, a.Hkv, a.P, a.D, l, c.src_page, kv, h, 0),
                            (size_t)c.rows * a.D * 2);
}

template <typename A>
void write_row(const A& a, int row, int page, int slot) {
    for (int l = 0; l < a.L; ++l)
        for (int kv = 0; kv < 2; ++kv)
            for (int h = 0; h < a.Hkv; ++h)
                std::memcpy(a.pool + row_at(a.num_pages, a.Hkv, a.P, a.D, l, page, kv, h, slot),
                            (kv ? a.v : a.k) + (((int64_t)l * a.n_total + row) * a.Hkv + h) * a.D,
                            (size_t)a.D * 2);
}

CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    return CUDA_SUCCESS;
}

}  // namespace

// ---- what the tests set and read ---------------------------------------------
enum { kAppend, kAppendBatch, kDecode, kPrefill, kCombine, kEvict };
#define EXPORT extern "C" __attribute__((visibility("default")))
EXPORT void fake_reset() {
    g_streams.clear();
    g_host.clear();
    g_races = 0;
    std::memset(g_count, 0, sizeof g_count);
    g_fail = -1;
    g_malloc_limit = ~size_t(0);
    g_copies_last = 0;
}
EXPORT void fake_fail(int kind) { g_fail = kind; }  // the next launch of this kind
EXPORT void fake_malloc_limit(int64_t bytes) { g_malloc_limit = bytes < 0 ? ~size_t(0) : (size_t)bytes; }
EXPORT void fake_copies_last(int last) { g_copies_last = last; }
EXPORT int64_t fake_count(int kind) { return g_count[kind]; }
EXPORT int64_t fake_races() { return g_races; }

// ---- launchers -----------------------------------------------------------------
namespace sq {

cudaError_t launch_append(AppendArgs& a, cudaStream_t st) {
    if (fails(kAppend)) return cudaErrorLaunchFailure;
    tick(st);
    for (int part = 0; part < 2; ++part) {
        if (part == g_copies_last && a.cow.rows > 0) copy_rows(a, a.cow);
        if (part != g_copies_last)
            for (int t = 0; t < a.n_tok; ++t)
                write_row(a, a.tok_begin + t, a.pages[(a.pos0 + t) / a.P - a.page_index0],
                          (a.pos0 + t) % a.P);
    }
    return cudaSuccess;
}

cudaError_t launch_append_batch(AppendBatchArgs& a, cudaStream_t st) {
    if (fails(kAppendBatch)) return cudaErrorLaunchFailure;
    tick(st);
    for (int part = 0; part < 2; ++part)
        if (part == g_copies_last)
            for (int i = 0; i < a.n_cow; ++i) copy_rows(a, a.cow[i]);
        else
            for (int i = 0; i < a.n; ++i) write_row(a, a.row0 + i, a.page[i], a.slot[i]);
    return cudaSuccess;
}

cudaError_t launch_decode(const CUtensorMap&, const DecodeArgs& a, int, int, cudaStream_t st) {
    if (fails(kDecode)) return cudaErrorLaunchFailure;
    const Clock& c = tick(st);
    use(st, c, a.segs, true);  // (the arrival words)
    use(st, c, a.part_o, true);
    return cudaSuccess;
}

cudaError_t launch_prefill(const CUtensorMap&, const CUtensorMap&, const PrefillShortArgs& a, int,
                           cudaStream_t st) {
    if (fails(kPrefill)) return cudaErrorLaunchFailure;
    const Clock& c = tick(st);
    use(st, c, a.tiles, false);
    bool split = false;
    for (int i = 0; i < a.n_items; ++i) split |= a.items[i].part >= 0;
    if (split) use(st, c, a.part_o, true);
    return cudaSuccess;
}

cudaError_t launch_prefill_combine(const PrefillCombineArgs& a, int, cudaStream_t st) {
    if (fails(kCombine)) return cudaErrorLaunchFailure;
    const Clock& c = tick(st);
    use(st, c, a.merges, false);
    use(st, c, a.part_o, false);
    return cudaSuccess;
}

cudaError_t launch_evict(const EvictArgs&, cudaStream_t st) {
    if (fails(kEvict)) return cudaErrorLaunchFailure;
    tick(st);
    return cudaSuccess;
}
cudaError_t launch_evict_inline(const EvictInlineArgs& a, cudaStream_t st) { return launch_evict(a, st); }
cudaError_t launch_read_probe(const void*, size_t, unsigned*, int, cudaStream_t) { return cudaSuccess; }
cudaError_t decode_prepare(int) { return cudaSuccess; }
cudaError_t prefill_prepare(int) { return cudaSuccess; }
cudaError_t evict_prepare() { return cudaSuccess; }
int decode_ctas_per_sm(int) { return 1; }
int evict_ctas_per_sm(int, int, int) { return 4; }
int64_t decode_partial_bytes(int32_t n_ent, int32_t G, int32_t D) {
    return (int64_t)n_ent * G * (D + 4) * (int64_t)sizeof(float);
}
int noalloc_scratch(void**) { return -5; }

}  // namespace sq

// ---- the runtime -----------------------------------------------------------------
extern "C" {

cudaError_t cudaMalloc(void** p, size_t n) {
    if (n > g_malloc_limit) return cudaErrorMemoryAllocation;
    *p = std::calloc(n, 1);
    g_blocks[(char*)*p] = {n, {}};
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    for (auto& s : g_streams) merge(g_host, s.second);
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    if (!p) return cudaSuccess;
    cudaDeviceSynchronize();
    g_blocks.erase((char*)p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return *p = std::malloc(n), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { return std::memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    return std::memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    use(st, tick(st), d, true);
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    *e = (cudaEvent_t)std::malloc(1);
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    g_events.erase(e);
    std::free(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) {
    return g_events[e] = g_streams[st], cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned) {
    return merge(g_streams[st], g_events[e]), cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return merge(g_host, g_events[e]), cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaErrorNotReady; }
cudaError_t cudaStreamSynchronize(cudaStream_t st) { return merge(g_host, g_streams[st]), cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    return *s = cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
    *fn = (void*)encode;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

}  // extern "C"
