// The plans' device memory (csrc/device_memory.h) on a fake CUDA runtime: pools that count, streams
// whose work "runs" when the test says so, allocations that fail on request.  Prints one line per
// case and exits non-zero at the first failure.  Built and run by tests/test_device_memory_host.py.
#include "device_memory.h"

#include <cstdio>
#include <cstdlib>
#include <set>
#include <vector>

namespace {

struct FakePool {
    int device;
    size_t used = 0, reserved = 0;
};
struct FakeEvent {
    int device;
    cudaStream_t st = nullptr;
    long at = -1;  // the stream's work before it
};
struct Alloc {
    FakePool *pool;
    size_t bytes;
};

int g_device = 0;
size_t g_total = size_t(1) << 38, g_room = size_t(1) << 38;  // device memory, and what all pools may reserve
std::map<cudaStream_t, long> g_issued, g_ran;                // work per stream
std::map<void *, Alloc> g_allocs;
std::vector<FakePool *> g_pools;
std::vector<std::pair<cudaStream_t, cudaEvent_t>> g_waits;
int g_syncs = 0, g_frees_async = 0, g_frees = 0, g_mallocs = 0, g_event_errors = 0;
std::set<cudaStream_t> g_capturing;
cudaStreamCaptureMode g_mode = cudaStreamCaptureModeGlobal;
int g_invalidated = 0;  // captures that a call of the thread would have ended
uintptr_t g_next = 0x1000;

size_t reserved_all() {
    size_t n = 0;
    for (auto *p : g_pools) n += p->reserved;
    return n;
}
bool event_passed(FakeEvent *e) { return e->at <= g_ran[e->st]; }

}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_device = d; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { *f = g_room; *t = g_total; return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *props) {
    auto *q = new FakePool{props->location.id};
    g_pools.push_back(q);
    *p = reinterpret_cast<cudaMemPool_t>(q);
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t p, cudaMemPoolAttr, void *v) {
    *static_cast<uint64_t *>(v) = reinterpret_cast<FakePool *>(p)->reserved;
    return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t keep) {
    auto *q = reinterpret_cast<FakePool *>(p);
    q->reserved = std::min(q->reserved, std::max(keep, q->used));
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void **ptr, size_t bytes, cudaMemPool_t p, cudaStream_t st) {
    auto *q = reinterpret_cast<FakePool *>(p);
    ++g_mallocs;
    const size_t grow = q->used + bytes > q->reserved ? q->used + bytes - q->reserved : 0;
    if (reserved_all() + grow > g_room) return cudaErrorMemoryAllocation;
    q->used += bytes;
    q->reserved = std::max(q->reserved, q->used);
    *ptr = reinterpret_cast<void *>(g_next += 0x1000);
    g_allocs[*ptr] = Alloc{q, bytes};
    ++g_issued[st];
    return cudaSuccess;
}
static cudaError_t release(void *ptr) {
    auto i = g_allocs.find(ptr);
    if (i == g_allocs.end()) {
        std::printf("a block freed twice\n");
        std::exit(1);
    }
    i->second.pool->used -= i->second.bytes;
    g_allocs.erase(i);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *ptr, cudaStream_t) {
    ++g_frees_async;
    if (g_allocs.count(ptr) && g_allocs[ptr].pool->device != g_device) ++g_event_errors;
    return release(ptr);
}
cudaError_t cudaFree(void *ptr) {
    ++g_frees;
    if (!g_capturing.empty() && g_mode != cudaStreamCaptureModeRelaxed) ++g_invalidated;
    return release(ptr);
}
cudaError_t cudaStreamSynchronize(cudaStream_t st) { ++g_syncs; g_ran[st] = g_issued[st]; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t st, cudaStreamCaptureStatus *s) {
    *s = g_capturing.count(st) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *m) { std::swap(*m, g_mode); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    *e = reinterpret_cast<cudaEvent_t>(new FakeEvent{g_device});
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete reinterpret_cast<FakeEvent *>(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) {
    auto *f = reinterpret_cast<FakeEvent *>(e);
    if (f->device != g_device) {
        ++g_event_errors;
        return cudaErrorInvalidResourceHandle;
    }
    f->st = st;
    f->at = ++g_issued[st];
    return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t e) {
    if (!g_capturing.empty() && g_mode != cudaStreamCaptureModeRelaxed) ++g_invalidated;
    return event_passed(reinterpret_cast<FakeEvent *>(e)) ? cudaSuccess : cudaErrorNotReady;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned) { g_waits.emplace_back(st, e); return cudaSuccess; }
}

using spg::Block;
using spg::DeviceMemory;

static cudaStream_t S(int i) { return reinterpret_cast<cudaStream_t>(uintptr_t(0x100 + i)); }
static const char *g_case = "";
#define CHECK(x)                                                        \
    do {                                                                \
        if (!(x)) {                                                     \
            std::printf("%s: line %d: %s\n", g_case, __LINE__, #x);     \
            return 1;                                                   \
        }                                                               \
    } while (0)
static Block get(DeviceMemory &m, size_t bytes, cudaStream_t st, bool temp = false, int device = 0, bool exact = false) {
    Block b;
    if (m.alloc(device, temp, bytes, exact, st, &b) != cudaSuccess) b.ptr = nullptr;
    return b;
}
static void reset() {
    for (auto *p : g_pools) delete p;
    g_pools.clear();
    g_allocs.clear();
    g_issued.clear();
    g_ran.clear();
    g_waits.clear();
    g_capturing.clear();
    g_syncs = g_frees_async = g_frees = g_mallocs = g_event_errors = g_invalidated = 0;
    g_device = 0;
    g_room = g_total;
}

constexpr size_t MB = size_t(1) << 20, GB = size_t(1) << 30;

static int large_blocks_go_back_to_the_driver() {
    reset();
    DeviceMemory m;
    Block a = get(m, 40 * GB, S(1)), b = get(m, 40 * GB, S(1)), t = get(m, 40 * GB, S(1), true), c = get(m, 10 * GB, S(1));
    CHECK(a.ptr && b.ptr && t.ptr && c.ptr);
    CHECK(a.from == b.from && a.from != t.from && a.from != c.from);  // by size and use
    CHECK(a.bytes >= 40 * GB && a.bytes <= 40 * GB + 40 * GB / 16);
    m.free(0, &a, 1, false, S(1));
    m.free(0, &c, 1, false, S(1));
    CHECK(g_frees_async == 2 && g_allocs.count(a.ptr) == 0);  // the driver has them: any allocation can get that memory
    Block d = get(m, 40 * GB - 1000, S(2));  // a nearly equal request finds the same pool
    CHECK(d.from == b.from && g_waits.empty());
    return 0;
}

static int small_blocks_follow_their_event() {
    reset();
    DeviceMemory m;
    Block a = get(m, 100000, S(1));
    m.free(0, &a, 1, false, S(1));
    CHECK(g_frees_async == 0);
    Block b = get(m, 99000, S(2));  // another stream, the last use has not run
    CHECK(b.ptr != a.ptr && g_waits.empty());
    Block t = get(m, 100000, S(1), true);  // temporaries apart from results
    CHECK(t.ptr != a.ptr);
    Block c = get(m, 99000, S(1));  // the same stream: at once, in order
    CHECK(c.ptr == a.ptr && g_waits.size() == 1 && g_waits[0].first == S(1));
    m.free(0, &c, 1, false, S(1));
    g_ran[S(1)] = g_issued[S(1)];
    Block d = get(m, 99000, S(2));  // now it has run
    CHECK(d.ptr == a.ptr);
    Block e = get(m, 60000, S(2)), f = get(m, 2 * MB, S(2));
    m.free(0, &f, 1, false, S(2));
    Block g = get(m, MB, S(2));  // not a block twice as large
    CHECK(g.ptr != f.ptr && e.ptr);
    return 0;
}

static int the_plans_device_is_current() {
    reset();
    DeviceMemory m;
    Block a = get(m, 100000, nullptr, false, 1), b = get(m, GB, nullptr, false, 1);
    CHECK(g_device == 0);
    m.free(1, &a, 1, false, nullptr);  // as a finaliser does, with device 0 current
    m.free(1, &b, 1, false, nullptr);
    CHECK(g_device == 0 && g_event_errors == 0);
    CHECK(reinterpret_cast<FakeEvent *>(get(m, 100000, nullptr, false, 1).freed)->device == 1);
    CHECK(m.trim(1, 0) == cudaSuccess && g_device == 0);
    return 0;
}

static int kept_blocks_are_bounded() {
    reset();
    DeviceMemory m;
    std::vector<Block> v;
    for (size_t i = 0; i < spg::CACHE_BLOCKS + 10; ++i) v.push_back(get(m, 8192, S(1)));
    for (auto &b : v) m.free(0, &b, 1, false, S(1));
    CHECK(g_frees_async + g_frees == 10 && g_allocs.size() == spg::CACHE_BLOCKS);
    for (int i = 0; i < 10; ++i) CHECK(g_allocs.count(v[i].ptr) == 0);  // the longest unused
    reset();
    DeviceMemory n;
    const size_t most = g_total / spg::CACHE_SHARE;
    v.clear();
    for (size_t k = 0; k < most / (64 * MB) + 5; ++k) v.push_back(get(n, 64 * MB, S(1)));
    for (auto &b : v) n.free(0, &b, 1, false, S(1));
    CHECK(g_allocs.size() * 64 * MB <= most);
    // blocks whose last use is on another stream and has not run stay: nothing waits for them
    v.clear();
    g_waits.clear();
    const size_t before = g_allocs.size();
    for (int k = 0; k < 8; ++k) v.push_back(get(n, 100 * MB, S(2)));
    for (auto &b : v) n.free(0, &b, 1, false, S(2));
    for (auto &w : g_waits) CHECK(w.first == reinterpret_cast<FakeEvent *>(w.second)->st || w.first == S(2));
    CHECK(before > 0);
    return 0;
}

static int a_full_device_is_tried_once_more() {
    reset();
    DeviceMemory m;
    Block small = get(m, MB, S(1)), big = get(m, 100 * GB, S(1), true);
    m.free(0, &small, 1, false, S(1));
    m.free(0, &big, 1, true, S(1));
    g_room = 120 * GB;
    Block a = get(m, 119 * GB, S(1));  // rounded it would not fit, and the other pool holds 100 GB
    CHECK(a.ptr && a.bytes == 119 * GB && g_syncs == 1);
    CHECK(g_allocs.count(small.ptr) == 0);
    Block b = get(m, 2 * GB, S(1));
    CHECK(!b.ptr && g_allocs.size() == 1);
    m.free(0, &a, 1, false, S(1));
    CHECK(get(m, 100 * GB, S(1)).ptr);  // a failure leaves nothing behind
    return 0;
}

static int trim_waits_for_nothing_and_keeps_what_it_may() {
    reset();
    DeviceMemory m;
    CHECK(m.trim(0, 0) == cudaSuccess && g_pools.empty());  // a device never used
    Block a = get(m, GB, S(1)), b = get(m, 2 * GB, S(1), true), held = get(m, 3 * GB, S(1)), s = get(m, MB, S(1)), p = get(m, MB, S(2));
    m.free(0, &a, 1, false, S(1));
    m.free(0, &b, 1, true, S(1));
    m.free(0, &s, 1, false, S(1));
    g_ran[S(1)] = g_issued[S(1)];
    m.free(0, &p, 1, false, S(2));  // its stream has not got there
    const size_t all = reserved_all();
    CHECK(m.trim(0, all) == cudaSuccess && reserved_all() == all);
    CHECK(m.trim(0, all - GB) == cudaSuccess && reserved_all() == all - GB);
    CHECK(g_allocs.count(s.ptr) == 1);  // kept blocks only when the pools' free memory is not enough
    CHECK(m.trim(0, 0) == cudaSuccess && g_syncs == 0 && g_waits.empty());
    CHECK(g_allocs.count(s.ptr) == 0 && g_allocs.count(p.ptr) == 1 && g_allocs.count(held.ptr) == 1);
    CHECK(reserved_all() == held.bytes + p.bytes);
    return 0;
}

static int pools_hold_at_most_half_for_others() {
    reset();
    DeviceMemory m;
    for (size_t k = 0; k < 12; ++k) {  // sizes that share no pool
        Block b = get(m, (20 + 2 * k) * GB, S(1));
        CHECK(b.ptr);
        m.free(0, &b, 1, false, S(1));
        CHECK(reserved_all() <= std::max(g_total / 2, b.bytes));
    }
    return 0;
}

static int a_free_inside_a_capture_keeps_nothing() {
    reset();
    DeviceMemory m;
    Block a = get(m, 100000, S(1));
    g_capturing.insert(S(1));
    m.free(0, &a, 1, false, S(1));
    CHECK(g_frees_async == 1 && g_allocs.empty());
    return 0;
}

static int a_free_beside_a_capture_leaves_it_valid() {
    reset();
    DeviceMemory m;
    std::vector<Block> v;
    for (size_t i = 0; i < spg::CACHE_BLOCKS + 10; ++i) v.push_back(get(m, 8192, S(1)));
    for (size_t i = 0; i < spg::CACHE_BLOCKS; ++i) m.free(0, &v[i], 1, false, S(1));
    g_ran[S(1)] = g_issued[S(1)];
    g_capturing.insert(S(2));
    for (size_t i = spg::CACHE_BLOCKS; i < v.size(); ++i) m.free(0, &v[i], 1, false, S(1));  // with evictions
    CHECK(g_frees == 10 && g_invalidated == 0 && g_mode == cudaStreamCaptureModeGlobal);
    return 0;
}

static int exact_blocks_are_of_just_their_bytes() {
    reset();
    DeviceMemory m;
    Block a = get(m, 100001, S(1), false, 0, true), b = get(m, GB + 1, S(1), false, 0, true);
    CHECK(a.bytes == 100001 && b.bytes == GB + 1);
    m.free(0, &a, 1, false, S(1));
    m.free(0, &b, 1, false, S(1));
    CHECK(g_frees_async == 2);
    return 0;
}

static size_t live_bytes() {
    size_t n = 0;
    for (auto &a : g_allocs) n += a.second.bytes;
    return n;
}

// A plan's arrays: several small ones, a middling and a large one, per lifetime.
static const size_t kArrays[] = {16, 4000, 64 * 1024, 64 * 1024 + 1, 700001, 3 * MB + 5, 300 * MB + 77};

static int a_plans_limit_is_of_the_memory_itself() {
    reset();
    DeviceMemory m;
    spg::PlanMemory warm;  // leaves kept blocks of nearly these sizes, some a little larger
    void *p = nullptr;
    for (int life = 0; life < 3; ++life)
        for (size_t n : kArrays) CHECK(warm.alloc(m, 0, S(1), n + n / 16, life, &p) == cudaSuccess);
    for (int life = 0; life < 3; ++life) warm.release(m, 0, S(1), life);
    CHECK(warm.held == 0);
    const size_t idle = live_bytes();
    size_t all = 0;
    for (size_t n : kArrays) all += 3 * n;
    spg::PlanMemory plan;
    plan.limit = (int64_t)all;  // fits exactly
    for (int life = 0; life < 3; ++life)
        for (size_t n : kArrays) {
            CHECK(plan.alloc(m, 0, S(1), n, life, &p) == cudaSuccess && p != nullptr);
            CHECK(live_bytes() - idle <= (size_t)plan.limit && (size_t)plan.held == live_bytes() - idle);
        }
    CHECK(plan.alloc(m, 0, S(1), 1, 0, &p) == cudaErrorMemoryAllocation && p == nullptr);
    plan.release(m, 0, S(1), 0);
    CHECK(plan.alloc(m, 0, S(1), all / 3, 1, &p) == cudaSuccess && plan.peak == plan.limit);
    spg::PlanMemory tiny;  // less than a shared block
    tiny.limit = 10000;
    const size_t before = live_bytes();
    CHECK(tiny.alloc(m, 0, S(1), 4000, 2, &p) == cudaSuccess && tiny.alloc(m, 0, S(1), 4000, 0, &p) == cudaSuccess);
    CHECK(live_bytes() - before <= 10000);
    return 0;
}

static int without_a_limit_blocks_are_little_larger() {
    reset();
    DeviceMemory m;
    spg::PlanMemory plan;
    void *p = nullptr;
    for (int k = 0; k < 40; ++k)
        for (int life = 0; life < 3; ++life) CHECK(plan.alloc(m, 0, S(1), kArrays[k % 7], life, &p) == cudaSuccess);
    CHECK(live_bytes() <= (size_t)plan.held + (size_t)plan.held / 16 + 3 * 512 * 1024 + 120 * 4096);
    CHECK(plan.blocks < 90);  // the small ones share
    return 0;
}

int main() {
    const struct {
        const char *name;
        int (*run)();
    } cases[] = {
#define CASE(f) {#f, f}
        CASE(large_blocks_go_back_to_the_driver),
        CASE(small_blocks_follow_their_event),
        CASE(the_plans_device_is_current),
        CASE(kept_blocks_are_bounded),
        CASE(a_full_device_is_tried_once_more),
        CASE(trim_waits_for_nothing_and_keeps_what_it_may),
        CASE(pools_hold_at_most_half_for_others),
        CASE(a_free_inside_a_capture_keeps_nothing),
        CASE(a_free_beside_a_capture_leaves_it_valid),
        CASE(exact_blocks_are_of_just_their_bytes),
        CASE(a_plans_limit_is_of_the_memory_itself),
        CASE(without_a_limit_blocks_are_little_larger),
    };
    for (auto &c : cases) {
        g_case = c.name;
        if (c.run() != 0) return 1;
        std::printf("%s: ok\n", c.name);
    }
    return 0;
}
