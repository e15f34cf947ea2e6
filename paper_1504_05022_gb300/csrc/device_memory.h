// Device memory of the plans, from stream-ordered pools of the driver.
//
// Large blocks (CLASS_MIN bytes or more) come from a pool of their size, in steps of a sixteenth to
// a thirty-second, where every free block fits, results and temporaries apart: a large block
// carved out of freed memory of other sizes makes a pool map it anew, which holds up the host
// for 0.7 ms per GB (30 of 106 ms on the 2^20 R-MAT when its results and temporaries shared one pool, 3.8
// of 11.6 ms for a batch of 20 pairs behind a product with 6 GB of C).  Freed, they stay with
// their pool: the driver hands them out again in stream order, and takes unused memory back by
// itself when any allocation of the process, here or elsewhere, finds the device full.  For other
// processes it is bounded: beyond half of the device's memory the pools longest unused give
// theirs back.
//
// Small blocks are kept by size above the pools, since a product makes 4 to 20 of them and the driver
// takes 1.7 us for each (a 64 x 64 Laplacian squared: 109 against 116 us): CACHE_BLOCKS of them and a
// CACHE_SHARE-th of the device's memory at most, which no other allocation can have meanwhile.  Each
// carries an event recorded when it was freed, which its next owner's stream waits for -- at
// once on the stream that freed it, on another one only when it has passed, so that streams do
// not come to wait for each other.
//
// Host code only; the plan's device is made current for every call.
#pragma once

#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <utility>
#include <vector>

namespace spg {

// Makes `device` current, and the device that was current before again.
class DeviceGuard {
  public:
    explicit DeviceGuard(int device) {
        err_ = cudaGetDevice(&before_);
        if (err_ == cudaSuccess && before_ != device) {
            err_ = cudaSetDevice(device);
            changed_ = err_ == cudaSuccess;
        }
    }
    ~DeviceGuard() {
        if (changed_) cudaSetDevice(before_);
    }
    DeviceGuard(const DeviceGuard &) = delete;
    DeviceGuard &operator=(const DeviceGuard &) = delete;
    cudaError_t error() const { return err_; }

  private:
    int before_ = 0;
    bool changed_ = false;
    cudaError_t err_ = cudaSuccess;
};

// While one lives, the thread's event queries and frees are no concern of a stream capture that this
// thread or another one has begun: they touch no capturing stream, but would invalidate a capture in
// the global mode (torch's), into which a finaliser may free a plan.
class OutsideCapture {
  public:
    OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode_); }
    ~OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode_); }
    OutsideCapture(const OutsideCapture &) = delete;
    OutsideCapture &operator=(const OutsideCapture &) = delete;

  private:
    cudaStreamCaptureMode mode_ = cudaStreamCaptureModeRelaxed;
};

constexpr size_t CLASS_MIN = size_t(128) << 20;
constexpr size_t CACHE_BLOCKS = 4096;  // a batch of 512 pairs in 64 waves holds about 2,600
constexpr size_t CACHE_SHARE = 256;

// The size a block of `bytes` is allocated with: steps of a sixteenth to a thirty-second.
inline size_t block_size(size_t bytes) {
    size_t step = 4096;
    while (step * 32 < bytes) step *= 2;
    return (bytes + step - 1) / step * step;
}

struct SizePool {
    cudaMemPool_t pool = nullptr;
    size_t live = 0;      // bytes allocated
    size_t reserved = 0;  // the most there were since it was trimmed
    uint64_t stamp = 0;   // last use
};

struct Block {
    void *ptr = nullptr;
    size_t bytes = 0;
    SizePool *from = nullptr;
    cudaEvent_t freed = nullptr;  // small blocks that were kept once
    cudaStream_t st = nullptr;    // where it was freed
    uint64_t stamp = 0;           // when
};

class DeviceMemory {
  public:
    // `exact`: of just these bytes (a plan with a limit).  An allocation that the driver cannot
    // meet is tried once more without rounding, when the stream's own frees have run.
    cudaError_t alloc(int device, bool temp, size_t bytes, bool exact, cudaStream_t st, Block *out) {
        DeviceGuard g(device);
        if (g.error() != cudaSuccess) return g.error();
        const size_t size = exact ? bytes : block_size(bytes);
        if (!exact && size < CLASS_MIN && take_kept(device, temp, size, st, out)) return cudaSuccess;
        cudaError_t e = take(device, temp, !exact && size >= CLASS_MIN ? size : 0, size, st, out);
        if (e == cudaErrorMemoryAllocation) {
            cudaGetLastError();
            if (cudaStreamSynchronize(st) != cudaSuccess) {
                cudaGetLastError();
                return e;
            }
            trim(device, 0);
            e = take(device, temp, 0, bytes, st, out);
        }
        return e;
    }

    // Stream-ordered on st, where the blocks' last use is.
    void free(int device, const Block *blocks, size_t n, bool temp, cudaStream_t st) {
        if (n == 0) return;
        DeviceGuard g(device);
        OutsideCapture relaxed;
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        // inside a capture of st itself nothing is kept: an event of the capture orders nothing outside
        cudaError_t e = g.error();
        if (e == cudaSuccess) e = cudaStreamIsCapturing(st, &capture);
        bool may_keep = e == cudaSuccess && capture == cudaStreamCaptureStatusNone;
        std::lock_guard<std::mutex> lk(mu_);
        Device &d = devices_[device];
        for (size_t k = 0; k < n; ++k) {
            Block b = blocks[k];
            const bool keep = may_keep && b.bytes < CLASS_MIN && b.bytes == block_size(b.bytes);
            if (keep && b.freed == nullptr) {
                e = cudaEventCreateWithFlags(&b.freed, cudaEventDisableTiming);
                if (e != cudaSuccess) b.freed = nullptr;
            }
            if (keep && e == cudaSuccess) e = cudaEventRecord(b.freed, st);
            if (keep && e == cudaSuccess) {
                b.st = st;
                b.stamp = ++clock_;
                d.oldest.emplace(b.stamp, std::make_pair(&d.kept[temp], d.kept[temp].emplace(b.bytes, b)));
                d.kept_bytes += b.bytes;
                while ((d.oldest.size() > CACHE_BLOCKS || d.kept_bytes > d.limit / (CACHE_SHARE / 2)) && drop_oldest(d, st)) {
                }
                continue;
            }
            may_keep = may_keep && e == cudaSuccess;
            give(b, [&] { cudaFreeAsync(b.ptr, st); });
        }
        if (e != cudaSuccess) cudaGetLastError();  // of these calls only
    }

    // Unused memory back to the system until the device's pools hold at most `keep` bytes; waits
    // for nothing: memory whose last use has not run yet stays.
    cudaError_t trim(int device, size_t keep) {
        std::lock_guard<std::mutex> lk(mu_);
        auto f = devices_.find(device);
        if (f == devices_.end()) return cudaSuccess;  // never used
        Device &d = f->second;
        DeviceGuard g(device);
        if (g.error() != cudaSuccess) return g.error();
        for (int pass = 0; pass < 2; ++pass) {  // the pools' free memory, then with the kept blocks'
            size_t held = 0;
            for (auto &p : d.pools) held += reserved_of(p.second);
            if (held <= keep) return cudaSuccess;
            if (pass == 1)
                for (auto i = d.oldest.begin(); i != d.oldest.end();) {
                    const auto next = std::next(i);
                    if (passed(i->second.second->second)) drop(d, i);
                    i = next;
                }
            for (auto &p : d.pools) {
                if (held <= keep) return cudaSuccess;
                const size_t before = reserved_of(p.second);
                const cudaError_t e = give_back(p.second, before - std::min(before, held - keep));
                if (e != cudaSuccess) return e;
                held -= before - std::min(before, reserved_of(p.second));
            }
        }
        return cudaSuccess;
    }

    // Memory that the device's pools hold without use, and the kept blocks.
    size_t unused(int device) {
        std::lock_guard<std::mutex> lk(mu_);
        auto f = devices_.find(device);
        if (f == devices_.end()) return 0;
        size_t n = f->second.kept_bytes;
        for (auto &p : f->second.pools) {
            const size_t r = reserved_of(p.second);
            n += r - std::min(r, p.second.live);
        }
        return n;
    }

  private:
    using Kept = std::multimap<size_t, Block>;
    struct Device {
        size_t limit = 0;  // half of the device's memory
        std::map<std::pair<size_t, bool>, SizePool> pools;  // by size (0: any) and use
        Kept kept[2];                                       // free small blocks of results, temporaries
        std::map<uint64_t, std::pair<Kept *, Kept::iterator>> oldest;  // and by age
        size_t kept_bytes = 0;
    };
    std::mutex mu_;
    std::map<int, Device> devices_;
    uint64_t clock_ = 0;

    static size_t reserved_of(const SizePool &p) {
        uint64_t r = 0;
        if (cudaMemPoolGetAttribute(p.pool, cudaMemPoolAttrReservedMemCurrent, &r) == cudaSuccess) return (size_t)r;
        cudaGetLastError();
        return p.reserved;
    }
    static cudaError_t give_back(SizePool &p, size_t keep) {
        const cudaError_t e = cudaMemPoolTrimTo(p.pool, keep);
        if (e == cudaSuccess) p.reserved = std::max(p.live, reserved_of(p));
        return e;
    }

    static bool passed(const Block &b) {
        if (cudaEventQuery(b.freed) == cudaSuccess) return true;
        cudaGetLastError();
        return false;
    }
    template <typename F>
    void give(const Block &b, F release) {
        if (b.freed) cudaEventDestroy(b.freed);
        release();
        b.from->live -= b.bytes;
        b.from->stamp = ++clock_;
    }
    // A kept block leaves: its last use is over, or it is freed in the order of st.
    Block forget(Device &d, std::map<uint64_t, std::pair<Kept *, Kept::iterator>>::iterator i) {
        const Block b = i->second.second->second;
        i->second.first->erase(i->second.second);
        d.oldest.erase(i);
        d.kept_bytes -= b.bytes;
        return b;
    }
    void drop(Device &d, std::map<uint64_t, std::pair<Kept *, Kept::iterator>>::iterator i) {
        const Block b = forget(d, i);
        give(b, [&] { cudaFree(b.ptr); });  // of a pool's block: waits for nothing
    }
    // The longest kept block whose last use is over, or is on st, back to its pool; false without one.
    bool drop_oldest(Device &d, cudaStream_t st) {
        for (auto i = d.oldest.begin(); i != d.oldest.end(); ++i) {
            if (passed(i->second.second->second)) {
                drop(d, i);
                return true;
            }
            if (i->second.second->second.st == st) {
                const Block b = forget(d, i);
                cudaStreamWaitEvent(st, b.freed, 0);
                give(b, [&] { cudaFreeAsync(b.ptr, st); });
                return true;
            }
        }
        return false;
    }
    // A kept block of `size` or up to an eighth more for stream st, or false.
    bool take_kept(int device, bool temp, size_t size, cudaStream_t st, Block *out) {
        std::lock_guard<std::mutex> lk(mu_);
        Device &d = devices_[device];
        Kept &m = d.kept[temp];
        for (auto i = m.lower_bound(size); i != m.end() && i->first <= size + size / 8; ++i) {
            if (i->second.st != st && !passed(i->second)) continue;
            if (cudaStreamWaitEvent(st, i->second.freed, 0) != cudaSuccess) {
                cudaGetLastError();
                return false;
            }
            *out = forget(d, d.oldest.find(i->second.stamp));
            return true;
        }
        return false;
    }

    // The pool of a size, made when it is first asked for (the device is current).
    cudaError_t pool_of(int device, bool temp, size_t size, Device **dev, SizePool **out) {
        Device &d = devices_[device];
        if (d.limit == 0) {
            size_t free_b = 0, total_b = 0;
            const cudaError_t e = cudaMemGetInfo(&free_b, &total_b);
            if (e != cudaSuccess) return e;
            d.limit = std::max<size_t>(total_b / 2, 1);
        }
        SizePool &p = d.pools[{size, temp}];
        if (p.pool == nullptr) {
            cudaMemPoolProps props;
            std::memset(&props, 0, sizeof(props));
            props.allocType = cudaMemAllocationTypePinned;
            props.handleTypes = cudaMemHandleTypeNone;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = device;
            cudaError_t e = cudaMemPoolCreate(&p.pool, &props);
            uint64_t keep = UINT64_MAX;  // freed memory stays with the pool
            if (e == cudaSuccess) {
                e = cudaMemPoolSetAttribute(p.pool, cudaMemPoolAttrReleaseThreshold, &keep);
                if (e != cudaSuccess) cudaMemPoolDestroy(p.pool);
            }
            if (e != cudaSuccess) {
                d.pools.erase({size, temp});
                return e;
            }
        }
        *dev = &d;
        *out = &p;
        return cudaSuccess;
    }

    cudaError_t take(int device, bool temp, size_t size, size_t bytes, cudaStream_t st, Block *out) {
        Device *d = nullptr;
        SizePool *p = nullptr;
        {
            std::lock_guard<std::mutex> lk(mu_);
            const cudaError_t e = pool_of(device, temp, size, &d, &p);
            if (e != cudaSuccess) return e;
            p->live += bytes;
            p->stamp = ++clock_;
        }
        const cudaError_t e = cudaMallocFromPoolAsync(&out->ptr, bytes, p->pool, st);  // may map memory: others go on
        std::lock_guard<std::mutex> lk(mu_);
        if (e != cudaSuccess) {
            p->live -= bytes;
            return e;
        }
        out->bytes = bytes;
        out->from = p;
        if (p->live <= p->reserved) return cudaSuccess;
        p->reserved = p->live;
        // it grew: the pools longest unused give memory back while all hold more than the limit
        size_t held = 0;
        for (auto &q : d->pools) held += q.second.reserved;
        while (held > d->limit) {
            SizePool *old = nullptr;
            for (auto &q : d->pools)
                if (q.second.reserved > q.second.live && (old == nullptr || q.second.stamp < old->stamp)) old = &q.second;
            if (old == nullptr) break;
            const size_t before = old->reserved;
            if (give_back(*old, old->live) != cudaSuccess) cudaGetLastError();
            if (old->reserved >= before) break;  // its frees have not run yet
            held -= before - old->reserved;
        }
        return cudaSuccess;
    }
};

// When a plan's array is released.
constexpr int LIFE_SYMBOLIC = 0;  // when spgemm_symbolic returns
constexpr int LIFE_NUMERIC = 1;   // when spgemm_numeric returns
constexpr int LIFE_PLAN = 2;      // by spgemm_free

// The device memory of one plan, by lifetime (symbolic: stage-1 and binning scratch; numeric: C~,
// merge pools and lists; plan: the rest).  Arrays of at most SMALL bytes share blocks of CHUNK
// bytes: a product on a few thousand rows makes 5 allocations instead of 21, which had taken a
// sixth of its time.  held and peak count what the arrays ask for.  A plan with a limit gets
// blocks of just those bytes, one per array, so that the limit is of the memory itself; the
// blocks of other plans are up to a sixteenth (kept ones an eighth) larger, and their shared
// blocks hold up to CHUNK bytes more per lifetime.
class PlanMemory {
  public:
    int64_t limit = 0;  // bytes, 0: none
    int64_t held = 0, peak = 0;
    int64_t blocks = 0;  // taken so far

    cudaError_t alloc(DeviceMemory &m, int device, cudaStream_t st, size_t bytes, int life, void **p) {
        *p = nullptr;
        if (bytes == 0) bytes = 16;
        if (limit > 0 && held + (int64_t)bytes > limit) return cudaErrorMemoryAllocation;
        Life &l = life_[life];
        const size_t need = (bytes + 255) & ~size_t(255);
        if (need > SMALL || limit > 0) {
            const cudaError_t e = block(m, device, st, bytes, life, p);
            if (e != cudaSuccess) return e;
        } else {
            if (l.room < need) {
                void *q = nullptr;
                const cudaError_t e = block(m, device, st, CHUNK, life, &q);
                if (e != cudaSuccess) return e;
                l.open = static_cast<char *>(q);
                l.room = CHUNK;
            }
            *p = l.open;
            l.open += need;
            l.room -= need;
        }
        l.bytes += (int64_t)bytes;
        held += (int64_t)bytes;
        peak = std::max(peak, held);
        return cudaSuccess;
    }

    // Stream-ordered on st.
    void release(DeviceMemory &m, int device, cudaStream_t st, int life) {
        Life &l = life_[life];
        m.free(device, l.blocks.data(), l.blocks.size(), life != LIFE_PLAN, st);
        held -= l.bytes;
        l = Life{};
    }

  private:
    static constexpr size_t CHUNK = 512 * 1024, SMALL = 64 * 1024;
    struct Life {
        std::vector<Block> blocks;
        int64_t bytes = 0;     // asked for
        char *open = nullptr;  // rest of the last shared block
        size_t room = 0;
    };
    Life life_[3];

    cudaError_t block(DeviceMemory &m, int device, cudaStream_t st, size_t bytes, int life, void **p) {
        Block b;
        const cudaError_t e = m.alloc(device, life != LIFE_PLAN, bytes, limit > 0, st, &b);
        ++blocks;
        if (e != cudaSuccess) return e;
        life_[life].blocks.push_back(b);
        *p = b.ptr;
        return cudaSuccess;
    }
};

}  // namespace spg
