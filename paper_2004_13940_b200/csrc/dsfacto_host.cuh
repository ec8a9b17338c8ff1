// Host-side services of the library: the device memory pool and the transfers between pageable caller memory and
// the device.
#pragma once
#include <cuda_runtime.h>
#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <condition_variable>
#include <cstdint>
#include <cstring>
#include <initializer_list>
#include <map>
#include <mutex>
#include <new>
#include <thread>
#include <unordered_map>
#include <vector>

namespace dsf {

// ------------------------------------------------------------------------------------------
// Device memory.  cudaMalloc and cudaFree cost 0.4 and 0.3 ms whatever the size, and a load makes some thirty of
// each: a load of 2.6 M entries spent nine tenths of its time there.  Freed blocks are kept per device, up to a
// 64th of its memory, and handed out again for requests of about their size; they go back to the driver when an
// allocation fails, when the bound is reached (those that have been idle longest), and with trim().
// A block is freed only after the work that used it has finished (callers synchronise their stream first), so it may
// be handed to any thread and stream.
// ------------------------------------------------------------------------------------------
class DevicePool {
public:
    static DevicePool &get() {
        static DevicePool *pool = new DevicePool;   // (never destroyed: handles may outlive static destruction)
        return *pool;
    }
    cudaError_t alloc(void **out, size_t bytes) {
        *out = nullptr;
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const size_t unit = bytes > ((size_t)1 << 20) ? (size_t)1 << 21 : 4096;   // large blocks are mapped in 2 MB pages anyway
        const size_t size = (std::max<size_t>(bytes, 1) + unit - 1) / unit * unit;
        {
            std::lock_guard<std::mutex> lock(mu_);
            try {
                std::multimap<size_t, Idle> &idle = idle_[dev];
                const auto it = idle.lower_bound(size);
                if (it != idle.end() && it->first <= size + size / 4) {
                    live_[it->second.ptr] = {it->first, dev};
                    *out = it->second.ptr;
                    idle_bytes_[dev] -= it->first;
                    idle.erase(it);
                    return cudaSuccess;
                }
            } catch (const std::bad_alloc &) { return cudaErrorMemoryAllocation; }
        }
        e = cudaMalloc(out, size);
        if (e == cudaErrorMemoryAllocation) {
            cudaGetLastError();
            trim();
            e = cudaMalloc(out, size);
        }
        if (e != cudaSuccess) return e;
        try {
            std::lock_guard<std::mutex> lock(mu_);
            live_[*out] = {size, dev};
        } catch (const std::bad_alloc &) {
            cudaFree(*out);
            *out = nullptr;
            return cudaErrorMemoryAllocation;
        }
        return cudaSuccess;
    }
    void free(void *ptr) {
        if (!ptr) return;
        for (;;) {
            void *go = ptr;   // back to the driver: this block, or the ones that have been idle longest, to make room for it
            {
                std::lock_guard<std::mutex> lock(mu_);
                const auto it = live_.find(ptr);
                if (it != live_.end()) {
                    const Block b = it->second;
                    try {
                        const size_t most = bound(b.dev);
                        size_t &held = idle_bytes_[b.dev];
                        std::multimap<size_t, Idle> &idle = idle_[b.dev];
                        if (held + b.bytes <= most) {
                            idle.emplace(b.bytes, Idle{ptr, ++clock_});
                            held += b.bytes;
                            live_.erase(it);
                            return;
                        }
                        if (b.bytes <= most) {
                            auto old = idle.begin();
                            for (auto q = idle.begin(); q != idle.end(); ++q)
                                if (q->second.since < old->second.since) old = q;
                            go = old->second.ptr;
                            held -= old->first;
                            idle.erase(old);
                        }
                    } catch (const std::bad_alloc &) {}   // (no room in the lists)
                    if (go == ptr) live_.erase(it);
                }
            }
            cudaFree(go);
            if (go == ptr) return;
        }
    }
    // idle bytes on the current device
    size_t idle_bytes() {
        int dev = 0;
        cudaGetDevice(&dev);
        std::lock_guard<std::mutex> lock(mu_);
        const auto it = idle_bytes_.find(dev);
        return it == idle_bytes_.end() ? 0 : it->second;
    }
    void trim() {
        std::map<int, std::multimap<size_t, Idle>> go;
        {
            std::lock_guard<std::mutex> lock(mu_);
            go.swap(idle_);
            for (auto &held : idle_bytes_) held.second = 0;
        }
        for (auto &d : go)
            for (auto &b : d.second) cudaFree(b.second.ptr);
    }

private:
    struct Block { size_t bytes; int dev; };
    struct Idle { void *ptr; uint64_t since; };
    size_t bound(int dev) {   // (mu_ is held)
        auto it = bound_.find(dev);
        if (it == bound_.end()) {
            size_t free_b = 0, total_b = 0;
            if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) total_b = 0;
            it = bound_.emplace(dev, total_b / 64).first;
        }
        return it->second;
    }
    std::mutex mu_;
    std::map<int, std::multimap<size_t, Idle>> idle_;
    uint64_t clock_ = 0;
    std::map<int, size_t> idle_bytes_, bound_;
    std::unordered_map<void *, Block> live_;
};

// Page-locked host memory on 2 MB pages: 64 MB take 5 ms (touched by several threads, then registered) against 29 ms
// of cudaHostAlloc, which locks 4 KB pages.  bytes: a multiple of 2 MB.  NULL if it cannot be had.
constexpr size_t kHugePage = (size_t)2 << 20;
inline char *locked_alloc(size_t bytes) {
    char *raw = static_cast<char *>(mmap(nullptr, bytes + kHugePage, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0));
    if (raw == MAP_FAILED) return nullptr;
    char *p = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(raw) + kHugePage - 1) / kHugePage * kHugePage);
    if (p > raw) munmap(raw, (size_t)(p - raw));
    if (raw + kHugePage > p) munmap(p + bytes, (size_t)(raw + kHugePage - p));
    madvise(p, bytes, MADV_HUGEPAGE);
    const int pages = (int)(bytes / kHugePage), workers = pages >= 8 ? 4 : 1;
    auto touch = [=](int w) { for (int k = w; k < pages; k += workers) p[(size_t)k * kHugePage] = 0; };
    std::thread team[4];
    for (int w = 1; w < workers; ++w)
        try { team[w] = std::thread(touch, w); } catch (...) {}   // (registering touches what is left)
    touch(0);
    for (std::thread &t : team)
        if (t.joinable()) t.join();
    if (cudaHostRegister(p, bytes, cudaHostRegisterPortable | cudaHostRegisterMapped) != cudaSuccess) {
        cudaGetLastError();
        munmap(p, bytes);
        return nullptr;
    }
    return p;
}
inline void locked_free(char *p, size_t bytes) {
    cudaHostUnregister(p);
    munmap(p, bytes);
}

// ------------------------------------------------------------------------------------------
// Result buffers: page-locked memory that the Python binding hands out as arrays, so that results arrive at the
// link's speed and no page is touched for the first time on the way (71 MB of parameters: 2.5 -> 1.4 ms, 2.7 MB: 0.20
// -> 0.06 ms).  At most 512 MB exist at a time, in use or idle (beyond that a caller gets NULL and takes ordinary
// memory), at most 256 MB of them idle; trim() gives the idle ones back.
// ------------------------------------------------------------------------------------------
class ResultBuffers {
public:
    static ResultBuffers &get() {
        static ResultBuffers *r = new ResultBuffers;
        return *r;
    }
    void *alloc(size_t bytes) {
        const size_t size = size_of(bytes);
        std::lock_guard<std::mutex> lock(mu_);
        auto it = idle_.lower_bound(size);
        if (it == idle_.end() || (size > kSmallMost ? it->first > size + size / 4 : it->first != size)) {
            const size_t region = std::max(size, kHugePage);
            if (total_ + region > kMost) return nullptr;
            char *p = locked_alloc(region);
            if (!p) return nullptr;
            total_ += region;
            const int parts = (int)(region / size);
            for (int k = 0; k < parts; ++k) idle_.emplace(size, Part{p + (size_t)k * size, p});
            regions_[p] = {region, 0};
            idle_bytes_ += region;
            it = idle_.lower_bound(size);
        }
        const Part part = it->second;
        live_[part.ptr] = {it->first, part.region};
        regions_[part.region].live += 1;
        idle_bytes_ -= it->first;
        idle_.erase(it);
        return part.ptr;
    }
    void free(void *ptr) {
        std::lock_guard<std::mutex> lock(mu_);
        const auto it = live_.find(static_cast<char *>(ptr));
        if (it == live_.end()) return;
        idle_.emplace(it->second.bytes, Part{it->first, it->second.region});
        idle_bytes_ += it->second.bytes;
        regions_[it->second.region].live -= 1;
        live_.erase(it);
        if (idle_bytes_ > kMostIdle) release_idle();
    }
    void trim() {
        std::lock_guard<std::mutex> lock(mu_);
        release_idle();
    }

private:
    static constexpr size_t kMost = (size_t)512 << 20, kMostIdle = (size_t)256 << 20, kSmallMost = (size_t)1 << 20;
    struct Part { char *ptr, *region; };
    struct Live { size_t bytes; char *region; };
    struct RegionUse { size_t bytes; int live; };
    static size_t size_of(size_t bytes) {   // up to 1 MB a power of two (several share a page), then whole pages
        if (bytes > kSmallMost) return (bytes + kHugePage - 1) / kHugePage * kHugePage;
        size_t s = (size_t)32 << 10;
        while (s < bytes) s *= 2;
        return s;
    }
    void release_idle() {   // (mu_ is held) every region no part of which is in use
        for (auto it = idle_.begin(); it != idle_.end();) {
            if (regions_[it->second.region].live == 0) {
                idle_bytes_ -= it->first;
                it = idle_.erase(it);
            } else {
                ++it;
            }
        }
        for (auto it = regions_.begin(); it != regions_.end();) {
            if (it->second.live == 0) {
                locked_free(it->first, it->second.bytes);
                total_ -= it->second.bytes;
                it = regions_.erase(it);
            } else {
                ++it;
            }
        }
    }
    std::mutex mu_;
    std::multimap<size_t, Part> idle_;
    std::unordered_map<char *, Live> live_;
    std::map<char *, RegionUse> regions_;
    size_t total_ = 0, idle_bytes_ = 0;
};

// ------------------------------------------------------------------------------------------
// Transfers.  A copy between pageable memory and the device goes through the driver's staging buffer in one
// thread: 11 GB/s, and 5 GB/s into memory that has not been touched yet.  Large copies are therefore cut into regions
// that the calling thread and a few helpers take one after another, each through two page-locked slots of its own.
// 328 MB to the device, 4 threads: 43 GB/s (8 threads: 40; slots of 512 / 256 / 128 KB instead of 1 MB: 32 / 22 /
// 16, every copy costs the driver some 10 us); 67 MB into fresh memory, 8 threads: 34 GB/s (4 threads: 19, page
// faults).  The helpers sleep between transfers; nobody waits for a helper that has not woken up yet,
// so a busy machine costs bandwidth, not a stall.  One transfer at a time has the helpers; another thread's that
// finds them taken goes through the driver, beside the first (a request must not wait for a data set to pass).
// ------------------------------------------------------------------------------------------
struct Piece {            // one array of a transfer
    void *dev;
    void *host;
    size_t bytes;
};
class Courier {
public:
    static Courier &get() {
        static Courier *c = new Courier;   // (never destroyed: its helpers sleep until the process ends)
        return *c;
    }
    static constexpr size_t kSlot = (size_t)1 << 20, kRegion = (size_t)2 << 20;   // of what one copy moves; of what a thread takes
    static constexpr int kMostPieces = 8;
    // Smaller arrays go through the driver: 1 MB to the device takes 0.08 ms either way, 2.7 MB back 0.20 ms through
    // the driver and 0.28 ms with helpers that have to wake up first.
    static constexpr size_t kWorth = (size_t)1 << 20, kWorthBack = (size_t)6 << 20;
    // Copies the pieces on the stream.  From the device: on return host memory has been written.  To the device: copies
    // may still be under way, and page-locked host memory of the caller's is read by them, so the caller waits for the
    // stream before it gives host memory back.
    cudaError_t move(bool to_device, std::initializer_list<Piece> pieces, cudaStream_t st) { return move(to_device, pieces.begin(), (int)pieces.size(), st); }
    cudaError_t move(bool to_device, const Piece *pieces, int count, cudaStream_t st) {
        cudaError_t e = cudaSuccess;
        Piece large[kMostPieces];
        int nlarge = 0;
        for (int q = 0; q < count; ++q) {
            const Piece &p = pieces[q];
            if (p.bytes == 0) continue;
            bool direct = p.bytes < (to_device ? kWorth : kWorthBack);
            if (!direct) {   // page-locked caller memory needs no detour
                cudaPointerAttributes at{};
                if (cudaPointerGetAttributes(&at, p.host) != cudaSuccess) cudaGetLastError();
                else direct = at.type == cudaMemoryTypeHost || at.type == cudaMemoryTypeManaged;
            }
            if (!direct && nlarge < kMostPieces) { large[nlarge++] = p; continue; }
            e = to_device ? cudaMemcpyAsync(p.dev, p.host, p.bytes, cudaMemcpyHostToDevice, st)
                          : cudaMemcpyAsync(p.host, p.dev, p.bytes, cudaMemcpyDeviceToHost, st);
            if (e != cudaSuccess) return e;
        }
        if (nlarge > 0 && (e = staged(to_device, large, nlarge, st)) != cudaSuccess) return e;
        return to_device ? cudaSuccess : cudaStreamSynchronize(st);
    }

private:
    struct Lane {          // the page-locked slots of one thread
        char *slot[2] = {nullptr, nullptr};
        cudaEvent_t ev[2] = {nullptr, nullptr};
        bool busy[2] = {false, false};
    };
    struct Region { char *dev, *host; size_t bytes; };
    cudaError_t staged(bool to_device, const Piece *pieces, int count, cudaStream_t st) {
        std::unique_lock<std::mutex> one(transfer_, std::try_to_lock);
        cudaError_t e = cudaErrorNotReady;
        if (one.owns_lock()) {
            try {
                size_t most = 0;
                for (int q = 0; q < count; ++q) most += pieces[q].bytes / kSlot + 32;
                regions_.reserve(most);
                e = prepare();
            } catch (const std::bad_alloc &) { e = cudaErrorMemoryAllocation; }
            if (e != cudaSuccess) cudaGetLastError();
        }
        if (e != cudaSuccess) {   // another thread's transfer has them, or no page-locked memory or threads to be had: the driver's way
            for (int q = 0; q < count; ++q) {
                const Piece &p = pieces[q];
                if ((e = to_device ? cudaMemcpyAsync(p.dev, p.host, p.bytes, cudaMemcpyHostToDevice, st)
                                   : cudaMemcpyAsync(p.host, p.dev, p.bytes, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
                    return e;
            }
            return cudaSuccess;
        }
        regions_.clear();
        size_t all = 0, total = 0;
        for (int q = 0; q < count; ++q) total += pieces[q].bytes;
        for (int q = 0; q < count; ++q) {
            const Piece &p = pieces[q];
            char *d = static_cast<char *>(p.dev), *h = static_cast<char *>(p.host), *end = h + p.bytes;
            while (h < end) {
                size_t n;
                if (to_device) {   // small ones at the start, so that the link has work soon, and at the end, so that little is left then
                    n = all < ((size_t)2 << 20) ? kSlot / 4 : total - all < ((size_t)6 << 20) ? kSlot / 2 : kSlot;
                } else {           // on 2 MB boundaries: a huge page is touched by one thread
                    n = kRegion - reinterpret_cast<uintptr_t>(h) % kRegion;
                }
                n = std::min(n, (size_t)(end - h));
                all += n;
                regions_.push_back({d, h, n});
                d += n;
                h += n;
            }
        }
        to_device_ = to_device;
        stream_ = st;
        next_.store(0);
        error_.store(cudaSuccess);
        {
            std::lock_guard<std::mutex> lock(mu_);
            open_ = true;
            ++job_;
        }
        wake_.notify_all();
        work(lanes_[0]);
        std::unique_lock<std::mutex> lock(mu_);
        open_ = false;                                   // helpers that wake up now find nothing
        idle_.wait(lock, [&] { return active_ == 0; });   // those at work finish the region they have
        return (cudaError_t)error_.load();
    }
    void work(Lane &lane) {
        int turn = 0;
        auto note = [&](cudaError_t e) { if (e != cudaSuccess) error_.store(e); return e == cudaSuccess; };
        char *out[2] = {nullptr, nullptr};   // from the device: where the slot's contents go
        size_t out_n[2] = {0, 0};
        auto settle = [&](int t) {           // the copy that last used slot t has finished; its contents are passed on
            if (!lane.busy[t]) return;
            note(cudaEventSynchronize(lane.ev[t]));
            lane.busy[t] = false;
            if (out[t]) { std::memcpy(out[t], lane.slot[t], out_n[t]); out[t] = nullptr; }
        };
        for (size_t r; error_.load() == cudaSuccess && (r = next_.fetch_add(1)) < regions_.size();) {
            const Region &g = regions_[r];
            for (size_t at = 0; at < g.bytes; at += kSlot) {
                const size_t n = std::min(kSlot, g.bytes - at);
                settle(turn);
                if (to_device_) {
                    std::memcpy(lane.slot[turn], g.host + at, n);
                    if (!note(cudaMemcpyAsync(g.dev + at, lane.slot[turn], n, cudaMemcpyHostToDevice, stream_))) break;
                } else {
                    if (!note(cudaMemcpyAsync(lane.slot[turn], g.dev + at, n, cudaMemcpyDeviceToHost, stream_))) break;
                    out[turn] = g.host + at;
                    out_n[turn] = n;
                }
                if (!note(cudaEventRecord(lane.ev[turn], stream_))) break;
                lane.busy[turn] = true;
                turn ^= 1;
            }
        }
        if (!to_device_) { settle(turn); settle(turn ^ 1); }
    }
    cudaError_t prepare() {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (pid_ != getpid()) {   // first use, or the child of a fork, which has no helpers
            pid_ = getpid();
            lanes_.clear();
        }
        if (!lanes_.empty() && dev == device_) return cudaSuccess;
        // (events belong to a device: a process that works on several gets new ones when it changes over)
        const bool fresh = lanes_.empty();
        if (fresh) {
            const unsigned cores = std::max(2u, std::thread::hardware_concurrency());
            lanes_.resize(std::min(8u, cores / 2));
            if (!(arena_ = locked_alloc(lanes_.size() * 2 * kSlot))) { lanes_.clear(); return cudaErrorMemoryAllocation; }
            for (size_t k = 0; k < lanes_.size(); ++k)
                for (int t = 0; t < 2; ++t) lanes_[k].slot[t] = arena_ + (2 * k + t) * kSlot;
        }
        for (Lane &l : lanes_)
            for (int t = 0; t < 2; ++t) {
                if (l.ev[t]) { cudaEventSynchronize(l.ev[t]); cudaEventDestroy(l.ev[t]); }
                l.busy[t] = false;
                l.ev[t] = nullptr;
                if ((e = cudaEventCreateWithFlags(&l.ev[t], cudaEventDisableTiming)) != cudaSuccess) {
                    if (fresh) lanes_.clear();
                    device_ = -1;
                    return e;
                }
            }
        device_ = dev;
        if (fresh)
            for (size_t k = 1; k < lanes_.size(); ++k) {
                try { std::thread([this, k] { help(k); }).detach(); } catch (...) { lanes_.resize(k); break; }
            }
        return cudaSuccess;
    }
    void help(size_t k) {
        uint64_t seen = 0;
        int dev = -1;
        std::unique_lock<std::mutex> lock(mu_);
        for (;;) {
            wake_.wait(lock, [&] { return open_ && job_ != seen; });
            seen = job_;
            if (to_device_ && k >= 4) continue;
            ++active_;
            lock.unlock();
            if (dev != device_) { dev = device_; cudaSetDevice(dev); }
            work(lanes_[k]);
            lock.lock();
            if (--active_ == 0) idle_.notify_all();
        }
    }
    std::mutex transfer_, mu_;
    std::condition_variable wake_, idle_;
    bool open_ = false;
    uint64_t job_ = 0;
    int active_ = 0, device_ = -1;
    pid_t pid_ = 0;
    char *arena_ = nullptr;
    std::vector<Lane> lanes_;
    std::vector<Region> regions_;
    bool to_device_ = false;
    cudaStream_t stream_ = nullptr;
    std::atomic<size_t> next_{0};
    std::atomic<int> error_{0};
};

// Page-locked, mapped memory of a handle: what kernels report to the host, and small inputs and results.  Page-locking
// costs 0.45 ms per megabyte, so blocks of handles that are gone are kept for the next ones, eight of them at most.
constexpr size_t kMailboxBytes = (size_t)128 << 10;
class Mailboxes {
public:
    static Mailboxes &get() {
        static Mailboxes *m = new Mailboxes;
        return *m;
    }
    void *take() {
        {
            std::lock_guard<std::mutex> lock(mu_);
            if (!idle_.empty()) {
                void *p = idle_.back();
                idle_.pop_back();
                return p;
            }
        }
        void *p = nullptr;
        if (cudaHostAlloc(&p, kMailboxBytes, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        return p;
    }
    void give(void *p) {
        if (!p) return;
        {
            std::lock_guard<std::mutex> lock(mu_);
            try { if (idle_.size() < 8) { idle_.push_back(p); return; } } catch (const std::bad_alloc &) {}
        }
        cudaFreeHost(p);
    }
    void trim() {
        std::vector<void *> go;
        {
            std::lock_guard<std::mutex> lock(mu_);
            go.swap(idle_);
        }
        for (void *p : go) cudaFreeHost(p);
    }

private:
    std::mutex mu_;
    std::vector<void *> idle_;
};

}  // namespace dsf
