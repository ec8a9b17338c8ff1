// The host-side services of the library (csrc/dsfacto_host.cuh) by themselves, without a GPU: the CUDA runtime calls
// that they make are defined here, device memory is ordinary memory.  Built and run by test_host_services.py; the
// argument names the check, exit status 0 means that it holds.
#include "dsfacto_host.cuh"
#include "dsfacto_request.h"
#include "dsfacto_words.h"

#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <random>

// memory of the host may run out at any allocation of the library
static thread_local int t_left = -1;   // allocations until then (-1: never)

// ---- the runtime ----
static std::mutex g_mu;
static std::condition_variable g_cv;
static std::map<char *, size_t> g_device;          // device blocks alive
static size_t g_device_bytes = 0;
static const size_t kDeviceTotal = (size_t)64 << 20;   // of which the pool may keep a 64th
static cudaStream_t g_slow = nullptr;              // copies on this stream wait until g_go (10 s at most)
static bool g_go = false, g_gave_up = false;

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { *f = *t = kDeviceTotal; return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (g_device_bytes + n > kDeviceTotal) return cudaErrorMemoryAllocation;
    *p = std::malloc(n);
    { const int left = t_left; t_left = -1; g_device[(char *)*p] = n; t_left = left; }   // (the runtime has its own memory)
    g_device_bytes += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    std::lock_guard<std::mutex> lock(g_mu);
    const auto it = g_device.find((char *)p);
    if (it == g_device.end()) { std::puts("cudaFree of an unknown block"); std::exit(1); }
    g_device_bytes -= it->second;
    g_device.erase(it);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostRegister(void *, size_t, unsigned) { return cudaSuccess; }
cudaError_t cudaHostUnregister(void *) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = std::malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *at, const void *) { at->type = cudaMemoryTypeUnregistered; return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *to, const void *from, size_t n, cudaMemcpyKind, cudaStream_t st) {
    if (st != nullptr && st == g_slow) {
        std::unique_lock<std::mutex> lock(g_mu);
        if (!g_cv.wait_for(lock, std::chrono::seconds(10), [] { return g_go || g_gave_up; })) g_gave_up = true;
    }
    std::memcpy(to, from, n);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free((void *)e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
}

void *operator new(size_t n) {
    if (t_left == 0) throw std::bad_alloc();
    if (t_left > 0) --t_left;
    void *p = std::malloc(n);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

#define NEED(cond)                                                         \
    do {                                                                   \
        if (!(cond)) { std::printf("line %d: %s\n", __LINE__, #cond); return 1; } \
    } while (0)

// A transfer that takes long does not hold up another thread's, in either direction.
static int transfers(bool to_device) {
    using dsf::Courier;
    const size_t big = (size_t)24 << 20, small = (size_t)8 << 20;
    std::vector<char> a(big, 1), a2(big, 0), b(small, 2), b2(small, 0);
    const cudaStream_t slow = (cudaStream_t)&a, other = (cudaStream_t)&b;
    g_slow = slow;
    cudaError_t ea = cudaErrorUnknown;
    std::thread first([&] { ea = Courier::get().move(true, {{a2.data(), a.data(), big}}, slow); });
    std::this_thread::sleep_for(std::chrono::milliseconds(200));   // (the first is under way)
    const cudaError_t eb = Courier::get().move(to_device, {{to_device ? b2.data() : b.data(), to_device ? b.data() : b2.data(), small}}, other);
    { std::lock_guard<std::mutex> lock(g_mu); g_go = true; }
    g_cv.notify_all();
    first.join();
    NEED(!g_gave_up);
    NEED(ea == cudaSuccess && eb == cudaSuccess && a2 == a && b2 == b);
    return 0;
}

// Several threads at once: blocks handed out do not overlap, what is kept stays within its bound, all goes back.
static int threads() {
    using namespace dsf;
    std::atomic<int> wrong{0};
    auto work = [&](unsigned seed) {
        std::mt19937 rng(seed);
        std::vector<std::pair<char *, size_t>> dev, res;
        std::vector<char> src((size_t)3 << 20), dst(src.size());
        for (int step = 0; step < 400; ++step) {
            const size_t n = 1 + rng() % ((size_t)1 << (8 + rng() % 11));
            void *p = nullptr;
            if (DevicePool::get().alloc(&p, n) == cudaSuccess) { std::memset(p, (int)seed, n); dev.push_back({(char *)p, n}); }
            if (void *q = ResultBuffers::get().alloc(n)) { std::memset(q, (int)seed, n); res.push_back({(char *)q, n}); }
            void *m = Mailboxes::get().take();
            std::memset(m, (int)seed, kMailboxBytes);
            if (step % 40 == 0) {
                std::memset(src.data(), (int)(seed + step), src.size());
                void *d = nullptr;
                if (DevicePool::get().alloc(&d, src.size()) == cudaSuccess) {
                    if (Courier::get().move(true, {{d, src.data(), src.size()}}, nullptr) != cudaSuccess ||
                        Courier::get().move(false, {{d, dst.data(), src.size()}}, nullptr) != cudaSuccess || src != dst) ++wrong;
                    DevicePool::get().free(d);
                }
            }
            for (size_t k = 0; k < kMailboxBytes; k += 4096) if (((char *)m)[k] != (char)seed) ++wrong;
            Mailboxes::get().give(m);
            while (dev.size() > 8 || (step == 399 && !dev.empty())) {
                const auto b = dev[rng() % dev.size()];
                for (size_t k = 0; k < b.second; ++k) if (b.first[k] != (char)seed) { ++wrong; break; }
                DevicePool::get().free(b.first);
                dev.erase(std::find(dev.begin(), dev.end(), b));
            }
            while (res.size() > 4 || (step == 399 && !res.empty())) {
                const auto b = res[rng() % res.size()];
                for (size_t k = 0; k < b.second; ++k) if (b.first[k] != (char)seed) { ++wrong; break; }
                ResultBuffers::get().free(b.first);
                res.erase(std::find(res.begin(), res.end(), b));
            }
            if (step % 100 == 50) DevicePool::get().trim();
            if (DevicePool::get().idle_bytes() > kDeviceTotal / 64) ++wrong;
        }
    };
    std::vector<std::thread> team;
    for (unsigned k = 1; k <= 6; ++k) team.emplace_back(work, k);
    for (std::thread &t : team) t.join();
    NEED(wrong == 0);
    DevicePool::get().trim();
    ResultBuffers::get().trim();
    Mailboxes::get().trim();
    NEED(g_device.empty() && g_device_bytes == 0);
    return 0;
}

// Without host memory for its lists the pool reports an allocation as failed and gives a freed block back: nothing is
// thrown, nothing is lost.
static int no_host_memory() {
    using dsf::DevicePool;
    dsf::Mailboxes::get();
    DevicePool::get();
    for (int left = 0; left < 8; ++left) {
        void *p = nullptr, *q = nullptr;
        t_left = left;
        const cudaError_t e = DevicePool::get().alloc(&p, 5000);
        t_left = -1;
        NEED((e == cudaSuccess) == (p != nullptr));
        if (!p) NEED(e == cudaErrorMemoryAllocation && DevicePool::get().alloc(&p, 5000) == cudaSuccess);
        NEED(DevicePool::get().alloc(&q, 100000) == cudaSuccess);
        std::memset(p, 1, 5000);
        t_left = left;
        DevicePool::get().free(p);
        DevicePool::get().free(q);
        void *box = dsf::Mailboxes::get().take();
        dsf::Mailboxes::get().give(box);
        DevicePool::get().trim();
        t_left = -1;
        NEED(DevicePool::get().idle_bytes() == 0 && g_device.empty() && g_device_bytes == 0);
    }
    return 0;
}

// Small batches whose own bytes fit the mailbox are laid out in it, however unequal their rows, and every block, read as
// request_kernel reads it, holds its rows.
static int requests() {
    using namespace dsf;
    std::mt19937 rng(7);
    std::lognormal_distribution<double> uneven(2.0, 1.2);
    const size_t mail = kMailboxBytes - 256;
    int fitted = 0;
    for (int round = 0; round < 3000; ++round) {
        const bool labels = round % 2 == 1;
        const int64_t m = round < 40 ? 1 + round / 2 : 1 + (int64_t)(rng() % (1u << (4 + rng() % 11)));
        std::vector<int64_t> indptr(1, 0);
        for (int64_t i = 0; i < m; ++i) {
            int64_t len = round % 5 == 0 ? 8 : round % 5 == 1 ? (int64_t)uneven(rng) : round % 5 == 2 ? (int64_t)(rng() % 3) : round % 5 == 3 ? 0 : 26 + rng() % 51;
            if (i == m / 2) len += round % 3 == 0 ? 400 : round % 3 == 1 ? 0 : 1 + rng() % 9000;   // one long row
            indptr.push_back(indptr.back() + len);
        }
        const int64_t nnz = indptr.back();
        const size_t scores = labels ? 0 : ((size_t)m * 8 + 15) / 16 * 16;
        const size_t own = 8 * (size_t)(m + 1) + 8 * (size_t)nnz + 4 * (size_t)m;   // row pointers, entries, labels or scores
        const RequestLayout lay = scores < mail ? request_layout(m, nnz, labels, mail - scores, 8, 296) : RequestLayout();
        if (own <= mail) NEED(lay.rows > 0);
        if (lay.rows == 0) continue;
        ++fitted;
        NEED(lay.rows <= kMostBlockRows && lay.blocks <= kMostBlocks && (int64_t)lay.rows * lay.blocks >= m && (int64_t)lay.rows * (lay.blocks - 1) < m);
        std::vector<int32_t> indices((size_t)nnz), box((mail - scores) / 4 + 64, -1);
        std::vector<float> values((size_t)nnz), y((size_t)m);
        for (int32_t &j : indices) j = (int32_t)(rng() >> 1);
        for (float &x : values) x = (float)rng();
        for (float &x : y) x = (float)rng();
        uint16_t at[kMostBlocks + 1];
        const size_t largest = lay_out_request(box.data(), lay, m, indptr.data(), indices.data(), values.data(), labels ? y.data() : nullptr, at);
        size_t most = 0;
        for (size_t k = at[lay.blocks]; k < box.size(); ++k) NEED(box[k] == -1);   // nothing behind the last word
        NEED(4 * (size_t)((at[lay.blocks] + 3) / 4 * 4) <= mail - scores);         // nor is read, with the unit it lies in
        for (int b = 0; b < lay.blocks; ++b) {
            const int units = (at[b + 1] + 3) / 4 - at[b] / 4;
            most = std::max(most, (size_t)units * 16);
            std::vector<int32_t> block(box.begin() + at[b] / 4 * 4, box.begin() + at[b] / 4 * 4 + units * 4);
            const int64_t r0 = (int64_t)b * lay.rows;
            const int rows = (int)std::min<int64_t>(lay.rows, m - r0);
            const int32_t *ends = block.data() + at[b] % 4, *idx = ends + rows;
            const int entries = ends[rows - 1];
            NEED(entries == indptr[r0 + rows] - indptr[r0] && at[b + 1] - at[b] == rows * (labels ? 2 : 1) + 2 * entries);
            for (int r = 0; r < rows; ++r) {
                const int beg = r > 0 ? ends[r - 1] : 0, len = ends[r] - beg;
                NEED(len == indptr[r0 + r + 1] - indptr[r0 + r]);
                if (len == 0) continue;
                NEED(std::memcmp(idx + beg, indices.data() + indptr[r0 + r], 4 * (size_t)len) == 0);
                NEED(std::memcmp(idx + entries + beg, values.data() + indptr[r0 + r], 4 * (size_t)len) == 0);
            }
            if (labels) NEED(std::memcmp(idx + 2 * entries, y.data() + r0, 4 * (size_t)rows) == 0);
        }
        NEED(most == largest);
    }
    NEED(fitted > 1000);
    return 0;
}

// Scores that arrive one by one: the caller has all of them, or, where the kernel fails in between, none.
static int scores_in_words() {
    const int64_t m = 1000;
    const uint32_t number = 77;
    for (int64_t arriving : {(int64_t)0, (int64_t)1, m / 2, m - 1, m}) {
        std::vector<unsigned long long> words((size_t)m, (unsigned long long)(number - 1) << 32 | 5);
        std::vector<float> scores((size_t)m, -1.0f);
        const int rc = dsf::take_scores(words.data(), m, number, scores.data(), [&](auto arrived) {
            for (int64_t k = 0; k < arriving; ++k) {      // the last one first: order is nobody's promise
                const int64_t i = arriving == m ? m - 1 - k : k;
                const float f = (float)i + 0.5f;
                uint32_t bits;
                std::memcpy(&bits, &f, sizeof bits);
                const bool all = arrived();
                if (all) return 1;                        // too early
                words[(size_t)i] = (unsigned long long)number << 32 | bits;
            }
            return arrived() ? 0 : -5;
        });
        NEED(rc == (arriving == m ? 0 : -5));
        for (int64_t i = 0; i < m; ++i) NEED(scores[(size_t)i] == (arriving == m ? (float)i + 0.5f : -1.0f));
    }
    return 0;
}

int main(int argc, char **argv) {
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "transfers-in") return transfers(true);
    if (what == "transfers-out") return transfers(false);
    if (what == "threads") return threads();
    if (what == "no-host-memory") return no_host_memory();
    if (what == "requests") return requests();
    if (what == "scores") return scores_in_words();
    return 2;
}
