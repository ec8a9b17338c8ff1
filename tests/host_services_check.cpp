// The host-side services of the library (csrc/dsfacto_host.cuh) by themselves, without a GPU: the CUDA runtime calls
// that they make are defined here, device memory is ordinary memory.  Built and run by test_host_services.py; the
// argument names the check, exit status 0 means that it holds.
#include "dsfacto_host.cuh"

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

int main(int argc, char **argv) {
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "transfers-in") return transfers(true);
    if (what == "transfers-out") return transfers(false);
    if (what == "threads") return threads();
    if (what == "no-host-memory") return no_host_memory();
    return 2;
}
