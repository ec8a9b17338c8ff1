// Polling a word that a kernel writes to mapped host memory, on any host processor.
#pragma once
#include <atomic>

namespace dsf {

// between two looks: tells the core that this is a wait
inline void spin_pause() {
#if defined(__x86_64__) || defined(__i386__)
    __builtin_ia32_pause();
#elif defined(__aarch64__)
    asm volatile("yield" ::: "memory");
#endif
}
// after the last look: what the kernel wrote before the word is read after it (x86 keeps the order of loads by itself)
inline void spin_done() { std::atomic_thread_fence(std::memory_order_acquire); }

}  // namespace dsf
