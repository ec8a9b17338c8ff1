// The host's side of words that a kernel writes to mapped host memory: 64 bits each, the upper half the number of the report
// (or call) that they belong to, the lower 32 bits of its contents.
#pragma once
#include <cstdint>
#include <cstring>

namespace dsf {

inline uint32_t word_number(const unsigned long long &word) { return (uint32_t)(*const_cast<const volatile unsigned long long *>(&word) >> 32); }
// whether a word carries the number, and then its contents
inline bool take_word(const unsigned long long &word, uint32_t number, uint32_t &contents) {
    const unsigned long long x = *const_cast<const volatile unsigned long long *>(&word);
    contents = (uint32_t)x;
    return (uint32_t)(x >> 32) == number;
}
// Scores that arrive as words each.  wait(arrived) asks until all are there or the kernel has failed, and returns a status; the
// caller's array is written only when it has all of them.  Meanwhile they are moved together at the front of the words, where
// each has been taken before its place is written (after the wait, a second pass over 5000 words took 1.5 us of a call's 32).
template <class Wait>
int take_scores(unsigned long long *words, int64_t m, uint32_t number, float *scores, Wait wait) {
    char *taken = reinterpret_cast<char *>(words);
    int64_t at = 0;
    uint32_t bits;
    const int rc = wait([&]() {
        for (; at < m && take_word(words[at], number, bits); ++at) std::memcpy(taken + 4 * at, &bits, 4);
        return at == m;
    });
    if (!rc) std::memcpy(scores, taken, 4 * (size_t)m);
    return rc;
}

}  // namespace dsf
