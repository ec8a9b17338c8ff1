// A small scoring batch (a request) as the host lays it out in mapped memory for request_kernel.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <cstring>

namespace dsf {

// Blocks of consecutive rows, one per CTA, one behind the other without gaps.  A block of r rows and e entries is 32-bit words:
// ends[r] (where each row ends among the block's entries), then e columns, e values and, for held-out rows, r labels.  So a
// batch takes no more than its own bytes, however unequal its rows are.  Where each block lies goes along with the launch, so
// that a CTA still has its rows after one trip across the link (which costs 0.2 us of the 12.5 that a row of 39 entries takes).
// (When every block took the bytes of the largest one, 290 rows were the most of a batch of 8 entries a row with one of 400, and
// larger ones went by copies to the device.  Calls of dsfacto_predict / dsfacto_evaluate, K = 16, in us, so and now: 1000 rows
// of 8 entries with one of 400 75 / 66 -> 44 / 43, 300 rows of log-normal lengths of mean 40 78 / 68 -> 42 / 40, 1600 of mean
// 8 55 / 43 -> 38 / 40, one row of 9000 entries among 2000 empty ones 840 -> 364 / 278.)
constexpr int kMostBlockRows = 64;
constexpr int kMostBlocks = 320;     // of a batch (their places take 642 bytes of the kernel's parameters)
constexpr size_t kMostRequestBytes = (size_t)128 << 10;
static_assert(kMostRequestBytes / 4 <= 65535, "the place of a block fits 16 bits");
static_assert(kMostRequestBytes / 8 / kMostBlockRows < kMostBlocks, "a row takes eight bytes at least: its end, and its score or label");

struct RequestLayout {
    int rows = 0;        // of a block; 0: the batch does not fit
    int blocks = 0;
};
// 32-bit words in front of row r0, which entries[r0] entries precede
inline int64_t request_words(int64_t rows, int64_t entries, bool labels) { return rows * (labels ? 2 : 1) + 2 * entries; }
// room: bytes of the mailbox left for the rows, a multiple of 16; warps: of a CTA; ctas: the most that are to be launched
inline RequestLayout request_layout(int64_t m, int64_t nnz, bool labels, size_t room, int warps, int ctas) {
    RequestLayout r;
    const int64_t words = (int64_t)(std::min(room, kMostRequestBytes) / 4);
    if (m < 1 || m > words || nnz < 0 || nnz > words || request_words(m, nnz, labels) > words) return r;
    // a row per warp while that leaves no more CTAs than that
    const int64_t at_once = (int64_t)warps * std::min(ctas, kMostBlocks), per_warp = (m + at_once - 1) / at_once;
    const int rows = (int)std::min<int64_t>(warps * per_warp, kMostBlockRows), blocks = (int)((m + rows - 1) / rows);
    if (blocks > kMostBlocks) return r;
    r.rows = rows;
    r.blocks = blocks;
    return r;
}
// Rows that are known to be sound.  at[b]: the first word of block b, at[blocks]: the number of words.  Returns the bytes that
// the largest block takes with the 16-byte units it begins and ends in.
__attribute__((noinline)) inline size_t lay_out_request(int32_t *to, const RequestLayout &lay, int64_t m, const int64_t *indptr, const int32_t *indices, const float *values,
                              const float *y, uint16_t *at) {
    size_t largest = 0;
    int64_t word = 0;
    for (int b = 0; b < lay.blocks; ++b) {
        const int64_t r0 = (int64_t)b * lay.rows, r1 = std::min<int64_t>(m, r0 + lay.rows), e0 = indptr[r0];
        const size_t e = (size_t)(indptr[r1] - e0), rows = (size_t)(r1 - r0);
        int32_t *ends = to + word;
        for (size_t r = 0; r < rows; ++r) ends[r] = (int32_t)(indptr[r0 + 1 + (int64_t)r] - e0);
        int32_t *entries = ends + rows;
        if (e > 0) { std::memcpy(entries, indices + e0, 4 * e); std::memcpy(entries + e, values + e0, 4 * e); }
        if (y) std::memcpy(entries + 2 * e, y + r0, 4 * rows);
        at[b] = (uint16_t)word;
        const int64_t next = word + request_words((int64_t)rows, (int64_t)e, y != nullptr);
        largest = std::max(largest, (size_t)((next + 3) / 4 - word / 4) * 16);
        word = next;
    }
    at[lay.blocks] = (uint16_t)word;
    return largest;
}

}  // namespace dsf
