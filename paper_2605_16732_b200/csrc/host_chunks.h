// How dirotq_linear_host cuts a call into row chunks and in which order it enqueues them.  Plain C++: the order is written against an
// interface (Ops), so that it can be checked, failures included, without a device.
#pragma once
#include <algorithm>
#include <stddef.h>

namespace dirotq {

constexpr int kMaxHostChunks = 32;
constexpr int kMinPipelinedRows = 512;  // shorter calls stay in one piece

// A full chunk is about 8 MB of the larger side (smaller ones pay more for starting copies, about 15 us each, and, with few rows, more per
// row for the kernels), but a good quarter of a short call, and at least 256 rows.  The first one and the last ones are
// shorter: the first copy in, and the last rows' computation and copy out, overlap with nothing.  4608 x 3072 -> 3072: 915 us
// in four equal chunks, 850 tapered; 1024 x 3072 -> 3072 311 us in one piece, 236 in chunks.
// `xrow`, `yrow`: bytes of a token row in and out.  Returns the number of chunks, whose sizes it writes to `rows`.
inline int plan_host_chunks(int M, size_t xrow, size_t yrow, int rows[kMaxHostChunks]) {
    constexpr size_t CHUNK_BYTES = 8u << 20;
    auto rows128 = [](long r) { return (r + 127) / 128 * 128; };
    long base = static_cast<long>(CHUNK_BYTES / std::max(xrow, yrow));
    base = rows128(std::max(std::min(base, M * 10L / 37), std::max(256L, M / 24L)));  // (at most kMaxHostChunks in all)
    int n = 0;
    for (long m0 = 0, mc = 0; m0 < M; m0 += mc) {
        const long left = M - m0;
        mc = left <= std::max(384L, 2 * base / 5) ? left : std::max(256L, std::min(rows128(3 * left / 5), m0 ? base : rows128(3 * base / 5)));
        rows[n++] = static_cast<int>(mc);
    }
    return n;
}

// Enqueues the chunks: copy in, compute, copy out, chunk by chunk.  Whatever fails on the way, join() comes last: it orders the
// caller's stream behind every copy that was enqueued, so that the caller may reuse its buffers after synchronising that stream.
template <typename Ops>
bool run_host_chunks(const int* rows, int n, Ops& ops) {
    bool ok = ops.fork();
    for (int c = 0, m0 = 0; ok && c < n; m0 += rows[c++]) ok = ops.copy_in(c, m0, rows[c]) && ops.compute(c, m0, rows[c]) && ops.copy_out(c, m0, rows[c]);
    return ops.join(ok) && ok;
}

}  // namespace dirotq
