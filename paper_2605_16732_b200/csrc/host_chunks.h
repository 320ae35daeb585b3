// How dirotq_linear_host cuts a call into row chunks and in which order it enqueues them.  Plain C++: the order is written against an
// interface (Ops), so that it can be checked, failures included, without a device.
#pragma once
#include <algorithm>
#include <stddef.h>

namespace dirotq {

constexpr int kMaxHostChunks = 32;
constexpr int kMinPipelinedRows = 512;  // shorter calls stay in one piece

// What a chunk costs beside its bytes is about 15 us for starting its copies and, with few rows, more per row for the kernels (at
// least 256 rows); what it saves is overlap, of which the first copy in and the last rows' computation and copy out have none.  So a full
// chunk is about 8 MB of the larger side, of a short call a little over a quarter (10 / 37: 4608 rows of 3072 are 768 + 1280 + 1280 + 768 +
// 512, where an exact quarter leaves a sixth chunk of 128), of a long one at least M / 24 rows (the event tables hold 32 chunks), the first one
// three fifths of that, and the end is cut in fifths 3 : 2 while it is longer than 384 rows or two fifths of a chunk.
// Measured from pinned memory, us, before (one piece below 2048 rows, up to eight equal chunks above) / after: 3072 -> 3072 at 1024,
// 4608 and 9216 rows 386 / 258, 889 / 829, 1662 / 1578; 1152 -> 4608 at 1024 258 / 237; 12288 -> 12288 at 4608 3401 / 2872; the widest
// layers' many chunks each read their rotation again and still gain up to some 5000 rows: 12288 -> 3072 at 1024, 4608 and 9216
// 936 / 694, 2593 / 2504, 4700 / 4841.  Chunks that grow with the root of the call's bytes come out the same on average.
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
