// Host loops of the setup on several threads.
#pragma once

#include <algorithm>
#include <cstdint>
#include <exception>
#include <thread>
#include <vector>

namespace ams {

// f(begin, end, chunk) over [0, n) in at most 16 contiguous chunks of at least
// min_chunk items, one thread each (the caller runs the last one, and any that
// no thread could be had for).  f must not throw.  Returns the chunks used;
// chunk c always covers [n c / chunks, n (c + 1) / chunks).
constexpr int kMaxChunks = 16;
inline int host_chunks(int64_t n, int64_t min_chunk) {
    const int64_t hw = std::max(1u, std::thread::hardware_concurrency());
    return (int)std::max<int64_t>(1, std::min<int64_t>({hw, kMaxChunks, n / min_chunk}));
}
template <typename F>
inline int parallel_chunks(int64_t n, int64_t min_chunk, const F& f) {
    const int nc = host_chunks(n, min_chunk);
    std::vector<std::thread> th;
    th.reserve(nc);
    int c = 0;
    for (; c + 1 < nc; ++c) {
        const int64_t b = n * c / nc, e = n * (c + 1) / nc;
        try {
            th.emplace_back([&f, b, e, c] { f(b, e, c); });
        } catch (const std::exception&) {
            break;
        }
    }
    for (; c < nc; ++c) f(n * c / nc, n * (c + 1) / nc, c);
    for (auto& t : th) t.join();
    return nc;
}

}  // namespace ams
