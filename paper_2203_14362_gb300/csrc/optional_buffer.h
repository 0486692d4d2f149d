// A device buffer that speeds a call up but that it can do without.
#pragma once

#include <cstddef>
#include <cstdint>

namespace spx {

// Grows on demand.  A size that the device had no memory for is not asked for again
// at once (an attempt costs two failing allocations and a wait): not before memory
// is freed (retry) or kSkip calls later.  What is held stays where it is until a
// larger buffer has taken its place, so calls that fail to grow it disturb nothing.
struct OptionalBuffer {
    static constexpr uint32_t kSkip = 256;
    void *p = nullptr;
    size_t bytes = 0;
    size_t refused = SIZE_MAX; // the smallest size refused
    uint32_t skipped = 0;

    // `need` bytes, or null.  alloc(void **, size_t) is false without memory;
    // release(void *) waits for work that uses the buffer.
    template <class A, class R>
    void *want(size_t need, A alloc, R release)
    {
        if (bytes >= need)
            return p;
        if (need >= refused && ++skipped < kSkip)
            return nullptr;
        skipped = 0;
        void *q = nullptr;
        if (!alloc(&q, need)) {
            refused = need < refused ? need : refused;
            return nullptr;
        }
        if (p)
            release(p);
        p = q;
        bytes = need;
        retry();
        return p;
    }
    void retry()
    {
        refused = SIZE_MAX;
        skipped = 0;
    }
};

} // namespace spx
