// A device buffer that grows with what its calls need, and how it does so.
#pragma once

#include <algorithm>
#include <cstddef>

namespace fh {

struct DevBuf {
    void *p = nullptr;
    size_t cap = 0;
    template <class T> T *as() const { return reinterpret_cast<T *>(p); }
};

// b holds at least `bytes` afterwards, contents undefined if it had to grow.
// gen advances whenever the address a launch may have been captured with is
// given up or replaced: when the old buffer is released too, since the
// allocation after it can fail and leave every other buffer as it was.
// Memory: int alloc(void **, size_t), 0 on success; void release(void *).
template <class Memory> int grow(Memory &mem, DevBuf &b, size_t bytes, long long &gen) {
    if (b.p && b.cap >= bytes) return 0;
    if (b.p) {
        mem.release(b.p);
        b = DevBuf{};
        ++gen;
    }
    const size_t want = std::max<size_t>(bytes, 256);
    void *p = nullptr;
    const int e = mem.alloc(&p, want);
    if (e != 0) return e;
    b.p = p;
    b.cap = want;
    ++gen;
    return 0;
}

}  // namespace fh
