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
// spare (may be null): a buffer that its users can do without, released for b
// if there is no room.
// Memory: int alloc(void **, size_t), 0 on success; void release(void *).
template <class Memory> int grow(Memory &mem, DevBuf &b, size_t bytes, long long &gen, DevBuf *spare = nullptr) {
    auto give_up = [&](DevBuf &d) {
        mem.release(d.p);
        d = DevBuf{};
        ++gen;
    };
    if (b.p && b.cap >= bytes) return 0;
    if (b.p) give_up(b);
    const size_t want = std::max<size_t>(bytes, 256);
    void *p = nullptr;
    int e = mem.alloc(&p, want);
    if (e != 0 && spare && spare != &b && spare->p) {
        give_up(*spare);
        e = mem.alloc(&p, want);
    }
    if (e != 0) return e;
    b.p = p;
    b.cap = want;
    ++gen;
    return 0;
}

}  // namespace fh
