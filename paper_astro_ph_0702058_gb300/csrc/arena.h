// Several buffers of one owner in one allocation: each device or pinned
// allocation and its free cost the driver tens of microseconds (a context held
// 24 of them), which a caller that makes a context per call pays every time.
#pragma once

#include <cstddef>

namespace nb {

class Arena {
public:
    template <class T>
    void add(T **p, const size_t bytes)
    {
        static_assert(sizeof(T *) == sizeof(void *), "object pointers");
        at_[count_] = reinterpret_cast<void **>(p);
        offset_[count_++] = total_;
        total_ += (bytes + 255) / 256 * 256;
    }
    // alloc(void **, bytes) -> error code (0: success); on failure every pointer stays as it was.
    template <class Alloc>
    auto commit(void **base, Alloc &&alloc) const
    {
        const auto e = alloc(base, total_);
        if (!e)
            for (int k = 0; k < count_; ++k) *at_[k] = static_cast<char *>(*base) + offset_[k];
        return e;
    }

private:
    static constexpr int kMost = 32;  // more than any owner adds
    void **at_[kMost] = {};
    size_t offset_[kMost] = {};
    size_t total_ = 0;
    int count_ = 0;
};

}  // namespace nb
