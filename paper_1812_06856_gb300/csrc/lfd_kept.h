// A buffer whose words are left at a fixed value between uses, so that a use
// need not set them first.  Plain C++ (also compiled for the host by itself).
#pragma once
#include <stddef.h>

namespace lfd {

template <typename T>
struct KeptBuffer {
    T *p = nullptr;
    size_t cap = 0;
    bool clean = false;              // every word has the value once the enqueued work has run

    // Room for `bytes` by grow(&p, &cap, bytes).  What that allocates is not
    // clean, whatever fails after it.
    template <typename Grow>
    auto reserve(size_t bytes, Grow grow)
    {
        if (cap < bytes) clean = false;
        return grow((void **)&p, &cap, bytes);
    }
};

}  // namespace lfd
