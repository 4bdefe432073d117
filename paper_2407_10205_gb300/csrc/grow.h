// grow.h -- a device table that grows with the calls that need it (host code, no CUDA in it).
#pragma once
#include <cstddef>

namespace phia {

// Room for `need` entries at p, which has `cap`: the old table is released first.  After a failed
// allocation there is none, so that a later call for fewer entries does not take it for one.
template <typename T, typename Alloc, typename Release>
bool grow_table(T *&p, size_t &cap, size_t need, Alloc alloc, Release release) {
    if (need <= cap) return true;
    release(p);
    p = nullptr;
    cap = 0;
    if (!alloc(&p, need * sizeof(T))) {
        p = nullptr;
        return false;
    }
    cap = need;
    return true;
}

}  // namespace phia
