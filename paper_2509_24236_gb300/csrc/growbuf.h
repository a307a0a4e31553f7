// Device buffers that grow while others hold their addresses.  Host code only
// (allocation is passed in), compiled on its own by the host tests.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <initializer_list>
#include <vector>

namespace pf {

// Capacity of buffers of `cap` elements that must hold `need`: half as much
// again at least, so that the buffers retired on the way (below) hold at most
// twice what the last ones do.
inline long long grown_capacity(long long cap, long long need)
{
    return need <= cap ? cap : std::max(need, cap + (cap + 1) / 2);
}

struct Grow {
    void* p;       // where the pointer to replace stands (a pointer of any type)
    size_t bytes;  // of the new buffer
    bool zero;     // which starts as zeros
};

// Replaces each pointer by a new buffer.  The old ones are retired, not freed:
// a batch's launch tables and captured graphs hold their addresses and may be
// launched as long as the volume lives.  All or nothing: when an allocation
// fails the new buffers are freed and every pointer stays.
template <typename Alloc, typename Free>
auto grow_all(std::vector<void*>& retired, std::initializer_list<Grow> set, Alloc alloc, Free free)
{
    std::vector<void*> fresh;
    decltype(alloc(nullptr, size_t(0), false)) e{};
    for (const Grow& g : set) {
        void* q = nullptr;
        e = alloc(&q, g.bytes, g.zero);
        if (!q) {
            for (void* f : fresh) free(f);
            return e;
        }
        fresh.push_back(q);
    }
    size_t i = 0;
    for (const Grow& g : set) {
        void* old;
        std::memcpy(&old, g.p, sizeof(old));
        if (old) retired.push_back(old);
        std::memcpy(g.p, &fresh[i++], sizeof(old));
    }
    return e;
}

}  // namespace pf
