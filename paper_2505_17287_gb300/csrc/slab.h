// The device memory of one served case: a block taken once (the slab) that
// the case's allocations are carved from. Host-only bookkeeping: offsets and
// lengths, no device call.
#pragma once
#include <stddef.h>

#include <iterator>
#include <map>

namespace ibm {

constexpr size_t SLAB_ALIGN = 256;   // every carved block starts on a multiple

inline size_t slab_round(size_t bytes) { return (bytes + SLAB_ALIGN - 1) / SLAB_ALIGN * SLAB_ALIGN; }

struct Slab {
    char *base = nullptr;
    size_t bytes = 0;
    std::map<size_t, size_t> ranges;   // free: offset -> length, neighbours merged

    void open(void *p, size_t n) {
        base = (char *)p;
        bytes = p ? n / SLAB_ALIGN * SLAB_ALIGN : 0;
        ranges.clear();
        if (bytes) ranges[0] = bytes;
    }
    bool holds(const void *p) const { return base && (const char *)p >= base && (const char *)p < base + bytes; }

    // the first free range that holds n bytes, or null
    void *take(size_t n) {
        const size_t need = slab_round(n);
        for (auto it = ranges.begin(); it != ranges.end(); ++it) {
            if (it->second < need) continue;
            const size_t off = it->first, len = it->second;
            ranges.erase(it);
            if (len > need) ranges[off + need] = len - need;
            return base + off;
        }
        return nullptr;
    }

    // give back a block of n bytes that take() returned
    void give(void *p, size_t n) {
        size_t off = (size_t)((char *)p - base), len = slab_round(n);
        auto next = ranges.lower_bound(off);
        if (next != ranges.end() && next->first == off + len) {
            len += next->second;
            next = ranges.erase(next);
        }
        if (next != ranges.begin()) {
            auto prev = std::prev(next);
            if (prev->first + prev->second == off) {
                prev->second += len;
                return;
            }
        }
        ranges[off] = len;
    }
};

}  // namespace ibm
