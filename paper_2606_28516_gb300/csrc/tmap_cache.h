// Cache of encoded tensor maps (plain C++: the CPU tests compile it too).
#pragma once

#include <stdint.h>

#include <mutex>

namespace cm {

// What determines an encoded map entirely.
struct TmapKey {
    const void* base;
    int64_t rows, cols;
    int box_rows, box_chunks, elem;
    bool operator==(const TmapKey& o) const {
        return base == o.base && rows == o.rows && cols == o.cols && box_rows == o.box_rows &&
               box_chunks == o.box_chunks && elem == o.elem;
    }
};

// Up to CAP maps, found by a hash of their key, the oldest replaced first; one per process, shared by threads.
// Replacement in order misses every lookup of a program that cycles through more keys than fit, and a call
// encodes up to 40 (a layer of E = 16 experts: 16 expert matrices and three others, each also in boxes of
// half the rows, and x, z, t, W_g): 2,048 hold a model of 24 such layers with room for other token counts. 64
// held 12 sublayers of E = 8 at a third of its lookups. A miss is a call into the CUDA driver; a hit costs the lock, one or two
// comparisons and a copy of 128 bytes. Zero-initialised storage is an empty cache.
template <class Map, int CAP = 2048>
class TmapCache {
public:
    // The map of key k, from the cache or from encode(Map*) (0 on success, else its code is returned and
    // nothing is kept).
    template <class Encode>
    int get(Map* out, const TmapKey& k, Encode encode) {
        const std::lock_guard<std::mutex> lock(mu_);
        const int b = bucket(k);
        for (int i = head_[b]; i; i = e_[i - 1].next)
            if (e_[i - 1].key == k) {
                *out = e_[i - 1].map;
                return 0;
            }
        const int rc = encode(out);
        if (rc) return rc;
        Entry& e = e_[next_];
        if (used_ == CAP) {  // take the oldest out of its bucket's chain
            int* p = &head_[bucket(e.key)];
            while (*p != next_ + 1) p = &e_[*p - 1].next;
            *p = e.next;
        } else {
            ++used_;
        }
        e.key = k;
        e.map = *out;
        e.next = head_[b];
        head_[b] = next_ + 1;
        next_ = next_ + 1 == CAP ? 0 : next_ + 1;
        return 0;
    }

private:
    static constexpr int BUCKETS = 2 * CAP;
    struct Entry {
        Map map;
        TmapKey key;
        int next;  // 1 + index of the next entry of the bucket's chain, 0: none
    };
    static int bucket(const TmapKey& k) {
        uint64_t h = reinterpret_cast<uintptr_t>(k.base) >> 4;
        const uint64_t v[3] = {(uint64_t)k.rows, (uint64_t)k.cols,
                               (uint64_t)k.box_rows << 24 ^ (uint64_t)k.box_chunks << 8 ^ (uint64_t)k.elem};
        for (uint64_t x : v) h = (h ^ x) * 0x9E3779B97F4A7C15ull ^ h >> 29;
        return (int)((h * 0x9E3779B97F4A7C15ull >> 32) % BUCKETS);
    }
    std::mutex mu_;
    Entry e_[CAP];
    int head_[BUCKETS];  // 1 + index of the first entry, 0: none
    int next_, used_;
};

}  // namespace cm
