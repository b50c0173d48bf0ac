// arc_map.hpp -- the host mirror's map from an arc (a, b) to its weight and its slot in the
// E* superset: one open-addressing table (linear probing, at most half full, no removal;
// an update only adds arcs or changes them).  It is built from tens of thousands of arcs
// when a handle is made and asked a few times per update; with a node per arc in two
// std::unordered_map the host's part of bc_init_static was 9.6 ms of 16 at BA n = 4096.
#pragma once

#include <cstdint>
#include <vector>

namespace bcg {

class ArcMap {
public:
    struct Entry {
        uint64_t key = kFree;
        int64_t w = 0;
        int32_t slot = -1;   // in the E* superset; -1: not there
    };

    static uint64_t key_of(int32_t a, int32_t b) { return ((uint64_t)(uint32_t)a << 32) | (uint32_t)b; }

    int64_t size() const { return size_; }

    void reserve(int64_t count) {
        int bits = 4;
        while (((int64_t)1 << bits) < 2 * count) ++bits;
        if (((int64_t)1 << bits) > (int64_t)table_.size()) rehash(bits);
    }

    Entry* find(int32_t a, int32_t b) {
        if (table_.empty()) return nullptr;
        Entry& e = table_[place(key_of(a, b))];
        return e.key == kFree ? nullptr : &e;
    }

    // The entry of (a, b), made when there is none (*added tells).
    Entry& at(int32_t a, int32_t b, bool* added = nullptr) {
        if (2 * (size_ + 1) > (int64_t)table_.size()) reserve(2 * (size_ + 1));
        Entry& e = table_[place(key_of(a, b))];
        if (added) *added = e.key == kFree;
        if (e.key == kFree) {
            e.key = key_of(a, b);
            ++size_;
        }
        return e;
    }

    template <typename F>
    void each(F&& f) {
        for (Entry& e : table_)
            if (e.key != kFree) f((int32_t)(e.key >> 32), (int32_t)(e.key & 0xffffffffu), e);
    }

private:
    static constexpr uint64_t kFree = ~0ull;   // no arc: vertices are non-negative

    size_t place(uint64_t key) const {
        const size_t mask = table_.size() - 1;
        size_t i = (size_t)((key * 0x9E3779B97F4A7C15ull) >> shift_);
        while (table_[i].key != kFree && table_[i].key != key) i = (i + 1) & mask;
        return i;
    }

    void rehash(int bits) {
        std::vector<Entry> old((size_t)1 << bits);
        old.swap(table_);
        shift_ = 64 - bits;
        for (const Entry& e : old)
            if (e.key != kFree) table_[place(e.key)] = e;
    }

    std::vector<Entry> table_;
    int64_t size_ = 0;
    int shift_ = 64;
};

}  // namespace bcg
