// Cache of values that are pure functions of their keys (host only; the tensor maps of one host thread).
//
// An open-addressed table with linear probing.  It holds up to MAX_USED values and then starts over from nothing: a set of keys of
// up to that size that comes round again is found whole, in any order, which first-in-first-out replacement does not give
// once the set is one key larger than the cache.
#pragma once
#include <stddef.h>
#include <stdint.h>
#include <string.h>

namespace sf {

template <typename Key, typename Value, int SLOTS>
class MapCache {
    static_assert((SLOTS & (SLOTS - 1)) == 0, "a power of two");

public:
    static constexpr int MAX_USED = SLOTS / 4 * 3;

    // The value of `key`, or NULL.
    const Value* find(const Key& key) const {
        for (int s = home(key); full_[s]; s = (s + 1) & (SLOTS - 1))
            if (key_[s] == key) return &value_[s];
        return nullptr;
    }
    // `key` must not be in the table.
    void insert(const Key& key, const Value& value) {
        if (used_ == MAX_USED) {
            memset(full_, 0, sizeof(full_));
            used_ = 0;
        }
        int s = home(key);
        while (full_[s]) s = (s + 1) & (SLOTS - 1);
        full_[s] = true;
        key_[s] = key;
        value_[s] = value;
        ++used_;
    }

private:
    static int home(const Key& key) { return (int)((key.hash() * 0x9E3779B97F4A7C15ull) >> 40) & (SLOTS - 1); }
    bool full_[SLOTS] = {};
    int used_ = 0;
    Key key_[SLOTS];
    Value value_[SLOTS];
};

}  // namespace sf
