// What a thread has worked out for the calls it makes again and again: a table of Sets x Ways entries, of which a key may be in
// the Ways of one set; where these are taken, the one that has gone unused the longest gives way.  A key is compared whole, the
// hash only picks the set.  Host code without dependencies; one table per thread, so nothing is locked.
#pragma once
#include <cstddef>
#include <cstdint>

namespace sq {

inline uint32_t hash_words(const int64_t *w, size_t n)
{
    uint64_t h = n;
    for (size_t i = 0; i < n; i++) {
        h = (h ^ uint64_t(w[i])) * 0x9E3779B97F4A7C15ull;      // 2^64 over the golden ratio: the high bits depend on all of the word
        h ^= h >> 32;
    }
    return uint32_t(h);
}

template <typename Key, typename Value, unsigned Sets, unsigned Ways>
class Recent {
public:
    static_assert((Sets & (Sets - 1)) == 0, "a power of two");

    // the value kept for a key, nullptr where there is none
    const Value *find(uint32_t hash, const Key &key)
    {
        const unsigned s = hash & (Sets - 1);
        for (unsigned i = 0; i < Ways; i++)
            if (hash_[s][i] == hash && used_[s][i] && entries_[s][i].key == key) {
                used_[s][i] = ++clock_;
                return &entries_[s][i].value;
            }
        return nullptr;
    }
    const Value &keep(uint32_t hash, const Key &key, const Value &value)
    {
        const unsigned s = hash & (Sets - 1);
        unsigned oldest = 0;
        for (unsigned i = 1; i < Ways; i++)
            if (used_[s][i] < used_[s][oldest]) oldest = i;
        entries_[s][oldest] = {key, value};
        hash_[s][oldest] = hash;
        used_[s][oldest] = ++clock_;
        return entries_[s][oldest].value;
    }

private:
    struct Entry {
        Key key;
        Value value;
    };
    uint32_t hash_[Sets][Ways] = {};     // apart from the entries: a search reads little else
    uint64_t used_[Sets][Ways] = {};     // time of the last use, 0: empty
    Entry entries_[Sets][Ways] = {};
    uint64_t clock_ = 0;
};

}  // namespace sq
