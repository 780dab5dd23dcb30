// Bounded store of prepared operations: keys compared byte by byte, the entry that was not asked for longest leaves when a
// new one comes in.  (Emptying a full store instead would throw away, time and again, the operations that every call
// makes, as soon as one of a caller's buffers has a new address in each call.)  Plain C++.
#pragma once
#include <stdint.h>
#include <string.h>

#include <iterator>
#include <list>
#include <unordered_map>
#include <utility>

// Key: a trivially copyable struct without unset padding, a multiple of 8 bytes long.
template <typename Key, typename Value>
class PlanStore {
    static_assert(sizeof(Key) % 8 == 0, "hashed in words of 8 bytes");
    struct Entry {
        Key key;
        Value value;
    };
    using Order = std::list<Entry>;  // the latest used first
    Order order;
    std::unordered_multimap<uint64_t, typename Order::iterator> index;
    size_t limit;

    static uint64_t hash(const Key &k) {
        uint64_t h = 1469598103934665603ull;
        const char *c = reinterpret_cast<const char *>(&k);
        for (size_t i = 0; i < sizeof(k); i += 8) {
            uint64_t w;
            memcpy(&w, c + i, 8);
            h = (h ^ w) * 1099511628211ull;
            h ^= h >> 29;
        }
        return h;
    }

    void drop_last() {
        const auto last = std::prev(order.end());
        const auto range = index.equal_range(hash(last->key));
        for (auto it = range.first; it != range.second; ++it)
            if (it->second == last) {
                index.erase(it);
                break;
            }
        order.pop_back();
    }

public:
    explicit PlanStore(size_t most) : limit(most) {}

    // The value of a key, or null; good until the next put or clear.
    const Value *find(const Key &key) {
        const auto range = index.equal_range(hash(key));
        for (auto it = range.first; it != range.second; ++it)
            if (memcmp(&it->second->key, &key, sizeof(key)) == 0) {
                order.splice(order.begin(), order, it->second);
                return &it->second->value;
            }
        return nullptr;
    }

    // Keeps the value of a key that find does not know.  Without memory nothing is kept, and nothing thrown.
    void put(const Key &key, Value &&value) noexcept {
        while (!order.empty() && order.size() >= limit) drop_last();
        bool listed = false;
        try {
            order.push_front(Entry{key, std::move(value)});
            listed = true;
            index.emplace(hash(key), order.begin());
        } catch (...) {
            if (listed) order.pop_front();
        }
    }

    void clear() {
        index.clear();
        order.clear();
    }
    size_t size() const { return order.size(); }
};
