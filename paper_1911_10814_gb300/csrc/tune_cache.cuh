// tune_cache.cuh -- choices that timing has made, kept for the life of the
// process.  Internal header, plain C++.
#pragma once

#include <cstddef>
#include <list>
#include <map>
#include <mutex>
#include <utility>

namespace nbp {

// The first choice made for a key stays, so that every context that meets the
// key computes in the same order; of more than cap keys the one used longest
// ago leaves (every new tangent brings coarse levels of new shapes).  Safe
// with several threads.
template <typename K, typename V> class TuneCache {
public:
    explicit TuneCache(size_t cap) : cap_(cap) {}
    bool find(const K &key, V &value) {
        std::lock_guard<std::mutex> lock(mutex_);
        auto it = at_.find(key);
        if (it == at_.end()) return false;
        used_.splice(used_.begin(), used_, it->second);
        value = it->second->second;
        return true;
    }
    // the choice kept for key: value, or what another thread was first with
    V keep(const K &key, const V &value) {
        std::lock_guard<std::mutex> lock(mutex_);
        auto it = at_.find(key);
        if (it != at_.end()) {
            used_.splice(used_.begin(), used_, it->second);
            return it->second->second;
        }
        used_.emplace_front(key, value);
        at_[key] = used_.begin();
        if (at_.size() > cap_) {
            at_.erase(used_.back().first);
            used_.pop_back();
        }
        return value;
    }
    size_t size() {
        std::lock_guard<std::mutex> lock(mutex_);
        return at_.size();
    }

private:
    const size_t cap_;
    std::mutex mutex_;
    std::list<std::pair<K, V>> used_;   // most recently used first
    std::map<K, typename std::list<std::pair<K, V>>::iterator> at_;
};

}  // namespace nbp
