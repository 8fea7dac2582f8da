// A small map by string that keeps the entries used last (host code).
#pragma once
#include <stddef.h>

#include <algorithm>
#include <string>
#include <utility>
#include <vector>

namespace dotpe {

// At most `most` entries; put() gives back the one that has to leave, for the caller to
// destroy.  Entries lie in order of use, the last used at the end: a handful is searched.
template <typename V>
class LruMap {
 public:
  explicit LruMap(size_t most) : most_(most) {}

  // the value of `key`, now the last used, or null
  V *find(const std::string &key) {
    for (size_t k = 0; k < at_.size(); ++k)
      if (at_[k].first == key) {
        std::rotate(at_.begin() + k, at_.begin() + k + 1, at_.end());
        return &at_.back().second;
      }
    return nullptr;
  }
  // key (not held yet) -> value; true: `out` had to leave
  bool put(const std::string &key, V value, V *out) {
    bool full = at_.size() >= most_;
    if (full) {
      *out = at_.front().second;
      at_.erase(at_.begin());
    }
    at_.emplace_back(key, value);
    return full;
  }
  void erase(const std::string &key) {
    at_.erase(std::remove_if(at_.begin(), at_.end(), [&](const auto &e) { return e.first == key; }), at_.end());
  }
  size_t size() const { return at_.size(); }
  template <typename F>
  void for_each(F f) {
    for (auto &e : at_) f(e.second);
  }

 private:
  size_t most_;
  std::vector<std::pair<std::string, V>> at_;
};

}  // namespace dotpe
