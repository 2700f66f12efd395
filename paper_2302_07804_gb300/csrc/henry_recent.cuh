// A bounded map of built objects that gives up the least recently used one when
// it is full (host code).
#pragma once
#include <cstddef>
#include <cstdint>
#include <map>
#include <utility>

namespace hk {

template <typename Key, typename Value, size_t MAX>
class RecentMap {
  struct Entry {
    Value value;
    uint64_t used;  // the clock at its last use
  };
  std::map<Key, Entry> m_;
  uint64_t clock_ = 0;

 public:
  size_t size() const { return m_.size(); }
  // The object of this key, marked as used; NULL if there is none.
  Value* find(const Key& k) {
    auto f = m_.find(k);
    if (f == m_.end()) return nullptr;
    f->second.used = ++clock_;
    return &f->second.value;
  }
  // Keeps v, the object of a key that find() did not have.  A full map first
  // hands its least recently used object to drop().
  template <typename Drop>
  Value* insert(const Key& k, Value v, Drop&& drop) {
    if (m_.size() >= MAX) {
      auto oldest = m_.begin();
      for (auto i = m_.begin(); i != m_.end(); ++i)
        if (i->second.used < oldest->second.used) oldest = i;
      drop(oldest->second.value);
      m_.erase(oldest);
    }
    return &m_.emplace(k, Entry{std::move(v), ++clock_}).first->second.value;
  }
  template <typename Drop>
  void clear(Drop&& drop) {
    for (auto& e : m_) drop(e.second.value);
    m_.clear();
  }
};

}  // namespace hk
