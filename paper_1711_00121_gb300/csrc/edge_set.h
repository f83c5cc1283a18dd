// The edges of a graph as a set of 64-bit keys: open addressing with linear
// probing in one array, at most half full.
#pragma once

#include <cstddef>
#include <cstdint>
#include <utility>
#include <vector>

namespace sr {

class EdgeSet {
 public:
  size_t size() const { return n_; }

  // Room for m keys without growing.
  void reserve(size_t m) {
    size_t cap = 64;
    while (cap < 2 * m) cap *= 2;
    if (cap > slot_.size()) rehash(cap);
  }

  bool contains(uint64_t k) const {
    if (slot_.empty()) return false;
    for (size_t i = home(k);; i = (i + 1) & mask_) {
      if (slot_[i] == k) return true;
      if (slot_[i] == EMPTY) return false;
    }
  }

  // False if the key is there already.
  bool insert(uint64_t k) {
    if (2 * (n_ + 1) > slot_.size()) rehash(slot_.empty() ? 64 : 2 * slot_.size());
    size_t i = home(k);
    for (; slot_[i] != EMPTY; i = (i + 1) & mask_)
      if (slot_[i] == k) return false;
    slot_[i] = k;
    ++n_;
    return true;
  }

  // False if the key is absent.  Later keys of the probe run move back into the
  // gap, so that no marker of the removal is left.
  bool erase(uint64_t k) {
    if (slot_.empty()) return false;
    size_t i = home(k);
    for (; slot_[i] != k; i = (i + 1) & mask_)
      if (slot_[i] == EMPTY) return false;
    for (size_t j = (i + 1) & mask_; slot_[j] != EMPTY; j = (j + 1) & mask_)
      if (((j - home(slot_[j])) & mask_) >= ((j - i) & mask_)) {
        slot_[i] = slot_[j];
        i = j;
      }
    slot_[i] = EMPTY;
    --n_;
    return true;
  }

 private:
  static constexpr uint64_t EMPTY = ~0ull;  // ids are below 2^31: no key
  size_t home(uint64_t k) const { return (size_t)((k * 0x9E3779B97F4A7C15ull) >> shift_); }

  void rehash(size_t cap) {
    std::vector<uint64_t> old(cap, EMPTY);
    old.swap(slot_);
    mask_ = cap - 1;
    shift_ = 64;
    while (cap > 1) {
      cap /= 2;
      --shift_;
    }
    for (uint64_t k : old)
      if (k != EMPTY) {
        size_t i = home(k);
        while (slot_[i] != EMPTY) i = (i + 1) & mask_;
        slot_[i] = k;
      }
  }

  std::vector<uint64_t> slot_;
  size_t n_ = 0, mask_ = 0;
  int shift_ = 64;
};

}  // namespace sr
