// Device memory of calls that a solver repeats (tape, snapshots, gauge values of the adjoint), kept for its next call:
// allocating and freeing it cost as much as a small run's kernels. What a call does not ask for is no reason for it to
// fail: while memory is short, everything it has not claimed is given back, this pool's own first. Mem allocates and frees
// (get returns null when memory is short). Plain C++: the rules are checked on the host.
#pragma once
#include <cstddef>
#include <vector>

namespace hw {

template <class Mem>
class WorkPool {
 public:
  // A call claims what it uses between begin and end.
  void begin() {
    for (Entry& e : v_) e.claimed = false;
  }
  // At least `bytes` as number k, with any contents; null if they cannot be had. give_back() frees what others keep
  // and says whether there was any.
  template <class GiveBack>
  void* get(int k, std::size_t bytes, const GiveBack& give_back) {
    if (v_.size() <= (std::size_t)k) v_.resize(k + 1);
    Entry& e = v_[k];
    if (e.bytes < bytes) {
      drop(e);
      e.p = Mem::get(bytes);
      if (!e.p && release_unclaimed()) e.p = Mem::get(bytes);
      if (!e.p && give_back()) e.p = Mem::get(bytes);
      e.bytes = e.p ? bytes : 0;
    }
    e.claimed = e.p != nullptr;
    return e.p;
  }
  // Frees what the present call has not claimed; whether there was any.
  bool release_unclaimed() {
    bool any = false;
    for (Entry& e : v_)
      if (!e.claimed && e.p) {
        drop(e);
        any = true;
      }
    return any;
  }
  // The call's end (its stream has drained): frees what it needed beyond keep bytes in all.
  void end(std::size_t keep) {
    std::size_t held = 0;
    for (Entry& e : v_) {
      if (held + e.bytes > keep) drop(e);
      held += e.bytes;
      e.claimed = false;
    }
  }
  std::size_t held() const {
    std::size_t h = 0;
    for (const Entry& e : v_) h += e.bytes;
    return h;
  }

 private:
  struct Entry {
    void* p = nullptr;
    std::size_t bytes = 0;
    bool claimed = false;
  };
  static void drop(Entry& e) {
    if (e.p) Mem::put(e.p);
    e = Entry{};
  }
  std::vector<Entry> v_;
};

}  // namespace hw
