// Device memory of a session (host code only; the two functions that get and
// give back memory are passed in).
//
// Small buffers lie behind one another in slabs, which live as long as the
// session: most of a small query's creation and destruction was a driver call
// per buffer (5 states, 200 iterations: 700 us a query with an allocation each,
// 660 with slabs). Launch plans change size while the session lives, so their
// buffers are of a kind of their own (Plan): a small one keeps a place in a slab
// and moves only when it outgrows it, to one at least twice as large, so all
// places of a buffer together take less than 2 kMost; a large one is an
// allocation of its own that is given back when the plan changes.
#pragma once

#include <algorithm>
#include <cstddef>
#include <vector>

namespace imdp {

class Buffers {
 public:
  typedef void* (*Get)(size_t bytes);  // nullptr: no memory
  typedef void (*Put)(void* p);
  static constexpr size_t kSlab = 256 * 1024, kMost = 32 * 1024;

  struct Plan {
    void* place = nullptr;  // in a slab
    size_t room = 0;        // bytes there
    void* own = nullptr;    // an allocation of its own, while the contents need one
  };

  Buffers(Get get, Put put) : get_(get), put_(put) {}
  Buffers(const Buffers&) = delete;
  Buffers& operator=(const Buffers&) = delete;
  ~Buffers() {
    for (void* p : single_) put_(p);
    for (void* p : slabs_) put_(p);
  }

  // `bytes` for the session's lifetime (or until release); nullptr: no memory.
  void* alloc(size_t bytes) {
    bytes = rounded(bytes);
    return bytes <= kMost ? take(bytes) : single(bytes);
  }

  // Room for `bytes` in plan buffer `b`, whose contents are lost; nullptr: no memory.
  void* refit(Plan& b, size_t bytes) {
    bytes = rounded(bytes);
    drop(b);
    if (bytes > kMost) return b.own = single(bytes);
    if (bytes > b.room) {
      const size_t room = std::min(kMost, std::max(bytes, 2 * b.room));
      void* p = take(room);
      if (!p) return nullptr;  // (the smaller place stays for a smaller plan)
      b.place = p;
      b.room = room;
    }
    return b.place;
  }

  // Gives back what plan buffer `b` does not need while it is empty.
  void drop(Plan& b) {
    release(b.own);
    b.own = nullptr;
  }

  // Gives back a buffer of `alloc` when it is an allocation of its own (nothing
  // is done for one in a slab, or for nullptr).
  void release(void* p) {
    const auto it = std::find(single_.begin(), single_.end(), p);
    if (!p || it == single_.end()) return;
    single_.erase(it);
    put_(p);
  }

 private:
  static size_t rounded(size_t bytes) { return (std::max<size_t>(bytes, 1) + 255) & ~size_t(255); }
  void* single(size_t bytes) {
    void* p = get_(bytes);
    if (p) single_.push_back(p);
    return p;
  }
  void* take(size_t bytes) {
    if (bytes > left_) {
      void* p = get_(kSlab);
      if (!p) return nullptr;
      slabs_.push_back(p);
      at_ = (unsigned char*)p;
      left_ = kSlab;
    }
    void* t = at_;
    at_ += bytes;
    left_ -= bytes;
    return t;
  }

  Get get_;
  Put put_;
  // apart from one another: a slab's address is also that of its first buffer
  std::vector<void*> single_, slabs_;
  unsigned char* at_ = nullptr;
  size_t left_ = 0;
};

}  // namespace imdp
