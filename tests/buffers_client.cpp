// A session's use of its device memory (csrc/buffers.h), on host memory that is
// watched: buffers in use lie in live blocks, keep their contents, do not
// overlap, and the memory taken does not grow with the number of plan changes.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <random>
#include <utility>
#include <vector>

#include "buffers.h"

static std::map<char*, size_t> live;
static size_t held = 0;
static bool refuse = false;

static void* get(size_t n) {
  if (refuse) return nullptr;
  char* p = (char*)std::malloc(n);
  live[p] = n;
  held += n;
  return p;
}
static void put(void* p) {
  auto it = live.find((char*)p);
  if (it == live.end()) {
    std::printf("gave back a block that is not live\n");
    std::exit(1);
  }
  held -= it->second;
  live.erase(it);
  std::free(p);
}

struct Used {
  char* p;
  size_t n;
  unsigned char mark;
};

static void check(const std::vector<Used>& us, const char* what) {
  std::map<char*, size_t> at;
  for (const Used& u : us) {
    auto b = live.upper_bound(u.p);
    if (b == live.begin() || u.p + u.n > std::prev(b)->first + std::prev(b)->second) {
      std::printf("%s: a buffer outside every live block\n", what);
      std::exit(1);
    }
    at[u.p] = u.n;
    for (size_t i = 0; i < u.n; ++i)
      if ((unsigned char)u.p[i] != u.mark) {
        std::printf("%s: a buffer's contents were overwritten\n", what);
        std::exit(1);
      }
  }
  char* end = nullptr;
  for (auto& kv : at) {
    if (kv.first < end) {
      std::printf("%s: buffers overlap\n", what);
      std::exit(1);
    }
    end = kv.first + kv.second;
  }
}

static Used fill(void* p, size_t n) {
  static unsigned char next = 0;
  std::memset(p, ++next, n);
  return Used{(char*)p, n, next};
}

int main() {
  std::mt19937 rng(7);
  for (int first = 0; first < 120; first += 3) {
    imdp::Buffers mem(get, put);
    std::vector<Used> keep;
    // small buffers until a plan buffer may be the first of a slab
    for (int i = 0; i < first; ++i) {
      const size_t n = 1 + rng() % (i % 9 == 4 ? 40000 : 3000);
      keep.push_back(fill(mem.alloc(n), n));
    }
    const size_t before = held;
    imdp::Buffers::Plan plan[3];
    for (int change = 0; change < 100; ++change) {
      std::vector<Used> now = keep;
      for (auto& b : plan) {
        const size_t n = 1 + rng() % (change % 2 ? 9000 : (change % 7 == 0 ? 70000 : 30000));
        now.push_back(fill(mem.refit(b, n), n));
      }
      check(now, "plan change");
      if (held > before + 3 * (70000 + 256 + 2 * imdp::Buffers::kMost) + imdp::Buffers::kSlab) {
        std::printf("%zu bytes more after %d plan changes\n", held - before, change + 1);
        return 1;
      }
      if (change % 50 == 49) {  // buffers taken between plans
        const size_t n = 1 + rng() % 2000;
        keep.push_back(fill(mem.alloc(n), n));
      }
    }
    for (auto& b : plan) mem.drop(b);
    check(keep, "plans dropped");
    // no memory: nullptr, and what is there stays
    refuse = true;
    void* big = mem.alloc(1 << 20);
    imdp::Buffers::Plan none;
    void* own = mem.refit(none, 1 << 20);
    refuse = false;
    if (big || own) return 1;
    check(keep, "refused");
    void* one = mem.alloc(1 << 20);
    const size_t with = held;
    mem.release(one);
    mem.release(nullptr);
    if (!keep.empty()) mem.release(keep[0].p);
    if (held > with - (1 << 20)) return 1;
  }
  std::printf("held %zu\n", held);
  return held == 0 ? 0 : 1;
}
