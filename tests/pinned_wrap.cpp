// C wrappers around csrc/zmc_pinned.h with a counting source, built by test_pinned_cpu.py.
#include <cstdlib>

#include "zmc_pinned.h"

struct Counting {
  static int live, made, error;
  static int get(void** p, size_t) {
    if (error) return error;
    ++live;
    ++made;
    *p = std::malloc(1);
    return 0;
  }
  static void put(void* p) {
    --live;
    std::free(p);
  }
};
int Counting::live = 0, Counting::made = 0, Counting::error = 0;

using Pool = zmc::PinnedPool<Counting>;
extern "C" {
void* pool_new(size_t keep) { return new Pool(keep); }
int pool_take(void* pool, size_t bytes, void** p, size_t* got) {
  zmc::PinnedBuf b;
  const int e = static_cast<Pool*>(pool)->take(bytes, &b);
  *p = b.p;
  *got = b.bytes;
  return e;
}
void pool_give(void* pool, void* p, size_t bytes) {
  static_cast<Pool*>(pool)->give({static_cast<char*>(p), bytes});
}
int pool_live() { return Counting::live; }
int pool_made() { return Counting::made; }
void pool_fail(int error) { Counting::error = error; }
}
