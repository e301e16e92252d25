// An allocation that fails while an array grows: the array is empty afterwards, with
// capacity zero, and the next request, also a smaller one than the old capacity,
// allocates.  Prints "OK" and exits 0, or the failed line and exits 1.
#include "common.cuh"

#include <new>

#define CHECK(x) \
  if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; }

int main() {
  int* p = nullptr;
  size_t cap = 0;
  int live = 0;
  bool fail = false;
  auto alloc = [&](size_t n) -> int* {
    if (fail) throw std::bad_alloc();
    ++live;
    return new int[n];
  };
  auto release = [&](int* q) {
    --live;
    delete[] q;
  };
  rihf::regrow(p, cap, 100, alloc, release);
  CHECK(p && cap == 100 && live == 1);
  int* first = p;
  rihf::regrow(p, cap, 60, alloc, release);
  CHECK(p == first && cap == 100);
  fail = true;
  bool thrown = false;
  try {
    rihf::regrow(p, cap, 200, alloc, release);
  } catch (const std::bad_alloc&) {
    thrown = true;
  }
  CHECK(thrown && !p && cap == 0 && live == 0);
  fail = false;
  rihf::regrow(p, cap, 60, alloc, release);
  CHECK(p && cap == 60 && live == 1);
  p[59] = 1;
  release(p);
  printf("OK\n");
  return 0;
}
