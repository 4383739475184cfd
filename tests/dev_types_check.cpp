// Host check of the index arithmetic that the kernels share (csrc/dev_types.h):
// test code, built by tests/test_dev_types.py; no GPU code.
#include <cstdint>
#include <cstdio>
#include <initializer_list>
#include <limits>

#include "dev_types.h"

using namespace hm;

static int g_fails = 0;
#define CHECK(cond)                                                         \
  do {                                                                      \
    if (!(cond) && g_fails++ < 20) std::printf("FAIL line %d: %s\n", __LINE__, #cond); \
  } while (0)

// Every entry a program may have, times the right-hand sides a batch interleaves.
template <int VS>
static void offsets() {
  for (int64_t i : {int64_t(0), int64_t(1), (int64_t(1) << 31) / VS - 1, (int64_t(1) << 31) / VS, int64_t(1) << 30,
                    (int64_t)std::numeric_limits<int32_t>::max()})
    if (i <= std::numeric_limits<int32_t>::max()) CHECK(entry_offset<VS>((int32_t)i) == i * VS);
}

// Tries until a wait on `value(try)` gives up, at most `max`.
template <class F>
static int64_t tries(uint32_t limit, int64_t max, F value) {
  Patience p(limit);
  int64_t i = 0;
  while (i < max && p.again(value(i))) ++i;
  return i;
}

int main() {
  // a number that never moves: limit tries; one that moves within the limit: no end; one that stops: limit more
  CHECK(tries(100, 10000, [](int64_t) { return 7; }) == 99);
  CHECK(tries(100, 100000, [](int64_t i) { return (int)(i / 99); }) == 100000);
  CHECK(tries(100, 100000, [](int64_t i) { return (int)(i < 5000 ? i / 50 : 99); }) == 4950 + 99);
  CHECK(tries(100, 10000, [](int64_t) { return 0; }) == 99);
  offsets<1>();
  offsets<2>();
  offsets<4>();
  offsets<8>();
  std::printf(g_fails ? "FAILED %d\n" : "ok\n", g_fails);
  return g_fails != 0;
}
