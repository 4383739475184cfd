// Host check of the waits of the H-LU column items (LuProgram::citems): test code,
// built by tests/test_lu_pieces.py against the library's host objects; no GPU code.
// The kernel takes an item in pieces of 64 rows, forward from the first and backward
// from the last, and waits before each until lu_piece_need steps are finished: every
// row it then reads must be final, the waits must not go backwards, and the last one
// must be what the item's columns record.
// usage: lu_pieces_check <points file> n eps codec leaf
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "program.h"

using namespace hm;

static int g_fails = 0;
#define CHECK(cond)                                                         \
  do {                                                                      \
    if (!(cond) && g_fails++ < 20) std::printf("FAIL line %d: %s\n", __LINE__, #cond); \
  } while (0)

int main(int argc, char** argv) {
  if (argc != 6) return 2;
  const int64_t n = std::atoll(argv[2]);
  std::vector<double> pts(3 * n);
  FILE* f = std::fopen(argv[1], "rb");
  if (!f || std::fread(pts.data(), 8, 3 * n, f) != (size_t)(3 * n)) return 2;
  std::fclose(f);
  hm_build_params prm{};
  prm.kernel = HM_KERNEL_MATERN15;
  prm.eta = 2.0;
  prm.eps_build = std::atof(argv[3]);
  prm.leaf_size = std::atoi(argv[5]);
  prm.nthreads = 8;
  HostMatrix L, U;
  LuProgram P;
  if (!lu_factor_host(prm, pts.data(), n, L, U) || !build_lu_program(L, U, std::atoi(argv[4]), prm.eps_build, 1, P)) return 1;
  const int nl = (int)P.nleaves;
  // steps after which each row is final, from the steps themselves
  std::vector<int> fin[2];
  for (auto& v : fin) v.assign(n, 1 << 30);
  for (int s = 0; s < (int)P.steps.size(); ++s)
    for (int i = 0; i < P.steps[s].nr; ++i) fin[s < nl ? 0 : 1][P.steps[s].r0 + i] = s + 1;
  int64_t pieces = 0;
  for (const LuCItem& it : P.citems) {
    const bool fwd = it.bwd == 0;
    const int np = (it.nr + 63) / 64;
    int before = 0;
    std::vector<bool> read(it.nr, false);
    for (int k = 0; k < np; ++k, ++pieces) {
      const int p = fwd ? k : np - 1 - k, a = 64 * p, b = std::min(it.nr, a + 64);
      const int need = lu_piece_need(fwd, nl, P.rowleaf[it.r0 + a], P.rowleaf[it.r0 + b - 1]);
      CHECK(need >= before);
      before = need;
      for (int i = a; i < b; ++i) {
        CHECK(fin[it.bwd][it.r0 + i] <= need && !read[i]);
        read[i] = true;
      }
    }
    CHECK(std::count(read.begin(), read.end(), true) == it.nr);
    for (int j = it.c0; j < it.c0 + it.nc; ++j) CHECK(P.scols[j].need == before);
  }
  std::printf("items %zu pieces %lld\n", P.citems.size(), (long long)pieces);
  std::printf(g_fails ? "FAILED %d\n" : "ok\n", g_fails);
  return g_fails != 0;
}
