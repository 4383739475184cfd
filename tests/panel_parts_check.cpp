// Host check of the parts of a panel's shared row chunks (csrc/program.cpp, cta_part):
// test code, built by tests/test_panel_parts.py; no GPU code.  No range of a panel
// launch may be empty, and the tensor-core kernel's walk -- CTAs of consecutive ranges,
// a chunk's parts in one CTA taken as one -- must close every chunk once for each CTA
// that holds pieces of it, with numbers 0, 1, ... below the count it waits for, and
// sum every piece exactly once.
// usage: panel_parts_check <points file> n format eps codec leaf adm
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <vector>

#include "program.h"

using namespace hm;

static int g_fails = 0;
#define CHECK(cond)                                                         \
  do {                                                                      \
    if (!(cond) && g_fails++ < 20) std::printf("FAIL line %d: %s\n", __LINE__, #cond); \
  } while (0)

int main(int argc, char** argv) {
  if (argc != 8) return 2;
  const int64_t n = std::atoll(argv[2]);
  HostMatrix H;
  hm_build_params prm{};
  prm.kernel = HM_KERNEL_LAPLACE;
  prm.format = std::atoi(argv[3]);
  prm.eta = 2.0;
  prm.eps_build = std::atof(argv[4]);
  prm.leaf_size = std::atoi(argv[6]);
  prm.adm = std::atoi(argv[7]);
  prm.nthreads = 8;
  H.prm = prm;
  H.n = n;
  H.kparam = std::sqrt(4.0 * M_PI / (double)n);
  H.pts.resize(3 * n);
  FILE* f = std::fopen(argv[1], "rb");
  if (!f || std::fread(H.pts.data(), 8, 3 * n, f) != (size_t)(3 * n)) return 2;
  std::fclose(f);
  build_cluster_tree(H.pts.data(), n, prm.leaf_size, H.ct);
  build_block_tree(H.ct, prm.eta, H.blocks, prm.adm);
  build_lowrank_blocks(H, 8);
  if (prm.format == HM_FMT_UH || prm.format == HM_FMT_UH_SEP) build_uniform_bases(H, 8);
  if (prm.format == HM_FMT_H2) build_nested_bases(H, 8);
  Program P;
  if (!build_program(H, std::atoi(argv[5]), prm.eps_build, 1, 152, P)) return 1;
  int64_t shared = 0, merged = 0;
  for (const Launch& L : P.launches) {
    if (L.kind != Launch::RGEMV || L.n == 0) continue;
    const int32_t* wb = P.wbeg.data() + L.woff[MR_SHAPE];
    const int nrange = L.nw[MR_SHAPE];
    CHECK(wb[0] == L.off && wb[nrange] == L.off + L.n);
    for (int r = 0; r < nrange; ++r) CHECK(wb[r] < wb[r + 1]);
    auto chunk = [&](int64_t p) {   // the chunk's first row, from the piece's header
      PieceHdr h;
      std::memcpy(&h, P.pk.pay.data() + (uint64_t)P.pdesc[MR_SHAPE][p].off16 * 16u, sizeof h);
      return h.row0;
    };
    std::map<int32_t, int64_t> total;
    for (int64_t p = L.off; p < L.off + L.n; ++p) ++total[chunk(p)];
    for (int grid : {152, (nrange + 5) / 6, 1, 7}) {
      const int per = (nrange + grid - 1) / grid;
      std::map<int32_t, int64_t> summed;
      std::map<int32_t, std::set<int>> closed;
      std::map<int32_t, int> want;
      for (int c = 0; c < grid; ++c) {
        const int r0 = c * per, r1 = std::min(r0 + per, nrange);
        if (r0 >= nrange) continue;
        int range = r0;
        bool more = false;
        int64_t acc = 0;
        for (int64_t p = wb[r0]; p < wb[r1]; ++p) {
          if (p == wb[range + 1]) ++range;
          const PieceCopy& d = P.pdesc[MR_SHAPE][p];
          const uint32_t fl = (d.bytes_flags >> 16) & 0xffu;
          if ((fl & PD_FIRST) && !more) {
            CHECK(acc == 0);
            acc = 0;
          }
          ++acc;
          CtaPart cp{false, 0, 1};
          if ((fl & PD_LAST) && (fl & PD_SPLIT)) {
            cp = cta_part(range, d.split_part & 0xff, P.splits[d.split_part >> 8].nparts, per, r1);
            ++shared;
            merged += cp.more;
          }
          more = (fl & PD_LAST) ? cp.more : false;
          if (more) CHECK(p + 1 < wb[r1] && chunk(p + 1) == chunk(p));
          if ((fl & PD_LAST) && !more) {
            const int32_t ch = chunk(p);
            CHECK(cp.idx >= 0 && cp.idx < cp.nparts && closed[ch].insert(cp.idx).second);
            CHECK(!want.count(ch) || want[ch] == cp.nparts);
            want[ch] = cp.nparts;
            summed[ch] += acc;
            acc = 0;
          }
        }
        CHECK(acc == 0);
      }
      CHECK(summed == total);
      for (const auto& w : want) CHECK((int)closed[w.first].size() == w.second);
    }
  }
  std::printf("parts %lld merged %lld\n", (long long)shared, (long long)merged);
  std::printf(g_fails ? "FAILED %d\n" : "ok\n", g_fails);
  return g_fails != 0;
}
