// Host check of the device's H-LU schedule (LuProgram::steps / citems / scols):
// test code, built by tests/test_lu_schedule.py against the library's host
// objects; no GPU code.  It replays the schedule in FP64 with its own decoder,
// steps in order and every column item as soon as its last rows are solved, and
// checks that every value a step or item reads is final by the condition the
// kernel waits for (finished steps, coefficient counter), that the late columns
// are the ones of the step right before, and that the result equals the replay
// of the work list it was derived from.
// usage: lu_schedule_check <points file> n kernel eps codec leaf
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "program.h"

using namespace hm;

static int g_fails = 0;
#define CHECK(cond)                                                         \
  do {                                                                      \
    if (!(cond) && g_fails++ < 20) std::printf("FAIL line %d: %s\n", __LINE__, #cond); \
  } while (0)

static double value(const LuProgram& P, uint64_t off, uint16_t fb, uint16_t em, int r) {
  CodeHdr h;
  h.B = fb & 15;
  h.fmt = fb >> 4;
  h.e = em & 0xff;
  h.m = em >> 8;
  h.vmin = 1.0;
  uint64_t code = 0;
  for (int b = 0; b < h.B; ++b) code |= (uint64_t)P.pk.pay[off + (uint64_t)r * h.B + b] << (8 * b);
  return decode_value(code, h);
}

int main(int argc, char** argv) {
  if (argc != 7) return 2;
  const int64_t n = std::atoll(argv[2]);
  std::vector<double> pts(3 * n), b(n);
  FILE* f = std::fopen(argv[1], "rb");
  if (!f || std::fread(pts.data(), 8, 3 * n, f) != (size_t)(3 * n) || std::fread(b.data(), 8, n, f) != (size_t)n) return 2;
  std::fclose(f);
  hm_build_params prm{};
  prm.kernel = std::atoi(argv[3]);
  prm.eta = 2.0;
  prm.eps_build = std::atof(argv[4]);
  prm.leaf_size = std::atoi(argv[6]);
  prm.nthreads = 8;
  HostMatrix L, U;
  LuProgram P;
  if (!lu_factor_host(prm, pts.data(), n, L, U) || !build_lu_program(L, U, std::atoi(argv[5]), prm.eps_build, 1, P)) return 1;
  const int nl = (int)P.nleaves;
  CHECK((int)P.steps.size() == 2 * nl);
  // the work list, in order
  std::vector<double> lw(n, 0.0), lx(n, 0.0), lc(P.ncoef, 0.0);
  auto solve_tri = [&](bool fwd, int R, const std::vector<double>& T, std::vector<double>& r) {   // T[j R + i], scaled
    if (fwd) {
      for (int j = 0; j < R; ++j)
        for (int i = j + 1; i < R; ++i) r[i] -= T[(size_t)j * R + i] * r[j];
    } else {
      for (int j = R - 1; j >= 0; --j) {
        r[j] /= T[(size_t)j * R + j];
        for (int i = 0; i < j; ++i) r[i] -= T[(size_t)j * R + i] * r[j];
      }
    }
  };
  for (const LuItem& it : P.items) {
    const bool fwd = it.kind == LU_ROW_L || it.kind == LU_COL_L;
    std::vector<double>& v = fwd ? lw : lx;
    if (it.kind == LU_ROW_L || it.kind == LU_ROW_U) {
      std::vector<double> r(it.nr), T((size_t)it.nr * it.nr);
      for (int i = 0; i < it.nr; ++i) r[i] = fwd ? b[L.ct.perm[it.r0 + i]] : lw[it.r0 + i];
      for (int j = it.c0; j < it.c1; ++j) {
        const LuCol& c = P.cols[j];
        const double m = ((c.flags & LC_COEF) ? lc[c.mult] : v[c.mult]) * c.scale;
        for (int i = 0; i < it.nr; ++i) r[i] -= value(P, c.off, c.fb, c.em, i) * m;
      }
      for (int j = 0; j < it.nr; ++j)
        for (int i = 0; i < it.nr; ++i)
          T[(size_t)j * it.nr + i] = value(P, P.cols[it.tri + j].off, P.cols[it.tri + j].fb, P.cols[it.tri + j].em, i) *
                                     P.cols[it.tri + j].scale;
      solve_tri(fwd, it.nr, T, r);
      for (int i = 0; i < it.nr; ++i) v[it.r0 + i] = r[i];
    } else {
      for (int j = it.c0; j < it.c1; ++j) {
        const LuCol& c = P.cols[j];
        double s = 0;
        for (int i = 0; i < it.nr; ++i) s += value(P, c.off, c.fb, c.em, i) * v[it.r0 + i];
        lc[c.mult] = s * c.scale;
      }
    }
  }
  // the schedule; NaN marks what is not final yet
  std::vector<double> w(n, NAN), x(n, NAN), coef(P.ncoef, NAN);
  std::vector<int> cnt(P.nflags, 0);
  size_t ci = 0;
  for (int s = 0; s < (int)P.steps.size(); ++s) {
    const LuStep& S = P.steps[s];
    const bool fwd = s < nl;
    std::vector<double>& v = fwd ? w : x;
    CHECK(S.nr >= 1 && S.nr <= P.maxr && S.nr <= CHUNK_ROWS);
    CHECK(S.e0 <= S.e1 && S.e1 == S.l0 && S.l1 - S.l0 <= LU_LATE && S.need_rhs <= s);
    CHECK(S.t0 == S.l1 && S.t0 + S.nr <= (int)P.scols.size());
    std::vector<double> r(S.nr), T((size_t)S.nr * S.nr);
    for (int i = 0; i < S.nr; ++i) {
      CHECK(P.rowleaf[S.r0 + i] == (fwd ? s : 2 * nl - 1 - s));
      r[i] = fwd ? b[L.ct.perm[S.r0 + i]] : w[S.r0 + i];
    }
    for (int j = S.e0; j < S.l1; ++j) {
      const LuSCol& c = P.scols[j];
      CHECK(c.need <= s && (j < S.l0 || c.need == s));
      CHECK(j == S.e0 || P.scols[j - 1].need <= c.need);
      if (c.flag >= 0) CHECK(cnt[c.flag] == c.target);
      const double m = (c.flag >= 0 ? coef[c.mult] : v[c.mult]) * c.scale;
      CHECK(std::isfinite(m));
      for (int i = 0; i < S.nr; ++i) r[i] -= value(P, c.off, c.fb, c.em, i) * m;
    }
    for (int j = 0; j < S.nr; ++j) {
      const LuSCol& c = P.scols[S.t0 + j];
      for (int i = 0; i < S.nr; ++i) T[(size_t)j * S.nr + i] = value(P, c.off, c.fb, c.em, i) * c.scale;
    }
    solve_tri(fwd, S.nr, T, r);
    for (int i = 0; i < S.nr; ++i) v[S.r0 + i] = r[i];
    // column items whose rows are all solved, in list order
    for (; ci < P.citems.size(); ++ci) {
      const LuCItem& it = P.citems[ci];
      std::vector<double>& z = it.bwd ? x : w;
      const int need = it.bwd ? 2 * nl - P.rowleaf[it.r0] : P.rowleaf[it.r0 + it.nr - 1] + 1;
      if (need > s + 1) break;
      CHECK(it.nc >= 1 && it.nc <= 4 && it.bwd == (fwd ? 0 : 1));
      for (int j = it.c0; j < it.c0 + it.nc; ++j) {
        const LuSCol& c = P.scols[j];
        double t = 0;
        for (int i = 0; i < it.nr; ++i) t += value(P, c.off, c.fb, c.em, i) * z[it.r0 + i];
        CHECK(std::isfinite(t));
        coef[c.mult] = t * c.scale;
      }
      cnt[it.flag] += it.nc;
    }
  }
  CHECK(ci == P.citems.size());
  double d = 0, nn = 0;
  for (int64_t i = 0; i < n; ++i) {
    d += (x[i] - lx[i]) * (x[i] - lx[i]);
    nn += lx[i] * lx[i];
  }
  std::printf("diff %.3e steps %zu items %zu\n", std::sqrt(d / nn), P.steps.size(), P.citems.size());
  CHECK(std::sqrt(d / nn) < 1e-11);
  std::printf(g_fails ? "FAILED %d\n" : "ok\n", g_fails);
  return g_fails != 0;
}
