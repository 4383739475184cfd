// Triangular solves with compressed H-LU factors (Sec. 5, Conclusion: the
// triangular solves of an H-LU factorisation read the same compressed blocks
// as the product, with sequential dependencies between them).
//
// x = U^-1 L^-1 b for up to LU_MAX_RHS right-hand sides is ONE persistent
// cooperative launch over the schedule of schedule_lu (hlu.cpp).  What bounds it
// is the chain of leaf solves (two per leaf, forward then backward), not
// bandwidth or arithmetic: the factors of n = 2048 are 15 MB.  So the design
// keeps everything but the newest dependency off that chain:
//  * the leaf steps complete in list order, so "which leaves are solved" is one
//    number, the frontier.  One watcher warp per block polls it and republishes
//    it in shared memory; the workers wait there (no dependency lists, one
//    poller per block on the one hot line).
//  * row blocks (half of the grid) take whole leaf steps in order, up to
//    gridDim / 2 steps ahead of the frontier.  A step decodes its diagonal
//    triangle and its late columns (those that read the step right before it)
//    to FP64 in shared memory before it waits for anything, adds the early
//    columns as their multipliers become final (sorted by that moment), and has
//    only the late columns and the substitution left once the step before it
//    is published.  Lane = row there: no cross-lane reduction on the chain.
//  * column blocks (the other half) form the coefficients t_b = S_b X_b^T z of
//    the low-rank factor blocks, one warp per item of <= 4 columns, following
//    the frontier through the rows of the block's column cluster, so that only
//    the last 64 rows remain when its last leaf is solved.
//  * all right-hand sides of a launch share every decoded value, every wait and
//    every hop of the chain (FP64 vectors [entry][NR]).
// Measured (Matern cube n = 2048, leaf 32, 93 leaves, eps = 1e-6, 3 right-hand
// sides): 1.34 ms, 7.2 us per leaf step; 788 ms before, when one warp took a leaf
// (its dependencies polled one by one, two columns at a time from global
// memory, the triangle decoded inside the substitution) and each right-hand
// side was a launch.
//
// Every packed value is decoded with the float-float-tier decoders of the
// product kernels (exact: head + tail is the stored value) and the arithmetic
// is FP64; a right-hand side's operations and their order do not depend on NR.
//
// A step or item waits only for earlier ones in the work list, both kinds are
// claimed in list order and all blocks are resident: the earliest unfinished one
// never waits for anything unfinished, so the launch cannot stall.  Every wait is
// bounded by the time without a finished step (Patience), so that neither a long
// solve nor a GPU shared with other work runs into it; after the first that runs out
// the abort word makes all later ones return at once, and the launch runs to its end.
#include <cstdint>
#include <cuda_runtime.h>

#include "decode.cuh"

namespace hm {

constexpr int LU_NW = 8;                          // worker warps per block (and one watcher warp)
constexpr int LU_THREADS = (LU_NW + 1) * 32;

struct LuArgs {
  const LuSCol* cols;
  const LuStep* steps;
  int nsteps;
  const LuCItem* citems;
  int ncitems;
  const int32_t* rowleaf;   // leaf index of each row (cluster order)
  const int32_t* perm;
  int nl;                   // leaves: steps 0 .. nl - 1 forward, nl .. 2 nl - 1 backward
  const uint8_t* pay;
  const double* b;          // original order
  int64_t ldb;
  double* x;                // original order
  int64_t ldx;
  double* w;                // forward result [row][NR], cluster order
  double* xz;               // solution [row][NR], cluster order
  double* coef;             // coefficients of the low-rank factor blocks [k][NR]
  int* flags;               // coefficient counters (zeroed before the launch)
  int* frontier;            // NR times the number of finished steps
  unsigned* claim;          // [0] steps, [1] column items handed out
  int* abort;               // set on the first timeout: every other wait gives up
  int* err;
};

// The block's copy of the frontier in shared memory (-1 after an abort).
__device__ __forceinline__ int front_load(uint32_t a) {
  int v;
  asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void front_store(uint32_t a, int v) {
  asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release(int* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void lu_fail(const LuArgs& A) {
  atomicExch(A.abort, 1);
  latch_error(A.err, 99);
}

// Wait until `need` steps are finished (bounded: about 2 s without a step).
template <int NR>
__device__ __forceinline__ void wait_front(const LuArgs& A, uint32_t sf, int need) {
  Patience p(1u << 26);
  for (;;) {
    const int v = front_load(sf);
    if (v >= need * NR || v < 0) return;
    if (!p.again(v)) break;
  }
  lu_fail(A);
}

// Wait until the multiplier of column c is final.
template <int NR>
__device__ __forceinline__ void wait_col(const LuArgs& A, uint32_t sf, const LuSCol& c) {
  wait_front<NR>(A, sf, c.need);
  if (c.flag < 0) return;
  Patience p(1u << 16);
  for (;;) {   // 64 tries of an L2 round trip each, then a look at the frontier: about 2 s without a step
    for (int i = 0; i < 64; ++i)
      if (ld_acquire(A.flags + c.flag) >= c.target) return;
    const int v = front_load(sf);
    if (v < 0) return;
    if (!p.again(v)) break;
  }
  lu_fail(A);
}

// The 8 B bytes of rows 8 g .. 8 g + 7 of packed column c (a column's last group
// may read past its rows: the payload has slack, the rows are masked later).
__device__ __forceinline__ void lu_raw(const LuArgs& A, const LuSCol& c, int g, uint2 (&raw)[8]) {
  const int B = c.fb & 15;
  const uint2* src = reinterpret_cast<const uint2*>(A.pay + c.off + (uint64_t)g * RPL * B);
#pragma unroll
  for (int i = 0; i < 8; ++i) raw[i] = i < B ? __ldg(src + i) : make_uint2(0u, 0u);
}

template <int F, int B>
__device__ __forceinline__ void lu_decode8(const uint2 (&raw)[8], int e, int m, double (&v)[8]) {
  uint32_t w[2 * B], w0[B], w1[B];
#pragma unroll
  for (int i = 0; i < B; ++i) {
    w[2 * i] = raw[i].x;
    w[2 * i + 1] = raw[i].y;
  }
#pragma unroll
  for (int i = 0; i < B; ++i) {
    w0[i] = w[i];
    w1[i] = w[B + i];
  }
  float h[4], l[4];
  decode4<TIER_FF, F, B>(w0, e, m, h, l);
#pragma unroll
  for (int u = 0; u < 4; ++u) v[u] = (double)h[u] + (double)l[u];
  decode4<TIER_FF, F, B>(w1, e, m, h, l);
#pragma unroll
  for (int u = 0; u < 4; ++u) v[4 + u] = (double)h[u] + (double)l[u];
}

// Those 8 values exactly (FP64), unscaled.
__device__ __forceinline__ void lu_values(const LuArgs& A, const LuSCol& c, const uint2 (&raw)[8], double (&v)[8]) {
  const int e = c.em & 0xff, m = c.em >> 8;
  switch (c.fb) {
#define HM_LU(FF_, BB_) \
  case ((FF_) << 4) | (BB_): lu_decode8<FF_, BB_>(raw, e, m, v); break;
    HM_FORMATS(HM_LU)
#undef HM_LU
    default:
      latch_error(A.err, 2);
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = 0.0;
  }
}

__device__ __forceinline__ void workers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(LU_NW * 32) : "memory"); }

// Shared memory of a row block (doubles), for leaves of at most R rows.
struct LuSmem {
  double* tri;    // triangle: forward strictly lower by columns, backward upper by columns, 1 / U_jj on its diagonal
  double* late;   // late columns [k][R]
  double* part;   // row sums of the worker warps [warp][R][NR]
  double* res;    // b - early contributions [R][NR]
};

// One leaf step of NR right-hand sides by the block's workers.
template <int NR>
__device__ void lu_step(const LuArgs& A, int s, const LuSmem& M, uint32_t sf, int warp, int lane) {
  const LuStep S = A.steps[s];
  const int R = S.nr, G = (R + RPL - 1) / RPL, NS = 32 / G, slot = lane / G, q = lane - slot * G;
  const bool fwd = s < A.nl, slot_on = slot < NS;
  const double* vin = fwd ? A.w : A.xz;
  const int nlate = S.l1 - S.l0;
  // triangle and late columns to FP64 (no dependencies)
  for (int k = warp * NS + slot; slot_on && k < R + nlate; k += LU_NW * NS) {
    const bool is_tri = k < R;
    const LuSCol c = A.cols[is_tri ? S.t0 + k : S.l0 + (k - R)];
    uint2 raw[8];
    double v[8];
    lu_raw(A, c, q, raw);
    lu_values(A, c, raw, v);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = RPL * q + u;
      if (i >= R) continue;
      if (!is_tri)
        M.late[(k - R) * R + i] = v[u];
      else if (fwd) {
        if (i > k) M.tri[k * (2 * R - k - 1) / 2 + (i - k - 1)] = v[u] * c.scale;
      } else if (i <= k) {
        M.tri[k * (k + 1) / 2 + i] = i == k ? 1.0 / (v[u] * c.scale) : v[u] * c.scale;
      }
    }
  }
  // early columns: NS per warp and turn, in the order in which their multipliers become final
  double acc[8][NR];
#pragma unroll
  for (int u = 0; u < 8; ++u)
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[u][r] = 0.0;
  {
    const int step = LU_NW * NS;
    int k = S.e0 + warp * NS + slot;
    const int kend = slot_on ? S.e1 : S.e0;
    LuSCol c{}, cn{};
    uint2 raw[8] = {};
    if (k < kend) {
      c = A.cols[k];
      if (k + step < kend) cn = A.cols[k + step];
      lu_raw(A, c, q, raw);
    }
    for (; k < kend; k += step) {
      double v[8];
      lu_values(A, c, raw, v);
      const LuSCol cur = c;
      c = cn;
      if (k + step < kend) {   // the next turn's codes and the parameters of the one after it
        lu_raw(A, c, q, raw);
        if (k + 2 * step < kend) cn = A.cols[k + 2 * step];
      }
      wait_col<NR>(A, sf, cur);
      const double* src = (cur.flag >= 0 ? A.coef : vin) + (int64_t)cur.mult * NR;
      double mlt[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r) mlt[r] = __ldcg(src + r) * cur.scale;
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[u][r] = fma(v[u], mlt[r], acc[u][r]);
    }
    __syncwarp();
  }
  // over the column slots (pairwise tree), then the warps' sums to shared memory
  for (int off = 1; off < NS; off <<= 1) {
    const bool take = (slot & (2 * off - 1)) == 0 && slot + off < NS;
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const double t = __shfl_down_sync(HM_FULL, acc[u][r], off * G);
        if (take) acc[u][r] += t;
      }
  }
  if (slot == 0)
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (RPL * q + u < R)
#pragma unroll
        for (int r = 0; r < NR; ++r) M.part[((size_t)warp * R + RPL * q + u) * NR + r] = acc[u][r];
  workers_sync();
  if (!fwd) wait_front<NR>(A, sf, S.need_rhs);
  for (int i = warp * 32 + lane; i < R * NR; i += LU_NW * 32) {
    const int row = i / NR, r = i - row * NR;
    double t = fwd ? __ldg(A.b + __ldg(A.perm + S.r0 + row) + r * A.ldb) : __ldcg(A.w + (int64_t)S.r0 * NR + i);
    double p[LU_NW];
#pragma unroll
    for (int k = 0; k < LU_NW; ++k) p[k] = M.part[(size_t)k * R * NR + i];
    t -= ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
    M.res[i] = t;
  }
  workers_sync();   // part is free again
  // late columns: columns warp, warp + LU_NW, ... (lane kk waits for and loads the kk-th), rows by lane
  {
    const int mine = (nlate - warp + LU_NW - 1) / LU_NW;
    double ml[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) ml[r] = 0.0;
    if (lane < mine) {
      const LuSCol c = A.cols[S.l0 + warp + LU_NW * lane];
      wait_col<NR>(A, sf, c);
      const double* src = (c.flag >= 0 ? A.coef : vin) + (int64_t)c.mult * NR;
#pragma unroll
      for (int r = 0; r < NR; ++r) ml[r] = __ldcg(src + r) * c.scale;
    }
    __syncwarp();
    for (int j0 = 0; j0 < R; j0 += 32) {
      const int row = j0 + lane;
      double a[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r) a[r] = 0.0;
      for (int k = 0; k < mine; ++k) {
        const double v = row < R ? M.late[(warp + LU_NW * k) * R + row] : 0.0;
#pragma unroll
        for (int r = 0; r < NR; ++r) a[r] = fma(v, __shfl_sync(HM_FULL, ml[r], k), a[r]);
      }
      if (row < R)
#pragma unroll
        for (int r = 0; r < NR; ++r) M.part[((size_t)warp * R + row) * NR + r] = a[r];
    }
  }
  workers_sync();
  // substitution, one warp per right-hand side; lane holds rows lane, lane + 32, ...
  if (warp < NR) {
    const int r = warp;
    double z[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int row = 32 * j + lane;
      z[j] = 0.0;
      if (row < R) {
        double p[LU_NW];
#pragma unroll
        for (int k = 0; k < LU_NW; ++k) p[k] = M.part[((size_t)k * R + row) * NR + r];
        z[j] = M.res[row * NR + r] - (((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7])));
      }
    }
    if (fwd) {   // unit lower triangle: z_j final, then rows i > j lose L_ij z_j
#pragma unroll
      for (int jb = 0; jb < 4; ++jb) {
        const double* t = M.tri;
#pragma unroll 4
        for (int j = 32 * jb; j < min(R, 32 * jb + 32); ++j) {
          const double* col = t + (j * (2 * R - j - 1) / 2 - j - 1);
          const double zj = __shfl_sync(HM_FULL, z[jb], j & 31);
#pragma unroll
          for (int k = jb; k < 4; ++k) {
            const int i = 32 * k + lane;
            if (i > j && i < R) z[k] = fma(-col[i], zj, z[k]);
          }
        }
      }
    } else {     // upper triangle: x_j = r_j / U_jj, then rows i < j lose U_ij x_j
#pragma unroll
      for (int jb = 3; jb >= 0; --jb) {
#pragma unroll 4
        for (int j = min(R, 32 * jb + 32) - 1; j >= 32 * jb; --j) {
          const double* col = M.tri + j * (j + 1) / 2;
          const double xj = __shfl_sync(HM_FULL, z[jb], j & 31) * col[j];
#pragma unroll
          for (int k = 0; k <= jb; ++k) {
            const int i = 32 * k + lane;
            if (i < j) z[k] = fma(-col[i], xj, z[k]);
            if (i == j) z[k] = xj;
          }
        }
      }
    }
    double* out = fwd ? A.w : A.xz;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int row = 32 * j + lane;
      if (row < R) __stcg(out + ((int64_t)S.r0 + row) * NR + r, z[j]);
    }
    __syncwarp();   // the lanes' rows before lane 0's release
    if (lane == 0) {
      wait_front<NR>(A, sf, s);   // steps are published in order
      red_release(A.frontier, 1);
    }
    if (!fwd)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int row = 32 * j + lane;
        if (row < R) A.x[__ldg(A.perm + S.r0 + row) + r * A.ldx] = z[j];
      }
  }
}

// One column item: coef[mult] = scale * sum_r X[r, j] z[r] for its <= 4 columns;
// lane (c = lane / 8, q = lane % 8) takes rows 8 q .. 8 q + 7 of column c of each
// 64-row piece, the pieces in the order in which their rows are solved.
template <int NR>
__device__ void lu_citem(const LuArgs& A, int ci, uint32_t sf, int lane) {
  const LuCItem it = A.citems[ci];
  const int cl = lane >> 3, q = lane & 7, np = (it.nr + 63) / 64;
  const bool on = cl < it.nc;
  const bool fwd = it.bwd == 0;
  const double* vin = fwd ? A.w : A.xz;
  LuSCol c{};
  if (on) c = A.cols[it.c0 + cl];
  double s[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) s[r] = 0.0;
  uint2 raw[8] = {};
  int need = 0;
  auto fetch = [&](int p) {   // codes and the required step of piece p
    const int a = 64 * p, b = min(it.nr, a + 64);
    if (on && a + RPL * q < it.nr) lu_raw(A, c, 8 * p + q, raw);
    need = lu_piece_need(fwd, A.nl, __ldg(A.rowleaf + it.r0 + a), __ldg(A.rowleaf + it.r0 + b - 1));
  };
  fetch(fwd ? 0 : np - 1);
  for (int k = 0; k < np; ++k) {
    const int p = fwd ? k : np - 1 - k, r0 = 64 * p + RPL * q;
    const bool have = on && r0 < it.nr;
    const int nd = need;
    double v[8];
    if (have) lu_values(A, c, raw, v);
    if (k + 1 < np) fetch(fwd ? p + 1 : p - 1);
    wait_front<NR>(A, sf, nd);
    if (have) {
      const double* z = vin + ((int64_t)it.r0 + r0) * NR;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (r0 + u < it.nr)
#pragma unroll
          for (int r = 0; r < NR; ++r) s[r] = fma(v[u], __ldcg(z + u * NR + r), s[r]);
    }
  }
  __syncwarp();
#pragma unroll
  for (int o = 4; o >= 1; o >>= 1)
#pragma unroll
    for (int r = 0; r < NR; ++r) s[r] += __shfl_xor_sync(HM_FULL, s[r], o);
  if (on && q == 0)
#pragma unroll
    for (int r = 0; r < NR; ++r) __stcg(A.coef + (int64_t)c.mult * NR + r, s[r] * c.scale);
  __syncwarp();
  if (lane == 0) red_release(A.flags + it.flag, it.nc);
}

template <int NR>
__global__ void __launch_bounds__(LU_THREADS, 1) k_lusolve(LuArgs A, int row_blocks, int maxr) {
  extern __shared__ __align__(16) double lu_smem[];
  __shared__ int s_front, s_step;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t sf = smem_u32(&s_front);
  if (threadIdx.x == 0) s_front = 0;
  __syncthreads();
  if (warp == LU_NW) {   // the watcher
    if (lane == 0) {
      const int total = A.nsteps * NR;
      int v = 0;
      Patience p(1u << 24);
      for (uint32_t i = 0; v < total; ++i) {
        v = ld_acquire(A.frontier);
        if ((i & 31u) == 31u && *(volatile int*)A.abort) break;
        front_store(sf, v);
        if (!p.again(v)) break;
      }
      if (v < total) {   // an abort, or no step for seconds
        lu_fail(A);
        front_store(sf, -1);
      }
    }
    return;
  }
  if ((int)blockIdx.x < row_blocks) {
    LuSmem M;
    M.tri = lu_smem;
    M.late = M.tri + (size_t)maxr * (maxr + 1) / 2;
    M.part = M.late + (size_t)LU_LATE * maxr;
    M.res = M.part + (size_t)LU_NW * maxr * NR;
    for (;;) {
      workers_sync();
      if (threadIdx.x == 0) s_step = (int)atomicAdd(A.claim, 1u);
      workers_sync();
      const int s = s_step;
      if (s >= A.nsteps) return;
      lu_step<NR>(A, s, M, sf, warp, lane);
    }
  }
  for (;;) {
    int i = 0;
    if (lane == 0) i = (int)atomicAdd(A.claim + 1, 1u);
    i = __shfl_sync(HM_FULL, i, 0);
    if (i >= A.ncitems) return;
    lu_citem<NR>(A, i, sf, lane);
  }
}

static size_t lu_smem_bytes(int maxr, int nr) {
  return ((size_t)maxr * (maxr + 1) / 2 + (size_t)LU_LATE * maxr + (size_t)(LU_NW + 1) * maxr * nr) * sizeof(double);
}

// One launch for nr <= LU_MAX_RHS right-hand sides (original order, device) on
// stream st; ctl holds the coefficient counters, the frontier, two claim
// counters and the abort word (nflags + 4 ints, zeroed first).
cudaError_t launch_lusolve(int nblk, int nr, const LuSCol* cols, const LuStep* steps, int nsteps, const LuCItem* citems,
                           int ncitems, const int32_t* rowleaf, const int32_t* perm, int nl, int maxr,
                           const uint8_t* pay, const double* b, int64_t ldb, double* x, int64_t ldx, double* w,
                           double* xz, double* coef, int* ctl, int nflags, int* err, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(ctl, 0, (size_t)(nflags + 4) * sizeof(int), st);
  if (e != cudaSuccess) return e;
  LuArgs A{cols, steps, nsteps, citems, ncitems, rowleaf, perm, nl,   pay,          b,
           ldb,  x,     ldx,    w,      xz,      coef,    ctl,  ctl + nflags,
           reinterpret_cast<unsigned*>(ctl + nflags + 1), ctl + nflags + 3, err};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)nblk);
  cfg.blockDim = dim3(LU_THREADS);
  cfg.dynamicSmemBytes = lu_smem_bytes(maxr, nr);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const int row_blocks = ncitems > 0 ? nblk / 2 : nblk;
  switch (nr) {
    case 1: e = cudaLaunchKernelEx(&cfg, k_lusolve<1>, A, row_blocks, maxr); break;
    case 2: e = cudaLaunchKernelEx(&cfg, k_lusolve<2>, A, row_blocks, maxr); break;
    case 3: e = cudaLaunchKernelEx(&cfg, k_lusolve<3>, A, row_blocks, maxr); break;
    case 4: e = cudaLaunchKernelEx(&cfg, k_lusolve<4>, A, row_blocks, maxr); break;
    default: return cudaErrorInvalidValue;
  }
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int NR>
static cudaError_t lu_fit(int maxr, int& per_sm) {
  const size_t sm = lu_smem_bytes(maxr, NR);
  const cudaError_t e = cudaFuncSetAttribute(k_lusolve<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)lu_smem_bytes(CHUNK_ROWS, LU_MAX_RHS));
  if (e != cudaSuccess) return e;
  int n = 0;
  const cudaError_t o = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_lusolve<NR>, LU_THREADS, sm);
  per_sm = per_sm < n ? per_sm : n;
  return o;
}

// Blocks of the persistent solve that fit on the device at once (leaves of at most maxr rows).
int lusolve_max_blocks(int maxr) {
  int per_sm = 1 << 20, dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (lu_fit<1>(maxr, per_sm) != cudaSuccess || lu_fit<2>(maxr, per_sm) != cudaSuccess ||
      lu_fit<3>(maxr, per_sm) != cudaSuccess || lu_fit<4>(maxr, per_sm) != cudaSuccess)
    return 0;
  return per_sm * nsm;
}

}  // namespace hm
