// Batches of a few right-hand sides: y := alpha*M*X + beta*y for 2 .. 8 columns
// (FP32 tier, where a panel of 32 costs as much as about 6 single products) and
// for any number of columns in the float-float tier, NV columns per pass.
//
// A single product is bound by the decode, not by HBM, and r single products
// decode the matrix r times.  A pass streams and decodes it once for its NV
// columns, with the work ranges, the pieces and -- per column -- the arithmetic of
// the single-product kernels (kernels.cu): the same FP32 (or Dot2) operations in
// the same order inside a piece, so a column of a batch differs from its single
// product at most in the float-float order of the pieces of a chunk.
//  * vectors are interleaved, v[entry][LV] float-float, so that a piece's input
//    segment is one bulk copy and a multiplier row one or two 16-byte cp.async;
//  * k_cbatch: column dots.  Lane (g, q) as in the single kernel; the partials of a
//    round are exchanged as they come, in the reduce-scatter's tree (same sums),
//    so that 3 instead of 8 per right-hand side are live;
//  * k_gsum_b: segment sums, four groups of lanes per output, two sums a lane;
//  * k_rbatch: row chunks.  The multiplier rows are gathered straight from the
//    coefficients (source indices one piece ahead), so a batch needs no fan-out;
//  * fewer, fatter warps than the single kernels: the NV independent sums of a
//    lane hide the latency that 16 warps per SM hide there.
// Measured (AFLP): N = 131072, eps = 1e-6, 4 columns 0.473 ms, 8 columns 0.84 ms (0.88
// and 1.76 as single products); n = 32768, eps = 1e-8, 4 columns 0.48 ms (0.70).  The
// row chunks of 8 columns take all 255 registers of a thread (4 bytes spilled).
#include <cstdint>
#include <cuda_runtime.h>

#include "stream.cuh"

namespace hm {

template <int TIER, int NV>
struct BCfg {
  static constexpr int LV = NV;                            // columns of a vector row (2, 4, 8)
  static constexpr int SHAPE = NV * (TIER == TIER_FF ? 2 : 1) <= 4 ? 1 : 2;   // launch shape whose work ranges are used
  static constexpr int CW = CS_CFG_WARPS[SHAPE], RW = RS_CFG_WARPS[SHAPE];
  static constexpr int NS = 2;                             // stages per warp
  static constexpr int CSTAGE = STAGE_BYTES + SEG_ROWS * LV * 8;
  static constexpr int RSTAGE = STAGE_BYTES + PIECE_MAX_COLS * LV * 8;
  static constexpr size_t CSMEM = (size_t)CW * NS * (CSTAGE + 8) + 128;
  static constexpr size_t RSMEM = (size_t)RW * NS * (RSTAGE + 16 + 8) + 128;
  static_assert(CSMEM <= 227 * 1024 && RSMEM <= 227 * 1024, "shared memory per block");
};

// ---------------------------------------------------------------- gather, segment sums
// v[i][k] = x[perm[i] + k * ldx] as float-float, k < r; zero for k >= r.
template <int NV>
__global__ void k_gather_b(const double* __restrict__ x, int64_t ldx, int r, const int32_t* __restrict__ perm, int n,
                           float2* __restrict__ v) {
  pdl_trigger();
  pdl_wait();   // the pass before may still read the vectors
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)n * NV) return;
  const int i = (int)(t / NV), k = (int)(t % NV);
  const FF f = k < r ? ff_from_d(__ldcg(x + perm[i] + k * ldx)) : FF{0.f, 0.f};
  v[t] = make_float2(f.hi, f.lo);
}

// As the single product's segment sums -- partials p0 + k, p0 + k + 4, ... by lane
// group k, a fixed xor tree over the four groups -- with NV / 2 lanes per group,
// two right-hand sides (16 bytes) each: a lane has no more sums in flight than
// two, so that as many threads are resident as in the single kernel (N = 131072,
// width 8: 74 us with all sums in four lanes).
constexpr int GB_LANES = 4;
template <int NV>
__global__ void k_gsum_b(const GsumOut* __restrict__ outs, int nouts, const F2* __restrict__ pscale,
                         const float2* __restrict__ partial, F2 alpha, float2* __restrict__ v) {
  constexpr int KL = NV / 2, LANES = GB_LANES * KL;
  pdl_trigger();
  pdl_wait();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t i = t / LANES;
  const int k = (int)(t % LANES) / KL, kp = (int)(t % KL);
  const bool on = i < nouts;
  GsumOut O{};
  if (on) O = outs[i];
  FF s0 = {0.f, 0.f}, s1 = {0.f, 0.f};
  const float4* src = reinterpret_cast<const float4*>(partial) + kp;
  if (O.flags & 2) {
#pragma unroll 2
    for (int p = O.p0 + k; p < O.p1; p += GB_LANES) {
      const float4 x = __ldcg(src + (int64_t)p * KL);
      const F2 w = pscale[O.ps + (p - O.p0)];
      s0 = ff_add(s0, ff_mul(FF{x.x, x.y}, FF{w.hi, w.lo}));
      s1 = ff_add(s1, ff_mul(FF{x.z, x.w}, FF{w.hi, w.lo}));
    }
  } else {
#pragma unroll 4
    for (int p = O.p0 + k; p < O.p1; p += GB_LANES) {
      const float4 x = __ldcg(src + (int64_t)p * KL);
      s0 = ff_add(s0, FF{x.x, x.y});
      s1 = ff_add(s1, FF{x.z, x.w});
    }
  }
#pragma unroll
  for (int m = GB_LANES / 2; m >= 1; m >>= 1) {   // whole warps: every lane takes part
    const FF a = {__shfl_xor_sync(HM_FULL, s0.hi, m * KL), __shfl_xor_sync(HM_FULL, s0.lo, m * KL)};
    const FF b = {__shfl_xor_sync(HM_FULL, s1.hi, m * KL), __shfl_xor_sync(HM_FULL, s1.lo, m * KL)};
    s0 = (k & m) ? ff_add(a, s0) : ff_add(s0, a);
    s1 = (k & m) ? ff_add(b, s1) : ff_add(s1, b);
  }
  if (!on || k != 0) return;
  s0 = ff_mul(s0, FF{O.scale.hi, O.scale.lo});
  s1 = ff_mul(s1, FF{O.scale.hi, O.scale.lo});
  if (O.flags & 1) {
    s0 = ff_mul(s0, FF{alpha.hi, alpha.lo});
    s1 = ff_mul(s1, FF{alpha.hi, alpha.lo});
  }
  reinterpret_cast<float4*>(v)[(int64_t)O.out * KL + kp] = make_float4(s0.hi, s0.lo, s1.hi, s1.lo);
}

// ---------------------------------------------------------------- column dots
// 8 codes of decode class fb at a shared address, the class chosen around the
// decoder alone.  In the float-float tier the arithmetic of NV right-hand sides is
// several times the decoder's code: it exists once (class F < 0 below), because
// one copy for each class in use does not fit the instruction cache (NV = 4 column
// dots, n = 32768, eps = 1e-8: 515 us with the copies, 233 us so).
template <int TIER, int F, int B>
__device__ __forceinline__ void decode_b(uint32_t fb, uint32_t a, int e, int m, float (&h)[8], float (&l)[8]) {
  if constexpr (F >= 0) {
    if constexpr (TIER == TIER_F32) {
      float2 h2[4];
      decode8p<F, B>(a, e, m, h2);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        h[2 * u] = h2[u].x;
        h[2 * u + 1] = h2[u].y;
      }
    } else {
      decode8s<TIER, F, B>(a, e, m, h, l);
    }
  } else {
    switch (fb) {
#define HM_DA(FF_, BB_) \
  case ((FF_) << 4) | (BB_): decode_b<TIER, FF_, BB_>(fb, a, e, m, h, l); break;
      HM_FORMATS(HM_DA)
#undef HM_DA
      default:   // the caller has checked the class
        break;
    }
  }
}
__device__ __forceinline__ bool known_class(uint32_t fb) {
  bool ok = false;
#define HM_KC(FF_, BB_) ok = ok || fb == (((FF_) << 4) | (BB_));
  HM_FORMATS(HM_KC)
#undef HM_KC
  return ok;
}

// Dots of this lane's 8 rows of column j with NV right-hand sides.
template <int TIER, int F, int B, int NV>
__device__ __forceinline__ void cb_column(uint32_t fb, uint32_t col, uint32_t meta, bool valid, const float2 (&xh)[NV][4],
                                          const float2 (&xl)[TIER == TIER_FF ? NV : 1][4], float (&a)[NV],
                                          float (&ac)[NV]) {
  int e = 0, m = 0;
  if constexpr (F == 2 || F < 0) {
    const uint32_t em = lds32(meta) & 0xffffu;
    e = em & 0xff;
    m = em >> 8;
  }
  float h[8], l[8];
  decode_b<TIER, F, B>(fb, col, e, m, h, l);
  float2 h2[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) h2[u] = make_float2(h[2 * u], h[2 * u + 1]);
  if constexpr (TIER == TIER_F32) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      float2 a2 = __fmul2_rn(h2[0], xh[k][0]);
      a2 = __ffma2_rn(h2[1], xh[k][1], a2);
      a2 = __ffma2_rn(h2[2], xh[k][2], a2);
      a2 = __ffma2_rn(h2[3], xh[k][3], a2);
      a[k] = valid ? a2.x + a2.y : 0.f;
      ac[k] = 0.f;
    }
  } else {
    float2 n2[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) n2[u] = neg2(h2[u]);
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      float2 a2 = make_float2(0.f, 0.f), ac2 = a2;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        dot2_2(a2, ac2, h2[u], n2[u], make_float2(l[2 * u], l[2 * u + 1]), xh[k][u], xl[k][u]);
      a[k] = a2.x;
      ac[k] = ac2.x;
      pair_add<TIER>(a[k], ac[k], a2.y, ac2.y);
      if (!valid) {
        a[k] = 0.f;
        ac[k] = 0.f;
      }
    }
  }
}

// One column-dot piece: lanes (g, q) = (lane / 8, lane % 8) take rows 8q .. 8q + 7
// of the columns j0 + g + 4 t, t < 8, one step per turn of a rolled loop; the
// partials are exchanged as they come (bit 2 after every second step, bit 1 after
// every fourth, bit 0 at the end): the reduce-scatter tree of the single kernel
// with three partials live instead of eight, and one copy of the column's code
// (unrolled, the code of the classes in use does not fit the instruction cache).
template <int TIER, int F, int B, int NV>
__device__ __forceinline__ void cb_piece(uint32_t sa, uint32_t fb, int R, int nc, int flags, const float2 (&xh)[NV][4],
                                         const float2 (&xl)[TIER == TIER_FF ? NV : 1][4], int lane, F2 alpha,
                                         float2* __restrict__ partial, float2* __restrict__ vout) {
  const int g = lane >> 3, q = lane & 7;
  const uint32_t Bv = F < 0 ? fb & 15u : (uint32_t)B;
  const uint32_t stride = (((uint32_t)R + 15u) & ~15u) * Bv;
  const bool fin = (flags & ITEM_FINAL) != 0;
  const uint32_t cm = sa + (uint32_t)sizeof(CPieceHdr);
  const uint32_t sc = cm + 8u * nc;
  const uint32_t cb = cm + (fin ? 16u : 8u) * nc + RPL * q * Bv;
  const bool rows_on = RPL * q < R;
  for (int j0 = 0; j0 < nc; j0 += 32) {
    float a0[NV], a0c[NV], c0[NV], c0c[NV], d0[NV], d0c[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) a0[k] = a0c[k] = c0[k] = c0c[k] = d0[k] = d0c[k] = 0.f;
#pragma unroll 1
    for (int t = 0; t < 8; ++t) {
      float a[NV], ac[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) a[k] = ac[k] = 0.f;
      if (j0 + 4 * t < nc) {   // a step holding a column (same for the warp)
        const int j = j0 + g + 4 * t;
        const bool v = j < nc && rows_on;
        const uint32_t jj = v ? (uint32_t)j : 0u;
        cb_column<TIER, F, B, NV>(fb, cb + jj * stride, cm + 8u * jj, v, xh, xl, a, ac);
      }
      if (!(t & 1)) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          a0[k] = a[k];
          a0c[k] = ac[k];
        }
        continue;
      }
#pragma unroll
      for (int k = 0; k < NV; ++k) exchange<TIER>(a0[k], a0c[k], a[k], ac[k], (q & 4) != 0, 4, a[k], ac[k]);
      if (!(t & 2)) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          c0[k] = a[k];
          c0c[k] = ac[k];
        }
        continue;
      }
#pragma unroll
      for (int k = 0; k < NV; ++k) exchange<TIER>(c0[k], c0c[k], a[k], ac[k], (q & 2) != 0, 2, a[k], ac[k]);
      const bool last = t == 7 || j0 + 16 >= nc;   // (the other half holds no column)
      if (last) {
#pragma unroll
        for (int k = 0; k < NV; ++k)
          exchange<TIER>(t == 7 ? d0[k] : a[k], t == 7 ? d0c[k] : ac[k], t == 7 ? a[k] : 0.f, t == 7 ? ac[k] : 0.f,
                         (q & 1) != 0, 1, a[k], ac[k]);
      }
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        d0[k] = a[k];
        d0c[k] = ac[k];
      }
      if (last) break;
    }
    const int j = j0 + g + 4 * step_of_lane(q);
    if (j < nc) {
      const int64_t out = (int64_t)(int32_t)lds32(cm + 8u * j + 4u) * NV;
      float2* dst = (fin ? vout : partial) + out;
      float2 w[NV];
      FF s1 = {1.f, 0.f};
      if (fin) {
        const uint2 f = lds64(sc + 8u * j);
        s1 = FF{__uint_as_float(f.x), __uint_as_float(f.y)};
      }
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const float h = d0[k] + d0c[k];
        FF v = {h, d0c[k] - (h - d0[k])};
        if (fin) {
          v = ff_mul(v, s1);
          if (flags & ITEM_ALPHA) v = ff_mul(v, FF{alpha.hi, alpha.lo});
        }
        w[k] = make_float2(v.hi, v.lo);
      }
#pragma unroll
      for (int k = 0; k < NV; k += 2)
        *reinterpret_cast<float4*>(dst + k) = make_float4(w[k].x, w[k].y, w[k + 1].x, w[k + 1].y);
    }
  }
}

template <int TIER, int NV>
__global__ void __launch_bounds__(BCfg<TIER, NV>::CW * 32, 1)
    k_cbatch(const ItemCopy* __restrict__ cps, const int32_t* __restrict__ wbeg, int nwt,
             const uint8_t* __restrict__ pay, const float2* __restrict__ vec, F2 alpha, float2* __restrict__ partial,
             float2* __restrict__ vout, int* err) {
  using C = BCfg<TIER, NV>;
  constexpr int NS = C::NS, NW = C::CW, SSTR = C::CSTAGE;
  extern __shared__ __align__(128) uint8_t smem[];
  pdl_trigger();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gw = range_of<NW>(warp, nwt);
  if (gw >= nwt) return;
  const int p0 = wbeg[gw], n = wbeg[gw + 1] - p0;
  if (n <= 0) return;
  uint8_t* ring = smem + (size_t)warp * NS * SSTR;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)NW * NS * SSTR) + warp * NS;
  if (lane == 0) {
    for (int s = 0; s < NS; ++s) mbar_init(&bars[s], 1);
    mbar_init_fence();
  }
  __syncwarp();
  const uint32_t sring = smem_u32(ring);
  const ItemCopy zero{0, 0, -1, 0};
  ItemCopy dc = lane < n ? cps[p0 + lane] : zero;
  ItemCopy dn = 32 + lane < n ? cps[p0 + 32 + lane] : zero;
  int dbase = 0, issued = 0;
  const uint64_t pol = policy_evict_first();
  int32_t last_vin = -1, last_rows = -1;
  // all lanes; copies piece i (and, if `withx`, its input segment when it is a new one); returns whether it is
  auto issue = [&](int i, bool withx) {
    if (i - dbase >= 32) {
      dc = dn;
      dbase += 32;
      dn = dbase + 32 + lane < n ? cps[p0 + dbase + 32 + lane] : zero;
    }
    const int sl = i - dbase;
    const uint32_t off16 = __shfl_sync(HM_FULL, dc.off16, sl);
    const uint32_t bytes = __shfl_sync(HM_FULL, dc.bytes, sl);
    const int32_t vin = __shfl_sync(HM_FULL, dc.vin, sl);
    const int32_t nrows = __shfl_sync(HM_FULL, dc.nrows, sl);
    const bool newx = vin != last_vin || nrows != last_rows;
    last_vin = vin;
    last_rows = nrows;
    if (lane == 0) {
      const int s = i % NS;
      uint8_t* st = ring + s * SSTR;
      const uint32_t pb = pad16u(bytes), xb = newx ? (uint32_t)nrows * NV * 8u : 0u;
      fence_proxy_async();
      mbar_expect_tx(&bars[s], pb + xb);
      bulk_g2s_hint(st, pay + (uint64_t)off16 * 16u, pb, &bars[s], pol);
      if (newx && withx) bulk_g2s(st + STAGE_BYTES, vec + (int64_t)vin * NV, xb, &bars[s]);
    }
    issued = i + 1;
    return newx;
  };
  unsigned xs = 0;
  for (int i = 0; i < NS && i < n; ++i) xs |= (unsigned)issue(i, false) << i;
  pdl_wait();   // the input segments come from the previous kernel
  for (int i = 0; i < NS && i < n; ++i) {
    const int32_t vin = __shfl_sync(HM_FULL, dc.vin, i), nrows = __shfl_sync(HM_FULL, dc.nrows, i);
    if (lane == 0 && (xs >> i & 1u))
      bulk_g2s(ring + i * SSTR + STAGE_BYTES, vec + (int64_t)vin * NV, (uint32_t)nrows * NV * 8u, &bars[i]);
  }
  float2 xh[NV][4], xl[TIER == TIER_FF ? NV : 1][4];
  int32_t xv = -1, xr = -1;
  for (int i = 0; i < n; ++i) {
    const int s = i % NS;
    if (!mbar_wait(&bars[s], (uint32_t)((i / NS) & 1))) {
      latch_error(err, 99);
      drain<NS>(bars, i + 1, issued);
      return;
    }
    const uint32_t sa = sring + (uint32_t)(s * SSTR);
    const uint4 hw = lds128(sa);   // CPieceHdr
    const int32_t hvin = (int32_t)hw.x;
    const int R = (int)(hw.y & 0xffffu), nc = (int)(hw.y >> 16);
    const uint32_t fb = hw.z & 0xffffu, flags = hw.z >> 16;
    if (hvin != xv || R != xr) {   // a new input segment came with this piece
      const uint32_t xa = sa + STAGE_BYTES + (uint32_t)(RPL * (lane & 7) * NV * 8);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const bool in = RPL * (lane & 7) + u < R;
#pragma unroll
        for (int k = 0; k < NV; k += 2) {
          uint4 v = make_uint4(0u, 0u, 0u, 0u);
          if (in) v = lds128(xa + (uint32_t)((u * NV + k) * 8));
          float* h0 = u & 1 ? &xh[k][u / 2].y : &xh[k][u / 2].x;
          float* h1 = u & 1 ? &xh[k + 1][u / 2].y : &xh[k + 1][u / 2].x;
          *h0 = __uint_as_float(v.x);
          *h1 = __uint_as_float(v.z);
          if constexpr (TIER == TIER_FF) {
            float* l0 = u & 1 ? &xl[k][u / 2].y : &xl[k][u / 2].x;
            float* l1 = u & 1 ? &xl[k + 1][u / 2].y : &xl[k + 1][u / 2].x;
            *l0 = __uint_as_float(v.y);
            *l1 = __uint_as_float(v.w);
          }
        }
      }
      xv = hvin;
      xr = R;
    }
    if constexpr (TIER == TIER_FF) {
      if (known_class(fb))
        cb_piece<TIER, -1, 0, NV>(sa, fb, R, nc, (int)flags, xh, xl, lane, alpha, partial, vout);
      else
        latch_error(err, 1);
    } else {
      switch (fb) {
#define HM_CB(FF_, BB_) \
  case ((FF_) << 4) | (BB_): cb_piece<TIER, FF_, BB_, NV>(sa, fb, R, nc, (int)flags, xh, xl, lane, alpha, partial, vout); break;
        HM_FORMATS(HM_CB)
#undef HM_CB
        default:
          latch_error(err, 1);
      }
    }
    __syncwarp();
    if (issued < n) issue(issued, true);
  }
}

// ---------------------------------------------------------------- row chunks
// The piece's columns into this lane's 8 rows of NV right-hand sides, as the
// single kernel's rs_piece.
template <int TIER, int F, int B, int NV>
__device__ __forceinline__ void rb_piece(uint32_t sa, const PieceHdr& H, F2 alpha_ff, int lane, float2 (&ahi)[NV][4],
                                         float2 (&alo)[NV][4]) {
  const int R = H.nrows;
  int G, S, slot, q;
  lane_split(R, lane, G, S, slot, q);
  const bool tile = (H.flags & PH_TILE) != 0;
  const uint32_t Bv = F < 0 ? H.fb & 15u : (uint32_t)B;
  const uint32_t stride = pad8u((uint32_t)R * Bv);
  const uint32_t cm = sa + (uint32_t)sizeof(PieceHdr);
  const uint32_t cb = cm + (tile ? 0u : pad8u(2u * H.ncols)) + RPL * q * Bv;
  const uint32_t tbl = sa + STAGE_BYTES;
  const int e_t = H.em & 0xff, m_t = H.em >> 8;
  FF sc = {1.f, 0.f};
  if (tile) {
    sc = FF{H.scale.hi, H.scale.lo};
    if (H.flags & PH_TALPHA) sc = ff_mul(sc, FF{alpha_ff.hi, alpha_ff.lo});
  }
  const int nc = slot < S ? H.ncols : 0;
  float2 s2[NV][4], c2[TIER == TIER_FF ? NV : 1][4];
#pragma unroll
  for (int k = 0; k < NV; ++k)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      s2[k][u] = make_float2(0.f, 0.f);
      if constexpr (TIER == TIER_FF) c2[k][u] = make_float2(0.f, 0.f);
    }
#pragma unroll 1
  for (int j = slot; j < nc; j += S) {
    int e = e_t, m = m_t;
    if constexpr (F == 2 || F < 0) {
      if (!tile) {
        const uint32_t em = lds32((cm + 2u * j) & ~3u) >> (16u * (j & 1));
        e = em & 0xff;
        m = (em >> 8) & 0xff;
      }
    }
    float h[8], l[8];
    decode_b<TIER, F, B>(H.fb, cb + (uint32_t)j * stride, e, m, h, l);
    float2 h2[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) h2[u] = make_float2(h[2 * u], h[2 * u + 1]);
    if constexpr (TIER == TIER_F32) {
#pragma unroll
      for (int k = 0; k < NV; k += 2) {
        const uint4 t = lds128(tbl + (uint32_t)((j * NV + k) * 8));
        const float v0 = __uint_as_float(t.x) * sc.hi, v1 = __uint_as_float(t.z) * sc.hi;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          s2[k][u] = __ffma2_rn(h2[u], make_float2(v0, v0), s2[k][u]);
          s2[k + 1][u] = __ffma2_rn(h2[u], make_float2(v1, v1), s2[k + 1][u]);
        }
      }
    } else {
      float2 n2[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) n2[u] = neg2(h2[u]);
#pragma unroll
      for (int k = 0; k < NV; k += 2) {
        const uint4 t = lds128(tbl + (uint32_t)((j * NV + k) * 8));
        FF v[2] = {{__uint_as_float(t.x), __uint_as_float(t.y)}, {__uint_as_float(t.z), __uint_as_float(t.w)}};
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          if (tile) v[w] = ff_mul(v[w], sc);
          const float2 vh2 = make_float2(v[w].hi, v[w].hi), vl2 = make_float2(v[w].lo, v[w].lo);
#pragma unroll
          for (int u = 0; u < 4; ++u)
            dot2_2(s2[k + w][u], c2[k + w][u], h2[u], n2[u], make_float2(l[2 * u], l[2 * u + 1]), vh2, vl2);
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < NV; ++k)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if constexpr (TIER == TIER_F32)
        ff_add_f2(ahi[k][u], alo[k][u], s2[k][u]);
      else
        ff_add_dot2(ahi[k][u], alo[k][u], s2[k][u], c2[k][u]);
    }
}

struct RbArgs {
  const PieceCopy* cps;
  const uint8_t* pay;
  const float2* vec;
  F2 alpha_ff;
  double beta;
  double* y;
  int64_t ldy;
  int r;                    // columns of this pass (<= NV)
  int mode;
  const int32_t* perm;
  float2* vout;
  const F2* rowscale;
  F2* fix;                  // per right-hand side nfix slots of CHUNK_ROWS
  int64_t nfix;
  int32_t* fixcnt;          // per right-hand side nsplit counters
  int nsplit;
  const Split* splits;
  const int32_t* fan;       // source of fan-out slot fan_base + i
  int32_t fan_base;
  int* err;
};

template <int TIER, int NV>
__global__ void __launch_bounds__(BCfg<TIER, NV>::RW * 32, 1)
    k_rbatch(RbArgs A, const int32_t* __restrict__ wbeg, int nwt) {
  using C = BCfg<TIER, NV>;
  constexpr int NS = C::NS, NW = C::RW, SSTR = C::RSTAGE;
  extern __shared__ __align__(128) uint8_t smem[];
  pdl_trigger();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gw = range_of<NW>(warp, nwt);
  if (gw >= nwt) return;
  const int p0 = wbeg[gw], n = wbeg[gw + 1] - p0;
  if (n <= 0) return;
  uint8_t* ring = smem + (size_t)warp * NS * SSTR;
  int4* info = reinterpret_cast<int4*>(smem + (size_t)NW * NS * SSTR) + warp * NS;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)NW * NS * (SSTR + 16)) + warp * NS;
  if (lane == 0) {
    for (int s = 0; s < NS; ++s) mbar_init(&bars[s], 1 + 32);   // expect-tx arrival + 32 cp.async arrivals
    mbar_init_fence();
  }
  __syncwarp();
  const uint32_t sring = smem_u32(ring);
  const PieceCopy zero{0, 0, 0, -1};
  PieceCopy dc = lane < n ? A.cps[p0 + lane] : zero;
  PieceCopy dn = 32 + lane < n ? A.cps[p0 + 32 + lane] : zero;
  int dbase = 0, issued = 0;
  const uint64_t pol = policy_evict_first();
  // sources of a piece's multiplier rows lane and lane + 32, loaded one piece ahead
  int32_t src[2] = {0, 0};
  auto sources = [&](int i) {
    const int sl = i - dbase;   // < 64: within dc / dn
    const uint32_t bf = __shfl_sync(HM_FULL, sl < 32 ? dc.bytes_flags : dn.bytes_flags, sl & 31);
    const int32_t moff = __shfl_sync(HM_FULL, sl < 32 ? dc.moff : dn.moff, sl & 31);
    const int nc = (int)(bf >> 24);
    const bool fan_run = moff >= A.fan_base;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = lane + 32 * u;
      src[u] = j < nc ? (fan_run ? __ldg(A.fan + (moff - A.fan_base) + j) : moff + j) : 0;
    }
  };
  auto payload = [&](int i) {
    if (i - dbase >= 32) {
      dc = dn;
      dbase += 32;
      dn = dbase + 32 + lane < n ? A.cps[p0 + dbase + 32 + lane] : zero;
    }
    const int sl = i - dbase;
    const uint32_t off16 = __shfl_sync(HM_FULL, dc.off16, sl), bf = __shfl_sync(HM_FULL, dc.bytes_flags, sl);
    const int32_t sp = __shfl_sync(HM_FULL, dc.split_part, sl);
    const int s = i % NS;
    const uint32_t pb = pad16u(bf & 0xffffu);
    fence_proxy_async();
    if (lane == 0) {
      info[s] = make_int4((int)((bf >> 16) & 0xffu), sp, 0, 0);
      mbar_expect_tx(&bars[s], pb);
      bulk_g2s_hint(ring + s * SSTR, A.pay + (uint64_t)off16 * 16u, pb, &bars[s], pol);
    }
    __syncwarp();
    issued = i + 1;
  };
  auto rows = [&](int i) {   // src holds piece i's sources
    const int s = i % NS;
    const int nc = (int)(__shfl_sync(HM_FULL, dc.bytes_flags, i - dbase) >> 24);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = lane + 32 * u;
      if (j < nc) {
        const uint32_t dst = sring + (uint32_t)(s * SSTR + STAGE_BYTES + j * NV * 8);
        const float2* row = A.vec + (int64_t)src[u] * NV;
#pragma unroll
        for (int c = 0; c < NV / 2; ++c)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * c), "l"(row + 2 * c) : "memory");
      }
    }
    cp_arrive(&bars[s]);
    if (i + 1 < n) sources(i + 1);
  };
  sources(0);
  for (int i = 0; i < NS && i < n; ++i) payload(i);
  pdl_wait();   // multipliers and outputs depend on the previous kernels
  for (int i = 0; i < NS && i < n; ++i) rows(i);
  float2 ahi[NV][4], alo[NV][4];
#pragma unroll
  for (int k = 0; k < NV; ++k)
#pragma unroll
    for (int u = 0; u < 4; ++u) ahi[k][u] = alo[k][u] = make_float2(0.f, 0.f);
  for (int i = 0; i < n; ++i) {
    const int s = i % NS;
    if (!mbar_wait(&bars[s], (uint32_t)((i / NS) & 1))) {
      latch_error(A.err, 99);
      drain<NS>(bars, i + 1, issued);
      return;
    }
    const uint32_t sa = sring + (uint32_t)(s * SSTR);
    PieceHdr H;
    {
      const uint4 a = lds128(sa), b = lds128(sa + 16);
      H.row0 = (int32_t)a.x;
      H.nrows = (uint16_t)(a.y & 0xffffu);
      H.flags = (uint16_t)(a.y >> 16);
      H.fb = (uint16_t)(a.z & 0xffffu);
      H.em = (uint16_t)(a.z >> 16);
      H.vin0 = (int32_t)a.w;
      H.ncols = (uint16_t)(b.x & 0xffffu);
      H.scale = F2{__uint_as_float(b.z), __uint_as_float(b.w)};
    }
    const int4 rinfo = info[s];
    if (rinfo.x & PD_FIRST) {
#pragma unroll
      for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int u = 0; u < 4; ++u) ahi[k][u] = alo[k][u] = make_float2(0.f, 0.f);
    }
    if constexpr (TIER == TIER_FF) {
      if (known_class(H.fb))
        rb_piece<TIER, -1, 0, NV>(sa, H, A.alpha_ff, lane, ahi, alo);
      else
        latch_error(A.err, 2);
    } else {
      switch (H.fb) {
#define HM_RB(FF_, BB_) \
  case ((FF_) << 4) | (BB_): rb_piece<TIER, FF_, BB_, NV>(sa, H, A.alpha_ff, lane, ahi, alo); break;
        HM_FORMATS(HM_RB)
#undef HM_RB
        default:
          latch_error(A.err, 2);
      }
    }
    if (rinfo.x & PD_LAST) {
      const int fl = H.flags | ((rinfo.x & PD_SPLIT) ? 0x10000 : 0);
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        if (k >= A.r) break;
        AccR<RPL> a8;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          a8.v[2 * u] = FF{ahi[k][u].x, alo[k][u].x};
          a8.v[2 * u + 1] = FF{ahi[k][u].y, alo[k][u].y};
        }
        F2* fix = A.fix + (int64_t)k * A.nfix * CHUNK_ROWS;
        int32_t* cnt = A.fixcnt + (int64_t)k * A.nsplit;
        if (A.mode == MODE_Y)
          rs_emit<MODE_Y, RPL, NV>(a8, H.row0, H.nrows, fl, rinfo.y >> 8, rinfo.y & 0xff, lane, A.alpha_ff, A.beta,
                                   A.y + k * A.ldy, A.perm, nullptr, nullptr, fix, cnt, A.splits);
        else if (A.mode == MODE_VEC)
          rs_emit<MODE_VEC, RPL, NV>(a8, H.row0, H.nrows, fl, rinfo.y >> 8, rinfo.y & 0xff, lane, A.alpha_ff, A.beta,
                                     nullptr, A.perm, A.vout + k, A.rowscale, fix, cnt, A.splits);
        else
          rs_emit<MODE_VEC_ADD, RPL, NV>(a8, H.row0, H.nrows, fl, rinfo.y >> 8, rinfo.y & 0xff, lane, A.alpha_ff,
                                         A.beta, nullptr, A.perm, A.vout + k, A.rowscale, fix, cnt, A.splits);
      }
    }
    __syncwarp();
    if (issued < n) {
      payload(issued);
      rows(issued - 1);
    }
  }
}

// ---------------------------------------------------------------- launchers
#define HM_B_ALL(X) X(TIER_F32, 2) X(TIER_F32, 4) X(TIER_F32, 8) X(TIER_FF, 2) X(TIER_FF, 4)

cudaError_t batch_init() {
  cudaError_t e = cudaSuccess;
#define HM_BI(T, V)                                                                                              \
  if (e == cudaSuccess)                                                                                          \
    e = cudaFuncSetAttribute(k_cbatch<T, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BCfg<T, V>::CSMEM);  \
  if (e == cudaSuccess)                                                                                          \
    e = cudaFuncSetAttribute(k_rbatch<T, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BCfg<T, V>::RSMEM);
  HM_B_ALL(HM_BI)
#undef HM_BI
  return e;
}

// Launch shape whose work ranges a batch of nv columns uses.
int batch_shape(int tier, int nv) {
#define HM_BS(T, V) \
  if (tier == T && nv == V) return BCfg<T, V>::SHAPE;
  HM_B_ALL(HM_BS)
#undef HM_BS
  return -1;
}

cudaError_t launch_gather_b(int nv, const double* x, int64_t ldx, int r, const int32_t* perm, int n, float2* v,
                            cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const unsigned grid = (unsigned)(((int64_t)n * nv + 255) / 256);
  switch (nv) {
    case 2: return launch_pdl(k_gather_b<2>, grid, 256, 0, st, x, ldx, r, perm, n, v);
    case 4: return launch_pdl(k_gather_b<4>, grid, 256, 0, st, x, ldx, r, perm, n, v);
    case 8: return launch_pdl(k_gather_b<8>, grid, 256, 0, st, x, ldx, r, perm, n, v);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_gsum_b(int nv, const GsumOut* outs, int nouts, const F2* pscale, const float2* partial, F2 alpha,
                          float2* v, cudaStream_t st) {
  if (nouts <= 0) return cudaSuccess;
  const unsigned grid = (unsigned)(((int64_t)nouts * GB_LANES * (nv / 2) + 255) / 256);
  switch (nv) {
    case 2: return launch_pdl(k_gsum_b<2>, grid, 256, 0, st, outs, nouts, pscale, partial, alpha, v);
    case 4: return launch_pdl(k_gsum_b<4>, grid, 256, 0, st, outs, nouts, pscale, partial, alpha, v);
    case 8: return launch_pdl(k_gsum_b<8>, grid, 256, 0, st, outs, nouts, pscale, partial, alpha, v);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_cdot_b(int tier, int nv, const ItemCopy* items, const int32_t* wbeg, int nw, const uint8_t* pay,
                          const float2* vec, F2 alpha, float2* partial, float2* vout, int* err, cudaStream_t st) {
  if (nw <= 0) return cudaSuccess;
#define HM_BC(T, V)                                                                                              \
  if (tier == T && nv == V)                                                                                      \
    return launch_pdl(k_cbatch<T, V>, spread_blocks(nw, BCfg<T, V>::CW), BCfg<T, V>::CW * 32,        \
                      BCfg<T, V>::CSMEM, st, items, wbeg, nw, pay, vec, alpha, partial, vout, err);
  HM_B_ALL(HM_BC)
#undef HM_BC
  return cudaErrorInvalidValue;
}

cudaError_t launch_rgemv_b(int tier, int nv, int mode, const PieceCopy* pieces, const int32_t* wbeg, int nw,
                           const uint8_t* pay, float2* vec, F2 alpha_ff, double beta, double* y, int64_t ldy, int r,
                           const int32_t* perm, const F2* rowscale, F2* fix, int64_t nfix, int32_t* fixcnt, int nsplit,
                           const Split* splits, const int32_t* fan, int32_t fan_base, int* err, cudaStream_t st) {
  if (nw <= 0) return cudaSuccess;
  const RbArgs A{pieces, pay, vec,  alpha_ff, beta,   y,      ldy,    r,   mode,     perm, vec,
                 rowscale, fix, nfix, fixcnt,   nsplit, splits, fan, fan_base, err};
#define HM_BR(T, V)                                                                                              \
  if (tier == T && nv == V)                                                                                      \
    return launch_pdl(k_rbatch<T, V>, spread_blocks(nw, BCfg<T, V>::RW), BCfg<T, V>::RW * 32,        \
                      BCfg<T, V>::RSMEM, st, A, wbeg, nw);
  HM_B_ALL(HM_BR)
#undef HM_BR
  return cudaErrorInvalidValue;
}

}  // namespace hm
