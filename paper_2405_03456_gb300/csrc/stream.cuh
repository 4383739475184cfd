// Device code shared by the streaming kernels: the single-product kernels
// (kernels.cu) and the batch kernels of a few right-hand sides (batch.cu).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "decode.cuh"

namespace hm {

__device__ __forceinline__ uint32_t pad16u(uint32_t x) { return (x + 15u) & ~15u; }

// After a bounded wait gave up: wait (bounded) for the copies still in flight
// into this warp's stages [i, issued) so that none lands after the block exits.
template <int NS>
__device__ void drain(uint64_t* bars, int i, int issued, uint32_t it0 = 0) {
  for (int j = i; j < issued; ++j) {
    const uint32_t u = it0 + (uint32_t)j;
    mbar_wait(&bars[u % NS], (u / NS) & 1u, 50u);
  }
}

// Programmatic dependent launch: a kernel lets the next one in the stream start
// at once (its blocks take SM resources as they free up and run their prologue),
// and waits for the previous one (completed, memory visible) before it reads
// anything that kernel wrote.  Both are no-ops for ordinary launches.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Range of warp (or pair) w of this block.  A launch with fewer ranges than warps
// on the device gets one block per SM all the same and deals its ranges out over
// the blocks, so that a short launch uses every SM (16 ranges on one SM share its
// issue slots while others idle).  So does a launch whose last block is not full; one
// whose ranges fill its blocks exactly keeps neighbouring ranges together.
template <int NW>
__device__ __forceinline__ int range_of(int w, int nranges) {
  return (int)gridDim.x * NW > nranges ? w * (int)gridDim.x + (int)blockIdx.x : (int)blockIdx.x * NW + w;
}

// ---------------------------------------------------------------- column dots
// (s, c) += (s2, c2) for Dot2 pairs (TwoSum of the leading parts).
template <int TIER>
__device__ __forceinline__ void pair_add(float& s, float& c, float s2, float c2) {
  if constexpr (TIER == TIER_F32) {
    s += s2;
  } else {
    float t, e;
    two_sum(s, s2, t, e);
    s = t;
    c += c2 + e;
  }
}

// One exchange over lane bit `mask`: the lane keeps b if `up`, else a, sends the
// other and adds its partner's copy of what it kept.
template <int TIER>
__device__ __forceinline__ void exchange(float a, float ac, float b, float bc, bool up, int mask, float& p, float& pc) {
  const float got = __shfl_xor_sync(HM_FULL, up ? a : b, mask);
  float gotc = 0.f;
  if constexpr (TIER == TIER_FF) gotc = __shfl_xor_sync(HM_FULL, up ? ac : bc, mask);
  const float keep = up ? b : a, keepc = up ? bc : ac;
  p = keep;
  pc = keepc;
  pair_add<TIER>(p, pc, got, gotc);
}

// Column step (of a round of 8) whose total lane q = 0 .. 7 of a column's lanes
// holds after exchanges over bit 2 (steps 2 i, 2 i + 1), bit 1 (pairs of those),
// bit 0: the reversed bits of q.
__device__ __forceinline__ int step_of_lane(int q) { return ((q & 1) << 2) | (q & 2) | (q >> 2); }

// ---------------------------------------------------------------- row chunks
// Lane split of a row-chunk piece: G = ceil(R / 8) lanes per column, S = 32 / G
// column slots, lane = slot G + q.  The divisions by the runtime G go through a
// table: slot = (lane * ceil(1024 / G)) >> 10 is exact for lane < 1024 / G,
// which holds for lane < 32 and G <= 16.
__constant__ uint16_t c_div1024[17] = {0,    1024, 512, 342, 256, 205, 171, 147, 128,
                                       114,  103,  94,  86,  79,  74,  69,  64};
__constant__ uint8_t c_slots[17] = {0, 32, 16, 10, 8, 6, 5, 4, 4, 3, 3, 2, 2, 2, 2, 2, 2};
__device__ __forceinline__ void lane_split(int R, int lane, int& G, int& S, int& slot, int& q) {
  G = (R + RPL - 1) / RPL;
  S = c_slots[G];
  slot = (lane * (int)c_div1024[G]) >> 10;
  q = lane - slot * G;
}

// Float-float row sums of a lane (RL rows), passed by value to the emit path.
template <int RL>
struct AccR {
  FF v[RL];
};

// Write the finished rows g0 .. g0 + nr - 1 of a chunk (nr <= RL; a lane's rows).
// Every global load the rows need (y through perm, the old coefficients, the row
// scales) is issued before the first store, so the lane waits for one round trip
// instead of one per row.  Coefficient vectors stay in float-float arithmetic
// (FP64 instructions are scarce on this GPU); y takes the FP64 sum hi + lo.
// Coefficient entries are VS apart (batches interleave their right-hand sides).
template <int MODE, int RL, int VS = 1>
__device__ __forceinline__ void rs_store_rows(const AccR<RL>& acc, int g0, int nr, F2 alpha_ff, double beta,
                                              double* __restrict__ y, const int32_t* __restrict__ perm,
                                              float2* __restrict__ vout, const F2* __restrict__ rowscale,
                                              bool calpha) {
  if constexpr (MODE == MODE_Y) {
    int o[RL];
#pragma unroll
    for (int u = 0; u < RL; ++u) o[u] = u < nr ? __ldg(perm + g0 + u) : 0;
    double yo[RL];
#pragma unroll
    for (int u = 0; u < RL; ++u) yo[u] = (u < nr && beta != 0.0) ? y[o[u]] : 0.0;
#pragma unroll
    for (int u = 0; u < RL; ++u) {
      if (u < nr) {
        const double val = ff_to_d(acc.v[u]);
        y[o[u]] = (beta == 0.0) ? val : fma(beta, yo[u], val);
      }
    }
  } else {
    float2 old[RL], sc[RL];
#pragma unroll
    for (int u = 0; u < RL; ++u) {
      old[u] = (MODE == MODE_VEC_ADD && u < nr) ? __ldcg(vout + entry_offset<VS>(g0 + u)) : make_float2(0.f, 0.f);
      sc[u] = (rowscale && u < nr) ? __ldg(reinterpret_cast<const float2*>(rowscale + g0 + u)) : make_float2(1.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < RL; ++u) {
      if (u < nr) {
        FF v = acc.v[u];
        if constexpr (MODE == MODE_VEC_ADD) v = ff_add(v, FF{old[u].x, old[u].y});
        if (rowscale) v = ff_mul(v, FF{sc[u].x, sc[u].y});
        if (calpha) v = ff_mul(v, FF{alpha_ff.hi, alpha_ff.lo});
        vout[entry_offset<VS>(g0 + u)] = make_float2(v.hi, v.lo);
      }
    }
  }
}

// End of a warp's part of a chunk (hflags: piece header flags, bit 16 set when
// the chunk is shared by several warps): reduce the column slots (fixed order), then
// emit the rows, directly or through the fix-up of a chunk shared by warps (the
// last part to arrive sums all parts in a fixed order, so the result does not
// depend on which warp finishes last).
// Out of line: it runs once per part and keeps the piece loop compact.
template <int MODE, int RL, int VS = 1>
__device__ __noinline__ bool rs_emit(AccR<RL> acc, int row0, int R, int hflags, int split, int pidx, int lane,
                                     F2 alpha_ff, double beta, double* __restrict__ y,
                                     const int32_t* __restrict__ perm, float2* __restrict__ vout,
                                     const F2* __restrict__ rowscale, F2* __restrict__ fix,
                                     int32_t* __restrict__ fixcnt, const Split* __restrict__ splits) {
  static_assert(RL == RPL, "lanes hold RPL rows");
  int G, S, slot, q;
  lane_split(R, lane, G, S, slot, q);
  const int rows = slot < S ? min(RL, R - RL * q) : 0;
  const bool shared = (hflags & 0x10000) != 0;
  for (int turn = 0;; ++turn) {
    // pairwise tree over the S column slots (slot s takes s + off when s is a
    // multiple of 2 off): log2 S shuffle rounds, all rows of a round in flight
    for (int off = 1; off < S; off <<= 1) {
      float hi[RL], lo[RL];
#pragma unroll
      for (int u = 0; u < RL; ++u) {
        hi[u] = __shfl_down_sync(HM_FULL, acc.v[u].hi, off * G);
        lo[u] = __shfl_down_sync(HM_FULL, acc.v[u].lo, off * G);
      }
      if ((slot & (2 * off - 1)) == 0 && slot + off < S) {
#pragma unroll
        for (int u = 0; u < RL; ++u) acc.v[u] = ff_add(acc.v[u], FF{hi[u], lo[u]});
      }
    }
    if (!shared || turn == 1) break;
    const Split sp = splits[split];
    F2* mypart = fix + (size_t)(sp.slot0 + pidx) * CHUNK_ROWS + RL * q;   // split, pidx: from the piece's split / part word
    if (lane < G)
#pragma unroll
      for (int u = 0; u < RL; ++u)
        if (u < rows) mypart[u] = F2{acc.v[u].hi, acc.v[u].lo};
    __syncwarp();   // the part's rows before lane 0's release
    int last = 0;
    if (lane == 0) last = atom_add_acq_rel(&fixcnt[split], 1) == sp.nparts - 1;
    last = __shfl_sync(HM_FULL, last, 0);
    if (!last) return false;
    __syncwarp();   // lane 0's acquire before the lanes read the other parts
    // the parts dealt out over the slots, then the same tree: a small matrix has
    // chunks of more than ten parts, and one load round trip for each in turn was most
    // of its launch (H product, n = 4096: 30.2 us before, 22.4 us now)
#pragma unroll
    for (int u = 0; u < RL; ++u) acc.v[u] = FF{0.f, 0.f};
    const F2* base = fix + (size_t)sp.slot0 * CHUNK_ROWS + RL * q;
    if (slot < S)
#pragma unroll 1
      for (int k = slot; k < sp.nparts; k += S) {   // the rows of one part: independent loads, then the sums
        float2 v[RL];
#pragma unroll
        for (int u = 0; u < RL; ++u)
          v[u] = u < rows ? __ldcg(reinterpret_cast<const float2*>(base + (size_t)k * CHUNK_ROWS + u))
                          : make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < RL; ++u) acc.v[u] = ff_add(acc.v[u], FF{v[u].x, v[u].y});
      }
    if (lane == 0) fixcnt[split] = 0;   // ready for the next product
  }
  // slot 0 lanes hold the chunk's rows RL q .. RL q + RL - 1
  if (lane < G)
    rs_store_rows<MODE, RL, VS>(acc, row0 + RL * q, rows, alpha_ff, beta, y, perm, vout, rowscale,
                                (hflags & PH_CALPHA) != 0);
  return true;
}

// ---------------------------------------------------------------- launches
// Blocks of NW ranges each for nranges ranges (see range_of).
inline unsigned spread_blocks(int nranges, int NW) {
  int dev = 0, nsm = 1;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    nsm = 1;
  const int need = (nranges + NW - 1) / NW;
  return (unsigned)(need > nsm ? need : nranges < nsm ? nranges : nsm);
}

// Launch with programmatic stream serialization (see pdl_trigger / pdl_wait).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*k)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                       Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace hm
