// Shared pieces of the reduction kernels: how nodes are dealt to warps, and the
// deterministic sum of the warps' and blocks' parts.
//
// A warp takes a strip of rows of one group of 32 columns, so that the
// x weight of a lane is applied once per strip and the lanes that own a wall or
// centre-line column keep their sums to themselves.  FP64 instructions cost 16
// issue cycles a warp on this GPU's FP64 pipe, so the warp sums fold the slots
// into the lanes (6 additions for 4 slots instead of 20).  The last block to
// finish adds the block parts in a fixed order: one launch per reduction.
#pragma once

#include "islbm_internal.h"
#include "islbm_store.cuh"

namespace islbm {

constexpr int kRedThreads = 512, kRedWarps = kRedThreads / 32;

// Strips of the reductions: `rows` rows of `nx` columns over the warps of a grid.
struct RowStrips {
  int ncg, per, rows, tasks;   // column groups, rows per strip, rows, (group, strip) items
  int blocks;
};

inline RowStrips row_strips(int nx, long long rows, int max_blocks) {
  RowStrips t;
  t.ncg = (nx + 31) / 32;
  t.rows = (int)rows;
  const long long warps = (long long)max_blocks * kRedWarps;
  const long long strips = std::max<long long>(1, warps / t.ncg);
  t.per = (int)std::max<long long>(1, (rows + strips - 1) / strips);
  t.tasks = t.ncg * (int)((rows + t.per - 1) / t.per);
  t.blocks = std::min(max_blocks, (t.tasks + kRedWarps - 1) / kRedWarps);
  return t;
}

// FP64 value of an FP32 value; normal values are widened on the integer units.
__device__ __forceinline__ double to_d(double v) { return v; }
__device__ __forceinline__ double to_d(float v) {
  const unsigned b = __float_as_uint(v);
  if (((b >> 23) & 0xFFu) - 1u >= 254u) return (double)v;   // 0, subnormal, inf, NaN
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20))),
                          (int)(b << 29));
}

// Sums of four values over the warp: lane l returns the sum of v[l & 3].
__device__ __forceinline__ double warp_sum4(const double (&v)[4]) {
  const unsigned lane = threadIdx.x & 31u;
  const bool b0 = lane & 1u, b1 = lane & 2u;
  // lane bit 0 selects v[0], v[2] or v[1], v[3]; bit 1 the first or second of them
  double a = (b0 ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, b0 ? v[0] : v[1], 1);
  double b = (b0 ? v[3] : v[2]) + __shfl_xor_sync(0xffffffffu, b0 ? v[2] : v[3], 1);
  double r = (b1 ? b : a) + __shfl_xor_sync(0xffffffffu, b1 ? a : b, 2);
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  return r;
}

// The block's part of every slot from its warps' parts, then (in the last block)
// the totals, to `out` (host memory that the device can write).  Slot `max_slot`
// is combined by max.  `words`: [0] the step kernels' error flag, which goes to
// out[RED_STRIDE], and [3] the count of finished blocks, zero between launches.
__device__ __forceinline__ void reduce_finish(const double (*sh)[RED_STRIDE], int max_slot,
                                              double* partial, double* out, int* words) {
  __shared__ int last;
  __shared__ double part[kRedThreads];
  __syncthreads();
  const int k = threadIdx.x & (RED_STRIDE - 1), grp = threadIdx.x / RED_STRIDE;
  if (grp == 0) {
    double v = sh[0][k];
    for (int w = 1; w < kRedWarps; ++w) v = (k == max_slot) ? fmax(v, sh[w][k]) : v + sh[w][k];
    partial[(size_t)blockIdx.x * RED_STRIDE + k] = v;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&words[3], 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  double v = 0.0;
  for (int b = grp; b < (int)gridDim.x; b += kRedThreads / RED_STRIDE) {
    const double x = __ldcg(partial + (size_t)b * RED_STRIDE + k);
    v = (k == max_slot) ? fmax(v, x) : v + x;
  }
  part[threadIdx.x] = v;
  __syncthreads();
  if (grp == 0) {
    for (int g = 1; g < kRedThreads / RED_STRIDE; ++g) {
      const double x = part[g * RED_STRIDE + k];
      v = (k == max_slot) ? fmax(v, x) : v + x;
    }
    out[k] = v;
  }
  if (threadIdx.x == 0) {
    out[RED_STRIDE] = (double)words[0];
    words[3] = 0;
  }
}

// Constants of the velocities, formed on the host: an operation, or a comparison,
// on the FP64 pipe costs the field output of 1025^2 nodes 2 us.
struct Force {
  double gbeta, c;   // g beta, -g beta / 2
  int shift;         // whether T_s != 0
};
inline Force make_force(const Solver& s) {
  return Force{s.ph.gbeta, -0.5 * s.ph.gbeta, s.ph.Ts != 0.0 ? 1 : 0};
}

// Adds v to *p (time averages) or writes it.
template <bool ACC>
__device__ __forceinline__ void put_field(double* p, double v) {
  *p = ACC ? *p + v : v;
}

}  // namespace islbm
