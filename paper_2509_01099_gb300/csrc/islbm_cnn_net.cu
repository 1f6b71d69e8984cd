// The warm-start network's passes as fused layers (NHWC, FP32 activations and
// gradients, BF16 products with FP32 accumulation on the tensor cores).
//
// A chain of im2col, GEMM and elementwise kernels writes and reads nine BF16
// copies of every activation (302 MB for the 256^2 layer at 16 samples) and
// nine FP32 ones on the way back; a prediction spends its time on 27 launches.
// Here a convolution gathers its nine taps from a staged window of its input
// (ldmatrix takes one address a pixel, so the im2col matrix is never formed;
// the nearest-neighbour upsampling is a shift of the pixel coordinates), and
// bias, tanh, its derivative and the upsampling's adjoint are part of the
// products' kernels.  Measured on GB300, chain and fused: a training step of 16
// samples 7.03 and 0.70 ms, a prediction 445 and 50 us.
//
// The products are narrow (3 to 64 channels), so they stay on mma.sync with
// operands in the staged window: their roofline is the activations' bytes
// (about 0.5 GB a training step of 16).  What bounds the kernels is the staging
// (FP32 loads, conversion, shared-memory stores) and its latency.  Device time
// at 16 samples (cold caches): 256^2 layers forward 52 and 47 us, data gradient
// 46 and 60 us, weight gradient 58 and 94 us.
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <type_traits>

#include "islbm_internal.h"

namespace {

using bf16 = __nv_bfloat16;

constexpr int kMaxCh = 64;       // channels of a layer (wider networks: the GEMM chain)
constexpr int kMaxStages = 8;
constexpr int kTW = 16;          // tile columns: one m16 (or k16) row of pixels
constexpr int kFeat = 16;        // input features
constexpr int kMaxHidden = 512;
constexpr int kMaxSize = 256;      // pixels of an image row (its window is staged whole)

__device__ __forceinline__ unsigned sptr(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void ldsm4(unsigned (&r)[4], unsigned a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void ldsm4t(unsigned (&r)[4], unsigned a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void ldsm2(unsigned (&r)[2], unsigned a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void ldsm2t(unsigned (&r)[2], unsigned a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void mma16816(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                         unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ unsigned pack2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const unsigned*>(&v);
}
__device__ __forceinline__ float round_bf16(float v) {
  return __bfloat162float(__float2bfloat16(v));
}

// One convolution layer.  Forward: x [B, H >> up, W >> up, cin] -> y [B, H, W,
// cout] = act(conv(up(x)) + bias).  Backward: d [B, H, W, cout], x as forward.
struct Conv {
  const float* x;
  const bf16* w;        // [9 cin][cout], rows [dy][dx][c]
  const float* bias;
  const float* d;
  float* out;           // forward: y; data gradient: [B, H >> up, W >> up, cin]
  int B, H, W, cin, cout, up, act;
  int kchunk;           // forward: products summed together (see gemm_kchunk)
  int vx, vw, vd;       // 16-byte loads allowed for x, w and d (alignment, channels)
};

__host__ __device__ constexpr int up16(int c) { return (c + 15) / 16 * 16; }
// staged pixels carry 16 bytes of padding: ldmatrix rows of 8 pixels then fall
// into different banks for every channel count in use (pitches 48 to 144 bytes)
__host__ __device__ constexpr int pitch_of(int c) { return up16(c) + 8; }

// A load of an image.  The read-only path (__ldg) is for data that nothing
// writes while the kernel runs, and its loads are not ordered by grid_wait: not
// for an image that the launch before may still be writing when this kernel
// starts (LIVE), which takes ordinary loads.
template <bool LIVE, typename V>
__device__ __forceinline__ V load_image(const V* s) {
  if constexpr (LIVE) {
    return *s;
  } else {
    return __ldg(s);
  }
}

// Stages the window [wy0, wy0 + rows) x [wx0, wx0 + cols) of an NHWC FP32
// image of C channels as BF16 [pixel][pitch_of(C)]; zeros outside the image
// and in the padding channels.  LIVE: see load_image.
template <bool LIVE>
__device__ __forceinline__ void stage_window(bf16* dst, const float* img, int H, int W,
                                             int C, int wy0, int wx0, int rows, int cols, int vec,
                                             int tid, int threads) {
  // a thread keeps its four channels and walks the pixels, four loads in flight
  const int q = up16(C) / 4, pitch = pitch_of(C), step = threads / q, n = rows * cols;
  const int c = tid % q * 4, dr = step / cols, dk = step - dr * cols;
  int p = tid / q, r = p / cols, k = p - r * cols;
  if (p >= step) return;
  while (p < n) {
    float4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int y = wy0 + r, x = wx0 + k;
      v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (p + i * step < n && y >= 0 && y < H && x >= 0 && x < W) {
        const float* s = img + (y * W + x) * C + c;
        if (vec) {
          if (c < C) v[i] = load_image<LIVE>(reinterpret_cast<const float4*>(s));
        } else {
          if (c < C) v[i].x = load_image<LIVE>(s);
          if (c + 1 < C) v[i].y = load_image<LIVE>(s + 1);
          if (c + 2 < C) v[i].z = load_image<LIVE>(s + 2);
          if (c + 3 < C) v[i].w = load_image<LIVE>(s + 3);
        }
      }
      r += dr;
      k += dk;
      if (k >= cols) {
        k -= cols;
        ++r;
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (p + i * step < n)
        *reinterpret_cast<uint2*>(dst + (p + i * step) * pitch + c) =
            make_uint2(pack2(v[i].x, v[i].y), pack2(v[i].z, v[i].w));
    p += 4 * step;
  }
}

struct Tiles {
  int tx, ty, n;
  __host__ __device__ Tiles(int B, int H, int W, int rows)
      : tx((W + kTW - 1) / kTW), ty((H + rows - 1) / rows), n(tx * ty * B) {}
  __device__ __forceinline__ void at(int t, int rows, int& b, int& y0, int& x0) const {
    const int r = t / tx;
    x0 = (t - r * tx) * kTW;
    b = r / ty;
    y0 = (r - b * ty) * rows;
  }
};

// Forward layer.  4 warps; a warp's m16 tile is one row of 16 pixels, it owns
// MT rows; NT n8 tiles of output channels from 8 NT blockIdx.y.  Persistent
// over pixel tiles, the weights stay staged.
template <int NT, int MT>
__global__ void __launch_bounds__(128) k_conv_fwd(Conv p) {
  constexpr int TR = 4 * MT, NB = NT * 8, WP = NB + 8;
  extern __shared__ __align__(128) unsigned char smem[];
  const int CP = up16(p.cin), XP = pitch_of(p.cin);
  bf16* sw = reinterpret_cast<bf16*>(smem);
  bf16* sx = sw + 9 * CP * WP;
  const int n0 = blockIdx.y * NB;
  if (p.vw) {
    for (int e = threadIdx.x; e < 9 * CP * NT; e += 128) {
      const int r = e / NT, j = e - r * NT;
      const int tap = r / CP, c = r - tap * CP;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (c < p.cin && n0 + 8 * j < p.cout)
        v = __ldg(reinterpret_cast<const uint4*>(p.w + (size_t)(tap * p.cin + c) * p.cout + n0 + 8 * j));
      *reinterpret_cast<uint4*>(sw + r * WP + 8 * j) = v;
    }
  } else {
    for (int e = threadIdx.x; e < 9 * CP * NB; e += 128) {
      const int r = e / NB, j = e - r * NB;
      const int tap = r / CP, c = r - tap * CP;
      sw[r * WP + j] = (c < p.cin && n0 + j < p.cout) ? p.w[(size_t)(tap * p.cin + c) * p.cout + n0 + j]
                                                     : __float2bfloat16(0.f);
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Hx = p.H >> p.up, Wx = p.W >> p.up;
  const int rows = p.up ? TR / 2 + 2 : TR + 2, cols = p.up ? kTW / 2 + 2 : kTW + 2;
  const Tiles tl(p.B, p.H, p.W, TR);
  // ldmatrix: this lane's pixel (A) / channel row (B) and 8-wide column
  const int arow = lane & 15, acol = (lane >> 4) * 8;
  // the weights of the next layer may be staged while this one runs
  islbm::grid_launch_next();
  islbm::grid_wait();
  const unsigned bbase = sptr(sw) + 2u * (unsigned)((lane & 15) * WP + (NT > 1 ? (lane >> 4) * 8 : 0));
  for (int t = blockIdx.x; t < tl.n; t += gridDim.x) {
    int b, y0, x0;
    tl.at(t, TR, b, y0, x0);
    const int wy0 = (y0 - 1) >> p.up, wx0 = (x0 - 1) >> p.up;
    __syncthreads();   // the window of the tile before is read
    stage_window<true>(sx, p.x + (size_t)b * Hx * Wx * p.cin, Hx, Wx, p.cin, wy0, wx0, rows, cols,
                       p.vx, threadIdx.x, 128);
    __syncthreads();
    float acc[MT][NT][4], tot[MT][NT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[m][j][r] = tot[m][j][r] = 0.f;
    auto fold = [&]() {
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            tot[m][j][r] += acc[m][j][r];
            acc[m][j][r] = 0.f;
          }
    };
    int left = p.kchunk;
#pragma unroll 1
    for (int tap = 0; tap < 9; ++tap) {
      const int dy = tap / 3 - 1, dx = tap - (dy + 1) * 3 - 1;
      const int wx = ((x0 + arow + dx) >> p.up) - wx0;
      unsigned aaddr[MT];
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const int wy = ((y0 + warp * MT + m + dy) >> p.up) - wy0;
        aaddr[m] = sptr(sx) + 2u * (unsigned)((wy * cols + wx) * XP + acol);
      }
#pragma unroll 1
      for (int k = 0; k < CP; k += 16) {
        if (left == 0) {
          fold();
          left = p.kchunk;
        }
        left -= 16;
        unsigned af[MT][4];
#pragma unroll
        for (int m = 0; m < MT; ++m) ldsm4(af[m], aaddr[m] + 2u * (unsigned)k);
        const unsigned bk = bbase + 2u * (unsigned)((tap * CP + k) * WP);
        if constexpr (NT == 1) {
          unsigned bq[2];
          ldsm2t(bq, bk);
#pragma unroll
          for (int m = 0; m < MT; ++m) mma16816(acc[m][0], af[m], bq[0], bq[1]);
        } else {
#pragma unroll
          for (int j = 0; j < NT; j += 2) {
            unsigned bq[4];
            ldsm4t(bq, bk + 16u * (unsigned)j);
#pragma unroll
            for (int m = 0; m < MT; ++m) {
              mma16816(acc[m][j], af[m], bq[0], bq[1]);
              mma16816(acc[m][j + 1], af[m], bq[2], bq[3]);
            }
          }
        }
      }
    }
    fold();
    const int grp = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      const int y = y0 + warp * MT + m;
      if (y >= p.H) break;
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const int n = n0 + 8 * j + 2 * tig;
        if (n >= p.cout) continue;
        const bool two = n + 1 < p.cout;
        const float b0 = p.bias[n], b1 = two ? p.bias[n + 1] : 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int x = x0 + grp + 8 * h;
          if (x >= p.W) continue;
          float u = tot[m][j][2 * h] + b0, v = tot[m][j][2 * h + 1] + b1;
          if (p.act) {
            u = tanhf(u);
            v = tanhf(v);
          }
          float* o = p.out + (((size_t)b * p.H + y) * p.W + x) * p.cout + n;
          if (p.cout % 2 == 0) {
            *reinterpret_cast<float2*>(o) = make_float2(u, v);
          } else {
            o[0] = u;
            if (two) o[1] = v;
          }
        }
      }
    }
  }
}

// Data gradient of a layer, through the upsampling's adjoint and the tanh of
// the layer's input: out = up^T(conv^T(d)) (1 - x^2).  Row r of a warp's m16
// tile is pixel 2 r (r < 8) or 2 (r - 8) + 1 of two image rows, so the four
// pixels that the adjoint adds are in one thread's accumulators.
template <int NT>
__global__ void __launch_bounds__(128) k_conv_dgrad(Conv p) {
  constexpr int TR = 8, NB = NT * 8;
  extern __shared__ __align__(128) unsigned char smem[];
  const int KP = up16(p.cout), DP = pitch_of(p.cout);
  bf16* sw = reinterpret_cast<bf16*>(smem);   // [tap][input channel][DP]
  bf16* sd = sw + 9 * NB * DP;
  const int n0 = blockIdx.y * NB;
  if (p.vw) {
    const int q = KP / 8;
    for (int e = threadIdx.x; e < 9 * NB * q; e += 128) {
      const int r = e / q, k = (e - r * q) * 8;
      const int tap = r / NB, c = n0 + r - tap * NB;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (c < p.cin && k < p.cout)
        v = __ldg(reinterpret_cast<const uint4*>(p.w + (size_t)(tap * p.cin + c) * p.cout + k));
      *reinterpret_cast<uint4*>(sw + r * DP + k) = v;
    }
  } else {
    for (int e = threadIdx.x; e < 9 * NB * KP; e += 128) {
      const int r = e / KP, k = e - r * KP;
      const int tap = r / NB, c = n0 + r - tap * NB;
      sw[r * DP + k] = (c < p.cin && k < p.cout) ? p.w[(size_t)(tap * p.cin + c) * p.cout + k]
                                                 : __float2bfloat16(0.f);
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cols = kTW + 2;
  const Tiles tl(p.B, p.H, p.W, TR);
  const int r16 = lane & 15;
  const int apix = r16 < 8 ? 2 * r16 : 2 * (r16 - 8) + 1, acol = (lane >> 4) * 8;
  const unsigned bbase =
      sptr(sw) + 2u * (unsigned)(((lane & 7) + (NT > 1 ? (lane >> 4) * 8 : 0)) * DP +
                                 ((lane >> 3) & 1) * 8);
  const int grp = lane >> 2, tig = lane & 3;
  const int Hx = p.H >> p.up, Wx = p.W >> p.up;
  for (int t = blockIdx.x; t < tl.n; t += gridDim.x) {
    int b, y0, x0;
    tl.at(t, TR, b, y0, x0);
    __syncthreads();
    stage_window<false>(sd, p.d + (size_t)b * p.H * p.W * p.cout, p.H, p.W, p.cout, y0 - 1, x0 - 1,
                        TR + 2, cols, p.vd, threadIdx.x, 128);
    __syncthreads();
    float sum[2][NT][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int r = 0; r < 4; ++r) sum[m][j][r] = 0.f;
#pragma unroll 1
    for (int tap = 0; tap < 9; ++tap) {
      const int dy = tap / 3 - 1, dx = tap - (dy + 1) * 3 - 1;
      float acc[2][NT][4];
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int r = 0; r < 4; ++r) acc[m][j][r] = 0.f;
      unsigned aaddr[2];
#pragma unroll
      for (int m = 0; m < 2; ++m)
        aaddr[m] = sptr(sd) +
                   2u * (unsigned)(((2 * warp + m - dy + 1) * cols + apix - dx + 1) * DP + acol);
#pragma unroll 1
      for (int k = 0; k < KP; k += 16) {
        unsigned af[2][4];
#pragma unroll
        for (int m = 0; m < 2; ++m) ldsm4(af[m], aaddr[m] + 2u * (unsigned)k);
        const unsigned bk = bbase + 2u * (unsigned)(tap * NB * DP + k);
        if constexpr (NT == 1) {
          unsigned bq[2];
          ldsm2(bq, bk);
#pragma unroll
          for (int m = 0; m < 2; ++m) mma16816(acc[m][0], af[m], bq[0], bq[1]);
        } else {
#pragma unroll
          for (int j = 0; j < NT; j += 2) {
            unsigned bq[4];
            ldsm4(bq, bk + 2u * (unsigned)(8 * j * DP));
#pragma unroll
            for (int m = 0; m < 2; ++m) {
              mma16816(acc[m][j], af[m], bq[0], bq[1]);
              mma16816(acc[m][j + 1], af[m], bq[2], bq[3]);
            }
          }
        }
      }
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int r = 0; r < 4; ++r) sum[m][j][r] += acc[m][j][r];
    }
    auto put = [&](int y, int x, int c, float u, float v) {
      const size_t at = (((size_t)b * Hx + y) * Wx + x) * p.cin + c;
      if (p.cin % 2 == 0) {
        const float2 a = *reinterpret_cast<const float2*>(p.x + at);
        *reinterpret_cast<float2*>(p.out + at) =
            make_float2(u * (1.f - a.x * a.x), v * (1.f - a.y * a.y));
      } else {
        p.out[at] = u * (1.f - p.x[at] * p.x[at]);
        if (c + 1 < p.cin) p.out[at + 1] = v * (1.f - p.x[at + 1] * p.x[at + 1]);
      }
    };
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const int c = n0 + 8 * j + 2 * tig;
      if (c >= p.cin) continue;
      if (p.up) {
        const int y = y0 / 2 + warp, x = x0 / 2 + grp;
        if (y < Hx && x < Wx)
          put(y, x, c, sum[0][j][0] + sum[0][j][2] + sum[1][j][0] + sum[1][j][2],
              sum[0][j][1] + sum[0][j][3] + sum[1][j][1] + sum[1][j][3]);
      } else {
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int y = y0 + 2 * warp + m, x = x0 + 2 * grp + h;
            if (y < p.H && x < p.W) put(y, x, c, sum[m][j][2 * h], sum[m][j][2 * h + 1]);
          }
      }
    }
  }
}

// Weight gradients of a layer: dW[tap][c][n] = sum over pixels of
// up(x)(pixel + tap, c) d(pixel, n).  A block sums the pixels [k0, k0 + kchunk)
// of the image-linear order, in phases of `pr` image rows (about 256 pixels);
// one compute warp per row of three taps and 16 input channels holds its
// products with 8 NT output channels in registers, and the other warps stage
// the next phase meanwhile.  Blocks write their sums to
// part[block][9 cin][cout]; k_grad_sum adds them in order.
struct Wgrad {
  Conv c;
  float* part;
  int pr, phases, kp, kchunk, cw;   // rows and (padded) pixels of a phase, phases an image, compute warps
};

template <int NT>
__global__ void __launch_bounds__(512) k_conv_wgrad(Wgrad g) {
  const Conv& p = g.c;
  constexpr int NB = NT * 8, DPITCH = NB + 8;
  extern __shared__ __align__(128) unsigned char smem[];
  const int XP = pitch_of(p.cin), n0 = blockIdx.y * NB;
  const int Hx = p.H >> p.up, Wx = p.W >> p.up;
  const int rows = p.up ? g.pr / 2 + 2 : g.pr + 2, cols = Wx + 2;
  const int xsize = rows * cols * XP, dsize = g.kp * DPITCH;
  bf16* sx = reinterpret_cast<bf16*>(smem);
  bf16* sd = sx + 2 * xsize;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total = p.B * g.phases * g.kp;
  const int k0 = blockIdx.x * g.kchunk, k1 = min(total, k0 + g.kchunk);
  const int f0 = k0 / g.kp, f1 = (k1 + g.kp - 1) / g.kp;
  const int nn = min(NB, p.cout - n0);
  auto stage = [&](int f, int buf, int tid, int threads) {
    const int b = f / g.phases, y0 = (f - b * g.phases) * g.pr;
    stage_window<false>(sx + buf * xsize, p.x + (size_t)b * Hx * Wx * p.cin, Hx, Wx, p.cin,
                        (y0 - 1) >> p.up, -1, rows, cols, p.vx, tid, threads);
    const float* img = p.d + ((size_t)b * p.H + y0) * p.W * p.cout + n0;
    const int pixels = min(g.pr, p.H - y0) * p.W;
    bf16* dst = sd + buf * dsize;
    if (p.vd) {   // channels of a block are a multiple of 4
      constexpr int Q = NB / 4;
      const int n = tid % Q * 4, step = threads / Q;
      if (tid / Q < step)
        for (int q = tid / Q; q < g.kp; q += 4 * step) {
          float4 v[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            v[i] = q + i * step < pixels && n < nn
                       ? __ldg(reinterpret_cast<const float4*>(img + (q + i * step) * p.cout + n))
                       : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (q + i * step < g.kp)
              *reinterpret_cast<uint2*>(dst + (q + i * step) * DPITCH + n) =
                  make_uint2(pack2(v[i].x, v[i].y), pack2(v[i].z, v[i].w));
        }
    } else {
      const int n = tid % NB, step = threads / NB;
      if (tid / NB < step)
        for (int q = tid / NB; q < g.kp; q += 4 * step) {
          float v[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            v[i] = q + i * step < pixels && n < nn ? __ldg(img + (q + i * step) * p.cout + n) : 0.f;
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (q + i * step < g.kp) dst[(q + i * step) * DPITCH + n] = __float2bfloat16(v[i]);
        }
    }
  };
  float acc[3][NT][4];
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[m][j][r] = 0.f;
  const int dy = warp % 3 - 1, c0 = warp / 3 * 16;
  const int ak = (lane & 7) + (lane >> 4) * 8, am = ((lane >> 3) & 1) * 8;
  const int bk = lane & 15, bn = (lane >> 4) * 8;
  stage(f0, 0, threadIdx.x, blockDim.x);
  __syncthreads();
  for (int f = f0; f < f1; ++f) {
    const int buf = (f - f0) & 1;
    if (warp >= g.cw) {
      if (f + 1 < f1) stage(f + 1, buf ^ 1, threadIdx.x - 32 * g.cw, blockDim.x - 32 * g.cw);
    } else {
      const int b = f / g.phases, y0 = (f - b * g.phases) * g.pr;
      const int wy0 = (y0 - 1) >> p.up;
      const int q0 = max(0, k0 - f * g.kp), q1 = min(g.kp, k1 - f * g.kp);
      const unsigned xb = sptr(sx + buf * xsize) + 2u * (unsigned)(c0 + am);
      const unsigned db = sptr(sd + buf * dsize) + 2u * (unsigned)(bk * DPITCH + (NT > 1 ? bn : 0));
      int ry = (q0 + ak) / p.W, cx = (q0 + ak) - ry * p.W;
#pragma unroll 2
      for (int q = q0; q < q1; q += 16) {
        const int wy = ((y0 + min(ry, g.pr - 1) + dy) >> p.up) - wy0;
        unsigned af[3][4];
#pragma unroll
        for (int m = 0; m < 3; ++m)
          ldsm4t(af[m], xb + 2u * (unsigned)((wy * cols + ((cx + m - 1) >> p.up) + 1) * XP));
        const unsigned ba = db + 2u * (unsigned)(q * DPITCH);
#pragma unroll
        for (int j = 0; j + 1 < NT; j += 2) {
          unsigned bq[4];
          ldsm4t(bq, ba + 16u * (unsigned)j);
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            mma16816(acc[m][j], af[m], bq[0], bq[1]);
            mma16816(acc[m][j + 1], af[m], bq[2], bq[3]);
          }
        }
        if constexpr (NT % 2 == 1) {
          unsigned bq[2];
          ldsm2t(bq, sptr(sd + buf * dsize) + 2u * (unsigned)((q + bk) * DPITCH + 8 * (NT - 1)));
#pragma unroll
          for (int m = 0; m < 3; ++m) mma16816(acc[m][NT - 1], af[m], bq[0], bq[1]);
        }
        for (cx += 16; cx >= p.W; cx -= p.W) ++ry;
      }
    }
    __syncthreads();
  }
  if (warp >= g.cw) return;
  float* out = g.part + (size_t)blockIdx.x * 9 * p.cin * p.cout;
  const int grp = lane >> 2, tig = lane & 3;
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int c = c0 + grp + (r >= 2 ? 8 : 0), n = n0 + 8 * j + 2 * tig + (r & 1);
        if (c < p.cin && n < p.cout)
          out[((size_t)((dy + 1) * 3 + m) * p.cin + c) * p.cout + n] = acc[m][j][r];
      }
}

// Bias gradients of all layers in one launch: column sums of d [M][N], chunks
// of 2048 rows, eight interleaved row lanes of a chunk added in order (the sums
// of islbm_cnn_colsum, bit for bit).  A lane's additions are a serial chain, so
// its loads run 16 ahead of them.
constexpr int kSumRows = 2048;
struct SumSeg {
  const float* d;
  float* part;
  int M, N, first, per;   // first block, chunks of a block
};
struct SumSegs {
  SumSeg s[kMaxStages];
  int n;
};
__global__ void __launch_bounds__(512) k_bias_sum(SumSegs g) {
  int k = 0;
  while (k + 1 < g.n && (int)blockIdx.x >= g.s[k + 1].first) ++k;
  const SumSeg s = g.s[k];
  const int t = threadIdx.x, n = t % s.N, r = t / s.N % 8, sub = t / (8 * s.N);
  const long long chunk = (long long)((int)blockIdx.x - s.first) * s.per + sub;
  const long long m0 = chunk * kSumRows, m1 = m0 + kSumRows < s.M ? m0 + kSumRows : s.M;
  const bool on = sub < s.per && m0 < s.M;
  float sum = 0.f;
  if (on) {
    long long m = m0 + r;
    for (; m + 15 * 8 < m1; m += 16 * 8) {
      float v[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = __ldg(s.d + (m + 8 * i) * s.N + n);
#pragma unroll
      for (int i = 0; i < 16; ++i) sum += v[i];
    }
    for (; m < m1; m += 8) sum += __ldg(s.d + m * s.N + n);
  }
  __shared__ float sh[512];
  sh[t] = sum;
  __syncthreads();
  if (on && r == 0) {
    float v = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) v += sh[(sub * 8 + i) * s.N + n];
    s.part[chunk * s.N + n] = v;
  }
}

// Sums of the blocks' partial gradients in block order, all tensors in one launch.
struct GradSeg {
  const float* part;      // [blocks][values]
  float* out;
  int blocks, values, zeros, first;   // zeros: values behind them set to zero
};
struct GradSegs {
  GradSeg s[2 * kMaxStages + 4];
  int n;
};

__global__ void __launch_bounds__(64) k_grad_sum(GradSegs g) {
  int k = 0;
  while (k + 1 < g.n && (int)blockIdx.x >= g.s[k + 1].first) ++k;
  const GradSeg s = g.s[k];
  const int i = ((int)blockIdx.x - s.first) * 64 + threadIdx.x;
  if (i >= s.values + s.zeros) return;
  float v = 0.f;
  if (i < s.values) {
    int b = 0;
    for (; b + 64 <= s.blocks; b += 64) {
      float t[64];
#pragma unroll
      for (int j = 0; j < 64; ++j) t[j] = s.part[(size_t)(b + j) * s.values + i];
#pragma unroll
      for (int j = 0; j < 64; ++j) v += t[j];
    }
#pragma unroll 8
    for (; b < s.blocks; ++b) v += s.part[(size_t)b * s.values + i];
  }
  s.out[i] = v;
}

// ---- fully connected layers ----

// Both layers in one launch: a block keeps 64 columns of the second layer's
// weights and takes tiles of 16 samples (one m16 tile) one after the other: it
// computes the hidden layer of the tile, then its columns of the second one, a
// warp 16 of them.  The features come with the launch as kernel parameters (no
// host copy, no synchronisation): 32 samples, or up to 480 of a larger batch.
// Beyond kZCopy samples one copy into device memory precedes a single launch.
// (With a launch for every 32 samples, each staging the weights again, the
// forward pass of a 256 -> 64 layer and one convolution of 2^2 pixels took 264 us
// for 512 samples and 29.7 ms for 65,536; now 64 us and 0.42 ms, 140 us and 0.47
// ms layer by layer.)
constexpr int kFcB = 16;         // samples of a tile
constexpr int kZSmall = 32, kZLarge = 480;   // samples of a launch (2 and 30 KB of parameters)
constexpr int kZCopy = 4 * kZLarge;
template <int N>
struct ZArg {
  float z[N][kFeat];
  __device__ __forceinline__ float at(int b, int i) const { return z[b][i]; }
};
struct ZDevice {
  const float* z;
  __device__ __forceinline__ float at(int b, int i) const { return z[(size_t)b * kFeat + i]; }
};
struct Fc {
  const bf16 *w1, *w2;
  const float *b1, *b2;
  float *zk, *h1, *x0;           // zk may be null
  int B, hidden, n2, v1, v2;     // v1, v2: 16-byte loads of w1 and w2
  int kchunk;                    // hidden units summed together (see gemm_kchunk)
};

// rows x cols values at src (row pitch ld), BF16, into dst (row pitch dp); zeros
// beyond (rmax, cmax).  cols is a multiple of 8.
__device__ __forceinline__ void stage_matrix(bf16* dst, int dp, const bf16* __restrict__ src, int ld,
                                             int rows, int cols, int rmax, int cmax, int vec) {
  const int q = cols / 8;
#pragma unroll 8
  for (int e = threadIdx.x; e < rows * q; e += blockDim.x) {
    const int r = e / q, c = (e - r * q) * 8;
    if (vec) {
      uint4 v = make_uint4(0, 0, 0, 0);
      if (r < rmax && c < cmax) v = __ldg(reinterpret_cast<const uint4*>(src + (size_t)r * ld + c));
      *reinterpret_cast<uint4*>(dst + r * dp + c) = v;
    } else {
      for (int i = 0; i < 8; ++i)
        dst[r * dp + c + i] =
            r < rmax && c + i < cmax ? src[(size_t)r * ld + c + i] : __float2bfloat16(0.f);
    }
  }
}

__global__ void __launch_bounds__(256) k_round_features(float* z, size_t n) {
  const size_t e = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (e < n) z[e] = round_bf16(z[e]);
}

// Samples [b0, b1) of the batch; za holds theirs, ZDevice those of the whole batch.
template <typename Z>
__global__ void __launch_bounds__(128) k_fc_fwd(Fc p, const __grid_constant__ Z za, int b0, int b1) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int HP = up16(p.hidden), P = HP + 8;
  bf16* sw1 = reinterpret_cast<bf16*>(smem);     // [16][P]
  bf16* sh = sw1 + kFeat * P;                    // [16][P]
  bf16* sw2 = sh + kFcB * P;                     // [HP][72]
  bf16* sz = sw2 + HP * 72;                      // [16][24]
  const int n0 = blockIdx.x * 64, zb = std::is_same<Z, ZDevice>::value ? 0 : b0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = lane >> 2, tig = lane & 3;
  islbm::grid_launch_next();
  stage_matrix(sw1, P, p.w1, p.hidden, kFeat, HP, kFeat, p.hidden, p.v1);
  stage_matrix(sw2, 72, p.w2 + n0, p.n2, HP, 64, p.hidden, p.n2 - n0, p.v2);
  for (int t = blockIdx.y; t < (b1 - b0 + kFcB - 1) / kFcB; t += gridDim.y) {
    const int bb = b0 + t * kFcB, nb = min(kFcB, b1 - bb);
    for (int e = threadIdx.x; e < kFcB * kFeat; e += 128) {
      const int b = e / kFeat, i = e % kFeat;
      const bf16 v = __float2bfloat16(b < nb ? za.at(bb - zb + b, i) : 0.f);
      sz[b * 24 + i] = v;
      if (blockIdx.x == 0 && p.zk && b < nb)
        p.zk[(size_t)(bb + b) * kFeat + i] = __bfloat162float(v);
    }
    __syncthreads();
    unsigned az[4];
    ldsm4(az, sptr(sz) + 2u * (unsigned)((lane & 15) * 24 + (lane >> 4) * 8));
    for (int j = warp; j < HP / 8; j += 4) {
      unsigned bq[2];
      ldsm2t(bq, sptr(sw1) + 2u * (unsigned)((lane & 15) * P + 8 * j));
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      mma16816(acc, az, bq[0], bq[1]);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int b = grp + (r >= 2 ? 8 : 0), k = 8 * j + 2 * tig + (r & 1);
        float v = 0.f;
        if (k < p.hidden) {
          v = tanhf(acc[r] + p.b1[k]);
          if (blockIdx.x == 0 && b < nb) p.h1[(size_t)(bb + b) * p.hidden + k] = v;
        }
        sh[b * P + k] = __float2bfloat16(v);
      }
    }
    __syncthreads();
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}}, tot[2][4];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) tot[j][r] = 0.f;
    for (int k = 0, left = p.kchunk; k < HP; k += 16, left -= 16) {
      if (left == 0) {
        left = p.kchunk;
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            tot[j][r] += acc[j][r];
            acc[j][r] = 0.f;
          }
      }
      unsigned af[4], bq[4];
      ldsm4(af, sptr(sh) + 2u * (unsigned)((lane & 15) * P + k + (lane >> 4) * 8));
      ldsm4t(bq, sptr(sw2) + 2u * (unsigned)((k + (lane & 15)) * 72 + warp * 16 + (lane >> 4) * 8));
      mma16816(acc[0], af, bq[0], bq[1]);
      mma16816(acc[1], af, bq[2], bq[3]);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int b = grp + (r >= 2 ? 8 : 0), n = n0 + warp * 16 + 8 * j + 2 * tig + (r & 1);
        if (b < nb && n < p.n2)
          p.x0[(size_t)(bb + b) * p.n2 + n] = tanhf(tot[j][r] + acc[j][r] + p.b2[n]);
      }
    // (the next tile's features go to sz, read before the last barrier, and its
    // hidden layer to sh, behind the next one)
  }
}

// dh1 = (d2 W2^T) (1 - h1^2).  `share` of a block's 16 warps take the chunks of
// `kchunk` columns of one tile of 16 samples (grid x, which takes any batch) and 8
// hidden units (grid y), which are added in order; the block's 16 / share tiles
// are of the same samples.
__global__ void __launch_bounds__(512) k_fc_dh(const float* __restrict__ d2,
                                               const bf16* __restrict__ w2,
                                               const float* __restrict__ h1, float* __restrict__ dh1,
                                               int B, int hidden, int n2, int kchunk, int share) {
  __shared__ float part[16][kFcB * 8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = lane >> 2, tig = lane & 3;
  const int kb = blockIdx.y * (16 / share) * 8, bb = blockIdx.x * kFcB;
  const int k0 = kb + warp / share * 8, mine = warp % share;
  const int chunks = (n2 + kchunk - 1) / kchunk;
  const float* r0 = d2 + (size_t)min(bb + grp, B - 1) * n2;
  const float* r1 = d2 + (size_t)min(bb + grp + 8, B - 1) * n2;
  const bf16* wr = w2 + (size_t)min(k0 + grp, hidden - 1) * n2;
  float total[4] = {0.f, 0.f, 0.f, 0.f};   // of the values threadIdx.x + 512 i of the block's tiles
  for (int c0 = 0; c0 < chunks; c0 += share) {
    const int nc = min(share, chunks - c0);
    if (mine < nc && k0 < hidden) {
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      const int e = min(n2, (c0 + mine + 1) * kchunk);
#pragma unroll 4
      for (int n = (c0 + mine) * kchunk; n < e; n += 16) {
        const int c = n + 2 * tig;               // n2 is even: pairs are whole
        const bool in0 = c < e, in1 = c + 8 < e;
        auto pair = [&](const float* r, int at, bool in) {
          const float2 v = in ? *reinterpret_cast<const float2*>(r + at) : make_float2(0.f, 0.f);
          return pack2(v.x, v.y);
        };
        const unsigned a[4] = {pair(r0, c, in0), pair(r1, c, in0), pair(r0, c + 8, in1),
                               pair(r1, c + 8, in1)};
        mma16816(acc, a, in0 ? *reinterpret_cast<const unsigned*>(wr + c) : 0u,
                 in1 ? *reinterpret_cast<const unsigned*>(wr + c + 8) : 0u);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
        part[warp][(grp + (r >= 2 ? 8 : 0)) * 8 + 2 * tig + (r & 1)] = acc[r];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int v = threadIdx.x + 512 * i, tile = v / (kFcB * 8);
      if (tile < 16 / share && kb + tile * 8 < hidden)
        for (int c = 0; c < nc; ++c) total[i] += part[tile * share + c][v % (kFcB * 8)];
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int v = threadIdx.x + 512 * i, tile = v / (kFcB * 8);
    const int b = bb + v % (kFcB * 8) / 8, k = kb + tile * 8 + v % 8;
    if (tile < 16 / share && b < B && k < hidden) {
      const float h = h1[(size_t)b * hidden + k];
      dh1[(size_t)b * hidden + k] = total[i] * (1.f - h * h);
    }
  }
}

// Weight and bias gradients of both fully connected layers in one launch:
// dW[k][n] = sum_b bf16(a[b][k]) bf16(d[b][n]) and db[n] = sum_b d[b][n], summed
// as the chain sums them: the products in steps of 16 samples on the tensor
// cores and, where the chain splits K, in chunks of `kchunk` samples; the biases
// by eight interleaved lanes in chunks of kSumRows samples.  (One FP32 chain
// over the batch, as an earlier form summed both, has 1.2 times the RMS error at
// 16 samples and 3.8 times at 4,096.)  Chunks are blocks of their own; where
// there are several, dw and db are their partial sums, which k_grad_sum adds.
// A weight block takes 16 rows and 256 columns, a warp 32 of them, and reads
// its fragments from global memory; a bias block takes 32 columns.  Bound by the
// 4 MB that it writes and a launch's latency: 256 x 4096 weights of 16 samples 5.4
// us, as scalar products 7.7.
struct FcGrad {
  const float *a, *d;
  float *dw, *db;
  int K, N, gx, gy;              // column and row tiles
  int kchunk, wchunks, bchunks;
  __host__ __device__ int wblocks() const { return gx * gy * wchunks; }
  __host__ __device__ int bblocks() const { return (N + 31) / 32 * bchunks; }
};
__device__ __forceinline__ void fc_weight_block(const FcGrad& p, int t, int B) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = lane >> 2, tig = lane & 3;
  const int tile = t % (p.gx * p.gy), chunk = t / (p.gx * p.gy);
  const int n0 = tile % p.gx * 256 + warp * 32, k0 = tile / p.gx * 16;
  const int b1 = min((long long)B, (long long)(chunk + 1) * p.kchunk);
  float acc[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[j][r] = 0.f;
  // a pair of samples b, b + 1 of column c of x [B][C]
  auto pair = [&](const float* x, int C, int b, int c) {
    const float u = c < C && b < b1 ? __ldg(x + (size_t)b * C + c) : 0.f;
    const float v = c < C && b + 1 < b1 ? __ldg(x + (size_t)(b + 1) * C + c) : 0.f;
    return pack2(u, v);
  };
  for (int b0 = chunk * p.kchunk; b0 < b1; b0 += 16) {
    const int b = b0 + 2 * tig;
    const unsigned af[4] = {pair(p.a, p.K, b, k0 + grp), pair(p.a, p.K, b, k0 + grp + 8),
                            pair(p.a, p.K, b + 8, k0 + grp), pair(p.a, p.K, b + 8, k0 + grp + 8)};
    unsigned bf[4][2];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      bf[j][0] = pair(p.d, p.N, b, n0 + 8 * j + grp);
      bf[j][1] = pair(p.d, p.N, b + 8, n0 + 8 * j + grp);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) mma16816(acc[j], af, bf[j][0], bf[j][1]);
  }
  float* o = p.dw + (size_t)chunk * p.K * p.N;
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int k = k0 + grp + (r >= 2 ? 8 : 0), n = n0 + 8 * j + 2 * tig + (r & 1);
      if (k < p.K && n < p.N) o[(size_t)k * p.N + n] = acc[j][r];
    }
}
__device__ __forceinline__ void fc_bias_block(const FcGrad& p, int t, int B) {
  __shared__ float sh[8][33];
  const int lane = threadIdx.x & 31, row = threadIdx.x >> 5, tiles = (p.N + 31) / 32;
  const int chunk = t / tiles, n = t % tiles * 32 + lane;
  const long long b1 = min((long long)B, (long long)(chunk + 1) * kSumRows);
  float s = 0.f;
  if (n < p.N)
    for (long long b = (long long)chunk * kSumRows + row; b < b1; b += 8)
      s += __ldg(p.d + (size_t)b * p.N + n);
  sh[row][lane] = s;
  __syncthreads();
  if (row != 0 || n >= p.N) return;
  float v = 0.f;
#pragma unroll
  for (int r = 0; r < 8; ++r) v += sh[r][lane];
  p.db[(size_t)chunk * p.N + n] = v;
}
__global__ void __launch_bounds__(256) k_fc_wgrad(FcGrad l2, FcGrad l1, int B) {
  int t = blockIdx.x;
  if (t < l2.wblocks()) return fc_weight_block(l2, t, B);
  t -= l2.wblocks();
  if (t < l1.wblocks()) return fc_weight_block(l1, t, B);
  t -= l1.wblocks();
  const bool second = t < l2.bblocks();
  fc_bias_block(second ? l2 : l1, second ? t : t - l2.bblocks(), B);
}

// Adam over all tensors of the network in one launch (the arithmetic of
// islbm_cnn_adam); a block takes kAdamBlock values of one tensor.
constexpr int kMaxTensors = 32, kAdamBlock = 2048;
struct AdamTensor {
  float* w;
  bf16* wb;
  const float* g;
  float *m, *v;
  long long n;
  int first;
};
struct AdamSet {
  AdamTensor t[kMaxTensors];
  int n;
};
__global__ void __launch_bounds__(256)
    k_adam_all(const __grid_constant__ AdamSet a, float lr, float b1, float b2, float eps, float c1,
               float c2) {
  int k = 0;
  while (k + 1 < a.n && (int)blockIdx.x >= a.t[k + 1].first) ++k;
  const AdamTensor t = a.t[k];
  const long long e0 = (long long)((int)blockIdx.x - t.first) * kAdamBlock;
  const long long e1 = e0 + kAdamBlock < t.n ? e0 + kAdamBlock : t.n;
#pragma unroll 4
  for (long long e = e0 + threadIdx.x; e < e1; e += 256) {
    const float gg = t.g[e];
    const float mm = b1 * t.m[e] + (1.f - b1) * gg;
    const float vv = b2 * t.v[e] + (1.f - b2) * gg * gg;
    t.m[e] = mm;
    t.v[e] = vv;
    const float upd = lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    const float nw = t.w[e] - upd;
    t.w[e] = nw;
    if (t.wb) t.wb[e] = __float2bfloat16(nw);
  }
}

// ---- host side ----

int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    sms = 1;
  return sms;
}

// Shared memory is raised to the kernel's limit once (the sizes differ by call).
constexpr int kSmemLimit = 200 * 1024;
cudaError_t allow_smem(const void* k) {
  return islbm::launch_setup_once(
      k,
      [](const void* f, int*) {
        return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
      },
      nullptr);
}

// Products of a sum.  The layers round their activations and gradients to BF16
// between two products, so a sum in another order shows in the results (one
// BF16 rounding in some 10^4 flips).  These kernels keep the order of the GEMM
// chain (islbm_cnn_gemm_bf16): k ascending in steps of 16, in chunks that are
// added in order where that product splits K (mma.sync and tcgen05.mma add the
// 16 products of a step alike, bit for bit).
int gemm_kchunk(long long M, int N, int K, int sms) {
  const int bn = N <= 16 ? 16 : N <= 32 ? 32 : 64;
  const long long tiles = (N + bn - 1) / bn * ((M + 127) / 128);
  int split = 1;
  if (tiles < 2LL * sms && K >= 512)
    split = std::max(1, (int)std::min<long long>((2LL * sms + tiles - 1) / tiles, K / 256));
  return ((K + split - 1) / split + 63) / 64 * 64;
}

// The same for a product whose operands take the chain's tensor-core kernel
// (tc: leading dimensions in multiples of 8, K above 32) or its mma.sync one.
int chain_kchunk(long long M, int N, int K, bool tc, int sms) {
  if (tc && K > 32) return gemm_kchunk(M, N, K, sms);
  const long long tiles = (M + 63) / 64 * ((N + 63) / 64);
  long long split = 1;
  if (tiles < 2LL * sms && K >= 512)
    split = std::max(1LL, std::min((2LL * sms + tiles - 1) / tiles, (long long)K / 256));
  return (int)(((K + split - 1) / split + 31) / 32 * 32);
}

int round_nt(int n8) { return n8 <= 2 ? std::max(n8, 1) : n8 <= 4 ? 4 : n8 <= 6 ? 6 : 8; }

// CTAs of a persistent launch: as many as the shared memory lets an SM hold.
int persistent_grid(int tiles, size_t smem, int sms, int gy, int max_per_sm) {
  const int per = std::max(1, std::min<int>(max_per_sm, (int)(220 * 1024 / (smem + 1024))));
  return std::max(1, std::min(tiles, (per * sms + gy - 1) / gy));
}

// Output-channel tiles of a block: all of them, fewer where the pixel tiles
// alone would leave SMs idle (the staged window is then read several times).
int pick_nt(int channels, int tiles, int sms) {
  const int n8 = (channels + 7) / 8;
  int nt = round_nt(n8);
  while (nt > 2 && tiles * ((n8 + nt - 1) / nt) < sms) nt = nt == 8 ? 4 : nt == 6 ? 4 : 2;
  return nt;
}

template <int NT, int MT>
cudaError_t fwd_nt(const Conv& p, int sms, cudaStream_t st) {
  const void* f = reinterpret_cast<const void*>(k_conv_fwd<NT, MT>);
  const cudaError_t e = allow_smem(f);
  if (e != cudaSuccess) return e;
  constexpr int TR = 4 * MT;
  const int win = p.up ? (TR / 2 + 2) * (kTW / 2 + 2) : (TR + 2) * (kTW + 2);
  const size_t smem = 2 * ((size_t)9 * up16(p.cin) * (NT * 8 + 8) + (size_t)win * pitch_of(p.cin));
  const int gy = ((p.cout + 7) / 8 + NT - 1) / NT;
  const dim3 grid(persistent_grid(Tiles(p.B, p.H, p.W, TR).n, smem, sms, gy, 8), gy);
  // up to one tile a block, the launch and the staging of the weights are most
  // of a layer: the next one starts early (a prediction: 64 -> 46 us of device time)
  const bool serial = Tiles(p.B, p.H, p.W, TR).n <= 4 * sms;
  return islbm::launch_grid(serial, k_conv_fwd<NT, MT>, grid, 128, smem, st, p);
}

template <int NT>
cudaError_t fwd_mt(const Conv& p, int sms, cudaStream_t st) {
  // 8 x 16 pixel tiles; 4 x 16 while those fill less than two thirds of the SMs
  const int gy = ((p.cout + 7) / 8 + NT - 1) / NT;
  return Tiles(p.B, p.H, p.W, 8).n * gy * 3 < 2 * sms ? fwd_nt<NT, 1>(p, sms, st)
                                                      : fwd_nt<NT, 2>(p, sms, st);
}

cudaError_t conv_forward(const Conv& p, int sms, cudaStream_t st) {
  switch (pick_nt(p.cout, Tiles(p.B, p.H, p.W, 8).n, sms)) {
    case 1: return fwd_mt<1>(p, sms, st);
    case 2: return fwd_mt<2>(p, sms, st);
    case 4: return fwd_mt<4>(p, sms, st);
    case 6: return fwd_mt<6>(p, sms, st);
    default: return fwd_mt<8>(p, sms, st);
  }
}

template <int NT>
cudaError_t dgrad_nt(const Conv& p, int sms, cudaStream_t st) {
  const void* f = reinterpret_cast<const void*>(k_conv_dgrad<NT>);
  const cudaError_t e = allow_smem(f);
  if (e != cudaSuccess) return e;
  const size_t smem = 2 * (size_t)pitch_of(p.cout) * (9 * NT * 8 + 10 * (kTW + 2));
  const int gy = ((p.cin + 7) / 8 + NT - 1) / NT;
  const dim3 grid(persistent_grid(Tiles(p.B, p.H, p.W, 8).n, smem, sms, gy, 8), gy);
  k_conv_dgrad<NT><<<grid, 128, smem, st>>>(p);
  return cudaGetLastError();
}

cudaError_t conv_dgrad(const Conv& p, int sms, cudaStream_t st) {
  switch (pick_nt(p.cin, Tiles(p.B, p.H, p.W, 8).n, sms)) {
    case 1: return dgrad_nt<1>(p, sms, st);
    case 2: return dgrad_nt<2>(p, sms, st);
    case 4: return dgrad_nt<4>(p, sms, st);
    case 6: return dgrad_nt<6>(p, sms, st);
    default: return dgrad_nt<8>(p, sms, st);
  }
}

// Launch shape of a layer's weight gradient.
struct WgradPlan {
  int nt, gy, cw, warps, pr, phases, kp, kchunk, blocks, chunks;
  size_t smem, floats;   // floats: partial sums of all blocks
};
WgradPlan wgrad_plan(int B, int H, int cin, int cout, int up, int sms) {
  WgradPlan w;
  const int n8 = (cout + 7) / 8;
  w.gy = (n8 + 3) / 4;
  w.nt = (n8 + w.gy - 1) / w.gy;
  w.cw = 3 * (up16(cin) / 16);
  w.warps = 16;
  const size_t row = 2 * (size_t)pitch_of(cin) * ((H >> up) + 2);
  auto smem = [&]() {
    w.kp = up16(w.pr * H);
    const int rows = up ? w.pr / 2 + 2 : w.pr + 2;
    return 2 * (rows * row + 2 * (size_t)w.kp * (w.nt * 8 + 8));
  };
  // phases of about 512 pixels (neighbouring phases stage two rows twice), 256
  // where two of those do not fit
  for (int pixels = 512; pixels >= 256; pixels /= 2) {
    w.pr = std::min(H, std::max(1, pixels / H));
    if (up && w.pr % 2 && w.pr > 1) --w.pr;
    w.smem = smem();
    if (w.smem <= (size_t)kSmemLimit) break;
  }
  w.phases = (H + w.pr - 1) / w.pr;
  // the chunks of the GEMM chain's split
  const long long K = (long long)B * H * H;
  w.kchunk = chain_kchunk(up16(9 * cin), cout, (int)K, cout % 8 == 0, sms);
  w.blocks = (int)(((long long)B * w.phases * w.kp + w.kchunk - 1) / w.kchunk);
  w.chunks = (int)((K + kSumRows - 1) / kSumRows);
  w.floats = (size_t)w.blocks * 9 * cin * cout;
  return w;
}

template <int NT>
cudaError_t wgrad_nt(const Wgrad& g, const WgradPlan& w, cudaStream_t st) {
  const void* f = reinterpret_cast<const void*>(k_conv_wgrad<NT>);
  const cudaError_t e = allow_smem(f);
  if (e != cudaSuccess) return e;
  k_conv_wgrad<NT><<<dim3(w.blocks, w.gy), w.warps * 32, w.smem, st>>>(g);
  return cudaGetLastError();
}

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

// what the fused kernels take: up to 64 channels and 8 stages, an even second
// layer, 16-byte aligned tensors
bool net_ok(int stages, const int* ch, int base, int hidden, int batch, int sms) {
  if (stages < 1 || stages > kMaxStages || !ch || base < 1 || hidden < 1 || hidden > kMaxHidden ||
      batch < 1)
    return false;
  for (int s = 0; s <= stages; ++s)
    if (ch[s] < 1 || ch[s] > kMaxCh) return false;
  if ((long long)base * base * ch[0] % 2 != 0) return false;
  const long long size = (long long)base << (stages - 1);
  if (size > kMaxSize || batch * size * size > 1ll << 30) return false;
  int H = base;   // a weight gradient's phases have to fit shared memory
  for (int s = 0; s < stages; ++s) {
    const int up = s + 1 < stages;
    if (up) H *= 2;
    const WgradPlan w = wgrad_plan(batch, H, ch[s], ch[s + 1], up, sms);
    if (w.smem > (size_t)kSmemLimit) return false;
    // and its padded pixels a 32-bit index (images of 1 or 2 rows are padded most)
    if ((long long)batch * w.phases * w.kp + w.kchunk > INT_MAX) return false;
  }
  return true;
}

size_t round64(size_t n) { return (n + 63) / 64 * 64; }

// Scratch of a backward pass, in floats: the gradient image of every layer's
// input, dh1, partial sums.
struct BackPlan {
  size_t image[kMaxStages], total;
  WgradPlan w[kMaxStages];
  FcGrad l1, l2;           // chunks and tiles; the pointers are set by the launch
};
// The chunks of one fully connected layer's gradients, K inputs and N outputs.
FcGrad fc_plan(int K, int N, int batch, int sms) {
  FcGrad g{};
  g.K = K;
  g.N = N;
  g.gx = (N + 255) / 256;
  g.gy = (K + 15) / 16;
  g.kchunk = chain_kchunk(K, N, batch, K % 8 == 0 && N % 8 == 0, sms);
  g.wchunks = (batch + g.kchunk - 1) / g.kchunk;
  g.bchunks = (batch + kSumRows - 1) / kSumRows;
  return g;
}
// floats of its partial sums (none where there is one chunk)
size_t fc_floats(const FcGrad& g) {
  return (g.wchunks > 1 ? round64((size_t)g.wchunks * g.K * g.N) : 0) +
         (g.bchunks > 1 ? round64((size_t)g.bchunks * g.N) : 0);
}
BackPlan back_plan(int stages, const int* ch, int base, int hidden, int batch, int sms) {
  BackPlan b;
  b.l2 = fc_plan(hidden, base * base * ch[0], batch, sms);
  b.l1 = fc_plan(kFeat, hidden, batch, sms);
  b.total = round64((size_t)batch * hidden) + fc_floats(b.l2) + fc_floats(b.l1);
  int H = base;
  for (int s = 0; s < stages; ++s) {
    b.image[s] = round64((size_t)batch * H * H * ch[s]);
    const int up = s + 1 < stages;
    if (up) H *= 2;
    b.w[s] = wgrad_plan(batch, H, ch[s], ch[s + 1], up, sms);
    b.total += b.image[s] + round64(b.w[s].floats) + round64((size_t)b.w[s].chunks * ch[s + 1]);
  }
  return b;
}

Conv layer(int B, int H, int cin, int cout, int up, const float* x, const void* w) {
  Conv c{};
  c.x = x;
  c.w = static_cast<const bf16*>(w);
  c.B = B;
  c.H = c.W = H;
  c.cin = cin;
  c.cout = cout;
  c.up = up;
  c.vx = cin % 4 == 0 && aligned(x, 16);
  c.vw = cout % 8 == 0 && aligned(w, 16);
  c.kchunk = 1 << 30;
  return c;
}

template <typename Z>
cudaError_t fc_launch(const Fc& f, const Z& za, int b0, int b1, int sms, cudaStream_t st) {
  const int hp = up16(f.hidden), gx = (f.n2 + 63) / 64;
  const size_t smem = 2 * ((size_t)(kFeat + kFcB) * (hp + 8) + (size_t)hp * 72 + kFcB * 24);
  const cudaError_t e = allow_smem(reinterpret_cast<const void*>(k_fc_fwd<Z>));
  if (e != cudaSuccess) return e;
  // every tile its own block while that fills up to four blocks an SM
  const int gy = std::min((b1 - b0 + kFcB - 1) / kFcB, std::max(1, 4 * sms / gx));
  k_fc_fwd<<<dim3(gx, gy), 128, smem, st>>>(f, za, b0, b1);
  return cudaGetLastError();
}
template <int N>
cudaError_t fc_launches(const Fc& f, const float* z, int sms, cudaStream_t st) {
  for (int b0 = 0; b0 < f.B; b0 += N) {
    const int b1 = std::min(f.B, b0 + N);
    ZArg<N> za{};
    std::copy(z + (size_t)b0 * kFeat, z + (size_t)b1 * kFeat, &za.z[0][0]);
    const cudaError_t e = fc_launch(f, za, b0, b1, sms, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
cudaError_t fc_forward(const Fc& f, const float* z, int sms, cudaStream_t st) {
  if (f.B <= kZSmall) return fc_launches<kZSmall>(f, z, sms, st);
  // a copy from pageable memory cannot be captured into a graph
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (f.B > kZCopy && f.zk) {
    const cudaError_t e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess) return e;
  }
  if (f.B <= kZCopy || !f.zk || cap != cudaStreamCaptureStatusNone)
    return fc_launches<kZLarge>(f, z, sms, st);
  cudaError_t e =
      cudaMemcpyAsync(f.zk, z, (size_t)f.B * kFeat * sizeof(float), cudaMemcpyHostToDevice, st);
  // z may be freed once the call returns, and a copy from pageable memory need not
  // have read it by then where the device reads the host's pages itself
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  k_round_features<<<(int)(((size_t)f.B * kFeat + 255) / 256), 256, 0, st>>>(f.zk,
                                                                            (size_t)f.B * kFeat);
  Fc g = f;
  g.zk = nullptr;   // written; every block reads it
  return fc_launch(g, ZDevice{f.zk}, 0, f.B, sms, st);
}

islbm_status status_of(cudaError_t e) { return e == cudaSuccess ? ISLBM_OK : ISLBM_ERR_CUDA; }

}  // namespace

extern "C" islbm_status islbm_cnn_forward(int stages, const int* channels, int base, int hidden,
                                          const void* const* params, const float* z, int batch,
                                          float* zk, float* h1, float* const* acts, void* stream) {
  const int sms = sm_count();
  if (!net_ok(stages, channels, base, hidden, batch, sms) || !params || !z || !h1 || !acts)
    return ISLBM_ERR_ARG;
  for (int k = 0; k < 4 + 2 * stages; ++k)
    if (!params[k] || !aligned(params[k], 4)) return ISLBM_ERR_ARG;
  for (int s = 0; s <= stages; ++s)
    if (!acts[s] || !aligned(acts[s], 16)) return ISLBM_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Fc f{static_cast<const bf16*>(params[0]), static_cast<const bf16*>(params[2]),
       static_cast<const float*>(params[1]), static_cast<const float*>(params[3]), zk, h1, acts[0],
       batch, hidden, base * base * channels[0], hidden % 8 == 0 && aligned(params[0], 16),
       base * base * channels[0] % 8 == 0 && aligned(params[2], 16),
       chain_kchunk(batch, base * base * channels[0], hidden,
                    hidden % 8 == 0 && base * base * channels[0] % 8 == 0, sms)};
  cudaError_t e = fc_forward(f, z, sms, st);
  if (e != cudaSuccess) return status_of(e);
  int H = base;
  for (int s = 0; s < stages; ++s) {
    const int up = s + 1 < stages;
    if (up) H *= 2;
    Conv c = layer(batch, H, channels[s], channels[s + 1], up, acts[s], params[4 + 2 * s]);
    c.bias = static_cast<const float*>(params[5 + 2 * s]);
    c.out = acts[s + 1];
    c.act = up;
    c.kchunk = chain_kchunk((long long)batch * H * H, c.cout, up16(9 * c.cin), c.cout % 8 == 0, sms);
    e = conv_forward(c, sms, st);
    if (e != cudaSuccess) return status_of(e);
  }
  return ISLBM_OK;
}

extern "C" islbm_status islbm_cnn_backward_scratch(int stages, const int* channels, int base,
                                                   int hidden, int batch, unsigned long long* bytes) {
  const int sms = sm_count();
  if (!bytes || !net_ok(stages, channels, base, hidden, batch, sms)) return ISLBM_ERR_ARG;
  *bytes = back_plan(stages, channels, base, hidden, batch, sms).total * sizeof(float);
  return ISLBM_OK;
}

extern "C" islbm_status islbm_cnn_backward(int stages, const int* channels, int base, int hidden,
                                           const void* const* params, int batch, const float* zk,
                                           const float* h1, const float* const* acts,
                                           const float* dy, float* const* grads, float* scratch,
                                           void* stream) {
  const int sms = sm_count();
  if (!net_ok(stages, channels, base, hidden, batch, sms) || !params || !zk || !h1 || !acts || !dy ||
      !grads || !scratch || !aligned(scratch, 256))
    return ISLBM_ERR_ARG;
  for (int k = 0; k < 4 + 2 * stages; ++k)
    if (!params[k] || !grads[k] || !aligned(params[k], 4)) return ISLBM_ERR_ARG;
  for (int s = 0; s < stages; ++s)
    if (!acts[s] || !aligned(acts[s], 16)) return ISLBM_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const BackPlan bp = back_plan(stages, channels, base, hidden, batch, sms);
  float* at = scratch;
  auto take = [&](size_t n) {
    float* q = at;
    at += round64(n);
    return q;
  };
  float* dh1 = take((size_t)batch * hidden);
  GradSegs segs{};
  SumSegs sums{};
  int first = 0, sum_first = 0;
  auto add_seg = [&](const float* part, float* out, int blocks, int values, int zeros) {
    segs.s[segs.n++] = GradSeg{part, out, blocks, values, zeros, first};
    first += (values + zeros + 63) / 64;
  };
  cudaError_t e;
  const float* d = dy;
  for (int s = stages - 1; s >= 0; --s) {
    const int up = s + 1 < stages, cin = channels[s], cout = channels[s + 1];
    const int H = base << std::min(s + 1, stages - 1);
    Conv c = layer(batch, H, cin, cout, up, acts[s], params[4 + 2 * s]);
    c.d = d;
    c.vd = cout % 4 == 0 && aligned(d, 16);
    const WgradPlan& w = bp.w[s];
    float* part = take(w.floats);
    const Wgrad g{c, part, w.pr, w.phases, w.kp, w.kchunk, w.cw};
    switch (w.nt) {
      case 1: e = wgrad_nt<1>(g, w, st); break;
      case 2: e = wgrad_nt<2>(g, w, st); break;
      case 3: e = wgrad_nt<3>(g, w, st); break;
      default: e = wgrad_nt<4>(g, w, st); break;
    }
    if (e != cudaSuccess) return status_of(e);
    add_seg(part, grads[4 + 2 * s], w.blocks, 9 * cin * cout, (up16(9 * cin) - 9 * cin) * cout);
    float* bpart = take((size_t)w.chunks * cout);
    const int per = 512 / (8 * cout);
    sums.s[sums.n++] = SumSeg{d, bpart, batch * H * H, cout, sum_first, per};
    sum_first += (w.chunks + per - 1) / per;
    add_seg(bpart, grads[5 + 2 * s], w.chunks, cout, 0);
    c.out = take(bp.image[s]);
    e = conv_dgrad(c, sms, st);
    if (e != cudaSuccess) return status_of(e);
    d = c.out;
  }
  k_bias_sum<<<sum_first, 512, 0, st>>>(sums);
  const int n2 = base * base * channels[0];
  const int dh_chunk = chain_kchunk(batch, hidden, n2, n2 % 8 == 0, sms), dh_tiles = (hidden + 7) / 8;
  const int dh_x = (batch + kFcB - 1) / kFcB;
  // Warps of a tile: all 16 of a block, half of them at a time where there are
  // not as many chunks and the blocks still fill the GPU (a batch that fills it
  // by itself has one chunk, and 15 warps would be idle: the backward pass of 512
  // hidden units, 4,096 outputs and one convolution took 3.19 ms for 4,096 samples
  // and takes 1.37, for 16,384 36.0 and 5.3).
  int share = 16;
  while (share > 1 && share / 2 >= (n2 + dh_chunk - 1) / dh_chunk &&
         (long long)dh_x * dh_tiles * (share / 2) / 16 >= 2LL * sms)
    share /= 2;
  k_fc_dh<<<dim3(dh_x, (dh_tiles + 16 / share - 1) / (16 / share)), 512, 0, st>>>(
      d, static_cast<const bf16*>(params[2]), h1, dh1, batch, hidden, n2, dh_chunk, share);
  auto fc = [&](FcGrad g, const float* a, const float* dd, float* dw, float* db) {
    g.a = a;
    g.d = dd;
    g.dw = dw;
    g.db = db;
    if (g.wchunks > 1) {
      g.dw = take((size_t)g.wchunks * g.K * g.N);
      add_seg(g.dw, dw, g.wchunks, g.K * g.N, 0);
    }
    if (g.bchunks > 1) {
      g.db = take((size_t)g.bchunks * g.N);
      add_seg(g.db, db, g.bchunks, g.N, 0);
    }
    return g;
  };
  const FcGrad l2 = fc(bp.l2, h1, d, grads[2], grads[3]);
  const FcGrad l1 = fc(bp.l1, zk, dh1, grads[0], grads[1]);
  k_fc_wgrad<<<l2.wblocks() + l1.wblocks() + l2.bblocks() + l1.bblocks(), 256, 0, st>>>(l2, l1,
                                                                                       batch);
  k_grad_sum<<<first, 64, 0, st>>>(segs);
  return status_of(cudaGetLastError());
}

extern "C" islbm_status islbm_cnn_adam_all(int tensors, float* const* w, void* const* wb,
                                           const float* const* g, float* const* m, float* const* v,
                                           const long long* n, float lr, float b1, float b2,
                                           float eps, long long t, void* stream) {
  if (tensors < 1 || !w || !wb || !g || !m || !v || !n || t < 1) return ISLBM_ERR_ARG;
  for (int k = 0; k < tensors; ++k)
    if (!w[k] || !g[k] || !m[k] || !v[k] || n[k] < 1 || n[k] > (1ll << 40)) return ISLBM_ERR_ARG;
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  for (int k0 = 0; k0 < tensors; k0 += kMaxTensors) {
    AdamSet a{};
    a.n = std::min(kMaxTensors, tensors - k0);
    long long blocks = 0;
    for (int k = 0; k < a.n; ++k) {
      a.t[k] = AdamTensor{w[k0 + k], static_cast<bf16*>(wb[k0 + k]), g[k0 + k], m[k0 + k],
                          v[k0 + k], n[k0 + k], (int)blocks};
      blocks += (n[k0 + k] + kAdamBlock - 1) / kAdamBlock;
      if (blocks > INT_MAX) return ISLBM_ERR_ARG;
    }
    k_adam_all<<<(unsigned)blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(a, lr, b1, b2, eps,
                                                                               c1, c2);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return status_of(e);
  }
  return ISLBM_OK;
}
