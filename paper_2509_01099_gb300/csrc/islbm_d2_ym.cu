// Marching 2-D step kernel: several time steps in one pass over the state
// (Sec. 2.1 - 2.3; FP32 and the 16-bit storage forms, node-centred stencil).
//
// A CTA owns a strip of up to 64 - 2 (NS - 1) columns over a chunk of rows and
// marches through it two rows at a time.  NS groups of two warps work as a
// pipeline: group s computes time step s of the rows that group s - 1 has just
// finished (group 1 reads rows brought by TMA) and hands its rows on through a
// ring in shared memory; only the last group writes to global memory.  A thread
// keeps one column for the whole chunk.  In the FP16NEQ form one more group in
// front decodes every staged row once (the tile kernel decodes 1.4 rows for a
// row of results, between two CTA-wide barriers), and the rows handed on are
// encoded and decoded again in registers.
//
// Why.  The tile kernel (k_step_tma) moves the whole state through HBM once a
// step and needs 324 instructions a node, many of them twice: it interpolates
// 10 rows in x for 8 rows of results, and recomputes tables, flags and
// addresses for every tile.  Marching interpolates every row once (the rows of
// the y stencil stay in registers), two rows at a time with the paired FP32
// instructions, and sets up a column once; with NS = 2 the state crosses HBM
// once for two steps.
//
// Rows.  A group takes the rows of its source in pairs (R, R + 1) and then
// produces rows (R - 1, R), whose y stencils R - 2 .. R + 1 it has.  The row
// pairs of consecutive groups are therefore one row apart; a chunk that starts
// above the bottom wall has group s start 2 (NS - s) rows below it.  The clamped
// stencils at the walls (row 0: rows 0 .. 2; row n - 1: rows n - 3 .. n - 1)
// fit the window when row 0 is the first and row n - 1 the second of a produced
// pair: chunks that touch the top wall have an even number of rows.
//
// The operations and their order are those of tile_body, and intermediate rows
// are rounded to the storage type as a store would (stochastic rounding
// included), so the results are the same bits as single steps.
//
// Every wait is bounded; a wait that gives up raises the CTA's abort flag and
// the error flag, thread 0 waits for its copies in flight, and the CTA returns.
#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "islbm_d2_common.cuh"
#include "islbm_store.cuh"
#include "islbm_tma.cuh"

namespace islbm {
namespace {

constexpr int kYmW = 64;           // columns of a group
constexpr int kYmMinRows = 12;     // shortest chunk

template <typename S, int NS>
struct YmGeom {
  // FP16NEQ: one more group in front decodes the staged rows into a ring
  static constexpr bool NEQ = is_neq<S>::value;
  static constexpr int LEVELS = NS + (NEQ ? 1 : 0), RINGS = LEVELS - 1;
  static constexpr int COLUMNS = kYmW - 2 * (LEVELS - 1);   // widest strip
  static constexpr int HX = 16 / (int)sizeof(S);       // elements of a 16-byte chunk
  // staged row: the columns of the first group, with one halo column on each
  // side where it interpolates, from a 16-byte boundary
  static constexpr int TW = (kYmW + (NEQ ? 0 : 2) + HX - 1 + HX - 1) / HX * HX;
  static constexpr int MW = (kYmW + 3 + 3) / 4 * 4;    // FP16NEQ: row of the FP32 moments
  // row pitch of the rings between groups, whose rows are FP32 in every storage
  // form (rounded to it, so that the next group reads them without conversions)
  static constexpr int RW = kYmW + 2;
  static constexpr unsigned ROWS = 14u * 2u * TW * sizeof(S);
  static constexpr unsigned M_OFF = (ROWS + 127u) / 128u * 128u;
  static constexpr unsigned M_BYTES = NEQ ? 4u * 2u * MW * 4u : 0u;
  static constexpr unsigned LOADED = ROWS + M_BYTES;   // bytes a stage's copies bring
  static constexpr unsigned TMA_BYTES = M_OFF + M_BYTES;
  static constexpr unsigned RING_BYTES = (14u * 2u * RW * 4u + 127u) / 128u * 128u;
  static constexpr int DT = 3;                         // TMA stages (row pairs)
  static constexpr int DR = 4;               // row pairs of a ring
  static constexpr unsigned SMEM = DT * TMA_BYTES + RINGS * DR * RING_BYTES + 256;
  static constexpr int THREADS = LEVELS * 64;
  static constexpr int CTAS = NEQ ? 2 : NS == 2 ? 4 : 6;   // an SM's registers and shared memory
  static_assert(TMA_BYTES % 128 == 0, "stages keep the TMA's 128-byte alignment");
  static_assert((2 * DT + 2 * DR * RINGS) * 8 + 4 <= 256 - 16, "barriers and the flag");
};

// The items of a launch: strips of columns x chunks of rows, evenly split.
struct YmSched {
  int nstrip, nchunk;
  __host__ __device__ int row(int k, int n) const {   // first row of chunk k
    if (k >= nchunk) return n;
    const int r = (int)((long long)n * k / nchunk);
    return k > 0 && k == nchunk - 1 ? r - ((n - r) & 1) : r;   // the top chunk is even
  }
  __host__ __device__ int col(int k, int n) const { return (int)((long long)n * k / nstrip); }
};

// y tables of two rows, cy = +1 and -1.
struct YmTables {
  float4 p0, p1, m0, m1;
};

// Wait on `bar`; one that does not end in time raises the error flag and the
// CTA's abort flag, with which every later wait returns at once: the groups
// run to their ends without waiting (their results are void).
__device__ __noinline__ void ym_wait_slow(uint64_t* bar, unsigned phase, volatile int* abort,
                                          int* err) {
  if (*abort) return;
  if (!mbar_wait_or_abort(bar, phase, abort)) {
    if (!*abort) atomicExch(err, 1);
    *abort = 1;
  }
}
__device__ __forceinline__ void ym_wait(uint64_t* bar, unsigned phase, volatile int* abort,
                                        int* err) {
  if (!mbar_try_wait(bar, phase)) ym_wait_slow(bar, phase, abort, err);
}

// Group of step s (1 .. NS) of one item.  SRC: element type of the source rows
// (plane pitch PS, row pitch RS).  First rows are at `src_ring`.
template <typename S, int NS, int s>
struct YmGroup {
  using G = YmGeom<S, NS>;
  using Elem = S;
  static constexpr bool FIRST = s == 1, LAST = s == NS;
  static constexpr bool STAGED = FIRST && !G::NEQ;     // source: the TMA stages
  using T = std::conditional_t<STAGED, S, float>;      // type of the source rows
  static constexpr int RS = STAGED ? G::TW : G::RW;    // row pitch of the source
  static constexpr int PS = 2 * RS;                    // plane pitch of the source

  // per-thread state of the march
  float2 hp[8];       // previous row pair of the planes moving in y (x-interpolated)
  float sv[6];        // second row of the previous pair, the planes not moving in y
  float bb[2];        // raw planes 7, 8 of row 0
  float2 wp[3], wm[3];
  int ci, bp, bm;     // source columns: own, stencil bases of cx = +1, -1
  bool wW, wE, any;

  static __device__ __forceinline__ float2 own(const T* a, const T* b, int pl, int c) {
    return make_float2(to_f(a[pl * PS + c]), to_f(b[pl * PS + c]));
  }
  static __device__ __forceinline__ float2 interp(const T* a, const T* b, int pl, int c,
                                                  const float2 (&w)[3]) {
    return __ffma2_rn(w[2], own(a, b, pl, c + 2),
                      __ffma2_rn(w[1], own(a, b, pl, c + 1), __fmul2_rn(w[0], own(a, b, pl, c))));
  }

  __device__ __forceinline__ void setup(const P2<float>& p, int x, int src0) {
    const int xc = min(max(x, 0), p.nx - 1);
    const float4 a = __ldg(p.px[0] + xc), b = __ldg(p.px[1] + xc);
    wp[0] = make_float2(a.x, a.x);
    wp[1] = make_float2(a.y, a.y);
    wp[2] = make_float2(a.z, a.z);
    wm[0] = make_float2(b.x, b.x);
    wm[1] = make_float2(b.y, b.y);
    wm[2] = make_float2(b.z, b.z);
    ci = x - src0;
    bp = __float_as_int(a.w) - src0;
    bm = __float_as_int(b.w) - src0;
    if (!(ISLBM_IN_WINDOW(ci, RS) && ISLBM_IN_WINDOW(bp, RS - 2) && ISLBM_IN_WINDOW(bm, RS - 2)))
      ci = bp = bm = 0;
    wW = x == 0;
    wE = x == p.nx - 1;
    any = __any_sync(0xffffffffu, wW || wE);
#pragma unroll
    for (int k = 0; k < 8; ++k) hp[k] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 6; ++k) sv[k] = 0.f;
    bb[0] = bb[1] = 0.f;
  }

  // Takes source rows R (at a) and R + 1 (at b), produces rows R - 1 and R into
  // fn, gn (of the first call: nothing of use).  One copy of this code serves
  // every iteration, the walls' behind uniform branches: the groups run
  // different code at the same time, and with separate copies for the first
  // and last rows (and the loop unrolled) instruction fetch made the kernel
  // slower by a fifth.
  __device__ __forceinline__ void take(const P2<float>& p, const T* a, const T* b, int R,
                                       const YmTables& q, float2 (&fn)[9], float2 (&gn)[5]) {
    const bool bot = R == 1, top = R == p.ny - 1, edge = bot || top;
    // y pass of window slot k: rows R - 2, R - 1 (hp) and R, R + 1 (h)
    auto ypass = [&](int k, float2 h, bool plus, float2& out) {
      const float4 q0 = plus ? q.p0 : q.m0, q1 = plus ? q.p1 : q.m1;
      out.x = dot3(q0, hp[k].x, hp[k].y, h.x);
      out.y = dot3(q1, hp[k].y, h.x, h.y);
      if (edge) {
        if (bot && !plus) out.x = dot3(q0, hp[k].y, h.x, h.y);
        if (top && plus) out.y = dot3(q1, hp[k].x, hp[k].y, h.x);
      }
    };
    // planes that do not move in y
    auto still = [&](int k, float2 z, float2& out) {
      out = make_float2(sv[k], z.x);
      sv[k] = z.y;
    };
    still(0, own(a, b, 0, ci), fn[0]);
    still(1, own(a, b, 9, ci), gn[0]);
    float2 z1 = interp(a, b, 1, bp, wp), z3 = interp(a, b, 3, bm, wm);
    float2 t1 = interp(a, b, 10, bp, wp), t3 = interp(a, b, 12, bm, wm);
    if (any) {
      if (wW) {
        z1 = own(a, b, 3, ci);
        const float2 v = own(a, b, 12, ci);
        t1 = make_float2(p.abb_hot - v.x, p.abb_hot - v.y);
      }
      if (wE) {
        z3 = own(a, b, 1, ci);
        const float2 v = own(a, b, 10, ci);
        t3 = make_float2(p.abb_cold - v.x, p.abb_cold - v.y);
      }
    }
    still(2, z1, fn[1]);
    still(3, z3, fn[3]);
    still(4, t1, gn[1]);
    still(5, t3, gn[3]);
    // planes moving in y only
    auto straight = [&](int kp, int plp, int km, int plm, float2& outp, float2& outm) {
      const float2 h = own(a, b, plp, ci), g = own(a, b, plm, ci);
      ypass(kp, h, true, outp);
      ypass(km, g, false, outm);
      if (edge) {
        if (bot) outp.x = hp[km].y;
        if (top) outm.y = h.x;
      }
      hp[kp] = h;
      hp[km] = g;
    };
    straight(0, 2, 1, 4, fn[2], fn[4]);
    straight(2, 11, 3, 13, gn[2], gn[4]);
    // diagonals.  Next to an x-wall the window holds the raw bounce-back
    // partner instead of the interpolated plane, and its centre is the result.
    auto diag = [&](int k, int pl, int partner, bool plus_x, bool plus_y, float2& out) {
      float2 h = plus_x ? interp(a, b, pl, bp, wp) : interp(a, b, pl, bm, wm);
      ypass(k, h, plus_y, out);
      if (any) {
        if (plus_x ? wW : wE) {
          h = own(a, b, partner, ci);
          out = make_float2(hp[k].y, h.x);
        }
      }
      hp[k] = h;
    };
    diag(4, 5, 7, true, true, fn[5]);
    diag(5, 6, 8, false, true, fn[6]);
    diag(6, 7, 5, false, false, fn[7]);
    diag(7, 8, 6, true, false, fn[8]);
    if (edge) {
      if (bot) {
        fn[5].x = bb[0];
        fn[6].x = bb[1];
      }
      if (top) {
        fn[7].y = to_f(a[5 * PS + ci]);
        fn[8].y = to_f(a[6 * PS + ci]);
      }
    }
    if (R < 0) {
      bb[0] = to_f(b[7 * PS + ci]);
      bb[1] = to_f(b[8 * PS + ci]);
    }
  }
};

// One CTA's work: columns [x0, x1) and rows [ya, yb).
struct YmItem {
  int x0, x1, ya, yb;
};

template <typename S, int NS>
__device__ __forceinline__ void ym_item(const CUtensorMap* tmap, const CUtensorMap* tmap_m,
                                        S* __restrict__ fout, const P2<float>& p, const PairC& kc, unsigned first_step,
                                        int* err, const YmItem& item) {
  using G = YmGeom<S, NS>;
  constexpr int DT = G::DT, DR = G::DR, RINGS = G::RINGS;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* rings = smem_raw + DT * G::TMA_BYTES;
  // full / empty barriers of the TMA stages, then of each ring
  uint64_t* bars = reinterpret_cast<uint64_t*>(rings + RINGS * DR * G::RING_BYTES + 16);
  volatile int* abort = reinterpret_cast<volatile int*>(bars + 2 * DT + 2 * DR * RINGS);
  if (threadIdx.x == 0) {
    for (int k = 0; k < DT; ++k) {
      mbar_init(&bars[k], 1);
      mbar_init(&bars[DT + k], 2);
    }
    for (int k = 0; k < 2 * DR * RINGS; ++k) mbar_init(&bars[2 * DT + k], 2);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();

  const int x0 = item.x0, x1 = item.x1, ya = item.ya, yb = item.yb;
  const int nI = (yb - ya + 1) / 2;           // row pairs of the last group
  const bool at_bottom = ya == 0, at_top = yb == p.ny;
  // group s: iterations [first(s), last(s)], rows ya - 2 (NS - s) - 1 + 2 i, +1
  auto first = [&](int s) { return at_bottom ? NS - s : 0; };
  auto last = [&](int s) { return nI + (at_top ? NS - s : 2 * (NS - s)); };
  const int xa = (x0 - NS) & ~(G::HX - 1);    // first staged column

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Copies of group 1's iterations, by thread 0: one box of a row pair, all planes.
  const int copies = last(1) - first(1) + 1, row0 = ya - 2 * (NS - 1) - 1 + 2 * first(1);
  int issued = 0;
  auto issue = [&]() {
    const int st = issued % DT;
    unsigned char* dst = smem_raw + st * G::TMA_BYTES;
    mbar_expect_tx(&bars[st], G::LOADED);
    tma_load_3d(dst, tmap, xa, row0 + 2 * issued, 0, &bars[st]);
    if constexpr (G::NEQ)
      tma_load_3d(dst + G::M_OFF, tmap_m, (x0 - NS) & ~3, row0 + 2 * issued, 0, &bars[st]);
    ++issued;
  };
  if (threadIdx.x == 0) {
    asm volatile("prefetch.tensormap [%0];\n" ::"l"(tmap) : "memory");
    grid_launch_next();
    grid_wait();
    while (issued < min(DT, copies)) issue();
  }
  // Refill of the stage of the iteration before, which the other warp has
  // released by now or does within this iteration.
  auto refill = [&]() {
    const int u = issued - DT;
    ym_wait(&bars[DT + u % DT], (unsigned)(u / DT) & 1u, abort, err);
    if (!*abort) {
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      issue();
    }
  };
  // FP16NEQ: the staged row pairs as FP32 deviations, one column a thread.
  [[maybe_unused]] auto decode = [&]() {
    if constexpr (G::NEQ) {
      const int x = x0 - NS + (int)threadIdx.x;
      int hc = x - xa, mc = x - ((x0 - NS) & ~3);
      if (!(ISLBM_IN_WINDOW(hc, G::TW) && ISLBM_IN_WINDOW(mc, G::MW))) hc = mc = 0;
      uint64_t* tfull = bars + 2 * DT;
      uint64_t* tempty = tfull + DR;
      float t0, ti;
      trest(p.a_T, t0, ti);
      int ss = 0, ts = 0;
      unsigned sp = 0, tp = 1;
      for (int n = 0; n < copies; ++n) {
        ym_wait(&bars[ss], sp, abort, err);
        const unsigned char* stage = smem_raw + ss * G::TMA_BYTES;
        const unsigned short* h = reinterpret_cast<const unsigned short*>(stage) + hc;
        const float* m = reinterpret_cast<const float*>(stage + G::M_OFF) + mc;
        unsigned r[14];
#pragma unroll
        for (int k = 0; k < 14; ++k)
          r[k] = (unsigned)h[2 * k * G::TW] | ((unsigned)h[(2 * k + 1) * G::TW] << 16);
        float2 mm[4], f[9], g[5];
#pragma unroll
        for (int k = 0; k < 4; ++k) mm[k] = make_float2(m[2 * k * G::MW], m[(2 * k + 1) * G::MW]);
        neq_decode2x2(mm[0], mm[1], mm[2], mm[3], r, t0, ti, f, g);
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars[DT + ss]);
        if (threadIdx.x == 0 && n > 0 && issued < copies) refill();
        ym_wait(&tempty[ts], tp, abort, err);
        float* t = reinterpret_cast<float*>(rings + ts * G::RING_BYTES) + threadIdx.x;
#pragma unroll
        for (int k = 0; k < 14; ++k) {
          const float2 v = k < 9 ? f[k < 9 ? k : 0] : g[k < 9 ? 0 : k - 9];
          t[2 * k * G::RW] = v.x;
          t[(2 * k + 1) * G::RW] = v.y;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&tfull[ts]);
        if (++ss == DT) {
          ss = 0;
          sp ^= 1u;
        }
        if (++ts == DR) {
          ts = 0;
          tp ^= 1u;
        }
      }
    }
  };
  auto run = [&](auto step) {
    constexpr int s = decltype(step)::value;
    using Gr = YmGroup<S, NS, s>;
    using T = typename Gr::T;
    using St = Store<typename Gr::Elem>;
    constexpr bool FIRST = Gr::FIRST, LAST = Gr::LAST, STAGED = Gr::STAGED;
    constexpr int RT = G::NEQ ? s : s - 1;    // ring written; RT - 1: ring read
    const int c = threadIdx.x - 64 * RT;
    const int x = x0 - (NS - s) + c;
    const int src0 = STAGED ? xa : x0 - NS + s - 1;
    Gr g;
    g.setup(p, x, src0);
    uint64_t* sfull = STAGED ? bars : bars + 2 * DT + 2 * DR * (RT - 1);
    uint64_t* sempty = sfull + (STAGED ? DT : DR);
    uint64_t* tfull = bars + 2 * DT + 2 * DR * RT;
    uint64_t* tempty = tfull + DR;
    constexpr int DS = STAGED ? DT : DR;
    const unsigned char* src = STAGED ? smem_raw : rings + (RT - 1) * DR * G::RING_BYTES;
    constexpr unsigned SB = STAGED ? G::TMA_BYTES : G::RING_BYTES;
    unsigned char* target = rings + RT * DR * G::RING_BYTES;
    const int i0 = first(s), i1 = last(s);
    const bool mine = x >= x0 && x < x1;
    int ss = 0;              // source slot of this iteration's (first) row pair
    unsigned sp = 0;         // its phase
    int ts = 0;              // target slot
    unsigned tp = 1;         // phase of its empty barrier (1: the first use passes)
    // source rows of iteration i: FIRST: both of slot ss; else the second row of
    // pair i (slot ss) and the first row of pair i + 1 (the next slot)
    if (!FIRST && !at_bottom) ym_wait(&sfull[0], 0u, abort, err);
    // a bottom chunk has no pair i0: its first pair is taken as "next"
    int have = FIRST || !at_bottom ? 1 : 0;
    unsigned off = 0;        // byte offset of the last group's next output row
    if (LAST) off = (unsigned)(((size_t)ya * p.pitch + (mine ? x : x0)) * sizeof(S));
    const int first_row = ya - 2 * (NS - s) + 2 * i0;
    const float4 *tqp = p.py[0] + first_row, *tqm = p.py[1] + first_row;
    for (int i = i0; i <= i1; ++i) {
      const int R = ya - 2 * (NS - s) - 1 + 2 * i;
      // tables of rows R - 1 and R, loaded before the wait, which hides their latency
      YmTables q{};
      if (i > i0 && ISLBM_IN_WINDOW(R - 1, p.ny) && ISLBM_IN_WINDOW(R, p.ny)) {
        q = YmTables{__ldg(tqp), __ldg(tqp + 1), __ldg(tqm), __ldg(tqm + 1)};
        tqp += 2;
        tqm += 2;
      }
      const T *a, *b;
      int ns = ss;
      unsigned np = sp;
      if (FIRST) {
        ym_wait(&sfull[ss], sp, abort, err);
        a = reinterpret_cast<const T*>(src + ss * SB);
        b = a + Gr::RS;
      } else {
        if (have && ++ns == DS) {
          ns = 0;
          np ^= 1u;
        }
        // the pair after the last one of a chunk at the top wall does not exist
        // (row ny, which no result uses)
        if (!(at_top && i == i1)) ym_wait(&sfull[ns], np, abort, err);
        a = reinterpret_cast<const T*>(src + ss * SB) + Gr::RS;
        b = reinterpret_cast<const T*>(src + ns * SB);
      }
      float2 fn[9], gn[5];
      g.take(p, a, b, R, q, fn, gn);
      // the source rows are in registers: release stage / pair i
      __syncwarp();
      if (have && lane == 0) mbar_arrive(&sempty[ss]);
      if (STAGED && threadIdx.x == 0 && i > i0 && issued < copies) refill();
      if (FIRST) {
        if (++ss == DS) {
          ss = 0;
          sp ^= 1u;
        }
      } else {
        ss = ns;
        sp = np;
        have = 1;
      }
      if (i == i0) continue;
      float2 mm[4];
      collide_pair(fn, gn, kc, mm);
      auto val = [&](int k) { return k < 9 ? fn[k < 9 ? k : 0] : gn[k < 9 ? 0 : k - 9]; };
      const unsigned seed_step = first_step + (unsigned)(s - 1);
      [[maybe_unused]] unsigned rr[14];   // FP16NEQ: remainders of rows R - 1 (low halves) and R
      [[maybe_unused]] float t0, ti;
      if constexpr (G::NEQ) {
        trest(p.a_T, t0, ti);
        neq_remainders2x2(fn, gn, mm, t0, ti, rr);
      }
      if constexpr (LAST && G::NEQ) {
        if (mine) {
          char* o = reinterpret_cast<char*>(fout);
          const size_t ps = (size_t)p.plane * 2;
          char* om = o + 14 * ps;
#pragma unroll
          for (int k = 0; k < 14; ++k)
            *reinterpret_cast<unsigned short*>(o + k * ps + off) = (unsigned short)(rr[k] & 0xFFFFu);
#pragma unroll
          for (int k = 0; k < 4; ++k) *reinterpret_cast<float*>(om + 2 * (k * ps + off)) = mm[k].x;
          if (R < yb) {
            const size_t off1 = off + (size_t)p.pitch * 2;
#pragma unroll
            for (int k = 0; k < 14; ++k)
              *reinterpret_cast<unsigned short*>(o + k * ps + off1) = (unsigned short)(rr[k] >> 16);
#pragma unroll
            for (int k = 0; k < 4; ++k)
              *reinterpret_cast<float*>(om + 2 * (k * ps + off1)) = mm[k].y;
          }
        }
        off += (unsigned)(2 * p.pitch * sizeof(S));
      } else if constexpr (LAST) {
        if (mine) {
          char* o = reinterpret_cast<char*>(fout);
          const size_t ps = (size_t)p.plane * sizeof(S);
          unsigned r = sr_seed((size_t)(R - 1) * p.pitch + x, seed_step);
#pragma unroll
          for (int k = 0; k < 14; ++k)
            St::st_sr(reinterpret_cast<S*>(o + k * ps + off), val(k).x, sr_next(r));
          if (R < yb) {
            const unsigned off1 = off + (unsigned)(p.pitch * sizeof(S));
            unsigned r1 = sr_seed((size_t)R * p.pitch + x, seed_step);
#pragma unroll
            for (int k = 0; k < 14; ++k)
              St::st_sr(reinterpret_cast<S*>(o + k * ps + off1), val(k).y, sr_next(r1));
          }
        }
        off += (unsigned)(2 * p.pitch * sizeof(S));
      } else {
        ym_wait(&tempty[ts], tp, abort, err);
        float* t = reinterpret_cast<float*>(target + ts * G::RING_BYTES) + c;
        if constexpr (G::NEQ) {   // what the next step would read back
          neq_decode2x2(mm[0], mm[1], mm[2], mm[3], rr, t0, ti, fn, gn);
#pragma unroll
          for (int k = 0; k < 14; ++k) {
            t[k * 2 * G::RW] = val(k).x;
            t[k * 2 * G::RW + G::RW] = val(k).y;
          }
        } else {
          unsigned r = sr_seed((size_t)((long long)(R - 1) * p.pitch + x), seed_step);
          unsigned r1 = sr_seed((size_t)((long long)R * p.pitch + x), seed_step);
#pragma unroll
          for (int k = 0; k < 14; ++k) {
            t[k * 2 * G::RW] = St::rounded_sr(val(k).x, sr_next(r));
            t[k * 2 * G::RW + G::RW] = St::rounded_sr(val(k).y, sr_next(r1));
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&tfull[ts]);
        if (++ts == DR) {
          ts = 0;
          tp ^= 1u;
        }
      }
    }
  };
  constexpr int front = G::NEQ ? 2 : 0;    // warps of the decoding group
  if (warp < front)
    decode();
  else if (warp < front + 2)
    run(std::integral_constant<int, 1>{});
  else if constexpr (NS > 1)
    run(std::integral_constant<int, 2>{});
  // copies still in flight land before the CTA's shared memory is released
  if (threadIdx.x == 0)
    for (int k = max(0, issued - DT); k < issued; ++k)
      mbar_wait(&bars[k % DT], (unsigned)(k / DT) & 1u);
}

template <typename S, int NS, int MINB>
__global__ void __launch_bounds__(YmGeom<S, NS>::THREADS, MINB)
    k_step_ym(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CUtensorMap tmap_m,
              S* __restrict__ fout, P2<float> p, const __grid_constant__ PairC kc, int* err,
              YmSched sc) {
  const int strip = blockIdx.x % sc.nstrip, chunk = blockIdx.x / sc.nstrip;
  ym_item<S, NS>(&tmap, &tmap_m, fout, p, kc, p.step, err,
                 YmItem{sc.col(strip, p.nx), sc.col(strip + 1, p.nx), sc.row(chunk, p.ny),
                        sc.row(chunk + 1, p.ny)});
}

// Many cavities in one launch: a CTA's item names its cavity, whose parameters
// it copies to shared memory.
template <typename S>
struct alignas(128) YmCav {
  CUtensorMap map[2];   // row pairs of the cavity's two buffers
  S* out[2];            // output buffer when reading buffer 0 / 1
  P2<float> p;
  PairC kc;
};
struct YmBatchItem {
  YmItem at;
  int cav;
};

template <typename S, int NS, int MINB>
__global__ void __launch_bounds__(YmGeom<S, NS>::THREADS, MINB)
    k_step_ym_batch(const YmCav<S>* __restrict__ cavs, const YmBatchItem* __restrict__ items,
                    int parity, unsigned step, int* err) {
  __shared__ P2<float> p;
  __shared__ PairC kc;
  const YmBatchItem it = items[blockIdx.x];
  const YmCav<S>& cv = cavs[it.cav];
  static_assert(sizeof(P2<float>) % 4 == 0 && sizeof(PairC) % 4 == 0, "copied by words");
  for (int k = threadIdx.x; k < (int)(sizeof(P2<float>) / 4); k += blockDim.x)
    reinterpret_cast<int*>(&p)[k] = reinterpret_cast<const int*>(&cv.p)[k];
  for (int k = threadIdx.x; k < (int)(sizeof(PairC) / 4); k += blockDim.x)
    reinterpret_cast<int*>(&kc)[k] = reinterpret_cast<const int*>(&cv.kc)[k];
  S* out = cv.out[parity];
  // (the barrier that opens ym_item orders the copies before their use)
  ym_item<S, NS>(&cv.map[parity], nullptr, out, p, kc, step, err, it.at);
}

// Strips and chunks of a launch.  A CTA costs its rows and about kYmStart more
// (the rows below its chunk that the first groups compute, the pipeline's fill
// and drain).  kYmRow: relative time of a row with 1 .. 4 CTAs on an SM; the
// warps of few CTAs leave issue slots empty, so four CTAs take only 1.7 times
// as long as one (measured at 257^2 .. 4096^2 with 5 .. 71 chunks; 1024^2: 26
// chunks, three CTAs an SM, 16.6 us a step, 35 chunks, four, 15.9).
constexpr double kYmStart = 8.0;
constexpr double kYmRow[5] = {0.0, 0.25, 0.30, 0.345, 0.42};

inline YmSched ym_schedule(int nx, int ny, int w, int sms, int per_sm) {
  YmSched sc;
  sc.nstrip = (nx + w - 1) / w;
  sc.nchunk = 1;
  double best = 1e300;
  for (int c = ny % 2 ? 2 : 1; c <= ny / kYmMinRows; ++c) {
    const long long items = (long long)sc.nstrip * c;
    const long long slots = (long long)sms * per_sm, left = items % slots;
    const double rows = (double)((ny + c - 1) / c) + kYmStart;
    const double cost = rows * ((double)(items / slots) * kYmRow[std::min(per_sm, 4)] +
                                kYmRow[std::min<long long>(4, (left + sms - 1) / sms)]);
    if (cost < best - 1e-9) {
      best = cost;
      sc.nchunk = c;
    }
  }
  return sc;
}

template <typename S, int NS>
cudaError_t launch_ym(Solver& s) {
  using G = YmGeom<S, NS>;
  const auto k = k_step_ym<S, NS, G::CTAS>;
  int per_sm = 0;
  const cudaError_t e = launch_setup_once(
      reinterpret_cast<const void*>(k),
      [](const void* f, int* n) {
        cudaError_t e2 =
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
        if (e2 == cudaSuccess)
          e2 = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                                    cudaSharedmemCarveoutMaxShared);
        if (e2 == cudaSuccess)
          e2 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, G::THREADS, G::SMEM);
        return e2;
      },
      &per_sm);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const YmSched sc = ym_schedule(s.n[0], s.n[1], G::COLUMNS, s.sm_count, per_sm);
  const P2<float> p = make_params<float>(s);
  // a launch that fills the GPU's slots leaves the next one's early blocks only
  // those that come free; into a half-full GPU they would crowd on the SMs with
  // room (1024^2, 35 chunks, 595 of 608 slots: 15.9 -> 15.4 us a step; 26 chunks,
  // 442 slots: 16.6 -> 19.4 us)
  const bool serial = sc.nstrip * sc.nchunk >= s.sm_count * per_sm * 15 / 16;
  return launch_grid(serial, k, sc.nstrip * sc.nchunk, G::THREADS, G::SMEM, s.stream,
                     *reinterpret_cast<const CUtensorMap*>(s.tmap_y[s.cur]),
                     *reinterpret_cast<const CUtensorMap*>(s.tmap_ym[s.cur]),
                     static_cast<S*>(s.buf[s.cur ^ 1]), p, make_pair_constants(p), s.derr, sc);
}

}  // namespace

// Whether the marching kernel takes a mesh (at least two chunks of the shortest
// length, 32-bit offsets in a plane), and whether it is the faster one there.
//
// It is once its CTAs fill the GPU, and in the 16-bit forms, which are bound by
// their conversions and stochastic rounding in either kernel, on larger meshes
// only.  us a step, tile kernel and this one: FP32 512^2 6.5 / 7.0, 900^2 15.9 /
// 15.3, 1024^2 19.4 / 15.4, 2049^2 74 / 54, 4096^2 277 / 193; BF16 1024^2 18.2 /
// 18.4, 1400^2 32.4 / 30.6, 4096^2 246 / 234; FP16NEQ 775^2 17.7 / 13.7, 2049^2
// 104 / 84, 4096^2 385 / 310 (at two CTAs an SM: at three, 96 registers, it
// spills and takes 423).
//
// And its strips have to be about as full as the tile kernel's tiles: a strip is
// 62 columns (FP16NEQ 60), a tile 64, so a mesh 64 columns wide takes two half
// empty strips for one full tile.  With f, the columns of the strips over those
// of the tiles, measured time over the tile kernel's (columns x rows so that the
// nodes are as given):
//   FP32, 0.6M nodes: f = 0.97 (62, 124, 240 columns) 0.87-0.88, 1.09 (512) 0.92,
//     1.16 (320) 1.02, 1.29 (192) 1.11, 1.45 (128) 1.17, 1.94 (64) 1.35; from
//     1.2M on, where the tile kernel's two buffers leave L2: 1.16 0.69-0.85, 1.29
//     0.75-0.93, 1.45 0.93-1.04, 1.94 1.06-1.19
//   FP16NEQ: f = 0.94 0.75, 1.17 (256) 0.92-0.97, 1.25 (192) 0.97-1.02, 1.41 (128)
//     1.08-1.15, 1.88 (64) 1.40-1.49
//   FP16 / BF16 from 1.5M: f = 0.97 0.95, 1.03 (1024) 0.94-0.99, 1.05 (768)
//     0.96-1.02, 1.09 (512) 0.97-1.05, 1.16 1.04-1.12, 1.45 1.28-1.37, 1.94 1.47-1.58
// Up to 32 columns, one of a group's two warps computes nothing that is kept:
// FP16NEQ 0.98-1.05, FP16 1.11-1.20, BF16 1.02-1.06 (FP32 0.73-0.88).
constexpr long long kYmMinNodes = 600000, kYmMinNodes16 = 1500000;
constexpr long long kYmL2Nodes = 1100000;   // FP32: 2 x 56 bytes of these are the L2 cache
bool step_2d_ym_takes(int nx, int ny, int precision, size_t plane_bytes) {
  if (nx < 16 || ny < 2 * kYmMinRows + 2 || plane_bytes >= (size_t)1 << 31) return false;
  const long long nodes = (long long)nx * ny;
  const bool neq = precision == ISLBM_FP16NEQ;
  const int w = neq ? YmGeom<Neq16, 2>::COLUMNS : YmGeom<float, 2>::COLUMNS;
  const double f = (double)((nx + w - 1) / w * w) / ((nx + 63) / 64 * 64);
  if (precision == ISLBM_FP32)
    return nodes >= kYmMinNodes && f <= (nodes < kYmL2Nodes ? 1.15 : 1.3);
  if (neq) return nodes >= kYmMinNodes && nx > 32 && f <= 1.2;
  return nodes >= kYmMinNodes16 && nx > 32 && f <= 1.04;
}

// TMA boxes (x, y, planes) of a staged row pair: the populations, and the
// moments of the FP16NEQ form.
void step_2d_ym_box(int precision, unsigned (&box)[3], unsigned (&moments)[3]) {
  box[0] = (unsigned)(precision == ISLBM_FP32      ? YmGeom<float, 2>::TW
                      : precision == ISLBM_FP16NEQ ? YmGeom<Neq16, 2>::TW
                                                   : YmGeom<__half, 2>::TW);
  box[1] = moments[1] = 2;
  box[2] = 14;
  moments[0] = (unsigned)YmGeom<Neq16, 2>::MW;
  moments[2] = 4;
}

cudaError_t launch_step_2d_ym(Solver& s, int steps) {
  if (steps != 2) return cudaErrorInvalidValue;
  cudaError_t e = cudaErrorInvalidValue;
  switch (s.precision) {
    case ISLBM_FP32: e = launch_ym<float, 2>(s); break;
    case ISLBM_FP16DEV: e = launch_ym<__half, 2>(s); break;
    case ISLBM_BF16DEV: e = launch_ym<__nv_bfloat16, 2>(s); break;
    case ISLBM_FP16NEQ: e = launch_ym<Neq16, 2>(s); break;
  }
  if (e == cudaSuccess) s.cur ^= 1;
  return e;
}

namespace {

struct YmBatch : BatchGroup {
  using G = YmGeom<float, 2>;
  YmCav<float>* cavs = nullptr;
  YmBatchItem* items = nullptr;
  int nitems = 0;
  DevAllocator mem;
  cudaStream_t stream = nullptr;
  ~YmBatch() override {
    dev_free(mem, cavs, stream);
    dev_free(mem, items, stream);
    cudaStreamSynchronize(stream);
  }
  cudaError_t launch(cudaStream_t st, int parity, unsigned step, int* err) override {
    k_step_ym_batch<float, 2, 4><<<nitems, G::THREADS, G::SMEM, st>>>(cavs, items, parity, step,
                                                                     err);
    return cudaGetLastError();
  }
};

}  // namespace

// Two steps of FP32 cavities in one launch.  *out stays null where single steps
// (k_step_tma_batch) are the better choice: other storage forms, meshes below
// the kernel's limits, too few nodes to fill the GPU (step_2d_ym_takes), or strips
// and chunks that cost more than they save.
cudaError_t make_batch_pair_group(const std::vector<Solver*>& members, int precision, int sms,
                                  cudaStream_t stream, BatchGroup** out) {
  *out = nullptr;
  long long nodes = 0;
  for (const Solver* m : members) {
    nodes += m->nodes;
    if (m->n[0] < 16 || m->n[1] < 2 * kYmMinRows + 2 ||
        (size_t)m->plane * m->elem >= (size_t)1 << 31)
      return cudaSuccess;
  }
  if (precision != ISLBM_FP32 || nodes < kYmMinNodes) return cudaSuccess;
  const auto k = k_step_ym_batch<float, 2, 4>;
  int per_sm = 0;
  cudaError_t e = launch_setup_once(
      reinterpret_cast<const void*>(k),
      [](const void* f, int* n) {
        cudaError_t e2 = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)YmBatch::G::SMEM);
        if (e2 == cudaSuccess)
          e2 = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                                    cudaSharedmemCarveoutMaxShared);
        if (e2 == cudaSuccess)
          e2 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, YmBatch::G::THREADS,
                                                             YmBatch::G::SMEM);
        return e2;
      },
      &per_sm);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // one chunk length for all cavities: the rows of all items (and each item's
  // start) spread over the slots, and half a longest item of idle slots at the end
  auto sched = [](const Solver* m, int rows) {
    const int w = kYmW - 2;
    YmSched sc;
    sc.nstrip = (m->n[0] + w - 1) / w;
    const int most = m->n[1] / kYmMinRows;
    sc.nchunk = std::max(1 + m->n[1] % 2, std::min(most, (m->n[1] + rows / 2) / rows));
    return sc;
  };
  int best = 64;
  double best_cost = 1e300;
  for (int rows = 16; rows <= 1024; rows += 8) {
    double total = 0.0, longest = 0.0;
    for (const Solver* m : members) {
      const YmSched sc = sched(m, rows);
      total += (double)sc.nstrip * (m->n[1] + sc.nchunk * kYmStart);
      longest = std::max(longest, (double)m->n[1] / sc.nchunk + kYmStart);
    }
    const double cost = std::max(total / ((double)sms * per_sm) + 0.5 * longest, longest);
    if (cost < best_cost) {
      best_cost = cost;
      best = rows;
    }
  }
  // Rows that an SM's slot marches for one tile of a tile kernel's slot (two an
  // SM): this kernel takes about 0.42 us for a row of `best_cost` (0.34 to 0.47 over
  // 100 batches), the other 3.5 to 4.3 us for a tile while its two buffers are in
  // L2 and 3.0 to 4.5 beyond (a step each).  Measured, batches of 64^2 to 768^2 (rows a tile, time of pairs over single
  // steps): below 1.1M nodes 7.5-8.4 0.88-0.96, 8.7-9.8 1.02-1.21 (4 x 448^2 0.85),
  // 10.2-14 1.10-1.43; above 7.4-8.9 0.70-0.95, 9.1-9.9 0.92-0.95, 10.1-12.6 0.97-1.09.
  long long tiles = 0;
  for (const Solver* m : members) tiles += (long long)((m->n[0] + 63) / 64) * ((m->n[1] + 7) / 8);
  const double per_tile = nodes < kYmL2Nodes ? 8.5 : 10.0;
  if (best_cost * 2 * sms > per_tile * (double)tiles) return cudaSuccess;
  std::vector<YmCav<float>> cavs(members.size());
  std::vector<YmBatchItem> items;
  for (size_t c = 0; c < members.size(); ++c) {
    Solver& m = *members[c];
    std::memcpy(&cavs[c].map[0], m.tmap_y[0], sizeof(CUtensorMap));
    std::memcpy(&cavs[c].map[1], m.tmap_y[1], sizeof(CUtensorMap));
    cavs[c].out[0] = static_cast<float*>(m.buf[1]);
    cavs[c].out[1] = static_cast<float*>(m.buf[0]);
    cavs[c].p = make_params<float>(m);
    cavs[c].kc = make_pair_constants(cavs[c].p);
    const YmSched sc = sched(&m, best);
    for (int b = 0; b < sc.nchunk; ++b)
      for (int a = 0; a < sc.nstrip; ++a)
        items.push_back(YmBatchItem{YmItem{sc.col(a, m.n[0]), sc.col(a + 1, m.n[0]),
                                           sc.row(b, m.n[1]), sc.row(b + 1, m.n[1])},
                                    (int)c});
  }
  // long items first: the short ones fill the end
  std::stable_sort(items.begin(), items.end(), [](const YmBatchItem& a, const YmBatchItem& b) {
    return a.at.yb - a.at.ya > b.at.yb - b.at.ya;
  });
  auto* g = new YmBatch();
  g->nitems = (int)items.size();
  g->mem = current_allocator();
  g->stream = stream;
  e = dev_alloc(g->mem, reinterpret_cast<void**>(&g->cavs), cavs.size() * sizeof(cavs[0]), stream);
  if (e == cudaSuccess)
    e = dev_alloc(g->mem, reinterpret_cast<void**>(&g->items), items.size() * sizeof(items[0]),
                  stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(g->cavs, cavs.data(), cavs.size() * sizeof(cavs[0]),
                        cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(g->items, items.data(), items.size() * sizeof(items[0]),
                        cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) {
    delete g;
    return e;
  }
  *out = g;
  return cudaSuccess;
}

int bounds_flag_ym(int reset) {
#ifdef ISLBM_BOUNDS_CHECK
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_bounds_flag, sizeof(int)) != cudaSuccess) return -1;
  if (reset) {
    const int zero = 0;
    cudaMemcpyToSymbol(g_bounds_flag, &zero, sizeof(int));
  }
  return v;
#else
  (void)reset;
  return 0;
#endif
}

}  // namespace islbm
