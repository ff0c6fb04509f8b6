// Pipelined persistent 2D half steps (sm_103a); the arithmetic of the tile
// kernels (tile2d.cuh) cell for cell, so the results are bitwise the same;
// one block per SM, many steps per launch (steps2d_kernel).
//
// The grid is walked in half tiles of 128 x 8 cells through a ring of two to
// four shared-memory stages (as many as fit).  For a coming half tile one
// thread issues tiled TMA tensor copies into a free stage, one box per array:
// the stencil operand with its halo, the density tile (or the tissue index),
// every streamed array, the N mechanisms of a memory variable or of a
// relaxation map in one 3D box.  They complete on the stage's mbarrier while
// the computing threads work on the current half tile in another stage, two
// cells each, so up to ~190 KB stay in flight per SM without registers or load
// instructions of the computing threads.  The updated arrays are written back
// into the stage and leave for HBM as TMA tensor stores.
//
// Boundaries: the copies read zero outside the grid (the zero-outside rule of
// the operand halo); half tiles at the edge of the grid or in a C-PML strip
// (edge half tiles) also clamp the density tile to the last cell, take the
// C-PML coefficients of each axis from its strip, and store nothing outside
// the grid (zeros in the row padding).  Periodic grids take the tile kernels.
// Every storage takes this path, the uint16 tissue index while its tables fit
// in shared memory.
#include <numeric>
#include <type_traits>

#include "async.cuh"
#include "coef.cuh"
#include "maps.cuh"
#include "tmap.h"

namespace fw2 {

namespace {

constexpr int kHT = 8;              // rows of a half tile
constexpr int kCW = kTX + 8;        // staged operand columns x0-4 .. x0+TX+3 (= kPW)
constexpr int kArr = kHT * kTX;     // floats of one streamed array per half tile


// Storage of a map form: dense maps of type MT (float, bf16 or FP16), or a
// tissue index of type IT per cell.
template <typename Maps>
struct Form;
template <typename T>
struct Form<DenseMaps<T>> {
  static constexpr bool kIdx = false;
  using MT = T;
  using IT = unsigned char;
};
template <>
struct Form<IdxMaps> {
  static constexpr bool kIdx = true;
  using MT = float;
  using IT = unsigned char;
};
template <>
struct Form<IdxMaps16> {
  static constexpr bool kIdx = true;
  using MT = float;
  using IT = unsigned short;
};
template <typename Maps>
constexpr bool kWideIdx = std::is_same<Maps, IdxMaps16>::value;
// columns of a box one cell wider than a half tile, rows of 16 bytes: the
// density (and K) box x0 .. x0+TX+3 (float) or x0+TX+7 (16 bits), the index
// box x0 .. x0+TX+15 (uint8) or x0+TX+7 (uint16)
template <typename T>
constexpr int kWide = kTX + (sizeof(T) == 1 ? 16 : sizeof(T) == 2 ? 8 : 4);
// floats that n elements of T take
template <typename T>
__host__ __device__ constexpr int floats_of(int n) { return (n * (int)sizeof(T) + 3) / 4; }

// shared-memory regions start on 128-byte boundaries (TMA destinations)
__host__ __device__ constexpr int round32(int n) { return (n + 31) & ~31; }

// The tensor maps that a 2D half step uses: both half steps' then fit in 4 KB
// of kernel parameters.
constexpr int kMaps2d = 10;
struct StepMaps {
  CUtensorMap m[kMaps2d];
  explicit StepMaps(const PipeMaps &T) {
    for (int i = 0; i < kMaps2d; ++i) m[i] = T.m[i];
  }
};

// Work of one launch: the half tiles of the grid (tiles of 128 x 8 cells,
// x fastest).
struct Region {
  int nx, ny, Lx, Ly;  // grid, boundary width (at least the halo, 4)
  int ntx, nhy;        // tiles along x, half-tile rows
  unsigned inv_ntx;    // floor(2^32 / ntx), for the division by ntx
  // Half tiles of block b of `grid`: one per round of `grid` consecutive ones,
  // rotated by `rot` blocks from round to round.  Without the rotation a
  // block meets few columns (grid and ntx share factors: 152 blocks and 16 or
  // 32 columns), and those at the x edges, whose half tiles take longer, hold
  // up the rest: 12 % of a step of 2048 x 1024 cells of the index form (when
  // the rotation came in; such a step takes 61 us now).
  int rot;
  __host__ __device__ __forceinline__ int halves() const { return ntx * nhy; }
  __device__ __forceinline__ int slot(int round, int b, int grid) const {
    return (int)((b + (unsigned)round * (unsigned)rot) % (unsigned)grid);
  }
  __device__ __forceinline__ int rounds(int b, int grid) const {
    const int full = halves() / grid;
    return full + (slot(full, b, grid) < halves() - full * grid ? 1 : 0);
  }
  __device__ __forceinline__ void half_origin(int h, int &x0, int &y0) const {
    // the product's high word is at most two below the quotient
    int q = (int)__umulhi((unsigned)h, inv_ntx), r = h - q * ntx;
    if (r >= ntx) { ++q; r -= ntx; }
    if (r >= ntx) { ++q; r -= ntx; }
    x0 = r * kTX;
    y0 = q * kHT;
  }
  // a half tile clear of the boundary rules and of the C-PML strips
  __device__ __forceinline__ bool interior(int x0, int y0) const {
    return x0 >= Lx && x0 + kTX + Lx <= nx && y0 >= Ly && y0 + kHT + Ly <= ny;
  }
};

// ---------------------------------------------------------------- stages ---
// velocity: operand p rows y0-3 .. y0+kHT+3; density box rows y0 .. y0+kHT;
// float arrays [k32][kHT][kTX]; map arrays [kM][kHT][kTX] (dense) or the
// index box rows y0 .. y0+kHT; K box (dense, literal nonlinear system)
template <int N, typename Maps>
struct VelStage {
  using F = Form<Maps>;
  static constexpr bool kIdx = F::kIdx;
  static constexpr int k32 = 2 + 2 * N;             // v_x, v_y, psi_x[N], psi_y[N]
  static constexpr int kM = kIdx ? 0 : 1 + 2 * N;   // 1/kappa1, a1[N], b1[N]
  static constexpr int kPb = (kHT + 7) * kCW;                       // operand box
  static constexpr int kRb = (kHT + 1) * kWide<typename F::MT>;     // density box (elements)
  static constexpr int kIb = (kHT + 1) * kWide<typename F::IT>;     // index box (elements)
  static constexpr int kP = round32(kPb);
  static constexpr int kR = kIdx ? 0 : round32(floats_of<typename F::MT>(kRb));  // the index form looks it up
  static constexpr int oM = k32 * kArr;                             // maps, from the float arrays
  static constexpr int kS = oM + floats_of<typename F::MT>(kM * kArr);
  static constexpr int kI = kIdx ? floats_of<typename F::IT>(kIb) : 0;
  static constexpr int kK = kIdx ? 0 : kR;
  static constexpr int kFloats = round32(kP + kR + kS + kI + kK);
};

// pressure: v_x rows y0-1 .. y0+kHT, v_y rows y0-4 .. y0+kHT+2; float arrays;
// map arrays or the index of the half tile
template <int N, typename Maps>
struct PrsStage {
  using F = Form<Maps>;
  static constexpr bool kIdx = F::kIdx;
  static constexpr int k32 = 1 + 2 * N;             // p, psi_x[N], psi_y[N]
  static constexpr int kM = kIdx ? 0 : 3 + 2 * N;   // 1/kappa2, K, chi, a2[N], b2[N]
  static constexpr int kXb = (kHT + 2) * kCW;
  static constexpr int kYb = (kHT + 7) * kCW;
  static constexpr int kX = round32(kXb);
  static constexpr int kY = round32(kYb);
  static constexpr int oM = k32 * kArr;
  static constexpr int kS = oM + floats_of<typename F::MT>(kM * kArr);
  static constexpr int kI = kIdx ? floats_of<typename F::IT>(kArr) : 0;
  static constexpr int kFloats = round32(kX + kY + kS + kI);
};

// Bytes one stage receives through the tensor maps (the chi box only with
// the nonlinear term, the velocity's K box only with the literal system).
template <int N, typename Maps, bool VEL>
__host__ __device__ constexpr unsigned stage_bytes(bool nl, bool nl_vel) {
  using MT = typename Form<Maps>::MT;
  using IT = typename Form<Maps>::IT;
  if (VEL) {
    using S = VelStage<N, Maps>;
    return 4u * (S::kPb + S::k32 * kArr) + (S::kIdx ? (unsigned)sizeof(IT) * S::kIb
                                                    : (unsigned)sizeof(MT) * (S::kM * kArr + (nl_vel ? 2 : 1) * S::kRb));
  } else {
    using S = PrsStage<N, Maps>;
    return 4u * (S::kXb + S::kYb + S::k32 * kArr) +
           (S::kIdx ? (unsigned)sizeof(IT) * kArr : (unsigned)sizeof(MT) * kArr * (S::kM - (nl ? 0 : 1)));
  }
}

// The tensor copies of one half tile into a stage, in two parts (one thread,
// which also announces the stage's bytes on the stage's mbarrier).  The first
// part holds what only this half tile's own block writes (the updated arrays)
// and the maps; the second the stencil operand, which the neighbouring half
// tiles of the previous half step wrote.  Boxes may reach outside the grid:
// those cells read as zero.
template <int N, typename Maps, bool VEL, typename TM>
__device__ __forceinline__ void issue_own(const StepParams &P, const TM &T, float *st, uint64_t *bar, int x0,
                                          int y0) {
  fence_proxy_async_smem();
  if (VEL) {
    using S = VelStage<N, Maps>;
    constexpr int kMf = floats_of<typename Form<Maps>::MT>(kArr);  // floats of one map array
    if (!S::kIdx) tma_load_2d(st + S::kP, &T.m[1], x0, y0, bar);
    float *ss = st + S::kP + S::kR, *sm = ss + S::oM;
    tma_load_2d(ss, &T.m[2], x0, y0, bar);
    tma_load_2d(ss + kArr, &T.m[3], x0, y0, bar);
    if (N > 0) {
      tma_load_3d(ss + 2 * kArr, &T.m[4], x0, y0, 0, bar);
      tma_load_3d(ss + (2 + N) * kArr, &T.m[5], x0, y0, 0, bar);
    }
    if (!S::kIdx) {
      tma_load_2d(sm, &T.m[6], x0, y0, bar);
      if (N > 0) {
        tma_load_3d(sm + kMf, &T.m[7], x0, y0, 0, bar);
        tma_load_3d(sm + (1 + N) * kMf, &T.m[8], x0, y0, 0, bar);
      }
      if (P.nl_vel) tma_load_2d(ss + S::kS, &T.m[9], x0, y0, bar);  // K, density-box shape
    } else {
      tma_load_2d(ss + S::kS, &T.m[1], x0, y0, bar);  // tissue index
    }
  } else {
    using S = PrsStage<N, Maps>;
    constexpr int kMf = floats_of<typename Form<Maps>::MT>(kArr);
    float *ss = st + S::kX + S::kY, *sm = ss + S::oM;
    tma_load_2d(ss, &T.m[2], x0, y0, bar);
    if (N > 0) {
      tma_load_3d(ss + kArr, &T.m[3], x0, y0, 0, bar);
      tma_load_3d(ss + (1 + N) * kArr, &T.m[4], x0, y0, 0, bar);
    }
    if (!S::kIdx) {
      tma_load_2d(sm, &T.m[5], x0, y0, bar);
      tma_load_2d(sm + kMf, &T.m[6], x0, y0, bar);
      if (P.nl) tma_load_2d(sm + 2 * kMf, &T.m[7], x0, y0, bar);
      if (N > 0) {
        tma_load_3d(sm + 3 * kMf, &T.m[8], x0, y0, 0, bar);
        tma_load_3d(sm + (3 + N) * kMf, &T.m[9], x0, y0, 0, bar);
      }
    } else {
      tma_load_2d(ss + S::kS, &T.m[5], x0, y0, bar);  // tissue index
    }
  }
}
template <int N, typename Maps, bool VEL, typename TM>
__device__ __forceinline__ void issue_operand(const TM &T, float *st, uint64_t *bar, int x0, int y0) {
  if (VEL) {
    tma_load_2d(st, &T.m[0], x0 - 4, y0 - 3, bar);
  } else {
    tma_load_2d(st, &T.m[0], x0 - 4, y0 - 1, bar);
    tma_load_2d(st + PrsStage<N, Maps>::kX, &T.m[1], x0 - 4, y0 - 4, bar);
  }
}
template <int N, typename Maps, bool VEL, typename TM>
__device__ __forceinline__ void issue_stage(const StepParams &P, const TM &T, float *st, uint64_t *bar,
                                            int x0, int y0) {
  mbar_arrive_expect_tx(bar, stage_bytes<N, Maps, VEL>(P.nl != 0, P.nl_vel != 0));
  issue_own<N, Maps, VEL>(P, T, st, bar, x0, y0);
  issue_operand<N, Maps, VEL>(T, st, bar, x0, y0);
}

// Store the updated arrays of a half tile from its stage (one thread, after
// every thread's fence and a barrier): velocity v_x, v_y, psi1_x, psi1_y;
// pressure p, psi2_x, psi2_y.  The copies write nothing outside the grid.
template <int N, typename Maps, bool VEL, typename TM>
__device__ __forceinline__ void store_stage(const TM &T, const float *st, int x0, int y0) {
  if (VEL) {
    using S = VelStage<N, Maps>;
    const float *ss = st + S::kP + S::kR;
    tma_store_2d(&T.m[2], x0, y0, ss);
    tma_store_2d(&T.m[3], x0, y0, ss + kArr);
    if (N > 0) {
      tma_store_3d(&T.m[4], x0, y0, 0, ss + 2 * kArr);
      tma_store_3d(&T.m[5], x0, y0, 0, ss + (2 + N) * kArr);
    }
  } else {
    using S = PrsStage<N, Maps>;
    const float *ss = st + S::kX + S::kY;
    tma_store_2d(&T.m[2], x0, y0, ss);
    if (N > 0) {
      tma_store_3d(&T.m[3], x0, y0, 0, ss + kArr);
      tma_store_3d(&T.m[4], x0, y0, 0, ss + (1 + N) * kArr);
    }
  }
  bulk_commit();
}

// ------------------------------------------------------------ compute ---
// 512 threads per block, two consecutive x cells each: thread t of row ly
// (64 threads per row) owns cells x0 + 2t, x0 + 2t + 1.  Every cell sees the
// operations of the tile path in the same order, so results are bitwise the
// same.
constexpr int kThreads = 512;
constexpr int kStepThreads = kThreads + 32;  // and the warp that copies and stores (steps2d_kernel)

__device__ __forceinline__ float2 sld2(const float *s) { return *reinterpret_cast<const float2 *>(s); }
// One result pair of array `a` of the stage: results leave through the stage
// and TMA tensor stores (fewer store instructions than per-thread stores; the
// store of a unit overlaps the compute of the next).
__device__ __forceinline__ void put2(float *own, int a, float2 v) { *reinterpret_cast<float2 *>(own + a * kArr) = v; }
__device__ __forceinline__ float &el2(float2 &v, int e) { return e == 0 ? v.x : v.y; }
// ten consecutive shared-memory values from column c of a row (c even)
struct Win10 {
  float v[10];
};
__device__ __forceinline__ Win10 win10(const float *row, int c) {
  Win10 w;
  const float2 *r2 = reinterpret_cast<const float2 *>(row + c);
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const float2 t = r2[i];
    w.v[2 * i] = t.x;
    w.v[2 * i + 1] = t.y;
  }
  return w;
}

// x and y derivatives of the staged p at the faces of cells x0+lx, x0+lx+1
// (operand rows y0-3.., columns x0-4..; cell e sits at column lx + 4 + e)
__device__ __forceinline__ void vel_derivs2(const StepParams &P, const float *sp, int sy, int lx, float2 &Dx,
                                            float2 &Dy) {
  const Win10 w = win10(sp + sy * kCW, lx);  // columns lx .. lx+9
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    float d = 0.f;
#pragma unroll
    for (int m = 1; m <= 4; ++m) d = fmaf(P.gh[m - 1], w.v[4 + e + m] - w.v[4 + e - m + 1], d);
    el2(Dx, e) = d;
  }
  float2 col[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) col[m] = sld2(sp + (sy - 3 + m) * kCW + lx + 4);
  Dy = make_float2(0.f, 0.f);
#pragma unroll
  for (int m = 1; m <= 4; ++m) Dy = fma2(dup2(P.gh[m - 1]), sub2(col[3 + m], col[4 - m]), Dy);
  if (P.g11h != 0.f) {
    const Win10 up = win10(sp + (sy + 1) * kCW, lx), dn = win10(sp + (sy - 1) * kCW, lx);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      el2(Dx, e) += P.g11h * ((up.v[5 + e] - up.v[4 + e]) + (dn.v[5 + e] - dn.v[4 + e]));
      el2(Dy, e) += P.g11h * ((up.v[5 + e] - w.v[5 + e]) + (up.v[3 + e] - w.v[3 + e]));
    }
  }
}

// x and y derivatives of v_x (rows y0-1..), v_y (rows y0-4..) at the centres
__device__ __forceinline__ void prs_derivs2(const StepParams &P, const float *svx, const float *svy, int ly,
                                            int lx, float2 &Dx, float2 &Dy) {
  const Win10 w = win10(svx + (ly + 1) * kCW, lx);
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    float d = 0.f;
#pragma unroll
    for (int m = 1; m <= 4; ++m) d = fmaf(P.gh[m - 1], w.v[4 + e + m - 1] - w.v[4 + e - m], d);
    el2(Dx, e) = d;
  }
  float2 col[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) col[m] = sld2(svy + (ly + m) * kCW + lx + 4);
  Dy = make_float2(0.f, 0.f);
#pragma unroll
  for (int m = 1; m <= 4; ++m) Dy = fma2(dup2(P.gh[m - 1]), sub2(col[4 + m - 1], col[4 - m]), Dy);
  if (P.g11h != 0.f) {
    const Win10 up = win10(svx + (ly + 2) * kCW, lx), dn = win10(svx + ly * kCW, lx);
    const Win10 y0w = win10(svy + (ly + 4) * kCW, lx), y1w = win10(svy + (ly + 3) * kCW, lx);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      el2(Dx, e) += P.g11h * ((up.v[4 + e] - up.v[3 + e]) + (dn.v[4 + e] - dn.v[3 + e]));
      el2(Dy, e) += P.g11h * ((y0w.v[5 + e] - y1w.v[5 + e]) + (y0w.v[3 + e] - y1w.v[3 + e]));
    }
  }
}

// Per-tissue tables of the index forms in shared memory: fields K, rho, chi,
// 1/kappa1, 1/kappa2, then a1, b1, a2, b2 of the mechanisms (kSlots each),
// kStride entries per field.  uint8: the global table as it is.  uint16: the
// fields of the context's N mechanisms only, tab_stride entries each, while
// they fit next to two stages.
template <int N, typename Maps>
struct Table {
  static constexpr int kSlots = kWideIdx<Maps> ? N : kTabSlots;
  const float *t;
  int stride;
  __device__ __forceinline__ Table(const StepParams &P, const float *tab)
      : t(tab), stride(kWideIdx<Maps> ? P.tab_stride : kTissues) {}
  // field id: kTabK .. kTabIk2, or the relaxation field `group` (a1, b1, a2,
  // b2) of mechanism nu
  __device__ __forceinline__ const float *field(int f) const { return t + f * stride; }
  __device__ __forceinline__ const float *relax(int group, int nu) const {
    return t + (kTabRelax + group * kSlots + nu) * stride;
  }
};
template <typename IT>
__device__ __forceinline__ float2 look2(const float *field, const IT *cells) {
  if constexpr (sizeof(IT) == 1) {
    const uchar2 c = *reinterpret_cast<const uchar2 *>(cells);
    return make_float2(field[c.x], field[c.y]);
  } else {
    const ushort2 c = *reinterpret_cast<const ushort2 *>(cells);
    return make_float2(field[c.x], field[c.y]);
  }
}
// the table of the index forms into shared memory (all threads)
template <int N, typename Maps>
__device__ __forceinline__ void stage_table(const StepParams &P, float *tab, int tid) {
  if constexpr (kWideIdx<Maps>) {
    const int S4 = P.tab_stride / 4;
    float4 *dst = reinterpret_cast<float4 *>(tab);
    for (int f = 0; f < kTabRelax + 4 * N; ++f) {
      const int r = f - kTabRelax, g = f < kTabRelax ? f : kTabRelax + (N ? r / N * kTabSlots + r % N : 0);
      const float4 *src = reinterpret_cast<const float4 *>(P.table + (long long)g * P.tab_stride);
      for (int t = tid; t < S4; t += kThreads) dst[f * S4 + t] = __ldg(src + t);
    }
  } else if constexpr (Form<Maps>::kIdx) {
    const float4 *src = reinterpret_cast<const float4 *>(P.table);
    float4 *dst = reinterpret_cast<float4 *>(tab);
    for (int t = tid; t < kTableFields * kTissues / 4; t += kThreads) dst[t] = __ldg(src + t);
  }
}

// Pair of staged map values (16-bit maps: FP16 times the map's scale) and of
// decay factors (16-bit maps hold 1 - b): the tile path's loads.
__device__ __forceinline__ float2 ldm2(const float *m, float) { return sld2(m); }
__device__ __forceinline__ float2 ldm2(const __nv_bfloat16 *m, float) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(m));
}
__device__ __forceinline__ float2 ldm2(const __half *m, float sc) {
  const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(m));
  return make_float2(v.x * sc, v.y * sc);
}
__device__ __forceinline__ float2 ldbm2(const float *m, float) { return sld2(m); }
template <typename MT>
__device__ __forceinline__ float2 ldbm2(const MT *m, float sc) {
  const float2 v = ldm2(m, sc);
  return make_float2(1.f - v.x, 1.f - v.y);
}
__device__ __forceinline__ float ldm1(const float *m, float) { return *m; }
__device__ __forceinline__ float ldm1(const __nv_bfloat16 *m, float) { return __bfloat162float(*m); }
__device__ __forceinline__ float ldm1(const __half *m, float sc) { return __half2float(*m) * sc; }
// the same pairs of C-PML strip values in global memory (aligned pairs)
__device__ __forceinline__ float2 ldg2(const float *m) { return __ldg(reinterpret_cast<const float2 *>(m)); }
__device__ __forceinline__ float2 lds2(const float *m, float) { return ldg2(m); }
__device__ __forceinline__ float2 ldsb2(const float *m, float) { return ldg2(m); }
template <typename MT>
__device__ __forceinline__ float2 lds2(const MT *m, float sc) {
  const unsigned u = __ldg(reinterpret_cast<const unsigned *>(m));
  return ldm2(reinterpret_cast<const MT *>(&u), sc);
}
template <typename MT>
__device__ __forceinline__ float2 ldsb2(const MT *m, float sc) {
  const float2 v = lds2(m, sc);
  return make_float2(1.f - v.x, 1.f - v.y);
}

// Densities at the faces of a pair, read where the thread needs them: cells
// (lx, ly), (lx + 1, ly), (lx + 2, ly), (lx, ly + 1), (lx + 1, ly + 1) of the
// half tile.  Cells beyond the last one along an axis take that cell's value
// (rho_coord of the tile path).  Dense maps read the staged density box; the
// index form looks the staged index up in the table.
struct FaceRho {
  float r0, r1, r2, u0, u1;  // row ly: lx .. lx+2; row ly+1: lx, lx+1
};
template <int N, typename Maps, bool EDGE>
__device__ __forceinline__ FaceRho face_rho(const StepParams &P, const Table<N, Maps> &tab,
                                            const typename Form<Maps>::MT *sr, const typename Form<Maps>::IT *si,
                                            int x0, int y0, int lx, int ly) {
  int c0 = lx, c1 = lx + 1, c2 = lx + 2, r0 = ly, r1 = ly + 1;
  if (EDGE) {
    const int mx = P.nx - 1 - x0, my = P.ny - 1 - y0;  // last cell inside, tile coordinates
    c0 = min(c0, mx);
    c1 = min(c1, mx);
    c2 = min(c2, mx);
    r0 = min(r0, my);
    r1 = min(r1, my);
  }
  auto at = [&](int r, int cc) -> float {
    if constexpr (Form<Maps>::kIdx) return tab.field(kTabRho)[si[r * kWide<typename Form<Maps>::IT> + cc]];
    else return ldm1(sr + r * kWide<typename Form<Maps>::MT> + cc, P.ms[kMsRho]);
  };
  return FaceRho{at(r0, c0), at(r0, c1), at(r0, c2), at(r1, c0), at(r1, c1)};
}

// Momentum factors of the literal nonlinear system (Eq. general5) at the x
// and y faces of the pair: p from the staged operand (cell e at column
// lx + 4 + e of row sy; zero beyond the grid), K from the staged K box (dense
// maps; the density box's shape) or the staged index (index forms),
// neighbours clamped to the last cell.
template <int N, typename Maps, bool EDGE>
__device__ __forceinline__ void mom_factors2(const StepParams &P, const Table<N, Maps> &tab,
                                             const typename Form<Maps>::IT *si, const typename Form<Maps>::MT *sk,
                                             const float *sp, int sy, int lx, int ly, int x0, int y0, float2 &fx,
                                             float2 &fy) {
  const float *row = sp + sy * kCW + lx + 4, *up = sp + (sy + 1) * kCW + lx + 4;
  const int mx = P.nx - 1 - x0, my = P.ny - 1 - y0;
  const int r1 = EDGE ? min(ly + 1, my) : ly + 1;
  auto K = [&](int r, int cc) -> float {
    if constexpr (Form<Maps>::kIdx) return tab.field(kTabK)[si[r * kWide<typename Form<Maps>::IT> + cc]];
    else return ldm1(sk + r * kWide<typename Form<Maps>::MT> + cc, P.ms[kMsK]);
  };
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int c0 = EDGE ? min(lx + e, mx) : lx + e, c1 = EDGE ? min(lx + e + 1, mx) : lx + e + 1;
    const float Kc = K(ly, c0), Kx = K(ly, c1), Ky = K(r1, c0);
    el2(fx, e) = mom_factor(Kc, Kx, row[e], row[e + 1]);
    el2(fy, e) = mom_factor(Kc, Ky, row[e], up[e]);
  }
}

// a, b of mechanism nu along x at the two cells of an edge pair: from the x
// strip inside its C-PML region, else unchanged (coef_edge of the tile path;
// its zero beyond the grid only reaches cells that are masked)
template <int OP, typename Maps>
__device__ __forceinline__ void x_strip_coef2(const StepParams &P, int nu, int i0, int j, float2 &a, float2 &b) {
  using ST = typename Maps::StripT;
  const int L = P.L[0];
  if (!(L > 0 && (i0 < L || i0 + 1 >= P.nx - L))) return;
  const ST *sa = static_cast<const ST *>(OP == 1 ? P.sa1[0] : P.sa2[0]);
  const ST *sb = static_cast<const ST *>(OP == 1 ? P.sb1[0] : P.sb2[0]);
  const float s_a = P.ms[(OP == 1 ? kMsA1 : kMsA2) + nu], s_b = P.ms[(OP == 1 ? kMsB1 : kMsB2) + nu];
  const long long row = (long long)nu * P.strip_nu[0] + (long long)j * (2 * L);
  // both cells on one side of the strip: one aligned pair (i0 and the high
  // side's offset nx - 2L are even)
  int sc0 = -1;
  if (i0 + 1 < L) sc0 = i0;
  else if (i0 >= P.nx - L && i0 + 1 < P.nx && ((P.nx - 2 * L) & 1) == 0) sc0 = i0 - (P.nx - 2 * L);
  if (sc0 >= 0) {
    a = lds2(sa + row + sc0, s_a);
    b = ldsb2(sb + row + sc0, s_b);
    return;
  }
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int x = i0 + e;
    if (x >= P.nx) {
      el2(a, e) = 0.f;
      el2(b, e) = 0.f;
    } else {
      const int sc = strip_coord(x, P.nx, L);
      if (sc >= 0) {
        el2(a, e) = ldmap(sa, row + sc, s_a);
        el2(b, e) = ldb(sb, row + sc, s_b);
      }
    }
  }
}

// a, b along y at the two cells of an edge pair inside the y strip (an
// aligned pair: i0 even, pitch a multiple of 16)
template <int OP, typename Maps>
__device__ __forceinline__ void y_strip_coef2(const StepParams &P, int nu, int i0, int sc, float2 &a, float2 &b) {
  using ST = typename Maps::StripT;
  const ST *sa = static_cast<const ST *>(OP == 1 ? P.sa1[1] : P.sa2[1]);
  const ST *sb = static_cast<const ST *>(OP == 1 ? P.sb1[1] : P.sb2[1]);
  const long long off = (long long)nu * P.strip_nu[1] + (long long)sc * P.pitch + i0;
  a = lds2(sa + off, P.ms[(OP == 1 ? kMsA1 : kMsA2) + nu]);
  b = ldsb2(sb + off, P.ms[(OP == 1 ? kMsB1 : kMsB2) + nu]);
}

// C-PML coefficients of a pair of an edge half tile, every mechanism: the
// values of the x strip where bit e of `x` is set (zero beyond the grid: those
// cells are masked), those of the y strip where `y` is.  They depend on the
// position alone, so they are loaded before the half tile's copies are waited
// for.
template <int N>
struct EdgeCoef {
  float2 xa[N > 0 ? N : 1], xb[N > 0 ? N : 1], ya[N > 0 ? N : 1], yb[N > 0 ? N : 1];
  unsigned x;
  bool y;
};
template <int N, int OP, typename Maps>
__device__ __forceinline__ void load_edge(const StepParams &P, int x0, int y0, int tid, EdgeCoef<N> &c) {
  c.x = 0;
  c.y = false;
  const int i0 = x0 + 2 * (tid & 63), j = y0 + (tid >> 6), L = P.L[0];
  if (N == 0 || i0 >= P.nx || j >= P.ny) return;
  if (L > 0 && (i0 < L || i0 + 1 >= P.nx - L)) {
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (i0 + e >= P.nx || strip_coord(i0 + e, P.nx, L) >= 0) c.x |= 1u << e;
#pragma unroll
    for (int nu = 0; nu < N; ++nu) {
      c.xa[nu] = c.xb[nu] = make_float2(0.f, 0.f);
      x_strip_coef2<OP, Maps>(P, nu, i0, j, c.xa[nu], c.xb[nu]);
    }
  }
  const int sc = strip_coord(j, P.ny, P.L[1]);
  if (sc >= 0) {
    c.y = true;
#pragma unroll
    for (int nu = 0; nu < N; ++nu) y_strip_coef2<OP, Maps>(P, nu, i0, sc, c.ya[nu], c.yb[nu]);
  }
}
// the coefficients of mechanism nu along x and y: a, b of the cells, or the strips'
template <int N>
__device__ __forceinline__ void pick_edge(const EdgeCoef<N> &c, int nu, float2 a, float2 b, float2 &ax, float2 &bx,
                                          float2 &ay, float2 &by) {
  ax = make_float2((c.x & 1u) ? c.xa[nu].x : a.x, (c.x & 2u) ? c.xa[nu].y : a.y);
  bx = make_float2((c.x & 1u) ? c.xb[nu].x : b.x, (c.x & 2u) ? c.xb[nu].y : b.y);
  ay = c.y ? c.ya[nu] : a;
  by = c.y ? c.yb[nu] : b;
}

// Prefetch into L2 the C-PML strip rows an edge half tile will read (warp 0,
// when its copies are issued): otherwise they come straight from DRAM while
// the half tile computes.  OP: 1 velocity (a1, b1), 2 pressure (a2, b2).
__device__ __forceinline__ void l2_line(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
template <int N, int OP, typename ST>
__device__ __forceinline__ void prefetch_strips2(const StepParams &P, int x0, int y0, int lane) {
  if constexpr (N > 0) {
    constexpr int kLine = 128 / (int)sizeof(ST);  // elements of a 128-byte line
    const ST *sa[2], *sb[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      sa[q] = static_cast<const ST *>(OP == 1 ? P.sa1[q] : P.sa2[q]);
      sb[q] = static_cast<const ST *>(OP == 1 ? P.sb1[q] : P.sb2[q]);
    }
    const int Lx = P.L[0];
    if (Lx > 0 && (x0 < Lx || x0 + kTX > P.nx - Lx)) {
      for (int t = lane; t < kHT * N * 2; t += 32) {
        const int r = t % kHT, nu = (t / kHT) % N, ab = t / (kHT * N);
        const int y = y0 + r;
        if (y >= P.ny) continue;
        const ST *b = (ab ? sb[0] : sa[0]) + nu * P.strip_nu[0] + (long long)y * (2 * Lx);
        for (int o = 0; o < 2 * Lx; o += kLine) l2_line(b + o);
      }
    }
    const int Ly = P.L[1];
    if (Ly > 0) {
      for (int t = lane; t < kHT * N * 2; t += 32) {
        const int r = t % kHT, nu = (t / kHT) % N, ab = t / (kHT * N);
        const int y = y0 + r;
        const int sc = y < P.ny ? strip_coord(y, P.ny, Ly) : -1;
        if (sc < 0) continue;
        const ST *b = (ab ? sb[1] : sa[1]) + nu * P.strip_nu[1] + (long long)sc * P.pitch + x0;
        for (int o = 0; o < kTX && x0 + o < P.nx; o += kLine) l2_line(b + o);
      }
    }
  }
}

template <int N, typename Maps, bool EDGE>
__device__ __forceinline__ void vel_compute(const StepParams &P, const float *tab, float *st, int x0, int y0,
                                            int tid, const EdgeCoef<N> &edge) {
  using S = VelStage<N, Maps>;
  using MT = typename S::F::MT;
  using IT = typename S::F::IT;
  const Table<N, Maps> T(P, tab);
  const float *sp = st;
  const MT *sr = reinterpret_cast<const MT *>(st + S::kP);
  const float *ss = st + S::kP + S::kR;
  const IT *si = reinterpret_cast<const IT *>(ss + S::kS);
  const int t2 = tid & 63, ly = tid >> 6, lx = 2 * t2;
  const int i0 = x0 + lx, j = y0 + ly;
  if (EDGE && (i0 >= P.nx || j >= P.ny)) return;
  float *own = const_cast<float *>(ss) + ly * kTX + lx;
  float2 Dx, Dy;
  vel_derivs2(P, sp, ly + 3, lx, Dx, Dy);
  float2 k1, A[N > 0 ? N : 1], B[N > 0 ? N : 1];
  if constexpr (S::kIdx) {
    const IT *cell = si + ly * kWide<IT> + lx;
    k1 = look2(T.field(kTabIk1), cell);
#pragma unroll
    for (int nu = 0; nu < N; ++nu) {
      A[nu] = look2(T.relax(0, nu), cell);
      B[nu] = look2(T.relax(1, nu), cell);
    }
  } else {
    const MT *mp = reinterpret_cast<const MT *>(ss + S::oM) + ly * kTX + lx;
    k1 = ldm2(mp, P.ms[kMsIk1]);
#pragma unroll
    for (int nu = 0; nu < N; ++nu) {
      A[nu] = ldm2(mp + (1 + nu) * kArr, P.ms[kMsA1 + nu]);
      B[nu] = ldbm2(mp + (1 + N + nu) * kArr, P.ms[kMsB1 + nu]);
    }
  }
  // per-axis coefficients: in an edge pair the C-PML strips replace them
  float2 AX[N > 0 ? N : 1], BX[N > 0 ? N : 1], AY[N > 0 ? N : 1], BY[N > 0 ? N : 1];
#pragma unroll
  for (int nu = 0; nu < N; ++nu) {
    if (EDGE) {
      pick_edge<N>(edge, nu, A[nu], B[nu], AX[nu], BX[nu], AY[nu], BY[nu]);
    } else {
      AX[nu] = A[nu]; BX[nu] = B[nu]; AY[nu] = A[nu]; BY[nu] = B[nu];
    }
  }
  float2 vx = sld2(own), vy = sld2(own + kArr);
  const float2 wn = dup2(P.w_new), wo = dup2(P.w_old);
  float2 Sx = mul2(Dx, k1), Sy = mul2(Dy, k1);
#pragma unroll
  for (int nu = 0; nu < N; ++nu) {
    const float2 px = sld2(own + (2 + nu) * kArr), py = sld2(own + (2 + N + nu) * kArr);
    const float2 nx_ = fma2(BX[nu], px, mul2(AX[nu], Dx)), ny_ = fma2(BY[nu], py, mul2(AY[nu], Dy));
    const float2 tx = fma2(wn, nx_, mul2(wo, px)), ty = fma2(wn, ny_, mul2(wo, py));
    Sx = add2(Sx, tx);
    Sy = add2(Sy, ty);
    put2(own, 2 + nu, nx_);
    put2(own, 2 + N + nu, ny_);
  }
  const FaceRho fr = face_rho<N, Maps, EDGE>(P, T, sr, si, x0, y0, lx, ly);
  if (P.nl_vel) {
    float2 fx, fy;
    mom_factors2<N, Maps, EDGE>(P, T, si, reinterpret_cast<const MT *>(ss + S::kS), sp, ly + 3, lx, ly, x0, y0, fx, fy);
    vx.x = vel_upd(vx.x, qdiv(P.two_dt, fr.r0 + fr.r1), Sx.x, fx.x);
    vx.y = vel_upd(vx.y, qdiv(P.two_dt, fr.r1 + fr.r2), Sx.y, fx.y);
    vy.x = vel_upd(vy.x, qdiv(P.two_dt, fr.r0 + fr.u0), Sy.x, fy.x);
    vy.y = vel_upd(vy.y, qdiv(P.two_dt, fr.r1 + fr.u1), Sy.y, fy.y);
  } else {
    vx.x = vel_upd(vx.x, qdiv(P.two_dt, fr.r0 + fr.r1), Sx.x);
    vx.y = vel_upd(vx.y, qdiv(P.two_dt, fr.r1 + fr.r2), Sx.y);
    vy.x = vel_upd(vy.x, qdiv(P.two_dt, fr.r0 + fr.u0), Sy.x);
    vy.y = vel_upd(vy.y, qdiv(P.two_dt, fr.r1 + fr.u1), Sy.y);
  }
  put2(own, 0, vx);
  put2(own, 1, vy);
}

template <int N, typename Maps, bool EDGE>
__device__ __forceinline__ void prs_compute(const StepParams &P, const float *tab, float *st, int x0, int y0,
                                            int tid, const EdgeCoef<N> &edge) {
  using S = PrsStage<N, Maps>;
  using MT = typename S::F::MT;
  using IT = typename S::F::IT;
  const Table<N, Maps> T(P, tab);
  const float *sx = st, *sy = st + S::kX;
  float *ss = st + S::kX + S::kY;
  const int t2 = tid & 63, ly = tid >> 6, lx = 2 * t2;
  const int i0 = x0 + lx, j = y0 + ly;
  if (EDGE && (i0 >= P.nx || j >= P.ny)) return;
  float *own = ss + ly * kTX + lx;
  float2 Dx, Dy;
  prs_derivs2(P, sx, sy, ly, lx, Dx, Dy);
  float2 k2, K, ch = make_float2(0.f, 0.f), A[N > 0 ? N : 1], B[N > 0 ? N : 1];
  if constexpr (S::kIdx) {
    const IT *cell = reinterpret_cast<const IT *>(ss + S::kS) + ly * kTX + lx;
    k2 = look2(T.field(kTabIk2), cell);
    K = look2(T.field(kTabK), cell);
    if (P.nl) ch = look2(T.field(kTabChi), cell);
#pragma unroll
    for (int nu = 0; nu < N; ++nu) {
      A[nu] = look2(T.relax(2, nu), cell);
      B[nu] = look2(T.relax(3, nu), cell);
    }
  } else {
    const MT *mp = reinterpret_cast<const MT *>(ss + S::oM) + ly * kTX + lx;
    k2 = ldm2(mp, P.ms[kMsIk2]);
    K = ldm2(mp + kArr, P.ms[kMsK]);
    if (P.nl) ch = ldm2(mp + 2 * kArr, P.ms[kMsChi]);
#pragma unroll
    for (int nu = 0; nu < N; ++nu) {
      A[nu] = ldm2(mp + (3 + nu) * kArr, P.ms[kMsA2 + nu]);
      B[nu] = ldbm2(mp + (3 + N + nu) * kArr, P.ms[kMsB2 + nu]);
    }
  }
  // per-axis coefficients: in an edge pair the C-PML strips replace them
  float2 AX[N > 0 ? N : 1], BX[N > 0 ? N : 1], AY[N > 0 ? N : 1], BY[N > 0 ? N : 1];
#pragma unroll
  for (int nu = 0; nu < N; ++nu) {
    if (EDGE) {
      pick_edge<N>(edge, nu, A[nu], B[nu], AX[nu], BX[nu], AY[nu], BY[nu]);
    } else {
      AX[nu] = A[nu]; BX[nu] = B[nu]; AY[nu] = A[nu]; BY[nu] = B[nu];
    }
  }
  float2 p = sld2(own);
  const float2 wn = dup2(P.w_new), wo = dup2(P.w_old);
  float2 Sx = mul2(Dx, k2), Sy = mul2(Dy, k2);
#pragma unroll
  for (int nu = 0; nu < N; ++nu) {
    const float2 px = sld2(own + (1 + nu) * kArr), py = sld2(own + (1 + N + nu) * kArr);
    const float2 nx_ = fma2(BX[nu], px, mul2(AX[nu], Dx)), ny_ = fma2(BY[nu], py, mul2(AY[nu], Dy));
    const float2 tx = fma2(wn, nx_, mul2(wo, px)), ty = fma2(wn, ny_, mul2(wo, py));
    Sx = add2(Sx, tx);
    Sy = add2(Sy, ty);
    put2(own, 1 + nu, nx_);
    put2(own, 1 + N + nu, ny_);
  }
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    float upd = P.dt * el2(K, e) * (el2(Sx, e) + el2(Sy, e));
    if (P.nl) upd = qdiv(upd, fmaf(el2(ch, e), el2(p, e), 1.f));
    el2(p, e) -= upd;
  }
  put2(own, 0, p);
}

// Ring of stages: as many as fit next to the maps' table (2 .. 4).
template <int N, typename Maps, bool VEL>
struct Ring {
  static constexpr int kStage = VEL ? VelStage<N, Maps>::kFloats : PrsStage<N, Maps>::kFloats;
  static constexpr int kBudget = (224 * 1024 - 128) / 4 - Maps::kSmemFloats;  // floats
  static constexpr int kFit = kBudget / kStage;
  static constexpr int kStages = kFit > 4 ? 4 : kFit;
  // With four stages a stage is refilled one unit after its results were
  // stored (the store has read it by then: no wait on it), two units ahead
  // of its compute; with two or three, right after its store, kStages - 1
  // units ahead.
  static constexpr int kLag = kStages >= 4 ? 1 : 0;
  static constexpr int kAhead = kStages - 1 - kLag;
  static constexpr size_t kBytes = sizeof(float) * ((size_t)kStages * kStage + Maps::kSmemFloats) + 128;
  static_assert(kStages >= 2, "two stages must fit in shared memory");
  static_assert(kBytes + 1024 <= 227 * 1024, "stages and table leave 1 KB for static shared memory");
};

// Ring of the multi-step kernel: stages that hold either half step's half
// tile, as many as fit (2 .. 4).
template <int N, typename Maps>
struct StepRing {
  static constexpr int kV = VelStage<N, Maps>::kFloats, kP = PrsStage<N, Maps>::kFloats;
  static constexpr int kStage = kV > kP ? kV : kP;
  static constexpr int kTotal = (224 * 1024 - 128) / 4;  // floats
  // the uint16 form's table takes what two stages leave
  static constexpr int kTab = kWideIdx<Maps> ? kTotal - 2 * kStage : Maps::kSmemFloats;
  static constexpr int kFit = (kTotal - kTab) / kStage;
  static constexpr int kStages = kFit > 4 ? 4 : kFit;
  static constexpr size_t kBytes = sizeof(float) * ((size_t)kStages * kStage + kTab) + 128;
  static_assert(kStages >= 2, "two stages must fit in shared memory");
  static_assert(kBytes + 1024 <= 227 * 1024, "stages and table leave 1 KB for static shared memory");
};
// largest table stride of the uint16 index form whose fields fit (about 1480
// tissues with four mechanisms)
template <int N>
constexpr int kWideTissues = StepRing<N, IdxMaps16>::kTab / (kTabRelax + 4 * N) / 4 * 4;

// Which of a block's half tiles hold sources, per half step: one bit per
// round, looked up once per launch (a load per half tile in the loop would
// put a memory latency on every one of them).  Rounds beyond the bitmap are
// looked up each time.
constexpr int kSrcWords = 64;
struct SourceBits {
  unsigned w[2][kSrcWords];
  __device__ __forceinline__ bool get(int half, int round) const {
    return round >= 32 * kSrcWords || ((w[half][round >> 5] >> (round & 31)) & 1u);
  }
};
// Set the bits (one warp), once they are zero.
__device__ __forceinline__ void mark_sources(const StepIO &io, const Region &R, int per, SourceBits &bits, int lane) {
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    const int *unit = io.src[f].unit;
    if (!unit) continue;
    for (int r = lane; r < per && r < 32 * kSrcWords; r += 32) {
      const int u = r * (int)gridDim.x + R.slot(r, blockIdx.x, gridDim.x);
      if (__ldg(unit + u) < __ldg(unit + u + 1)) atomicOr(&bits.w[f == 0 ? 1 : 0][r >> 5], 1u << (r & 31));
    }
  }
}

// Add the sources of a half tile to its updated arrays in the stage (one
// warp, once every result is there): the entries of a target summed in their
// order, then added, as inject_kernel does.  Four targets a lane at a time:
// each is a chain of loads.
template <int N, typename Maps, bool VEL>
__device__ __forceinline__ void inject_unit(const StepIO &io, int u, long long n, float *st, int lane) {
  const float *row = io.signal + n * io.sig_cols;
  float *ss = VEL ? st + VelStage<N, Maps>::kP + VelStage<N, Maps>::kR
                  : st + PrsStage<N, Maps>::kX + PrsStage<N, Maps>::kY;
#pragma unroll
  for (int a = 0; a < (VEL ? 2 : 1); ++a) {
    const UnitSource &src = io.src[VEL ? 1 + a : 0];
    if (!src.unit) continue;
    const int t1 = __ldg(src.unit + u + 1);
    for (int t0 = __ldg(src.unit + u) + lane; t0 < t1; t0 += 128) {
      int b[4], e[4], pos[4];
      float v[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int t = t0 + 32 * m;
        const bool in = t < t1;
        b[m] = in ? __ldg(src.off + t) : 0;
        e[m] = in ? __ldg(src.off + t + 1) : 0;
        pos[m] = in ? __ldg(src.pos + t) : 0;
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) v[m] = b[m] < e[m] ? 0.f + __ldg(row + __ldg(src.col + b[m])) : 0.f;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        for (int c = b[m] + 1; c < e[m]; ++c) v[m] += __ldg(row + __ldg(src.col + c));
        if (t0 + 32 * m < t1) ss[a * kArr + pos[m]] += v[m];
      }
    }
  }
}

// Trace row of one step, groups spread over the blocks' last threads: the mean
// of p over a group's cells, summed in their order.  p was written by other
// SMs during this launch: read through L2, eight loads in flight.  (By the
// copying warp, on the path of its stores, a step of 250 x 186 took 1.2 us
// more.)  Long groups and many sensors are left to record_kernel
// (record_apart).
__device__ __forceinline__ void record_row(const StepIO &io, const float *p, long long n, int tid) {
  for (int g = blockIdx.x + (kThreads - 1 - tid) * gridDim.x; g < io.rec_groups; g += kThreads * gridDim.x) {
    const int b = __ldg(io.rec_off + g), e = __ldg(io.rec_off + g + 1);
    float s = 0.f;
    for (int i = b; i < e; i += 8) {
      float v[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) v[m] = i + m < e ? __ldcg(p + __ldg(io.rec_cell + i + m)) : 0.f;
#pragma unroll
      for (int m = 0; m < 8; ++m)
        if (i + m < e) s += v[m];
    }
    io.rec_out[n * io.rec_groups + g] = e > b ? s / (float)(e - b) : 0.f;
  }
}

// Phases ph0 .. ph1 - 1 of the time loop in one launch (phase 2n: velocity
// half step of step n with its v sources, 2n + 1: pressure half step with its
// p sources; the recording of step n runs in phase 2n + 2).  Block (32, 17),
// one per SM: sixteen warps compute, the last one issues the copies and
// stores and adds the sources.  More than one phase needs a cooperative
// launch, since the blocks wait for one another between phases.
//
// What bounds it: HBM on grids beyond L2 (4096^2, N = 4: 654 us a step, 0.92
// of the copy bandwidth on the step's bytes), the latency chain of a phase
// (operand copy, compute, store, grid barrier: about 4.4 us) on small ones.
// Four launches per step (two half steps, sources, recording) added to every
// one of them a start and a drain and left the SMs without copies in flight
// meanwhile; here the next phase's first half tiles are copied (all but the
// operand) while the barrier is under way, and sources and recording need no
// launch of their own.  The velocity phases walk the half tiles forwards and
// the pressure phases backwards, so each starts on the rows whose operand the
// previous one left in L2 (0.8 % at 1501 x 1237).
//
// A stage goes round full -> computed -> stored -> refilled.  The computing
// warps wait for "full" and announce "computed" each on its own, so that a
// warp starts on the next stage while others are still busy with the last one
// and nobody waits for a store to leave (10 % at 512^2 and 2048 x 1024 of the
// uint8 index, 4 % at 4096^2, over one barrier per half tile for all threads
// and copies issued by one of them).
//
// us a step with four launches of half-step kernels and now: 250 x 186 (N = 2)
// 20.6 and 8.8, 512^2 (N = 4) 28.8 and 15.7, 1501 x 1237 with cross taps 104
// and 75, 2048 x 1024 of the uint8 index 91 and 61, 4096^2 681 and 654.  A
// launch keeps its SMs to its end: contexts that step on several streams at
// once take turns unless their half tiles fit side by side (three of 250 x 186
// 5.4 and 2.6 us a step of each; three of 512^2, N = 2, 7.8 and 11.9).
template <int N, typename Maps>
__global__ void __launch_bounds__(kStepThreads, 1)
    steps2d_kernel(const StepParams P, const Region R, const __grid_constant__ StepMaps TV,
                   const __grid_constant__ StepMaps TP, const StepIO io, const long long ph0, const long long ph1) {
  using G = StepRing<N, Maps>;
  constexpr int kS = G::kStages, kStage = G::kStage;
  extern __shared__ __align__(128) float smem_raw[];
  __shared__ __align__(8) uint64_t full[kS], done[kS];
  __shared__ int blocked;
  __shared__ SourceBits sources;
  // TMA destinations need 128-byte alignment: round the base up (the launch
  // adds 128 bytes of slack)
  float *smem = reinterpret_cast<float *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  float *tab = smem + kS * kStage;
  const int tid = threadIdx.y * 32 + threadIdx.x;
  for (int i = tid; i < 2 * kSrcWords; i += kStepThreads) (&sources.w[0][0])[i] = 0u;
  if (tid == 0) {
    for (int q = 0; q < kS; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&done[q], kThreads / 32);
    }
    fence_mbarrier_init();
    // after a wait that gave up the state is incomplete: nothing runs until
    // the status is cleared
    blocked = ph1 - ph0 > 1 && status_of(P.status) != 0;
  }
  // this block's half tiles in every phase (at least one: grid <= half tiles)
  const int grid = (int)gridDim.x;
  const int per = R.rounds(blockIdx.x, grid);
  const int last_slot = R.slot(per - 1, blockIdx.x, grid);
  __syncthreads();
  if (blocked) return;
  // Walk over the jobs (phase, half tile): rounds upwards in velocity phases,
  // downwards in pressure phases; a job's stage is its number modulo kS.
  struct Walk {
    long long ph;
    int round, slot, x, y;  // origin of the half tile
    int stage;
    unsigned parity;        // of the stage's barriers for this job
  };
  auto start = [&] {
    Walk w{ph0, (ph0 & 1) ? per - 1 : 0, (ph0 & 1) ? last_slot : (int)blockIdx.x, 0, 0, 0, 0};
    R.half_origin(w.round * grid + w.slot, w.x, w.y);
    return w;
  };
  auto last_of_phase = [&](const Walk &w) { return w.round == ((w.ph & 1) ? 0 : per - 1); };
  auto next = [&](Walk &w) {
    if (last_of_phase(w)) {
      ++w.ph;  // the next phase starts where this one ended
    } else {
      const bool down = w.ph & 1;
      w.round += down ? -1 : 1;
      w.slot += down ? -R.rot : R.rot;
      if (w.slot < 0) w.slot += grid;
      if (w.slot >= grid) w.slot -= grid;
      R.half_origin(w.round * grid + w.slot, w.x, w.y);
    }
    if (++w.stage == kS) {
      w.stage = 0;
      w.parity ^= 1u;
    }
  };

  if (tid >= kThreads) {
    // ---------------------------------------------------- copies and stores
    const int lane = tid - kThreads;
    GridBarrier gb;
    gb.init(io.sync);
    Walk wi = start(), ws = wi;  // next job to issue, next job to store
    int ahead = 0;               // jobs issued and not stored
    Walk wd = wi;                // first job whose operand waits for the grid barrier
    int held = 0;                // and their number
    auto operand = [&](const Walk &w) {  // lane 0: the job may start once these have landed
      float *st = smem + w.stage * kStage;
      uint64_t *bar = &full[w.stage];
      if (w.ph & 1) {
        mbar_arrive_expect_tx(bar, stage_bytes<N, Maps, false>(P.nl != 0, P.nl_vel != 0));
        issue_operand<N, Maps, false>(TP, st, bar, w.x, w.y);
      } else {
        mbar_arrive_expect_tx(bar, stage_bytes<N, Maps, true>(P.nl != 0, P.nl_vel != 0));
        issue_operand<N, Maps, true>(TV, st, bar, w.x, w.y);
      }
    };
    // fill free stages, at most one phase ahead of the phase `ph` under way
    // (what a later phase updates is still being written)
    auto fill = [&](long long ph) {
      while (ahead < kS && wi.ph < ph1 && wi.ph <= ph + 1) {
        if (lane == 0) {
          float *st = smem + wi.stage * kStage;
          uint64_t *bar = &full[wi.stage];
          if (wi.ph & 1) issue_own<N, Maps, false>(P, TP, st, bar, wi.x, wi.y);
          else issue_own<N, Maps, true>(P, TV, st, bar, wi.x, wi.y);
          if (wi.ph == ph) operand(wi);
        }
        if (wi.ph != ph && held++ == 0) wd = wi;
        if (!R.interior(wi.x, wi.y)) {
          if (wi.ph & 1) prefetch_strips2<N, 2, typename Maps::StripT>(P, wi.x, wi.y, lane);
          else prefetch_strips2<N, 1, typename Maps::StripT>(P, wi.x, wi.y, lane);
        }
        ++ahead;
        next(wi);
      }
    };
    auto release_held = [&] {
      for (; held > 0; --held) {
        if (lane == 0) operand(wd);
        next(wd);
      }
    };
    fill(ph0);
    // With the source marks and the index table ahead of the first copies, and
    // the parameters above 4 KB, the two half steps of a step in launches of
    // their own took 16.6 us at 250 x 186 (N = 4, float; 12.9 now) and 36.5 at
    // 512 x 512 of the uint16 index with 1160 tissues (33.0).  (Marked by the
    // computing warps, steps in one launch took 1.7 % more at 250 x 186.)
    mark_sources(io, R, per, sources, lane);
    __syncwarp();
    bool ok = true;
#pragma unroll 1
    while (true) {
      ok = mbar_wait_bounded(&done[ws.stage], ws.parity);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      if ((ws.ph >> 1) < io.sig_steps && sources.get((int)(ws.ph & 1), ws.round)) {
        float *st = smem + ws.stage * kStage;
        const int u = ws.round * grid + ws.slot;
        if (ws.ph & 1) inject_unit<N, Maps, false>(io, u, ws.ph >> 1, st, lane);
        else inject_unit<N, Maps, true>(io, u, ws.ph >> 1, st, lane);
        fence_proxy_async_smem();
        __syncwarp();
      }
      if (lane == 0) {
        if (ws.ph & 1) store_stage<N, Maps, false>(TP, smem + ws.stage * kStage, ws.x, ws.y);
        else store_stage<N, Maps, true>(TV, smem + ws.stage * kStage, ws.x, ws.y);
      }
      --ahead;
      const long long ph = ws.ph;
      const bool last = last_of_phase(ws);
      next(ws);
      if (!last) {
        if (lane == 0) bulk_wait_read<0>();
        __syncwarp();
        fill(ph);
        continue;
      }
      if (ph + 1 == ph1) break;
      if (lane == 0) {
        bulk_wait_all();  // this block's results are in memory
        fence_proxy_async_all();
        gb.arrive();
      }
      __syncwarp();
      // copies of the next phase's first half tiles while the others arrive
      fill(ph);
      if (lane == 0) {
        ok = gb.wait(P.status);
        fence_proxy_async_all();
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      release_held();
      fill(ph + 1);
    }
    if (!ok) {
      // a wait gave up: let this block's copies land (a stage whose operand
      // was still held back gets it, so that its barrier can complete)
      if (lane == 0) report_status(P.status, kStatusWaitTimeout);
      release_held();
      for (; ahead > 0; --ahead) {
        mbar_wait_bounded(&full[ws.stage], ws.parity);
        next(ws);
      }
    }
    if (lane == 0) bulk_wait_all();
    return;
  }

  // ------------------------------------------------------------- compute ---
  if constexpr (Form<Maps>::kIdx) {
    stage_table<N, Maps>(P, tab, tid);
    asm volatile("bar.sync 1, %0;\n" ::"n"(kThreads) : "memory");
  }
  Walk w = start();
#pragma unroll 1
  while (true) {
    const bool vel = (w.ph & 1) == 0, interior = R.interior(w.x, w.y);
    EdgeCoef<N> edge;
    if (!interior) {
      if (vel) load_edge<N, 1, Maps>(P, w.x, w.y, tid, edge);
      else load_edge<N, 2, Maps>(P, w.x, w.y, tid, edge);
    }
    if (!mbar_wait_bounded(&full[w.stage], w.parity)) {
      if ((tid & 31) == 0) report_status(P.status, kStatusWaitTimeout);
      return;
    }
    const long long n = w.ph >> 1;
    // the previous step's trace row, before this warp's first half tile of the
    // velocity phase (the operand is there, so every block's p is complete)
    if (vel && w.round == 0 && w.ph != ph0 && io.rec_groups > 0 && n - 1 < io.rec_steps) record_row(io, P.p, n - 1, tid);
    float *cur = smem + w.stage * kStage;
    if (interior) {
      if (vel) vel_compute<N, Maps, false>(P, tab, cur, w.x, w.y, tid, edge);
      else prs_compute<N, Maps, false>(P, tab, cur, w.x, w.y, tid, edge);
    } else {
      if (vel) vel_compute<N, Maps, true>(P, tab, cur, w.x, w.y, tid, edge);
      else prs_compute<N, Maps, true>(P, tab, cur, w.x, w.y, tid, edge);
    }
    fence_proxy_async_smem();
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(&done[w.stage]);
    if (last_of_phase(w) && w.ph + 1 == ph1) return;
    next(w);
  }
}

// Batched half step over a unit table of several contexts (one group: same N
// and map kind, no periodic axis): entry (ctx, x0, y0, interior).  The
// contexts' step parameters and tensor maps sit in device memory (TMA reads
// the maps from there); a block copies a context's parameters to shared
// memory, and stages its tissue-index table, when the context changes.
// 512 threads and one barrier per unit: a warp of its own for the copies, as
// in steps2d_kernel, was slower here (12.1 against 11.2 ms for six contexts
// and 32 steps), since every context change empties the pipeline and leaves
// the index table to one warp.
template <int N, typename Maps, bool VEL>
__global__ void __launch_bounds__(kThreads, 1)
    pipe2d_batched_kernel(const StepParams *Ps, const PipeMaps *Ts, const int4 *units, const int *runs) {
  using G = Ring<N, Maps, VEL>;
  constexpr int kS = G::kStages, kStage = G::kStage;
  extern __shared__ __align__(128) float smem_raw[];
  __shared__ __align__(8) uint64_t bar[kS];
  __shared__ __align__(16) StepParams sP;
  __shared__ int ok[kS];  // per stage: thread 0 never rewrites a flag a thread has yet to read
  float *smem = reinterpret_cast<float *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  float *tab = smem + kS * kStage;
  const int tid = threadIdx.y * 32 + threadIdx.x;
  if (tid == 0) {
    for (int q = 0; q < kS; ++q) mbar_init(&bar[q], 1);
    fence_mbarrier_init();
  }
  __syncthreads();
  // a contiguous run of units per block (runs[b] .. runs[b + 1]; the host
  // balances the runs by the units' cost): consecutive units share a context
  // (one parameter and table load per context) and halo rows (L2)
  const int h_end = runs[blockIdx.x + 1];
  int h = runs[blockIdx.x];
  if (h >= h_end) return;
  unsigned phase = 0, pending = 0;
  // thread 0: the context whose tensor maps it last acquired (the runs of
  // units are contiguous per context, so each map is acquired about once)
  int fenced = -1;
  auto acquire = [&](int c) {
    if (c == fenced) return;
    for (int m = 0; m < kPipeMaps; ++m) fence_tensormap_acquire(&Ts[c].m[m]);
    fenced = c;
  };
  int hs = h;
  for (int q = 0; q < G::kAhead; ++q, ++hs) {
    if (hs >= h_end) break;
    if (tid == 0) {
      const int4 e = units[hs];
      acquire(e.x);
      issue_stage<N, Maps, VEL>(Ps[e.x], Ts[e.x], smem + q * kStage, &bar[q], e.y, e.z);
    }
    pending |= 1u << q;
  }
  int s = 0, cur = -1;
  // one barrier per unit: after the wait for stage s it also marks the previous
  // unit computed, so its stage is stored and refilled; a context change adds one
  int4 prev = make_int4(-1, 0, 0, 0);
#pragma unroll 1
  for (; h < h_end; ++h) {
    if (tid == 0) ok[s] = mbar_wait_bounded(&bar[s], (phase >> s) & 1u);
    __syncthreads();
    if (!ok[s]) {
      if (tid == 0) {
        report_status(Ps[units[h].x].status, kStatusWaitTimeout);
        for (int q = 0; q < kS; ++q)
          if (q != s && ((pending >> q) & 1u)) mbar_wait_bounded(&bar[q], (phase >> q) & 1u);
        bulk_wait_all();
      }
      return;
    }
    phase ^= 1u << s;
    pending &= ~(1u << s);
    const int sp = (s + kS - 1) % kS;       // the previous unit's stage
    const int q = (s + G::kAhead) % kS;     // the stage refilled now
    if (tid == 0 && prev.x >= 0) store_stage<N, Maps, VEL>(Ts[prev.x], smem + sp * kStage, prev.y, prev.z);
    const int4 e = units[h];
    if (e.x != cur) {
      // new context: parameters (and index table) into shared memory
      const int *src = reinterpret_cast<const int *>(Ps + e.x);
      int *dst = reinterpret_cast<int *>(&sP);
      for (int w = tid; w < (int)(sizeof(StepParams) / 4); w += kThreads) dst[w] = __ldg(src + w);
      __syncthreads();
      stage_table<N, Maps>(sP, tab, tid);
      __syncthreads();
      cur = e.x;
    }
    if (hs < h_end) {
      if (tid < 32) {
        const int4 en = units[hs];
        if (tid == 0) {
          bulk_wait_read<G::kLag>();
          acquire(en.x);
          issue_stage<N, Maps, VEL>(Ps[en.x], Ts[en.x], smem + q * kStage, &bar[q], en.y, en.z);
        }
        if (!en.w && en.x == cur) prefetch_strips2<N, VEL ? 1 : 2, typename Maps::StripT>(sP, en.y, en.z, tid);
      }
      pending |= 1u << q;
      ++hs;
    }
    float *stp = smem + s * kStage;
    EdgeCoef<N> edge;
    if (e.w) {
      if (VEL) vel_compute<N, Maps, false>(sP, tab, stp, e.y, e.z, tid, edge);
      else prs_compute<N, Maps, false>(sP, tab, stp, e.y, e.z, tid, edge);
    } else {
      load_edge<N, VEL ? 1 : 2, Maps>(sP, e.y, e.z, tid, edge);
      if (VEL) vel_compute<N, Maps, true>(sP, tab, stp, e.y, e.z, tid, edge);
      else prs_compute<N, Maps, true>(sP, tab, stp, e.y, e.z, tid, edge);
    }
    fence_proxy_async_smem();
    prev = e;
    s = (s + 1) % kS;
  }
  __syncthreads();
  if (tid == 0 && prev.x >= 0)
    store_stage<N, Maps, VEL>(Ts[prev.x], smem + ((s + kS - 1) % kS) * kStage, prev.y, prev.z);
  if (tid == 0) bulk_wait_all();
}

template <int N, typename Maps, bool VEL>
cudaError_t pipe_batched_launch(const StepParams *Ps, const PipeMaps *Ts, const int4 *units, const int *runs, int grid,
                                cudaStream_t st) {
  constexpr size_t bytes = Ring<N, Maps, VEL>::kBytes;
  cudaError_t e = cudaFuncSetAttribute(pipe2d_batched_kernel<N, Maps, VEL>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  pipe2d_batched_kernel<N, Maps, VEL><<<grid, dim3(32, kThreads / 32), bytes, st>>>(Ps, Ts, units, runs);
  return cudaGetLastError();
}

template <typename Maps, bool VEL>
cudaError_t pipe_batched_dispatch(const StepParams *Ps, const PipeMaps *Ts, const int4 *units, const int *runs,
                                  int n_relax, int grid, cudaStream_t st) {
  switch (n_relax) {
    case 0: return pipe_batched_launch<0, Maps, VEL>(Ps, Ts, units, runs, grid, st);
    case 1: return pipe_batched_launch<1, Maps, VEL>(Ps, Ts, units, runs, grid, st);
    case 2: return pipe_batched_launch<2, Maps, VEL>(Ps, Ts, units, runs, grid, st);
    case 3: return pipe_batched_launch<3, Maps, VEL>(Ps, Ts, units, runs, grid, st);
    case 4: return pipe_batched_launch<4, Maps, VEL>(Ps, Ts, units, runs, grid, st);
    default: return cudaErrorInvalidValue;
  }
}

template <int N, typename Maps>
cudaError_t steps_launch(const StepParams &P, const Region &R, int grid, const PipeMaps &vel, const PipeMaps &prs,
                         const StepIO &io, long long ph0, long long ph1, cudaStream_t st) {
  constexpr size_t bytes = StepRing<N, Maps>::kBytes;
  static_assert(sizeof(StepParams) + sizeof(Region) + 2 * sizeof(StepMaps) + sizeof(StepIO) + 128 <= 4096,
                "kernel parameters");
  const StepMaps TV(vel), TP(prs);
  cudaError_t e = cudaFuncSetAttribute(steps2d_kernel<N, Maps>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  const dim3 block(32, kStepThreads / 32);
  if (ph1 - ph0 == 1) {
    steps2d_kernel<N, Maps><<<grid, block, bytes, st>>>(P, R, TV, TP, io, ph0, ph1);
    return cudaGetLastError();
  }
  // the blocks wait for one another: all of them resident together
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, steps2d_kernel<N, Maps>, P, R, TV, TP, io, ph0, ph1);
}

template <typename Maps>
cudaError_t steps_dispatch(const StepParams &P, const Region &R, int grid, const PipeMaps &TV, const PipeMaps &TP,
                           const StepIO &io, long long ph0, long long ph1, cudaStream_t st) {
  switch (P.n_relax) {
    case 0: return steps_launch<0, Maps>(P, R, grid, TV, TP, io, ph0, ph1, st);
    case 1: return steps_launch<1, Maps>(P, R, grid, TV, TP, io, ph0, ph1, st);
    case 2: return steps_launch<2, Maps>(P, R, grid, TV, TP, io, ph0, ph1, st);
    case 3: return steps_launch<3, Maps>(P, R, grid, TV, TP, io, ph0, ph1, st);
    case 4: return steps_launch<4, Maps>(P, R, grid, TV, TP, io, ph0, ph1, st);
    default: return cudaErrorInvalidValue;
  }
}

Region region_of(const StepParams &P) {
  Region R{};
  R.nx = P.nx;
  R.ny = P.ny;
  R.Lx = P.L[0] > 4 ? P.L[0] : 4;
  R.Ly = P.L[1] > 4 ? P.L[1] : 4;
  R.ntx = (P.nx + kTX - 1) / kTX;
  R.nhy = (P.ny + kHT - 1) / kHT;
  R.inv_ntx = R.ntx == 1 ? 0xffffffffu : (unsigned)((1ull << 32) / R.ntx);
  return R;
}

}  // namespace

bool pipe2d_supported(const StepParams &P, int map_kind) {
  // the copies read zero outside the grid: the zero-outside boundary only
  if (P.nz != 1 || P.n_relax < 0 || P.n_relax > kPipe2dMaxRelax || P.periodic[0] || P.periodic[1]) return false;
  // uint16 index: the tables have to fit in shared memory (beyond that the
  // tile kernels read them through L2; 1160 tissues at 1536 x 2048: 191 us a
  // step there)
  if (map_kind == 3) {
    const int most[] = {kWideTissues<0>, kWideTissues<1>, kWideTissues<2>, kWideTissues<3>, kWideTissues<4>};
    return P.tab_stride <= most[P.n_relax];
  }
  return map_kind >= 0 && map_kind <= 4;
}

bool pipe2d_batched_supported(const StepParams &P, int map_kind) {
  return (map_kind == 0 || map_kind == 2) && pipe2d_supported(P, map_kind);
}

bool pipe2d_preferred(const StepParams &P, int map_kind) { return pipe2d_supported(P, map_kind); }

bool pipe2d_interior_half(const StepParams &P, int x0, int y0) {
  const int Lx = P.L[0] > 4 ? P.L[0] : 4, Ly = P.L[1] > 4 ? P.L[1] : 4;
  return x0 >= Lx && x0 + kTX + Lx <= P.nx && y0 >= Ly && y0 + kHT + Ly <= P.ny;
}

cudaError_t launch_pipe2d_batched(bool vel, const StepParams *Ps, const PipeMaps *Ts, const int4 *units,
                                  int n_units, const int *runs, int n_relax, int map_kind, int grid,
                                  cudaStream_t st) {
  if (n_units <= 0) return cudaSuccess;
  if (map_kind == 2)
    return vel ? pipe_batched_dispatch<IdxMaps, true>(Ps, Ts, units, runs, n_relax, grid, st)
               : pipe_batched_dispatch<IdxMaps, false>(Ps, Ts, units, runs, n_relax, grid, st);
  if (map_kind == 0)
    return vel ? pipe_batched_dispatch<DenseMaps<float>, true>(Ps, Ts, units, runs, n_relax, grid, st)
               : pipe_batched_dispatch<DenseMaps<float>, false>(Ps, Ts, units, runs, n_relax, grid, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_steps2d(const StepParams &P, int map_kind, int n_sm, const PipeMaps &vel, const PipeMaps &prs,
                           const StepIO &io, long long ph0, long long ph1, cudaStream_t st) {
  Region R = region_of(P);
  const long long nh = (long long)R.ntx * R.nhy;
  const int grid = (int)(nh < n_sm ? nh : n_sm);
  // a round advances every block by grid + rot columns: all columns in turn
  while (R.rot + 1 < grid && std::gcd(grid + R.rot, R.ntx) != 1) ++R.rot;
  if (map_kind == 2) return steps_dispatch<IdxMaps>(P, R, grid, vel, prs, io, ph0, ph1, st);
  if (map_kind == 0) return steps_dispatch<DenseMaps<float>>(P, R, grid, vel, prs, io, ph0, ph1, st);
  if (map_kind == 1) return steps_dispatch<DenseMaps<__nv_bfloat16>>(P, R, grid, vel, prs, io, ph0, ph1, st);
  if (map_kind == 3) return steps_dispatch<IdxMaps16>(P, R, grid, vel, prs, io, ph0, ph1, st);
  if (map_kind == 4) return steps_dispatch<DenseMaps<__half>>(P, R, grid, vel, prs, io, ph0, ph1, st);
  return cudaErrorInvalidValue;
}

namespace {

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encoder() {
  static EncodeTiled fn = [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<EncodeTiled>(f);
  }();
  return fn;
}

// tensor map over [ny][nx] (rank 2, row stride pitch) or [n3][ny][nx] (rank
// 3, plane stride s3 elements) of es-byte elements with a box of bx x by (x bz)
bool encode(CUtensorMap *m, const void *base, const StepParams &P, int rank, int n3, long long s3, int bx, int by,
            int bz, int es = 4) {
  const unsigned long long dims[3] = {(unsigned long long)P.nx, (unsigned long long)P.ny, (unsigned long long)n3};
  const unsigned long long strides[2] = {(unsigned long long)P.pitch * es, (unsigned long long)s3 * es};
  const unsigned box[3] = {(unsigned)bx, (unsigned)by, (unsigned)bz};
  return encode_tensor_map(m, base, es, rank, dims, strides, box);
}

}  // namespace

bool encode_tensor_map(CUtensorMap *m, const void *base, int elem_bytes, int rank, const unsigned long long *dims,
                       const unsigned long long *strides_bytes, const unsigned *box) {
  EncodeTiled fn = encoder();
  if (!fn || !base || rank < 2 || rank > 5) return false;
  cuuint64_t d[5], st[4];
  cuuint32_t b[5], e[5];
  for (int i = 0; i < rank; ++i) {
    d[i] = dims[i];
    b[i] = box[i];
    e[i] = 1;
  }
  for (int i = 0; i + 1 < rank; ++i) st[i] = strides_bytes[i];
  const CUtensorMapDataType t = elem_bytes == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                                : elem_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                  : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  return fn(m, t, (cuuint32_t)rank, const_cast<void *>(base), d, st, b, e, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

cudaError_t build_pipe2d_maps(const StepParams &P, int map_kind, PipeMaps *vel, PipeMaps *prs, const char **why) {
  *vel = PipeMaps{};
  *prs = PipeMaps{};
  if (!encoder()) {
    *why = "cuTensorMapEncodeTiled is not available from the driver";
    return cudaErrorInvalidValue;
  }
  const int N = P.n_relax;
  const long long S = P.npts_alloc;
  const bool dense = map_kind == 0 || map_kind == 1 || map_kind == 4;
  const int es = map_kind == 1 || map_kind == 4 ? 2 : 4;                     // bytes of a map value
  const int wide = es == 2 ? kWide<__half> : kWide<float>;                   // density box columns
  const int ies = map_kind == 3 ? 2 : 1;                                     // bytes of an index
  const int iwide = ies == 2 ? kWide<unsigned short> : kWide<unsigned char>; // index box columns
  bool ok = true;
  // velocity half step
  ok = ok && encode(&vel->m[0], P.p, P, 2, 1, S, kCW, kHT + 7, 1);
  if (dense) ok = ok && encode(&vel->m[1], P.rho, P, 2, 1, S, wide, kHT + 1, 1, es);
  else ok = ok && encode(&vel->m[1], P.tissue, P, 2, 1, S, iwide, kHT + 1, 1, ies);
  if (dense && P.nl_vel) ok = ok && encode(&vel->m[9], P.K, P, 2, 1, S, wide, kHT + 1, 1, es);
  ok = ok && encode(&vel->m[2], P.v[0], P, 2, 1, S, kTX, kHT, 1);
  ok = ok && encode(&vel->m[3], P.v[1], P, 2, 1, S, kTX, kHT, 1);
  if (N > 0) {
    ok = ok && encode(&vel->m[4], P.psi1[0], P, 3, N, S, kTX, kHT, N);
    ok = ok && encode(&vel->m[5], P.psi1[1], P, 3, N, S, kTX, kHT, N);
  }
  if (dense) {
    ok = ok && encode(&vel->m[6], P.ik1, P, 2, 1, S, kTX, kHT, 1, es);
    if (N > 0) {
      ok = ok && encode(&vel->m[7], P.a1, P, 3, N, S, kTX, kHT, N, es);
      ok = ok && encode(&vel->m[8], P.b1, P, 3, N, S, kTX, kHT, N, es);
    }
  }
  // pressure half step
  ok = ok && encode(&prs->m[0], P.v[0], P, 2, 1, S, kCW, kHT + 2, 1);
  ok = ok && encode(&prs->m[1], P.v[1], P, 2, 1, S, kCW, kHT + 7, 1);
  ok = ok && encode(&prs->m[2], P.p, P, 2, 1, S, kTX, kHT, 1);
  if (N > 0) {
    ok = ok && encode(&prs->m[3], P.psi2[0], P, 3, N, S, kTX, kHT, N);
    ok = ok && encode(&prs->m[4], P.psi2[1], P, 3, N, S, kTX, kHT, N);
  }
  if (!dense) ok = ok && encode(&prs->m[5], P.tissue, P, 2, 1, S, kTX, kHT, 1, ies);
  if (dense) {
    ok = ok && encode(&prs->m[5], P.ik2, P, 2, 1, S, kTX, kHT, 1, es);
    ok = ok && encode(&prs->m[6], P.K, P, 2, 1, S, kTX, kHT, 1, es);
    if (P.nl) ok = ok && encode(&prs->m[7], P.chi, P, 2, 1, S, kTX, kHT, 1, es);
    if (N > 0) {
      ok = ok && encode(&prs->m[8], P.a2, P, 3, N, S, kTX, kHT, N, es);
      ok = ok && encode(&prs->m[9], P.b2, P, 3, N, S, kTX, kHT, N, es);
    }
  }
  if (!ok) {
    *why = "cuTensorMapEncodeTiled rejected a map";
    return cudaErrorInvalidValue;
  }
  return cudaSuccess;
}

}  // namespace fw2
