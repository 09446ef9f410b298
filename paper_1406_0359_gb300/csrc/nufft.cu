// Kaiser-Bessel interpolation G of Phi = G F Z S (Section 4) and its adjoint
// G^H, over uv-sorted visibility tiles.
//
// Visibilities are binned once per operator into TB x TB tiles of the half
// oversampled grid (stable LSD radix sort on the tile id and cell) and cut into
// work items of at most `chunk` visibilities; a warp owns an item:
//   degrid: the tile's (TB+J)^2 grid patch is staged in shared memory by one
//           TMA tile load (the grid carries a J-wide halo, so the patch is
//           contiguous); every lane gathers its visibility's J x J taps.
//   grid:   groups of lanes sum runs of visibilities of one cell in registers,
//           then in patches in shared memory, flushed to the padded global grid
//           with vector atomics.
// Kernel weights come from a per-tap polynomial in the fractional offset
// (Chebyshev fit of the Kaiser-Bessel kernel, computed on the host).
#include <cstdio>
#include <algorithm>
#include <cstring>
#include <vector>

#include <initializer_list>

#include "internal.h"

namespace purify {

namespace {

// FP32 positions: the cell inside the tile in the top 7 bits, the offset in
// units of 2^-24 below them, 0 and 1 both included (a mirrored grid node has
// offset 1).
constexpr int kOffBits = 24, kCellShift = kOffBits + 1;
PD uint32_t encode_offset(int cell, double f) {
  return (uint32_t(cell) << kCellShift) | uint32_t(f * double(1u << kOffBits) + 0.5);
}
PD void decode(const Pos<float>& p, int& cu, float& fu, int& cv, float& fv) {
  constexpr float sc = 1.0f / float(1u << kOffBits);
  constexpr uint32_t mask = (1u << kCellShift) - 1u;
  cu = int(p.u >> kCellShift);
  cv = int(p.v >> kCellShift);
  fu = float(p.u & mask) * sc;
  fv = float(p.v & mask) * sc;
}
PD void decode(const Pos<double>& p, int& cu, double& fu, int& cv, double& fv) {
  const double a = floor(p.u), b = floor(p.v);
  cu = int(a);
  cv = int(b);
  fu = p.u - a;
  fv = p.v - b;
}

// Kernel weights of the J taps at fractional offset f.  The kernel is even,
// so tap J-1-a at f equals tap a at 1-f, i.e. its polynomial in x = 2f-1 is
// tap a's at -x: with P_a(x) = E_a(x^2) + x O_a(x^2) both taps of a pair come
// from one even and one odd Horner chain in x^2.
template <typename T> PD void kb_eval(const KbPoly<T>& kb, T f, T (&w)[kJ]) {
  constexpr int D = KbDeg<T>::value;
  const T x = T(2) * f - T(1);
  const T x2 = x * x;
#pragma unroll
  for (int a = 0; a < kJ / 2; ++a) {
    T e = kb.c[a][D - (D & 1)];
#pragma unroll
    for (int d = D - (D & 1) - 2; d >= 0; d -= 2) e = fma(e, x2, kb.c[a][d]);
    T o = kb.c[a][D - 1 + (D & 1)];
#pragma unroll
    for (int d = D - 1 + (D & 1) - 2; d >= 1; d -= 2) o = fma(o, x2, kb.c[a][d]);
    w[a] = fma(x, o, e);
    w[kJ - 1 - a] = fma(-x, o, e);
  }
}

// One lane's staged visibility record (kGrRec values)
// written as 16-byte vectors: at the 80-byte (FP32) lane stride each
// quarter-warp's vector stores hit distinct bank groups, where scalar stores at
// that stride collide four ways.
PD void stage_store(float* st, const float (&wu)[kJ], const float (&wv)[kJ], float e0, float e1) {
  float4* d = reinterpret_cast<float4*>(st);
  d[0] = make_float4(wu[0], wu[1], wu[2], wu[3]);
  d[1] = make_float4(wu[4], wu[5], wu[6], wu[7]);
  d[2] = make_float4(wv[0], wv[1], wv[2], wv[3]);
  d[3] = make_float4(wv[4], wv[5], wv[6], wv[7]);
  *reinterpret_cast<float2*>(d + 4) = make_float2(e0, e1);
}
PD void stage_store(double* st, const double (&wu)[kJ], const double (&wv)[kJ], double e0, double e1) {
  double2* d = reinterpret_cast<double2*>(st);
#pragma unroll
  for (int a = 0; a < kJ / 2; ++a) {
    d[a] = make_double2(wu[2 * a], wu[2 * a + 1]);
    d[kJ / 2 + a] = make_double2(wv[2 * a], wv[2 * a + 1]);
  }
  d[kJ] = make_double2(e0, e1);
}
static_assert(kJ == 8, "stage_store writes 2J + 2 values");

// ---------------------------------------------------------------------------
// Warp-per-item forms of degridding and gridding (the ball block and the
// operator calls).  Each warp owns one work item end to end: its own TMA-staged
// patch and mbarrier (degridding) or its own accumulator patch (gridding), so
// there are no CTA-wide barriers and no cross-warp merges; items are ordered
// largest first so the hardware's CTA scheduling balances the load.
// Two warps per CTA: a CTA of 8 holds its shared memory and registers until its
// longest item ends (1024^2 / 4M points: Phi 99.7 against 108.4 us, Phi^H 155
// against 160); single-warp CTAs measured the same alone, but a batch's grid of
// the largest instance's items per instance launches twice as many (16
// instances: 1227 against 1215 us an iteration).
constexpr int kWItems = 2;  // items (warps) per CTA

// Row pitch (cells) of the staged patch.  A warp's lanes read cells of one
// grid row after another; FP32 cells are 8 bytes and served per half-warp (16
// cells), so at a pitch of 8 mod 16 the 8 cells of two neighbouring tile rows
// fall on disjoint banks (a tile of 16 is a half-warp wide by itself).  FP64
// cells are served per quarter-warp; two more columns spread their rows.
template <typename T> __host__ __device__ constexpr int patch_pitch(int TB) {
  return sizeof(T) == 4 ? 24 : TB + kJ + 2;
}
template <typename T> __host__ __device__ inline size_t warp_patch_elems(int TB) {
  return size_t(TB + kJ) * patch_pitch<T>(TB);
}

template <typename C>
PD bool warp_stage_patch(C* patch, uint64_t* bar, const CUtensorMap* map, int tu, int tv, int TB, uint32_t bytes,
                         int lane, int* err) {
  if (lane == 0) {
    mbar_init(bar, 1);
    fence_barrier_init();
    mbar_arrive_expect_tx(bar, bytes);
    const int cw = int(sizeof(C) / 8);
    tma_load_2d(patch, map, tv * TB * cw, tu * TB, bar);
  }
  __syncwarp();
  const bool ok = mbar_wait_bounded(bar, 0, err);
  return __all_sync(0xffffffffu, ok) != 0;
}

// Degridding: one lane per visibility, its kernel weights in registers, its
// J x J cells gathered from the warp's staged patch; visibilities are sorted by
// cell, so a warp's lanes read neighbouring cells.  Bound by the shared-memory
// pipe: 64 cells of 8 bytes at 128 bytes a clock are 4 cycles per visibility, the
// pipe is 85% busy and issue, with the taps as packed pairs, 53%.  The form with
// four lanes per visibility staged every weight through shared memory and
// summed by shuffles, 7.8 cycles: 141 us a launch against 80 (1024^2,
// M = 4,194,304).
// sum_b w[b] row[b] over a footprint row, FP32 as packed (re, im) pairs.
template <typename C> struct TapRow;
template <> struct TapRow<double2> {
  double w[kJ];
  PD void set(const double (&v)[kJ]) {
#pragma unroll
    for (int b = 0; b < kJ; ++b) w[b] = v[b];
  }
  PD void add(double2& acc, double wu, const double2* row) const {
    double2 h = make_double2(0.0, 0.0);
#pragma unroll
    for (int b = 0; b < kJ; ++b) {
      const double2 c = row[b];
      h.x = fma(w[b], c.x, h.x);
      h.y = fma(w[b], c.y, h.y);
    }
    acc.x = fma(wu, h.x, acc.x);
    acc.y = fma(wu, h.y, acc.y);
  }
};
template <> struct TapRow<float2> {
  unsigned long long w[kJ];  // (w, w)
  PD void set(const float (&v)[kJ]) {
#pragma unroll
    for (int b = 0; b < kJ; ++b) asm("mov.b64 %0, {%1, %1};" : "=l"(w[b]) : "f"(v[b]));
  }
  PD void add(float2& acc, float wu, const float2* row) const {
    unsigned long long h = 0ull;
#pragma unroll
    for (int b = 0; b < kJ; ++b) {
      const unsigned long long c = *reinterpret_cast<const unsigned long long*>(row + b);
      asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(h) : "l"(w[b]), "l"(c));
    }
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(h));
    acc.x = fmaf(wu, x, acc.x);
    acc.y = fmaf(wu, y, acc.y);
  }
};

template <typename T, typename Src>
__global__ void __launch_bounds__(32 * kWItems) k_degrid_w(Src src, KbPoly<T> kb, const __grid_constant__ CUtensorMap map0) {
  typedef typename cplx_t<T>::type C;
  decltype(auto) a = src.get();
  const Geometry& g = a.g;
  const int n_items = a.n_items;
  const int* __restrict__ perm = a.perm;
  const DegridEp<C>& dep = a.dep;
  const CUtensorMap* map = Src::kTable ? a.map : &map0;
  extern __shared__ __align__(128) unsigned char sm_raw[];
  __shared__ __align__(8) uint64_t bars[kWItems];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int item = blockIdx.x * kWItems + warp;
  if (item >= n_items) return;
  const WorkItem it = a.items[item];
  const int tu = it.tile / g.ntv, tv = it.tile - tu * g.ntv;
  const int PP = patch_pitch<T>(g.TB);
  const size_t pe = warp_patch_elems<T>(g.TB);
  C* patch = reinterpret_cast<C*>(sm_raw) + warp * pe;
  if (Src::kTable && lane == 0) tensormap_acquire(map);
  const Pos<T>* __restrict__ pos = a.pos;
  int i = it.begin + lane;
  Pos<T> p = pos[min(i, it.end - 1)];  // the first positions arrive beside the patch
  pdl_wait();  // (items and positions are the operator's, written at its set-up)
  if (!warp_stage_patch(patch, &bars[warp], map, tu, tv, g.TB, uint32_t(pe * sizeof(C)), lane, a.err)) return;
  const bool ball = dep.mode == DG_BALL;
  Acc<T> p0, p1;
  for (; i - lane < it.end; i += 32) {
    const int is = min(i, it.end - 1);
    // the epilogue's operands and the next positions are on their way while the taps are summed
    C z = cz<C>(), yv = cz<C>();
    int pm = 0;
    if (ball) {
      z = dep.z[is];
      yv = dep.ys[is];
    } else if (dep.mode == DG_STORE_PERM) {
      pm = perm[is];
    }
    const Pos<T> cur = p;
    p = pos[min(i + 32, it.end - 1)];
    int cu, cv;
    T fu, fv, wu[kJ], wv[kJ];
    decode(cur, cu, fu, cv, fv);
    kb_eval(kb, fu, wu);
    kb_eval(kb, fv, wv);
    TapRow<C> taps;
    taps.set(wv);
    const C* row = patch + cu * PP + cv;
    C acc = cz<C>();
#pragma unroll
    for (int r = 0; r < kJ; ++r, row += PP) taps.add(acc, wu[r], row);
    if (i >= it.end) continue;
    if (ball) {
      const T nu = T(dep.nu);
      const C v = cmk<C>(fma(nu, acc.x, z.x), fma(nu, acc.y, z.y));
      dep.z[i] = v;
      const T dx = fma(-nu, yv.x, v.x), dy = fma(-nu, yv.y, v.y);
      p0.add_prod(dx, dx);
      p0.add_prod(dy, dy);
      const T ex = acc.x - yv.x, ey = acc.y - yv.y;
      p1.add_prod(ex, ex);
      p1.add_prod(ey, ey);
    } else if (dep.mode == DG_STORE_PERM) {
      dep.y[perm_index(pm)] = perm_value(pm, acc);
    } else {
      dep.y[i] = acc;
    }
  }
  __syncwarp();
  pdl_trigger();
  if (ball) {
    warp_merge(p0);
    warp_merge(p1);
    if (lane == 0 && dep.acc) {
      double* acc = dep.acc + 2 * (item % kBallAcc);
      atomicAdd(acc, p0.value());
      atomicAdd(acc + 1, p1.value());
    } else if (lane == 0) {
      reinterpret_cast<Acc<T>*>(dep.part0)[item] = p0;
      reinterpret_cast<Acc<T>*>(dep.part1)[item] = p1;
    }
  }
}

// Gridding: the warp splits its item into two contiguous slices, one per group
// of 16 lanes; a lane of a group sums four cells (one row and column parity) of
// its visibility's J x J footprint in registers for as long as the group's cell
// stays the same, and adds the run to the group's own patch of plain cells in
// shared memory (no atomics, nothing shared between groups) when it changes.
// The patches are merged at the end, one vector atomic per two cells.  Two
// visibilities take 8 FMAs a lane; bound by instruction issue (70%) and the
// shared-memory pipe (69%, some 6 cycles a visibility).  One visibility at
// a time on 32 lanes took 165 us a launch, this form 115 (1024^2, M =
// 4,194,304, half grid); four groups of 8 lanes win where cells are full (512^2:
// 128 against 149 us for Phi^H) but hold 16 warps an SM and lose elsewhere (187
// against 150).
constexpr int kGroups = 2;
constexpr int kGrLanes = 32 / kGroups;      // lanes of a group: 8 rows x 2 column parities
constexpr int kGrCols = 8 * kJ / kGrLanes;  // columns per lane
constexpr int kGrRec = 2 * kJ + 4;          // staged record: wu[J], wv[J], u.re, u.im, pad
constexpr int kGrStage = kGrLanes * kGrRec + 8;  // a group's records; the pad puts the groups on distinct banks
template <typename T> struct __align__(2 * sizeof(T)) GCell { T x, y; };
// Row stride 2 mod 16 or 10 mod 16 (even): the 8 rows x 2 neighbouring columns
// that a group's 16 lanes update at once (8-byte FP32 cells) fall on 16
// distinct bank pairs; pairs of cells stay 16-byte aligned.
__host__ __device__ constexpr int grid_row_stride(int TB) { return TB + kJ + 2; }
template <typename T> __host__ __device__ inline size_t grid_patch_cells(int TB) {
  return size_t(TB + kJ) * grid_row_stride(TB);
}
template <typename T> __host__ __device__ inline size_t grid_warp_bytes(int TB) {
  return kGroups * (grid_patch_cells<T>(TB) * sizeof(GCell<T>) + kGrStage * sizeof(T));
}

// One lane's sums of W complex cells of one column parity, FP32 as packed pairs of
// columns (an FMA of two by one instruction, same rounding).
template <typename T, int W> struct RowAcc;
template <int W> struct RowAcc<double, W> {
  double x[W], y[W];
  PD void zero() {
#pragma unroll
    for (int b = 0; b < W; ++b) x[b] = y[b] = 0.0;
  }
  PD void add(const double* wv, double ax, double ay) {
#pragma unroll
    for (int b = 0; b < W; ++b) {
      x[b] = fma(wv[b], ax, x[b]);
      y[b] = fma(wv[b], ay, y[b]);
    }
  }
  PD void flush(GCell<double>* c) {
#pragma unroll
    for (int b = 0; b < W; ++b) {
      c[2 * b].x += x[b];
      c[2 * b].y += y[b];
    }
  }
};
template <int W> struct RowAcc<float, W> {
  unsigned long long x[W / 2], y[W / 2];
  PD void zero() {
#pragma unroll
    for (int b = 0; b < W / 2; ++b) x[b] = y[b] = 0ull;
  }
  static PD void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
  }
  PD void add(const float* wv, float ax, float ay) {
    unsigned long long px, py, w[W / 2];
    asm("mov.b64 %0, {%1, %1};" : "=l"(px) : "f"(ax));
    asm("mov.b64 %0, {%1, %1};" : "=l"(py) : "f"(ay));
    if constexpr (W == 2) {
      w[0] = *reinterpret_cast<const unsigned long long*>(wv);
    } else {
#pragma unroll
      for (int b = 0; b < W / 4; ++b) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(wv + 4 * b);
        w[2 * b] = v.x;
        w[2 * b + 1] = v.y;
      }
    }
#pragma unroll
    for (int b = 0; b < W / 2; ++b) {
      fma2(x[b], w[b], px);
      fma2(y[b], w[b], py);
    }
  }
  PD void flush(GCell<float>* c) {
    GCell<float> k[W];
#pragma unroll
    for (int b = 0; b < W; ++b) k[b] = c[2 * b];
#pragma unroll
    for (int b = 0; b < W / 2; ++b) {
      float x0, x1, y0, y1;
      asm("mov.b64 {%0, %1}, %2;" : "=f"(x0), "=f"(x1) : "l"(x[b]));
      asm("mov.b64 {%0, %1}, %2;" : "=f"(y0), "=f"(y1) : "l"(y[b]));
      k[2 * b].x += x0;
      k[2 * b].y += y0;
      k[2 * b + 1].x += x1;
      k[2 * b + 1].y += y1;
    }
#pragma unroll
    for (int b = 0; b < W; ++b) c[2 * b] = k[b];
  }
};

PD void cell_pair(float2 (&c)[2], const GCell<float>* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  c[0] = make_float2(v.x, v.y);
  c[1] = make_float2(v.z, v.w);
}
PD void cell_pair(double2 (&c)[2], const GCell<double>* p) {
  c[0] = make_double2(p[0].x, p[0].y);
  c[1] = make_double2(p[1].x, p[1].y);
}
// Two neighbouring merged cells into the grid (16-byte aligned for FP32).
PD void atomic_add_pair(float2* p, float2 a, float2 b) {
  atomicAdd(reinterpret_cast<float4*>(p), make_float4(a.x, a.y, b.x, b.y));
}
PD void atomic_add_pair(double2* p, double2 a, double2 b) {
  atomicAdd(&p[0].x, a.x);
  atomicAdd(&p[0].y, a.y);
  atomicAdd(&p[1].x, b.x);
  atomicAdd(&p[1].y, b.y);
}

template <typename T, typename Src>
__global__ void __launch_bounds__(32 * kWItems) k_grid_w(Src src, KbPoly<T> kb) {
  typedef typename cplx_t<T>::type C;
  decltype(auto) a = src.get();
  const Geometry& g = a.g;
  const int n_items = a.n_items;
  const Pos<T>* __restrict__ pos = a.pos;
  const int* __restrict__ perm = a.perm;
  const GridPro<C>& gpro = a.gpro;
  extern __shared__ __align__(128) unsigned char sm_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int item = blockIdx.x * kWItems + warp;
  if (item >= n_items) return;
  const WorkItem it = a.items[item];
  const int tu = it.tile / g.ntv, tv = it.tile - tu * g.ntv;
  const int PW = g.TB + kJ, PS = grid_row_stride(g.TB);
  const int cells = int(grid_patch_cells<T>(g.TB));
  unsigned char* wbase = sm_raw + warp * grid_warp_bytes<T>(g.TB);
  GCell<T>* patches = reinterpret_cast<GCell<T>*>(wbase);
  T* stage = reinterpret_cast<T*>(patches + kGroups * cells);
  const int grp = lane / kGrLanes, q = lane % kGrLanes;
  const int r = q % kJ, h = q / kJ;  // the lane's footprint row and column parity
  // this group's slice; the first positions (and permutation) travel while the patches are zeroed
  const int cnt = it.end - it.begin, per = (cnt + kGroups - 1) / kGroups;
  const int lo = it.begin + min(cnt, grp * per), hi = it.begin + min(cnt, (grp + 1) * per);
  int i = lo + q;
  Pos<T> p = pos[min(i, it.end - 1)];
  int pm = gpro.mode == GP_PERM ? perm[min(i, it.end - 1)] : 0;
  {
    uint4* zp = reinterpret_cast<uint4*>(patches);  // cells are even in number
    const int nz = kGroups * cells * int(sizeof(GCell<T>)) / 16;
    for (int e = lane; e < nz; e += 32) zp[e] = make_uint4(0, 0, 0, 0);
  }
  pdl_wait();
  T scale = 0;
  if (gpro.mode == GP_BALL) scale = T(gpro.block_scale ? gpro.block_scale[it.pad] : gpro.scalars[gpro.scale_idx]);
  GCell<T>* mine = patches + grp * cells + r * PS + h;
  T* gst = stage + grp * kGrStage;
  int run = -1, last = -1;  // the current run's cell; the slice's last staged cell
  RowAcc<T, kGrCols> acc;
  acc.zero();
  for (int b = 0; b < per; b += kGrLanes, i += kGrLanes) {
    const bool valid = i < hi;
    const int is = min(i, it.end - 1);
    C u = cz<C>(), yv = cz<C>();
    if (gpro.mode == GP_PERM) {
      u = perm_value(pm, gpro.y[perm_index(pm)]);
    } else if (gpro.mode == GP_SORTED) {
      u = gpro.y[is];
    } else {
      u = gpro.z[is];
      yv = gpro.ys[is];
    }
    const Pos<T> cur = p;
    p = pos[min(i + kGrLanes, it.end - 1)];
    if (gpro.mode == GP_PERM) pm = perm[min(i + kGrLanes, it.end - 1)];
    int cu, cv;
    T fu, fv, wu[kJ], wv[kJ];
    decode(cur, cu, fu, cv, fv);
    kb_eval(kb, fu, wu);
    kb_eval(kb, fv, wv);
    if (gpro.mode == GP_BALL) {  // v = z, c = nu y: project, keep the dual, grid 2r - v
      const C v = u;
      const T nu = T(gpro.nu);
      const T cx = nu * yv.x, cy = nu * yv.y;
      const T rx = fma(v.x - cx, scale, cx), ry = fma(v.y - cy, scale, cy);
      if (valid) gpro.z[i] = cmk<C>(v.x - rx, v.y - ry);
      u = cmk<C>(T(2) * rx - v.x, T(2) * ry - v.y);
    }
    if (!valid) u = cz<C>();  // adds nothing, changes no cell
    int cell = cu * PS + cv;
    int before = __shfl_up_sync(0xffffffffu, cell, 1, kGrLanes);
    if (q == 0) before = last;
    const unsigned changes = __ballot_sync(0xffffffffu, valid && cell != before);
    last = __shfl_sync(0xffffffffu, cell, kGrLanes - 1, kGrLanes);
    __syncwarp();  // the previous batch's records are read
    {
      T* st = gst + q * kGrRec;
      const T wo[kJ] = {wv[0], wv[2], wv[4], wv[6], wv[1], wv[3], wv[5], wv[7]};
      stage_store(st, wu, wo, u.x, u.y);
    }
    __syncwarp();
    const int nj = min(kGrLanes, per - b);
    static_assert(kGroups == 2, "the first record of either group");
    constexpr unsigned kFirst = 0x00010001u;
#pragma unroll 4
    for (int j = 0; j < nj; ++j) {
      if (changes & (kFirst << j)) {
        const int next = __shfl_sync(0xffffffffu, cell, j, kGrLanes);
        if ((changes >> (grp * kGrLanes + j)) & 1u) {
          if (run >= 0) {
            acc.flush(mine + run);
            acc.zero();
          }
          run = next;
        }
      }
      const T* rec = gst + j * kGrRec;
      const T w = rec[r];
      acc.add(rec + kJ + h * kGrCols, w * rec[2 * kJ], w * rec[2 * kJ + 1]);
    }
  }
  if (run >= 0) acc.flush(mine + run);
  pdl_trigger();
  __syncwarp();
  // pairs of cells, 8 (tiles of 8) or 12 of 16 (tiles of 16) lanes to a row
  const int ls = g.TB == 8 ? 3 : 4, pc = 2 * (lane & ((1 << ls) - 1));
  if (pc < PW) {
    C* dst = a.Q + size_t(tu * g.TB) * g.KC + (tv * g.TB + pc);
    for (int pr = lane >> ls; pr < PW; pr += 32 >> ls) {
      const GCell<T>* k = patches + pr * PS + pc;
      C v[2] = {cz<C>(), cz<C>()};
#pragma unroll
      for (int z = 0; z < kGroups; ++z) {
        C c[2];
        cell_pair(c, k + z * cells);
        v[0] = cadd(v[0], c[0]);
        v[1] = cadd(v[1], c[1]);
      }
      if (v[0].x != 0 || v[0].y != 0 || v[1].x != 0 || v[1].y != 0) atomic_add_pair(dst + size_t(pr) * g.KC, v[0], v[1]);
    }
  }
}

// ----------------------------------------------------------------- binning
// Grid cell and fractional offset of a uv sample: t = u K / (2 pi), cell =
// floor(t) taken modulo K, f = t - floor(t) in [0, 1).  The expression order
// matches the plain definition so that samples lying exactly on grid nodes
// fall in the same cell.
PD void grid_cell(double u, int K, int& cell, double& f) {
  const double t = (u * double(K)) / (2.0 * 3.14159265358979323846);
  const double fl = floor(t);
  f = t - fl;
  long long c = (long long)fl % K;
  if (c < 0) c += K;
  cell = int(c);
}
// Cell and offset of both axes, reflected into the half grid when the column
// cell is in [K/2, K) (and fold is set); returns whether it was.
PD bool grid_cells(const double* uv, int64_t m, int K, bool fold, int (&cell)[2], double (&f)[2]) {
  grid_cell(uv[2 * m], K, cell[0], f[0]);
  grid_cell(uv[2 * m + 1], K, cell[1], f[1]);
  const bool mirror = fold && cell[1] >= K / 2;
  if (mirror)
    for (int a = 0; a < 2; ++a) {
      cell[a] = K - 1 - cell[a];
      f[a] = 1.0 - f[a];
    }
  return mirror;
}

// Sort key: tile id, then the cell inside the tile (row-major), so that a
// tile's visibilities come grouped by grid cell.
// With visibility blocks (Eq. 4) the block index leads the key, so that every
// work item lies in one block.
__global__ void k_bin_keys(const double* __restrict__ uv, const int* __restrict__ blocks, int64_t M, int K, int TB,
                           int lb, int ntv, int tbits, bool fold, uint32_t* __restrict__ keys,
                           int* __restrict__ vals) {
  const int64_t m = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (m >= M) return;
  int c[2];
  double f[2];
  const bool mirror = grid_cells(uv, m, K, fold, c, f);
  const uint32_t tile = uint32_t((c[0] / TB) * ntv + (c[1] / TB));
  const uint32_t blk = blocks ? uint32_t(blocks[m]) : 0u;
  keys[m] = (blk << (tbits + 2 * lb)) | (tile << (2 * lb)) | (uint32_t(c[0] % TB) << lb) | uint32_t(c[1] % TB);
  vals[m] = mirror ? ~int(m) : int(m);
}

constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;

__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint32_t* __restrict__ keys, int64_t M, int shift,
                                                             int nblocks, int* __restrict__ hist) {
  __shared__ int h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = int64_t(blockIdx.x) * kSortTile;
  for (int k = 0; k < kSortItems; ++k) {
    const int64_t i = base + int64_t(k) * kSortThreads + threadIdx.x;
    if (i < M) atomicAdd(&h[(keys[i] >> shift) & 255u], 1);
  }
  __syncthreads();
  hist[int64_t(threadIdx.x) * nblocks + blockIdx.x] = h[threadIdx.x];
}

// Exclusive scan of a[0..L) in place, three phases: per-chunk sums, a scan of
// the chunk sums by one block, and per-chunk scans offset by their chunk's
// prefix (all loads and stores coalesced).  total (if not null) receives the
// sum of all L values.  Needs L <= kScanChunk * 1024.
constexpr int kScanT = 256, kScanE = 16, kScanChunk = kScanT * kScanE;

__device__ __forceinline__ int block_excl_scan_int(int v, int* sh /*[32]*/, int* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) sh[w] = incl;
  __syncthreads();
  if (w == 0) {
    int x = lane < nw ? sh[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += u;
    }
    sh[lane] = x;  // inclusive prefix of warp sums
  }
  __syncthreads();
  const int before = w > 0 ? sh[w - 1] : 0;
  if (total) *total = sh[nw - 1];
  __syncthreads();
  return before + incl - v;
}

__global__ void __launch_bounds__(kScanT) k_scan_reduce(const int* __restrict__ a, int64_t L, int* __restrict__ bsum) {
  __shared__ int sh[32];
  const int64_t base = int64_t(blockIdx.x) * kScanChunk;
  int v = 0;
#pragma unroll
  for (int j = 0; j < kScanE; ++j) {
    const int64_t i = base + threadIdx.x + int64_t(j) * kScanT;
    if (i < L) v += a[i];
  }
  int tot = 0;
  block_excl_scan_int(v, sh, &tot);
  if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024) k_scan_top(int* __restrict__ bsum, int B, int* __restrict__ total) {
  __shared__ int sh[32];
  const int v = int(threadIdx.x) < B ? bsum[threadIdx.x] : 0;
  int tot = 0;
  const int ex = block_excl_scan_int(v, sh, &tot);
  if (int(threadIdx.x) < B) bsum[threadIdx.x] = ex;
  if (threadIdx.x == 0 && total) *total = tot;
}

__global__ void __launch_bounds__(kScanT) k_scan_down(int* __restrict__ a, int64_t L, const int* __restrict__ bsum) {
  __shared__ int tile[kScanChunk + kScanChunk / 32];
  __shared__ int sh[32];
  auto pad = [](int e) { return e + (e >> 5); };
  const int64_t base = int64_t(blockIdx.x) * kScanChunk;
#pragma unroll
  for (int j = 0; j < kScanE; ++j) {
    const int e = threadIdx.x + j * kScanT;
    tile[pad(e)] = base + e < L ? a[base + e] : 0;
  }
  __syncthreads();
  int loc[kScanE];
  int run = 0;
#pragma unroll
  for (int k = 0; k < kScanE; ++k) {
    loc[k] = run;
    run += tile[pad(threadIdx.x * kScanE + k)];
  }
  const int off = block_excl_scan_int(run, sh, nullptr) + bsum[blockIdx.x];
#pragma unroll
  for (int k = 0; k < kScanE; ++k) tile[pad(threadIdx.x * kScanE + k)] = loc[k] + off;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kScanE; ++j) {
    const int e = threadIdx.x + j * kScanT;
    if (base + e < L) a[base + e] = tile[pad(e)];
  }
}

// Exclusive scan of a[0..L) in place by one 1024-thread block (fallback for
// L beyond the three-phase limit); total -> *total.
__global__ void __launch_bounds__(1024) k_scan(int* __restrict__ a, int64_t L, int* __restrict__ total) {
  __shared__ int sums[1024];
  const int64_t per = (L + 1023) / 1024;
  const int64_t lo = int64_t(threadIdx.x) * per;
  const int64_t hi = lo + per < L ? lo + per : L;
  int s = 0;
  for (int64_t i = lo; i < hi; ++i) s += a[i];
  sums[threadIdx.x] = s;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    const int v = threadIdx.x >= off ? sums[threadIdx.x - off] : 0;
    __syncthreads();
    sums[threadIdx.x] += v;
    __syncthreads();
  }
  int run = threadIdx.x > 0 ? sums[threadIdx.x - 1] : 0;
  for (int64_t i = lo; i < hi; ++i) {
    const int v = a[i];
    a[i] = run;
    run += v;
  }
  if (threadIdx.x == 1023 && total) *total = sums[1023];
}

// bsum: scratch of at least 1024 ints.
inline void launch_scan(int* a, int64_t L, int* total, int* bsum, cudaStream_t s) {
  const int64_t B = (L + kScanChunk - 1) / kScanChunk;
  if (B <= 1024) {
    k_scan_reduce<<<int(B > 0 ? B : 1), kScanT, 0, s>>>(a, L, bsum);
    k_scan_top<<<1, 1024, 0, s>>>(bsum, int(B > 0 ? B : 1), total);
    k_scan_down<<<int(B > 0 ? B : 1), kScanT, 0, s>>>(a, L, bsum);
  } else {
    k_scan<<<1, 1024, 0, s>>>(a, L, total);
  }
}

__global__ void __launch_bounds__(kSortThreads) k_radix_scatter(const uint32_t* __restrict__ kin,
                                                                const int* __restrict__ vin, int64_t M, int shift,
                                                                int nblocks, const int* __restrict__ offs,
                                                                uint32_t* __restrict__ kout, int* __restrict__ vout) {
  constexpr int NW = kSortThreads / 32;
  __shared__ int running[256];
  __shared__ int wcount[NW][256];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  running[threadIdx.x] = offs[int64_t(threadIdx.x) * nblocks + blockIdx.x];
  for (int k = 0; k < NW; ++k) wcount[k][threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = int64_t(blockIdx.x) * kSortTile;
  const unsigned lt = (1u << lane) - 1u;
  for (int round = 0; round < kSortItems; ++round) {
    const int64_t i = base + int64_t(round) * kSortThreads + threadIdx.x;
    const bool valid = i < M;
    uint32_t key = 0;
    int val = 0;
    int d = 256;  // sentinel digit for the ragged tail
    if (valid) {
      key = kin[i];
      val = vin[i];
      d = int((key >> shift) & 255u);
    }
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int rank = __popc(peers & lt);
    if (valid && rank == 0) wcount[w][d] = __popc(peers);
    __syncthreads();
    if (valid) {
      int pos = running[d] + rank;
      for (int k = 0; k < w; ++k) pos += wcount[k][d];
      kout[pos] = key;
      vout[pos] = val;
    }
    __syncthreads();
    int add = 0;
    for (int k = 0; k < NW; ++k) {
      add += wcount[k][threadIdx.x];
      wcount[k][threadIdx.x] = 0;
    }
    running[threadIdx.x] += add;
    __syncthreads();
  }
}

__global__ void k_tile_bounds(const uint32_t* __restrict__ keys, int64_t M, int shift, int* __restrict__ start,
                              int* __restrict__ end) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= M) return;
  const uint32_t k = keys[i] >> shift;
  if (i == 0 || (keys[i - 1] >> shift) != k) start[k] = int(i);
  if (i == M - 1 || (keys[i + 1] >> shift) != k) end[k] = int(i + 1);
}

__global__ void k_chunk_counts(const int* __restrict__ start, const int* __restrict__ end, int ntiles, int chunk,
                               int* __restrict__ cnt) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ntiles) return;
  const int c = end[t] - start[t];
  cnt[t] = (c + chunk - 1) / chunk;
}

// Bins are (block, tile) pairs, bin = block * tiles_per_block + tile; the
// item records the tile and (in `pad`) the block.
__global__ void k_fill_items(const int* __restrict__ start, const int* __restrict__ end,
                             const int* __restrict__ off, int nbins, int tiles_per_block, int chunk,
                             WorkItem* __restrict__ items) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nbins) return;
  const int s = start[t], e = end[t];
  int o = off[t];
  for (int b = s; b < e; b += chunk, ++o) {
    WorkItem w;
    w.tile = t % tiles_per_block;
    w.begin = b;
    w.end = min(e, b + chunk);
    w.pad = t / tiles_per_block;
    items[o] = w;
  }
}

template <typename T>
__global__ void k_encode(const double* __restrict__ uv, const int* __restrict__ perm, int64_t M, int K, int TB,
                         Pos<T>* __restrict__ pos);
template <>
__global__ void k_encode<float>(const double* __restrict__ uv, const int* __restrict__ perm, int64_t M, int K, int TB,
                                Pos<float>* __restrict__ pos) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= M) return;
  int cell[2];
  double f[2];
  grid_cells(uv, perm_index(perm[i]), K, true, cell, f);
  Pos<float> p;
  p.u = encode_offset(cell[0] % TB, f[0]);
  p.v = encode_offset(cell[1] % TB, f[1]);
  pos[i] = p;
}
template <>
__global__ void k_encode<double>(const double* __restrict__ uv, const int* __restrict__ perm, int64_t M, int K, int TB,
                                 Pos<double>* __restrict__ pos) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= M) return;
  int c[2];
  double f[2];
  grid_cells(uv, perm_index(perm[i]), K, true, c, f);
  Pos<double> p;
  // cell + f may round up to the next integer when f is within an ulp of 1
  // (and a mirrored f may be 1): keep the sum inside the cell
  p.u = fmin(double(c[0] % TB) + f[0], nextafter(double(c[0] % TB + 1), 0.0));
  p.v = fmin(double(c[1] % TB) + f[1], nextafter(double(c[1] % TB + 1), 0.0));
  pos[i] = p;
}

// Positions on the grid of twice the resolution (K = 2 Kc) from the cells of
// the Kc grid: t = 2 (cell_c + f_c) exactly, so that tile (cell / TB) of the
// fine grid equals tile (cell_c / (TB/2)) of the coarse one and the coarse
// binning's items and order serve the fine grid unchanged.
template <typename T>
__global__ void k_encode_x2(const double* __restrict__ uv, const int* __restrict__ perm, int64_t M, int Kc, int TB,
                            Pos<T>* __restrict__ pos) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= M) return;
  int cell[2];
  double fr[2];
  grid_cells(uv, perm_index(perm[i]), Kc, true, cell, fr);
  for (int a = 0; a < 2; ++a) {
    const double t2 = 2.0 * fr[a];  // exact
    const double up = t2 >= 1.0 ? 1.0 : 0.0;
    cell[a] = (2 * cell[a] + int(up)) % TB;
    fr[a] = t2 - up;
  }
  Pos<T> p;
  if constexpr (sizeof(T) == 4) {
    p.u = encode_offset(cell[0], fr[0]);
    p.v = encode_offset(cell[1], fr[1]);
  } else {
    p.u = fmin(double(cell[0]) + fr[0], nextafter(double(cell[0] + 1), 0.0));
    p.v = fmin(double(cell[1]) + fr[1], nextafter(double(cell[1] + 1), 0.0));
  }
  pos[i] = p;
}

}  // namespace

template <typename T> cudaError_t configure_nufft() {
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = raise_smem_limit(k_degrid_w<T, ArgVal<DegridArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_grid_w<T, ArgVal<GridArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_degrid_w<T, ArgTab<DegridArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_grid_w<T, ArgTab<GridArgs<T>>>);
  return e;
}
template cudaError_t configure_nufft<float>();
template cudaError_t configure_nufft<double>();

cudaError_t set_wait_spins_nufft(uint32_t spins) { return set_module_wait_spins(spins); }

template <typename T> int degrid_patch_pitch(int TB) { return patch_pitch<T>(TB); }
template int degrid_patch_pitch<float>(int);
template int degrid_patch_pitch<double>(int);

template <typename T>
void launch_degrid(const Geometry& g, const CUtensorMap& map, const WorkItem* items, int n_items, const Pos<T>* pos,
                   const int* perm, const KbPoly<T>& kb, const DegridEp<typename cplx_t<T>::type>& ep, int* err,
                   cudaStream_t s) {
  if (n_items <= 0) return;
  const size_t sm = kWItems * warp_patch_elems<T>(g.TB) * sizeof(typename cplx_t<T>::type);
  ArgVal<DegridArgs<T>> src{DegridArgs<T>{g, nullptr, items, n_items, pos, perm, ep, err}};
  launch_pdl(k_degrid_w<T, ArgVal<DegridArgs<T>>>, (n_items + kWItems - 1) / kWItems, 32 * kWItems, sm, s, src, kb, map);
}

template <typename T>
void launch_degrid_batch(const DegridArgs<T>* tab, int count, int max_items, int max_tb, const KbPoly<T>& kb,
                         cudaStream_t s) {
  if (max_items <= 0 || count <= 0) return;
  const size_t sm = kWItems * warp_patch_elems<T>(max_tb) * sizeof(typename cplx_t<T>::type);
  CUtensorMap unused;
  std::memset(&unused, 0, sizeof(unused));
  ArgTab<DegridArgs<T>> src{tab};
  k_degrid_w<T><<<dim3((max_items + kWItems - 1) / kWItems, count), 32 * kWItems, sm, s>>>(src, kb, unused);
}

template <typename T>
void launch_grid(const Geometry& g, const WorkItem* items, int n_items, const Pos<T>* pos, const int* perm,
                 const KbPoly<T>& kb, const GridPro<typename cplx_t<T>::type>& pro, typename cplx_t<T>::type* Q,
                 cudaStream_t s) {
  if (n_items <= 0) return;
  ArgVal<GridArgs<T>> src{GridArgs<T>{g, items, n_items, pos, perm, pro, Q}};
  launch_pdl(k_grid_w<T, ArgVal<GridArgs<T>>>, (n_items + kWItems - 1) / kWItems, 32 * kWItems,
             kWItems * grid_warp_bytes<T>(g.TB), s, src, kb);
}

template <typename T>
void launch_grid_batch(const GridArgs<T>* tab, int count, int max_items, int max_tb, const KbPoly<T>& kb,
                       cudaStream_t s) {
  if (max_items <= 0 || count <= 0) return;
  ArgTab<GridArgs<T>> src{tab};
  k_grid_w<T><<<dim3((max_items + kWItems - 1) / kWItems, count), 32 * kWItems,
                kWItems * grid_warp_bytes<T>(max_tb), s>>>(src, kb);
}

template <typename T>
void launch_encode_x2(const double* uv, const int* perm, int64_t M, int Kc, int TB, Pos<T>* pos, cudaStream_t s) {
  const int tb = 256;
  k_encode_x2<T><<<int((M + tb - 1) / tb), tb, 0, s>>>(uv, perm, M, Kc, TB, pos);
}

// Fields of a binning key: block, tile, cell row and column inside the tile.
struct KeyBits { int lb, tbits, bits; };
static KeyBits key_bits(int TB, int tiles_per_block, int R) {
  KeyBits k{0, 0, 0};
  while ((1 << k.lb) < TB) ++k.lb;
  while ((1 << k.tbits) < tiles_per_block) ++k.tbits;
  int rbits = 0;
  while ((1 << rbits) < (R > 1 ? R : 1)) ++rbits;
  k.bits = 2 * k.lb + k.tbits + rbits;
  return k;
}

// Stable radix sort of (key, value) pairs by the low `bits` bits; the sorted
// values end in `vals`, the sorted keys at `keys` (which may move to `k1`).
static cudaError_t sort_pairs(uint32_t*& keys, uint32_t* k1, int* vals, int* v1, int64_t M, int bits, int nblocks,
                              int* hist, int* bsum, cudaStream_t s) {
  uint32_t* kout = k1;
  int* vin = vals;
  int* vout = v1;
  for (int shift = 0; shift < bits; shift += 8) {
    k_radix_hist<<<nblocks, kSortThreads, 0, s>>>(keys, M, shift, nblocks, hist);
    launch_scan(hist, int64_t(256) * nblocks, nullptr, bsum, s);
    k_radix_scatter<<<nblocks, kSortThreads, 0, s>>>(keys, vin, M, shift, nblocks, hist, kout, vout);
    std::swap(keys, kout);
    std::swap(vin, vout);
  }
  if (vin != vals) return cudaMemcpyAsync(vals, vin, M * sizeof(int), cudaMemcpyDeviceToDevice, s);
  return cudaGetLastError();
}

int sort_order_plain(const double* uv, int64_t M, const Geometry& g, int* order, cudaStream_t s, const int* blocks) {
  const int nt = g.K / g.TB;
  const KeyBits kb = key_bits(g.TB, nt * nt, blocks ? 64 : 1);
  const int nblocks = int((M + kSortTile - 1) / kSortTile), tb = 256;
  uint32_t *k0 = nullptr, *k1 = nullptr;
  int *v1 = nullptr, *hist = nullptr, *bsum = nullptr;
  cudaError_t e = setup_alloc(&k0, M * sizeof(uint32_t), s);
  if (e == cudaSuccess) e = setup_alloc(&k1, M * sizeof(uint32_t), s);
  if (e == cudaSuccess) e = setup_alloc(&v1, M * sizeof(int), s);
  if (e == cudaSuccess) e = setup_alloc(&hist, size_t(256) * nblocks * sizeof(int), s);
  if (e == cudaSuccess) e = setup_alloc(&bsum, 1024 * sizeof(int), s);
  if (e == cudaSuccess) {
    k_bin_keys<<<int((M + tb - 1) / tb), tb, 0, s>>>(uv, blocks, M, g.K, g.TB, kb.lb, nt, kb.tbits, false, k0, order);
    uint32_t* kin = k0;
    e = sort_pairs(kin, k1, order, v1, M, kb.bits, nblocks, hist, bsum, s);
  }
  for (void* t : {static_cast<void*>(k0), static_cast<void*>(k1), static_cast<void*>(v1), static_cast<void*>(hist),
                  static_cast<void*>(bsum)})
    if (t) cudaFreeAsync(t, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e == cudaSuccess ? 0 : (e == cudaErrorMemoryAllocation ? -2 : -3);
}

__global__ void k_slot_blocks(const WorkItem* __restrict__ items, const int* __restrict__ perm,
                              int* __restrict__ blocks) {
  const WorkItem it = items[blockIdx.x];
  for (int i = it.begin + int(threadIdx.x); i < it.end; i += blockDim.x) blocks[perm_index(perm[i])] = it.pad;
}
void launch_slot_blocks(const WorkItem* items, int n_items, const int* perm, int* blocks, cudaStream_t s) {
  if (n_items > 0) k_slot_blocks<<<n_items, 128, 0, s>>>(items, perm, blocks);
}

template <typename T>
int build_bins(const double* uv, int64_t M, const Geometry& g, int chunk, Pos<T>* pos, int* perm,
               WorkItem** items_out, int* n_items_out, cudaStream_t s, const int* blocks, int R,
               cudaMemPool_t items_pool) {
  const int tiles_per_block = (g.K / g.TB) * g.ntv;
  const int ntiles = tiles_per_block * (R > 1 ? R : 1);  // bins
  const KeyBits kb = key_bits(g.TB, tiles_per_block, R);
  const int lb = kb.lb;
  const int nblocks = int((M + kSortTile - 1) / kSortTile);
  uint32_t *k0 = nullptr, *k1 = nullptr;
  int *v1 = nullptr, *hist = nullptr, *tstart = nullptr, *tend = nullptr, *cnt = nullptr, *total = nullptr;
  int* bsum = nullptr;
  WorkItem* items = nullptr;
  int rc = 0;
  int h_total = 0;
  auto fail = [&](cudaError_t e) {
    if (e != cudaSuccess && rc == 0) rc = (e == cudaErrorMemoryAllocation) ? -2 : -3;
  };
  // temporaries from the set-up pool (no device-wide synchronisation on
  // release, reused across operator creations)
  fail(setup_alloc(&k0, M * sizeof(uint32_t), s));
  fail(setup_alloc(&k1, M * sizeof(uint32_t), s));
  fail(setup_alloc(&v1, M * sizeof(int), s));
  fail(setup_alloc(&hist, size_t(256) * nblocks * sizeof(int), s));
  fail(setup_alloc(&tstart, size_t(ntiles) * sizeof(int), s));
  fail(setup_alloc(&tend, size_t(ntiles) * sizeof(int), s));
  fail(setup_alloc(&cnt, size_t(ntiles) * sizeof(int), s));
  fail(setup_alloc(&total, sizeof(int), s));
  fail(setup_alloc(&bsum, 1024 * sizeof(int), s));
  if (rc == 0) {
    const int tb = 256;
    k_bin_keys<<<int((M + tb - 1) / tb), tb, 0, s>>>(uv, R > 1 ? blocks : nullptr, M, g.K, g.TB, lb, g.ntv,
                                                     kb.tbits, true, k0, perm);
    uint32_t* kin = k0;
    fail(sort_pairs(kin, k1, perm, v1, M, kb.bits, nblocks, hist, bsum, s));
    fail(cudaMemsetAsync(tstart, 0, size_t(ntiles) * sizeof(int), s));
    fail(cudaMemsetAsync(tend, 0, size_t(ntiles) * sizeof(int), s));
    // bin index = key >> 2 lb = block << tbits | tile; with tiles_per_block a power of
    // two this equals block * tiles_per_block + tile
    k_tile_bounds<<<int((M + tb - 1) / tb), tb, 0, s>>>(kin, M, 2 * lb, tstart, tend);
    k_chunk_counts<<<(ntiles + tb - 1) / tb, tb, 0, s>>>(tstart, tend, ntiles, chunk, cnt);
    launch_scan(cnt, ntiles, total, bsum, s);
    fail(cudaMemcpyAsync(&h_total, total, sizeof(int), cudaMemcpyDeviceToHost, s));
    fail(cudaStreamSynchronize(s));
    fail(cudaGetLastError());
  }
  if (rc == 0) {
    const size_t ib = size_t(h_total > 0 ? h_total : 1) * sizeof(WorkItem);
    fail(items_pool ? cudaMallocFromPoolAsync(reinterpret_cast<void**>(&items), ib, items_pool, s)
                    : cudaMalloc(&items, ib));
    if (rc == 0) {
      const int tb = 256;
      k_fill_items<<<(ntiles + tb - 1) / tb, tb, 0, s>>>(tstart, tend, cnt, ntiles, tiles_per_block, chunk, items);
      k_encode<T><<<int((M + tb - 1) / tb), tb, 0, s>>>(uv, perm, M, g.K, g.TB, pos);
      fail(cudaStreamSynchronize(s));
      fail(cudaGetLastError());
      // largest items first (stable): whole-warp items then finish together
      if (rc == 0 && h_total > 1) {
        std::vector<WorkItem> h(h_total), o(h_total);
        fail(cudaMemcpyAsync(h.data(), items, h.size() * sizeof(WorkItem), cudaMemcpyDeviceToHost, s));
        fail(cudaStreamSynchronize(s));
        // stable counting sort by length, longest first (lengths <= chunk)
        std::vector<int> first(size_t(chunk) + 2, 0);
        for (const WorkItem& w : h) first[size_t(chunk - (w.end - w.begin)) + 1] += 1;
        for (size_t k = 1; k < first.size(); ++k) first[k] += first[k - 1];
        for (const WorkItem& w : h) o[size_t(first[size_t(chunk - (w.end - w.begin))]++)] = w;
        fail(cudaMemcpyAsync(items, o.data(), o.size() * sizeof(WorkItem), cudaMemcpyHostToDevice, s));
        fail(cudaStreamSynchronize(s));
      }
    }
  }
  for (void* t : {static_cast<void*>(k0), static_cast<void*>(k1), static_cast<void*>(v1), static_cast<void*>(hist),
                  static_cast<void*>(bsum), static_cast<void*>(tstart), static_cast<void*>(tend),
                  static_cast<void*>(cnt), static_cast<void*>(total)})
    if (t) cudaFreeAsync(t, s);
  if (rc != 0) {
    if (items_pool) cudaFreeAsync(items, s);
    else cudaFree(items);
    return rc;
  }
  *items_out = items;
  *n_items_out = h_total;
  return 0;
}

#define INST(T)                                                                                              \
  template void launch_degrid<T>(const Geometry&, const CUtensorMap&, const WorkItem*, int, const Pos<T>*,      \
                                 const int*, const KbPoly<T>&, const DegridEp<cplx_t<T>::type>&, int*,          \
                                 cudaStream_t);                                                                \
  template void launch_grid<T>(const Geometry&, const WorkItem*, int, const Pos<T>*, const int*,                \
                               const KbPoly<T>&, const GridPro<cplx_t<T>::type>&, cplx_t<T>::type*,             \
                               cudaStream_t);                                                                  \
  template void launch_degrid_batch<T>(const DegridArgs<T>*, int, int, int, const KbPoly<T>&, cudaStream_t);    \
  template void launch_grid_batch<T>(const GridArgs<T>*, int, int, int, const KbPoly<T>&, cudaStream_t);        \
  template void launch_encode_x2<T>(const double*, const int*, int64_t, int, int, Pos<T>*, cudaStream_t);     \
  template int build_bins<T>(const double*, int64_t, const Geometry&, int, Pos<T>*, int*, WorkItem**, int*,     \
                             cudaStream_t, const int*, int, cudaMemPool_t);
INST(float)
INST(double)
#undef INST

}  // namespace purify
