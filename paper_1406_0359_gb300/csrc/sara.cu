// SARA dictionary Psi = [Dirac, Db1, ..., Db8] / 3 (Section 2.2) on the GPU,
// or a sub-dictionary of it (Section 4's BP = Dirac, BPDb8 = Db8, ...): the q
// selected bases, each scaled by 1/sqrt(q), coefficients basis-major in
// increasing basis order (Dirac first).
//
// Analysis (Psi^H): one launch per wavelet level covers all selected
// Daubechies filters (blockIdx.z = filter slot; the first level's also the Dirac
// block).  A CTA stages its periodic input tile once in shared memory, filters the rows (axis 1) into low/high halves, then the
// columns (axis 0), and writes the three detail sub-bands of the level to their
// Mallat positions; the low-low band goes to a scratch band for the next level
// (or to its final place at the last level).  Convention, per axis:
//     lo[k] = sum_m h[m] x[(2k + m) mod L],   hi[k] = sum_m g[m] x[(2k + m) mod L].
// Synthesis (Psi) is the exact adjoint, one launch per level from the coarsest;
// the finest level is fused across all eight filters and the Dirac block, so
// the image is written once.
//
// SDMM fusions (Algorithm 1, blocks i = 1, 2): the analysis epilogue applies
// the l1 proximity operator to v = Psi^H x_hat + z_1 (soft threshold at
// gamma w), updates z_1 and emits 2 r_1 - v_1 for the synthesis, plus FP64
// partial sums of the objective ||W Psi^H x_hat||_1; the final synthesis
// epilogue applies the positivity block and writes x_1 + x_2.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/purify.h"
#include "host_math.h"
#include "internal.h"

namespace purify {

namespace {

constexpr int kTH = 16;  // analysis: output coefficients per tile side
constexpr int kTO = 32;  // synthesis: output samples per tile side
constexpr int kThr = 256;

// Periodic index i mod L (the integer modulo only off the common in-range case).
PD int wrap(int i, int L) {
  if (i >= 0 && i < L) return i;
  i %= L;
  return i < 0 ? i + L : i;
}

// Final coefficient epilogue: plain store or fused l1 prox.
template <typename T> struct CoefOut {
  T* c;           // plain: Psi^H x [9][n][n]
  int prox;       // 0: plain, 1: l1 block
  T* z1;
  const T* w;
  T* cs;          // prox output 2r - v
  T gamma;
};

template <typename T> PD void emit(const CoefOut<T>& o, size_t idx, T alpha, Acc<T>& part) {
  if (!o.prox) {
    o.c[idx] = alpha;
    return;
  }
  const T wj = o.w ? o.w[idx] : T(1);
  const T v = alpha + o.z1[idx];
  const T thr = o.gamma * wj;
  const T av = fabs(v);
  const T r = av > thr ? copysign(av - thr, v) : T(0);
  o.z1[idx] = v - r;
  o.cs[idx] = T(2) * r - v;
  part.add_prod(wj, fabs(alpha));
}

// emit for NE coefficients at once: every w and z_1 load precedes the first
// store (the stores may alias them, which would otherwise serialise one memory
// round trip per coefficient).
template <int NE, typename T>
PD void emit_n(const CoefOut<T>& o, const size_t (&idx)[NE], const T (&alpha)[NE], int ne, Acc<T>& part) {
  if (!o.prox) {
#pragma unroll
    for (int k = 0; k < NE; ++k)
      if (k < ne) o.c[idx[k]] = alpha[k];
    return;
  }
  T wj[NE], z[NE];
#pragma unroll
  for (int k = 0; k < NE; ++k) {
    wj[k] = (k < ne && o.w) ? o.w[idx[k]] : T(1);
    z[k] = k < ne ? o.z1[idx[k]] : T(0);
  }
#pragma unroll
  for (int k = 0; k < NE; ++k) {
    if (k >= ne) continue;
    const T v = alpha[k] + z[k];
    const T thr = o.gamma * wj[k];
    const T av = fabs(v);
    const T r = av > thr ? copysign(av - thr, v) : T(0);
    o.z1[idx[k]] = v - r;
    o.cs[idx[k]] = T(2) * r - v;
    part.add_prod(wj[k], fabs(alpha[k]));
  }
}

template <typename T> struct AnaArgs {
  const T* in;
  size_t in_stride;  // elements between filters' input bands (0: shared input)
  int L;             // input band side
  int n;
  T* s_out;          // LL scratch [filter slot][H*H]
  int last;          // LL band is final
  int slot0;         // coefficient block of filter slot 0 (1 when the Dirac basis is selected)
  int nf;            // filter slots
  int fid[kMaxDb];   // Daubechies filter (K - 1) of each filter slot
  T scale;           // 1 / sqrt(number of bases)
  CoefOut<T> out;
  double* partials;  // per-CTA objective partials, Acc<T> in double slots (prox only)
};

template <typename T, int F>
__device__ void ana_body(const AnaArgs<T>& A, const T* __restrict__ h, const T* __restrict__ g, int z, T* sm,
                         double* red) {
  constexpr int W = 2 * kTH + F - 2;
  T* X = sm;
  T* lo = X + W * W;
  T* hi = lo + W * kTH;
  const int L = A.L, H = L / 2, n = A.n;
  const int r0 = blockIdx.y * kTH, c0 = blockIdx.x * kTH;
  const T* in = A.in + size_t(z) * A.in_stride;
  {
    // warps take rows, lanes columns: each lane wraps its few columns once
    constexpr int NC = (W + 31) / 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int cols[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) cols[k] = wrap(2 * c0 + lane + 32 * k, L);
    for (int ir = wid; ir < W; ir += kThr / 32) {
      const T* row = in + size_t(wrap(2 * r0 + ir, L)) * L;
#pragma unroll
      for (int k = 0; k < NC; ++k)
        if (lane + 32 * k < W) X[ir * W + lane + 32 * k] = row[cols[k]];
    }
  }
  __syncthreads();
  // row filtering, CB consecutive outputs per item: they share F + 2 CB - 2 inputs
  constexpr int CB = 4;
  for (int e = threadIdx.x; e < W * (kTH / CB); e += kThr) {
    const int ir = e / (kTH / CB), cg = e - ir * (kTH / CB);
    const T* xr = X + ir * W + 2 * CB * cg;
    T xv[F + 2 * CB - 2];
#pragma unroll
    for (int k = 0; k < F + 2 * CB - 2; ++k) xv[k] = xr[k];
#pragma unroll
    for (int b = 0; b < CB; ++b) {
      T sl = 0, sh = 0;
#pragma unroll
      for (int m = 0; m < F; ++m) {
        sl = fma(h[m], xv[2 * b + m], sl);
        sh = fma(g[m], xv[2 * b + m], sh);
      }
      lo[ir * kTH + CB * cg + b] = sl;
      hi[ir * kTH + CB * cg + b] = sh;
    }
  }
  __syncthreads();
  // Large FP64 levels are bound by the FP64 units: the next level's CTAs, started
  // early, pile up on the SMs that finish first (Db8, 4 levels, n = 512: 87 us
  // against 75); after the last level whatever follows may start
  if (sizeof(T) == 4 || A.n <= 256 || A.last) pdl_trigger();
  Acc<T> part;
  const int r = threadIdx.x / kTH, c = threadIdx.x - r * kTH;
  const int R = r0 + r, Cc = c0 + c;
  if (R < H && Cc < H) {
    T ll = 0, lh = 0, hl = 0, hh = 0;
#pragma unroll
    for (int m = 0; m < F; ++m) {
      const T a = lo[(2 * r + m) * kTH + c], b = hi[(2 * r + m) * kTH + c];
      ll = fma(h[m], a, ll);
      lh = fma(h[m], b, lh);
      hl = fma(g[m], a, hl);
      hh = fma(g[m], b, hh);
    }
    const size_t base = size_t(A.slot0 + z) * n * n;
    const T sc = A.scale;
    const size_t idx[4] = {base + size_t(R) * n + (H + Cc), base + size_t(H + R) * n + Cc,
                           base + size_t(H + R) * n + (H + Cc), base + size_t(R) * n + Cc};
    const T val[4] = {lh * sc, hl * sc, hh * sc, ll * sc};
    emit_n<4>(A.out, idx, val, A.last ? 4 : 3, part);
    if (!A.last) A.s_out[size_t(z) * H * H + size_t(R) * H + Cc] = ll;
  }
  if (A.partials) {
    const Acc<T> t = block_merge<kThr>(part, red);
    if (threadIdx.x == 0)
      reinterpret_cast<Acc<T>*>(A.partials)[(size_t(z) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t;
  }
}

// The Dirac block c_0 = x / sqrt(q) of the pixels under a level-1 tile of TO x TO
// outputs (filter slot nf of that level's launch).
template <typename T, int TO> __device__ void ana_dirac(const AnaArgs<T>& A, int z, double* red) {
  constexpr int S = 2 * TO;
  const int n = A.n, r0 = blockIdx.y * S, c0 = blockIdx.x * S;
  Acc<T> part;
  for (int e0 = threadIdx.x; e0 < S * S; e0 += 4 * kThr) {
    size_t idx[4];
    T val[4];
    int ne = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int e = e0 + k * kThr, r = r0 + e / S, c = c0 + e % S;
      const bool in = r < n && c < n;
      idx[k] = in ? size_t(r) * n + c : 0;
      val[k] = in ? A.in[idx[k]] * A.scale : T(0);
      ne += in;
    }
    if (ne == 4) {
      emit_n<4>(A.out, idx, val, 4, part);
    } else {  // a tile past the image's edge
      for (int k = 0; k < 4; ++k) {
        const int e = e0 + k * kThr;
        if (r0 + e / S < n && c0 + e % S < n) emit(A.out, idx[k], val[k], part);
      }
    }
  }
  if (A.partials) {
    const Acc<T> t = block_merge<kThr>(part, red);
    if (threadIdx.x == 0)
      reinterpret_cast<Acc<T>*>(A.partials)[(size_t(z) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t;
  }
}

// One analysis level; blockIdx.z = instance * nz + slot: the nf filters and, on
// the first level with the Dirac basis, its block (nz = nf + 1).
template <typename T, typename Src>
__global__ void __launch_bounds__(kThr) k_ana_level(const __grid_constant__ Src src, int nz, DbFilters<T> f) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ double red[32];
  T* sm = reinterpret_cast<T*>(sm_raw);
  const int inst = int(blockIdx.z) / nz, z = int(blockIdx.z) - inst * nz;
  decltype(auto) A = src.get_at(inst);
  pdl_wait();
  if (z == A.nf) {
    ana_dirac<T, kTH>(A, z, red);
    return;
  }
  const int k = A.fid[z];
  const T* h = f.h[k];
  const T* g = f.g[k];
  switch (k) {
    case 0: ana_body<T, 2>(A, h, g, z, sm, red); break;
    case 1: ana_body<T, 4>(A, h, g, z, sm, red); break;
    case 2: ana_body<T, 6>(A, h, g, z, sm, red); break;
    case 3: ana_body<T, 8>(A, h, g, z, sm, red); break;
    case 4: ana_body<T, 10>(A, h, g, z, sm, red); break;
    case 5: ana_body<T, 12>(A, h, g, z, sm, red); break;
    case 6: ana_body<T, 14>(A, h, g, z, sm, red); break;
    default: ana_body<T, 16>(A, h, g, z, sm, red); break;
  }
}

// Fine analysis levels (FP32, band sides with enough 32 x 32 output tiles to
// fill the chip): the same arithmetic on four times the outputs per CTA.  A row
// item gives 4 low and 4 high outputs from F + 6 inputs, a column item 4 x 4
// sub-band outputs from 2 (F + 6): 57 instead of 72 instructions per output, the
// input's halo read 1.5 instead of 2.1 times, shared memory read by conflict-free
// 8-byte (rows 2 mod 4 words apart) and 4-byte accesses.  Bound by instruction
// issue: level 1 of a 1024^2 image 26 us against 36 with 16 x 16 tiles.
constexpr int kFA = 32;                     // output coefficients per tile side
constexpr int kFP = kFA + 4;                // pitch of the row-filtered halves
template <int F> struct FineAna {
  static constexpr int W = 2 * kFA + F - 2;                 // input tile side
  static constexpr int WP = (W / 2) % 2 ? W : W + 2;        // its pitch
  static constexpr size_t smem = size_t(W * WP + 2 * W * kFP) * sizeof(float);
};

template <int F>
__device__ void ana_fine_body(const AnaArgs<float>& A, const float* __restrict__ h, const float* __restrict__ g, int z,
                              float* sm, double* red) {
  constexpr int W = FineAna<F>::W, WP = FineAna<F>::WP, NI = F + 6;
  float* X = sm;
  float* lo = X + W * WP;
  float* hi = lo + W * kFP;
  const int L = A.L, H = L / 2, n = A.n;
  const int r0 = blockIdx.y * kFA, c0 = blockIdx.x * kFA;
  const float* in = A.in + size_t(z) * A.in_stride;
  const bool al = (reinterpret_cast<size_t>(in) & 7) == 0;  // a caller's image need not be
  for (int e = threadIdx.x; e < W * (W / 2); e += kThr) {
    const int ir = e / (W / 2), pc = e - ir * (W / 2);
    const float* src = in + size_t((2 * r0 + ir) & (L - 1)) * L + ((2 * (c0 + pc)) & (L - 1));
    float2 v;
    if (al) v = *reinterpret_cast<const float2*>(src);
    else v = make_float2(src[0], src[1]);
    *reinterpret_cast<float2*>(X + ir * WP + 2 * pc) = v;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < W * (kFA / 4); e += kThr) {
    const int cg = e / W, ir = e - cg * W;
    float xv[NI];
#pragma unroll
    for (int k = 0; k < NI; k += 2) {
      const float2 v = *reinterpret_cast<const float2*>(X + ir * WP + 8 * cg + k);
      xv[k] = v.x;
      xv[k + 1] = v.y;
    }
    float sl[4], sh[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      sl[b] = sh[b] = 0.f;
#pragma unroll
      for (int m = 0; m < F; ++m) {
        sl[b] = fmaf(h[m], xv[2 * b + m], sl[b]);
        sh[b] = fmaf(g[m], xv[2 * b + m], sh[b]);
      }
    }
    *reinterpret_cast<float4*>(lo + ir * kFP + 4 * cg) = make_float4(sl[0], sl[1], sl[2], sl[3]);
    *reinterpret_cast<float4*>(hi + ir * kFP + 4 * cg) = make_float4(sh[0], sh[1], sh[2], sh[3]);
  }
  __syncthreads();
  pdl_trigger();
  static_assert(kThr == kFA * kFA / 4, "one column item per thread");
  const int c = threadIdx.x % kFA, rg = threadIdx.x / kFA;
  const int R = r0 + 4 * rg, Cc = c0 + c;
  float v[4][4];  // [ll, lh, hl, hh][output row]
  {
    float xv[NI];
#pragma unroll
    for (int k = 0; k < NI; ++k) xv[k] = lo[(8 * rg + k) * kFP + c];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      v[0][b] = v[2][b] = 0.f;
#pragma unroll
      for (int m = 0; m < F; ++m) {
        v[0][b] = fmaf(h[m], xv[2 * b + m], v[0][b]);
        v[2][b] = fmaf(g[m], xv[2 * b + m], v[2][b]);
      }
    }
#pragma unroll
    for (int k = 0; k < NI; ++k) xv[k] = hi[(8 * rg + k) * kFP + c];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      v[1][b] = v[3][b] = 0.f;
#pragma unroll
      for (int m = 0; m < F; ++m) {
        v[1][b] = fmaf(h[m], xv[2 * b + m], v[1][b]);
        v[3][b] = fmaf(g[m], xv[2 * b + m], v[3][b]);
      }
    }
  }
  Acc<float> part;
  const size_t base = size_t(A.slot0 + z) * n * n + size_t(R) * n + Cc;
  const size_t off[4] = {0, size_t(H), size_t(H) * n, size_t(H) * n + H};
#pragma unroll
  for (int q = 1; q < 5; ++q) {  // lh, hl, hh, then ll where it is final
    if (q == 4 && !A.last) break;
    size_t idx[4];
    float val[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      idx[b] = base + off[q & 3] + size_t(b) * n;
      val[b] = v[q & 3][b] * A.scale;
    }
    emit_n<4>(A.out, idx, val, 4, part);
  }
  if (!A.last) {
#pragma unroll
    for (int b = 0; b < 4; ++b) A.s_out[size_t(z) * H * H + size_t(R + b) * H + Cc] = v[0][b];
  }
  if (A.partials) {
    const Acc<float> t = block_merge<kThr>(part, red);
    if (threadIdx.x == 0)
      reinterpret_cast<Acc<float>*>(A.partials)[(size_t(z) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t;
  }
}

template <typename Src>
__global__ void __launch_bounds__(kThr, 4) k_ana_fine(const __grid_constant__ Src src, int nz, DbFilters<float> f) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ double red[32];
  float* sm = reinterpret_cast<float*>(sm_raw);
  const int inst = int(blockIdx.z) / nz, z = int(blockIdx.z) - inst * nz;
  decltype(auto) A = src.get_at(inst);
  pdl_wait();
  if (z == A.nf) {
    ana_dirac<float, kFA>(A, z, red);
    return;
  }
  switch (A.fid[z]) {
    case 0: ana_fine_body<2>(A, f.h[0], f.g[0], z, sm, red); break;
    case 1: ana_fine_body<4>(A, f.h[1], f.g[1], z, sm, red); break;
    case 2: ana_fine_body<6>(A, f.h[2], f.g[2], z, sm, red); break;
    case 3: ana_fine_body<8>(A, f.h[3], f.g[3], z, sm, red); break;
    case 4: ana_fine_body<10>(A, f.h[4], f.g[4], z, sm, red); break;
    case 5: ana_fine_body<12>(A, f.h[5], f.g[5], z, sm, red); break;
    case 6: ana_fine_body<14>(A, f.h[6], f.g[6], z, sm, red); break;
    default: ana_fine_body<16>(A, f.h[7], f.g[7], z, sm, red); break;
  }
}

// Dirac block of a dictionary without wavelets: c_0 = x (with the prox epilogue when fused).
template <typename T> struct DiracArgs {
  const T* x;
  size_t N;
  T scale;
  CoefOut<T> out;
  double* partials;
};
template <typename T, typename Src>
__global__ void __launch_bounds__(kThr) k_dirac(Src src) {
  __shared__ double red[32];
  decltype(auto) a = src.get();
  const T* __restrict__ x = a.x;
  const size_t N = a.N;
  const T scale = a.scale;
  const CoefOut<T>& out = a.out;
  double* partials = a.partials;
  Acc<T> part;
  const size_t i = size_t(blockIdx.x) * kThr + threadIdx.x;
  if (i < N) emit(out, i, x[i] * scale, part);
  if (partials) {
    const Acc<T> t = block_merge<kThr>(part, red);
    if (threadIdx.x == 0) reinterpret_cast<Acc<T>*>(partials)[blockIdx.x] = t;
  }
}

template <typename T> struct SynArgs {
  const T* c;       // final coefficients [q][n][n] (plain Psi^H layout)
  const T* s_in;    // LL band from the coarser synthesis level, or null (LL is final in c)
  int H;            // coefficient band side; output side L = 2H
  int n;
  T* s_out;         // [filter slot][L*L] (intermediate levels)
  int slot0;        // coefficient block of filter slot 0 (1 when the Dirac basis is selected)
  int nf;           // selected Daubechies filters
  int fid[kMaxDb];  // Daubechies filter (K - 1) of each filter slot
  T scale;          // 1 / sqrt(number of bases)
  // finest level (fused over filters):
  int pos_block;    // apply the positivity block
  T* x_out;
  const T* xh;
  T* z2;
};

// Output samples of thread t in a synthesis tile: acc[2 q + p] is row
// il = e / (kTO/2), column jl = 2 (e mod kTO/2) + p of item e = t + q kThr.
PD void syn_out_pos(int q, int& il, int& jl) {
  const int e = int(threadIdx.x) + (q >> 1) * kThr;
  il = e / (kTO / 2);
  jl = 2 * (e % (kTO / 2)) + (q & 1);
}
constexpr int kUP = 48;  // row pitch of the upsampled rows (16 mod 32: two rows of a warp's reads hit distinct banks)

// One filter's level synthesis of the output tile (i0, j0).  Upsampling along
// rows then columns; outputs 2j and 2j + 1 of either pass read the same
// inputs (rows / columns j - t + F/2), so each item computes both parities.
template <typename T, int F>
__device__ void syn_body(const SynArgs<T>& S, const T* __restrict__ h, const T* __restrict__ g, int z, T* sm,
                         int i0, int j0, T (&acc)[kTO * kTO / kThr], bool accumulate) {
  constexpr int CT = kTO / 2 + F / 2, HF = F / 2;
  static_assert(CT <= kUP && kTO * kTO / kThr == 4, "tile shape");
  T* LLt = sm;
  T* LHt = LLt + CT * CT;
  T* HLt = LHt + CT * CT;
  T* HHt = HLt + CT * CT;
  T* Ulo = HHt + CT * CT;      // [kTO][kUP]
  T* Uhi = Ulo + kTO * kUP;
  const int H = S.H, n = S.n, L = 2 * H;
  const T* cb = S.c + size_t(S.slot0 + z) * n * n;
  const int rb = i0 / 2 - F / 2, cbase = j0 / 2 - F / 2;
  {
    // warps take rows, lanes columns (CT <= 24 columns)
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int lc = lane;
    const int c = wrap(cbase + lc, H);
    const T* sb = S.s_in ? S.s_in + size_t(z) * H * H : nullptr;
    for (int lr = wid; lr < CT; lr += kThr / 32) {
      if (lc >= CT) continue;
      const int r = wrap(rb + lr, H);
      const int e = lr * CT + lc;
      LLt[e] = sb ? sb[size_t(r) * H + c] : cb[size_t(r) * n + c];
      LHt[e] = cb[size_t(r) * n + (H + c)];
      HLt[e] = cb[size_t(H + r) * n + c];
      HHt[e] = cb[size_t(H + r) * n + (H + c)];
    }
  }
  __syncthreads();
  // rows il = 2j + par: U(il, lc) = sum_t h[par + 2t] LL(j - t + HF, lc) + g[par + 2t] HL(...)
  for (int e = threadIdx.x; e < (kTO / 2) * CT; e += kThr) {
    const int j = e / CT, lc = e - j * CT;
    const int o = (j + HF) * CT + lc;
    T ul0 = 0, ul1 = 0, uh0 = 0, uh1 = 0;
#pragma unroll
    for (int t = 0; t < HF; ++t) {
      const T a = LLt[o - t * CT], b = HLt[o - t * CT], c = LHt[o - t * CT], d = HHt[o - t * CT];
      ul0 = fma(h[2 * t], a, fma(g[2 * t], b, ul0));
      ul1 = fma(h[2 * t + 1], a, fma(g[2 * t + 1], b, ul1));
      uh0 = fma(h[2 * t], c, fma(g[2 * t], d, uh0));
      uh1 = fma(h[2 * t + 1], c, fma(g[2 * t + 1], d, uh1));
    }
    Ulo[(2 * j) * kUP + lc] = ul0;
    Ulo[(2 * j + 1) * kUP + lc] = ul1;
    Uhi[(2 * j) * kUP + lc] = uh0;
    Uhi[(2 * j + 1) * kUP + lc] = uh1;
  }
  __syncthreads();
  // columns jl = 2j + par: X(il, jl) = sum_t h[par + 2t] Ulo(il, j - t + HF) + g[par + 2t] Uhi(...)
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int e = threadIdx.x + q * kThr;
    const int il = e / (kTO / 2), j = e % (kTO / 2);
    const int o = il * kUP + j + HF;
    T v0 = 0, v1 = 0;
#pragma unroll
    for (int t = 0; t < HF; ++t) {
      const T a = Ulo[o - t], b = Uhi[o - t];
      v0 = fma(h[2 * t], a, fma(g[2 * t], b, v0));
      v1 = fma(h[2 * t + 1], a, fma(g[2 * t + 1], b, v1));
    }
    if (accumulate) {
      acc[2 * q] += v0;
      acc[2 * q + 1] += v1;
    } else if (i0 + il < L && j0 + 2 * j + 1 < L) {
      T* dst = S.s_out + size_t(z) * L * L + size_t(i0 + il) * L + (j0 + 2 * j);
      dst[0] = v0;
      dst[1] = v1;
    }
  }
  __syncthreads();
}

template <typename T>
__device__ void syn_dispatch(const SynArgs<T>& S, const DbFilters<T>& f, int z, int k, T* sm, int i0, int j0,
                             T (&acc)[kTO * kTO / kThr], bool accumulate) {
  const T* h = f.h[k];
  const T* g = f.g[k];
  switch (k) {
    case 0: syn_body<T, 2>(S, h, g, z, sm, i0, j0, acc, accumulate); break;
    case 1: syn_body<T, 4>(S, h, g, z, sm, i0, j0, acc, accumulate); break;
    case 2: syn_body<T, 6>(S, h, g, z, sm, i0, j0, acc, accumulate); break;
    case 3: syn_body<T, 8>(S, h, g, z, sm, i0, j0, acc, accumulate); break;
    case 4: syn_body<T, 10>(S, h, g, z, sm, i0, j0, acc, accumulate); break;
    case 5: syn_body<T, 12>(S, h, g, z, sm, i0, j0, acc, accumulate); break;
    case 6: syn_body<T, 14>(S, h, g, z, sm, i0, j0, acc, accumulate); break;
    default: syn_body<T, 16>(S, h, g, z, sm, i0, j0, acc, accumulate); break;
  }
}

// Intermediate synthesis level: blockIdx.z = instance * nf + filter slot,
// output band -> scratch.
template <typename T, typename Src>
__global__ void __launch_bounds__(kThr) k_syn_level(const __grid_constant__ Src src, int nf, DbFilters<T> f) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  T* sm = reinterpret_cast<T*>(sm_raw);
  const int inst = int(blockIdx.z) / nf, z = int(blockIdx.z) - inst * nf;
  decltype(auto) S = src.get_at(inst);
  T acc[kTO * kTO / kThr];
  pdl_wait();
  syn_dispatch(S, f, z, S.fid[z], sm, blockIdx.y * kTO, blockIdx.x * kTO, acc, false);
}

// Finest level: all selected filters and the Dirac block summed into the
// image (ALL: the eight filters in slots 0..7, unrolled); the common scale
// 1/sqrt(q) is applied here, once.
template <typename T, bool ALL, typename Src>
__global__ void __launch_bounds__(kThr) k_syn_final(const __grid_constant__ Src src, DbFilters<T> f) {
  decltype(auto) S = src.get_at(int(blockIdx.z));
  extern __shared__ __align__(16) unsigned char sm_raw[];
  T* sm = reinterpret_cast<T*>(sm_raw);
  const int i0 = blockIdx.y * kTO, j0 = blockIdx.x * kTO;
  T acc[kTO * kTO / kThr];
#pragma unroll
  for (int q = 0; q < kTO * kTO / kThr; ++q) acc[q] = 0;
  pdl_wait();
  if constexpr (ALL) {
#pragma unroll
    for (int k = 0; k < kMaxDb; ++k) syn_dispatch(S, f, k, k, sm, i0, j0, acc, true);
  } else {
    for (int z = 0; z < S.nf; ++z) syn_dispatch(S, f, z, S.fid[z], sm, i0, j0, acc, true);
  }
  const int n = S.n;
#pragma unroll
  for (int q = 0; q < kTO * kTO / kThr; ++q) {
    int il, jl;
    syn_out_pos(q, il, jl);
    if (i0 + il >= n || j0 + jl >= n) continue;
    const size_t idx = size_t(i0 + il) * n + (j0 + jl);
    const T x1 = (S.slot0 ? acc[q] + S.c[idx] : acc[q]) * S.scale;  // Dirac block
    if (S.pos_block) {
      const T v2 = S.xh[idx] + S.z2[idx];
      const T r2 = v2 > T(0) ? v2 : T(0);
      S.z2[idx] = v2 - r2;
      S.x_out[idx] = x1 + (T(2) * r2 - v2);
    } else {
      S.x_out[idx] = x1;
    }
  }
}

// Fine synthesis levels (FP32, 64 x 64 output tiles): the same arithmetic with
// the tile's halo read 1.6 instead of 2.3 times and both passes in items of 8
// (columns) and 16 (rows) outputs, 4 loads per output and filter instead of 12;
// the next filter's sub-bands arrive by asynchronous copies while one is
// transformed (two barriers per filter, no exposed load).  Bound by instruction
// issue: the finest level of a 1024^2 image 31 us against 47, the next 12 against 20.
constexpr int kFS = 64;             // output samples per tile side
constexpr int kFThr = 320;          // threads: one column item (at most 40 x 8) each
constexpr int kFC = kFS / 2 + 8;    // coefficient tile side, at most
constexpr int kFU = 42;             // pitch of the upsampled rows (2 mod 4 words)
constexpr size_t kFineSynBand = 4 * size_t(kFC) * kFC;  // the four sub-band tiles
constexpr size_t kFineSynU = 2 * size_t(kFS) * kFU;
constexpr int kFItems = kFS * kFS / 8;                   // row items of 8 outputs
constexpr int kFQ = (kFItems + kFThr - 1) / kFThr;       // per thread, at most
constexpr int kFAcc = 8 * kFQ;

PD void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
PD void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> PD void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Start the copies of filter slot z's sub-band tiles (HF = half its length).
PD void syn_fine_load(const SynArgs<float>& S, int z, int HF, float* band, int i0, int j0) {
  const int CT = kFS / 2 + HF, H = S.H, n = S.n;
  const float* cb = S.c + size_t(S.slot0 + z) * n * n;
  const float* sb = S.s_in ? S.s_in + size_t(z) * H * H : cb;
  const int sp = S.s_in ? H : n;  // pitch of the low band
  const int rb = i0 / 2 - HF, cbase = j0 / 2 - HF;
  for (int lr = int(threadIdx.x) >> 5; lr < CT; lr += kFThr / 32) {
    const int r = (rb + lr) & (H - 1);
    for (int lc = int(threadIdx.x) & 31; lc < CT; lc += 32) {
      const int c = (cbase + lc) & (H - 1), e = lr * kFC + lc;
      cp_async4(band + e, sb + size_t(r) * sp + c);
      cp_async4(band + kFC * kFC + e, cb + size_t(r) * n + (H + c));
      cp_async4(band + 2 * kFC * kFC + e, cb + size_t(H + r) * n + c);
      cp_async4(band + 3 * kFC * kFC + e, cb + size_t(H + r) * n + (H + c));
    }
  }
  cp_async_commit();
}

// One filter's contribution to the thread's outputs: acc[8 q + k] is row il,
// column 8 jg + k of item e = tid + q kFThr = jg kFS + il.
template <int F>
__device__ void syn_fine_body(const float* __restrict__ h, const float* __restrict__ g, const float* band, float* U,
                              float (&acc)[kFAcc]) {
  constexpr int HF = F / 2, CT = kFS / 2 + HF;
  static_assert(CT * (kFS / 8) <= kFThr, "one column item per thread");
  if (int(threadIdx.x) < CT * (kFS / 8)) {
    const int e = threadIdx.x, jg = e / CT, lc = e - jg * CT;
#pragma unroll
    for (int hb = 0; hb < 2; ++hb) {  // the low, then the high column band
      const float* a = band + hb * kFC * kFC + (4 * jg + 1) * kFC + lc;
      const float* b = a + 2 * kFC * kFC;
      float av[HF + 3], bv[HF + 3];
#pragma unroll
      for (int k = 0; k < HF + 3; ++k) {
        av[k] = a[k * kFC];
        bv[k] = b[k * kFC];
      }
      float* u = U + hb * kFS * kFU + 8 * jg * kFU + lc;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float u0 = 0.f, u1 = 0.f;
#pragma unroll
        for (int t = 0; t < HF; ++t) {
          const float x = av[j + HF - 1 - t], y = bv[j + HF - 1 - t];
          u0 = fmaf(h[2 * t], x, fmaf(g[2 * t], y, u0));
          u1 = fmaf(h[2 * t + 1], x, fmaf(g[2 * t + 1], y, u1));
        }
        u[(2 * j) * kFU] = u0;
        u[(2 * j + 1) * kFU] = u1;
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kFQ; ++q) {
    const int e = int(threadIdx.x) + q * kFThr, il = e % kFS, jg = e / kFS;
    if (e >= kFItems) break;
    constexpr int NL = (HF + 5) / 2 * 2;  // columns 4 jg .. 4 jg + HF + 3, in pairs
    float lv[NL], hv[NL];
#pragma unroll
    for (int k = 0; k < NL; k += 2) {
      const float2 a = *reinterpret_cast<const float2*>(U + il * kFU + 4 * jg + k);
      const float2 b = *reinterpret_cast<const float2*>(U + kFS * kFU + il * kFU + 4 * jg + k);
      lv[k] = a.x;
      lv[k + 1] = a.y;
      hv[k] = b.x;
      hv[k + 1] = b.y;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float v0 = 0.f, v1 = 0.f;
#pragma unroll
      for (int t = 0; t < HF; ++t) {
        const float x = lv[j + HF - t], y = hv[j + HF - t];
        v0 = fmaf(h[2 * t], x, fmaf(g[2 * t], y, v0));
        v1 = fmaf(h[2 * t + 1], x, fmaf(g[2 * t + 1], y, v1));
      }
      acc[8 * q + 2 * j] += v0;
      acc[8 * q + 2 * j + 1] += v1;
    }
  }
}
PD void syn_fine_dispatch(const DbFilters<float>& f, int k, const float* band, float* U, float (&acc)[kFAcc]) {
  switch (k) {
    case 0: syn_fine_body<2>(f.h[0], f.g[0], band, U, acc); break;
    case 1: syn_fine_body<4>(f.h[1], f.g[1], band, U, acc); break;
    case 2: syn_fine_body<6>(f.h[2], f.g[2], band, U, acc); break;
    case 3: syn_fine_body<8>(f.h[3], f.g[3], band, U, acc); break;
    case 4: syn_fine_body<10>(f.h[4], f.g[4], band, U, acc); break;
    case 5: syn_fine_body<12>(f.h[5], f.g[5], band, U, acc); break;
    case 6: syn_fine_body<14>(f.h[6], f.g[6], band, U, acc); break;
    default: syn_fine_body<16>(f.h[7], f.g[7], band, U, acc); break;
  }
}

// The tile's outputs through shared memory (tile[kFS][kFS + 4]) to rows of
// float4: sink(row, column, values).
template <typename Sink> PD void syn_fine_out(float* tile, const float (&acc)[kFAcc], Sink sink) {
  constexpr int TP = kFS + 4;
#pragma unroll
  for (int q = 0; q < kFQ; ++q) {
    const int e = int(threadIdx.x) + q * kFThr, il = e % kFS, jg = e / kFS;
    if (e >= kFItems) break;
    float4* d = reinterpret_cast<float4*>(tile + il * TP + 8 * jg);
    d[0] = make_float4(acc[8 * q], acc[8 * q + 1], acc[8 * q + 2], acc[8 * q + 3]);
    d[1] = make_float4(acc[8 * q + 4], acc[8 * q + 5], acc[8 * q + 6], acc[8 * q + 7]);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < kFS * kFS / 4; e += kFThr) {
    const int il = e / (kFS / 4), j = 4 * (e % (kFS / 4));
    sink(il, j, *reinterpret_cast<const float4*>(tile + il * TP + j));
  }
}

// Intermediate level: blockIdx.z = instance * nf + filter slot.
template <typename Src>
__global__ void __launch_bounds__(kFThr, 2) k_syn_fine(const __grid_constant__ Src src, int nf, DbFilters<float> f) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  float* band = reinterpret_cast<float*>(sm_raw);
  float* U = band + kFineSynBand;
  const int inst = int(blockIdx.z) / nf, z = int(blockIdx.z) - inst * nf;
  decltype(auto) S = src.get_at(inst);
  const int i0 = blockIdx.y * kFS, j0 = blockIdx.x * kFS, L = 2 * S.H;
  pdl_wait();
  syn_fine_load(S, z, S.fid[z] + 1, band, i0, j0);
  float acc[kFAcc];
#pragma unroll
  for (int q = 0; q < kFAcc; ++q) acc[q] = 0.f;
  cp_async_wait<0>();
  __syncthreads();
  syn_fine_dispatch(f, S.fid[z], band, U, acc);
  pdl_trigger();
  float* dst = S.s_out + size_t(z) * L * L + size_t(i0) * L + j0;
  syn_fine_out(band, acc, [&](int il, int j, float4 v) { *reinterpret_cast<float4*>(dst + size_t(il) * L + j) = v; });
}

// Finest level: all selected filters and the Dirac block summed into the image.
template <typename Src>
__global__ void __launch_bounds__(kFThr, 2) k_syn_fine_final(const __grid_constant__ Src src, DbFilters<float> f) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  float* band = reinterpret_cast<float*>(sm_raw);  // two sub-band buffers
  float* U = band + 2 * kFineSynBand;
  decltype(auto) S = src.get_at(int(blockIdx.z));
  const int i0 = blockIdx.y * kFS, j0 = blockIdx.x * kFS, n = S.n;
  float acc[kFAcc];
#pragma unroll
  for (int q = 0; q < kFAcc; ++q) acc[q] = 0.f;
  pdl_wait();
  syn_fine_load(S, 0, S.fid[0] + 1, band, i0, j0);
  for (int z = 0; z < S.nf; ++z) {
    if (z + 1 < S.nf) {
      syn_fine_load(S, z + 1, S.fid[z + 1] + 1, band + ((z + 1) & 1) * kFineSynBand, i0, j0);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    syn_fine_dispatch(f, S.fid[z], band + (z & 1) * kFineSynBand, U, acc);
  }
  __syncthreads();
  const bool al = (reinterpret_cast<size_t>(S.x_out) & 15) == 0 && (reinterpret_cast<size_t>(S.c) & 15) == 0;
  syn_fine_out(band, acc, [&](int il, int j, float4 v4) {
    const size_t idx = size_t(i0 + il) * n + (j0 + j);
    float v[4] = {v4.x, v4.y, v4.z, v4.w}, d[4] = {0.f, 0.f, 0.f, 0.f}, o[4];
    if (S.slot0) {  // Dirac block
      if (al) *reinterpret_cast<float4*>(d) = *reinterpret_cast<const float4*>(S.c + idx);
      else
        for (int k = 0; k < 4; ++k) d[k] = S.c[idx + k];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = (v[k] + d[k]) * S.scale;
    if (S.pos_block) {  // (the solver's arrays are aligned)
      const float4 x4 = *reinterpret_cast<const float4*>(S.xh + idx);
      float4 z4 = *reinterpret_cast<const float4*>(S.z2 + idx);
      const float xv[4] = {x4.x, x4.y, x4.z, x4.w};
      float zv[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float v2 = xv[k] + zv[k], r2 = v2 > 0.f ? v2 : 0.f;
        zv[k] = v2 - r2;
        o[k] += 2.f * r2 - v2;
      }
      *reinterpret_cast<float4*>(S.z2 + idx) = make_float4(zv[0], zv[1], zv[2], zv[3]);
    }
    if (al) *reinterpret_cast<float4*>(S.x_out + idx) = make_float4(o[0], o[1], o[2], o[3]);
    else
      for (int k = 0; k < 4; ++k) S.x_out[idx + k] = o[k];
  });
}
constexpr size_t kFineSynSmem = (kFineSynBand + kFineSynU) * sizeof(float);
constexpr size_t kFineFinalSmem = (2 * kFineSynBand + kFineSynU) * sizeof(float);

template <typename T> size_t ana_smem(int F) {
  const int W = 2 * kTH + F - 2;
  return size_t(W * W + 2 * W * kTH) * sizeof(T);
}
template <typename T> size_t syn_smem(int F) {
  const int CT = kTO / 2 + F / 2;
  return size_t(4 * CT * CT + 2 * kTO * kUP) * sizeof(T);
}

inline int cdiv(int a, int b) { return (a + b - 1) / b; }
// Whether a level takes the large-tile kernels: FP32, whole tiles, and enough
// CTAs for two per SM (below that the small tiles' four times as many CTAs hide
// the latency better).
constexpr int kFineCtas = 2 * 152;
constexpr int kFinalFineSlots = 2;  // the final level's CTAs go through all filters: one per SM is enough
template <typename T> inline bool fine_tiles(int side, int tile, int slots) {
  return sizeof(T) == 4 && side % tile == 0 && (side / tile) * (side / tile) * slots >= kFineCtas;
}

// Launch plan of one analysis (Dirac block, then one launch per level) and
// one synthesis (coarse levels, then the fused finest level), shared by the
// single-operator path (arguments by value) and the batch (device tables).
template <typename T> struct AnaPlan {
  bool dirac;
  DiracArgs<T> d;
  int nb0;
  int levels;
  AnaArgs<T> a[16];
  dim3 grid[16];  // z = nz
  int nz[16];     // slots per instance: the filters, and the Dirac block on the first level
  bool fine[16];
  int np;         // objective partials written
};
template <typename T>
AnaPlan<T> plan_analysis(const SaraPlan<T>& P, const T* x, const CoefOut<T>& out, double* partials) {
  AnaPlan<T> pl{};
  const int n = P.n;
  const size_t N = size_t(n) * n;
  pl.dirac = P.dirac != 0 && P.nf == 0;  // with wavelets it rides along with their first level
  pl.nb0 = int((N + kThr - 1) / kThr);
  pl.d = DiracArgs<T>{x, N, P.scale, out, partials};
  int np = pl.dirac && partials ? pl.nb0 : 0;
  pl.levels = P.nf > 0 ? P.levels : 0;
  const T* in = x;
  size_t in_stride = 0;
  T* bufs[2] = {P.s0, P.s1};
  for (int lev = 1; lev <= pl.levels; ++lev) {
    const int L = n >> (lev - 1), H = L / 2;
    AnaArgs<T>& A = pl.a[lev - 1];
    A.in = in;
    A.in_stride = in_stride;
    A.L = L;
    A.n = n;
    A.s_out = bufs[lev & 1];
    A.last = lev == P.levels;
    A.slot0 = P.dirac;
    A.nf = P.nf;
    for (int z = 0; z < kMaxDb; ++z) A.fid[z] = P.fid[z];
    A.scale = P.scale;
    A.out = out;
    A.partials = partials ? partials + np : nullptr;
    pl.fine[lev - 1] = fine_tiles<T>(H, kFA, P.nf);
    const int th = pl.fine[lev - 1] ? kFA : kTH;
    pl.nz[lev - 1] = P.nf + (lev == 1 ? P.dirac : 0);
    pl.grid[lev - 1] = dim3(cdiv(H, th), cdiv(H, th), pl.nz[lev - 1]);
    if (partials) np += int(pl.grid[lev - 1].x * pl.grid[lev - 1].y * pl.grid[lev - 1].z);
    in = A.s_out;
    in_stride = size_t(H) * H;
  }
  pl.np = np;
  return pl;
}

template <typename T> struct SynPlan {
  int levels;  // coarse levels (launches before the final one)
  SynArgs<T> a[16];
  dim3 grid[16];
  bool fine[16];
  SynArgs<T> fin;
  dim3 fgrid;
  bool all;       // the eight filters: the unrolled final kernel
  bool fin_fine;
};
template <typename T>
SynPlan<T> plan_synthesis(const SaraPlan<T>& P, const T* c, T* x, int pos_block, const T* xh, T* z2) {
  SynPlan<T> pl{};
  const int n = P.n;
  T* bufs[2] = {P.s0, P.s1};
  const T* s_in = nullptr;
  auto select = [&](SynArgs<T>& S) {
    S.slot0 = P.dirac;
    S.nf = P.nf;
    for (int z = 0; z < kMaxDb; ++z) S.fid[z] = P.fid[z];
    S.scale = P.scale;
  };
  int k = 0;
  for (int lev = P.levels; lev >= 2 && P.nf > 0; --lev, ++k) {
    const int H = n >> lev, L = 2 * H;
    SynArgs<T>& S = pl.a[k];
    S = SynArgs<T>{};
    S.c = c;
    S.s_in = s_in;
    S.H = H;
    S.n = n;
    S.s_out = bufs[lev & 1];
    select(S);
    pl.fine[k] = fine_tiles<T>(L, kFS, P.nf);
    const int to = pl.fine[k] ? kFS : kTO;
    pl.grid[k] = dim3(cdiv(L, to), cdiv(L, to), P.nf);
    s_in = S.s_out;
  }
  pl.levels = k;
  SynArgs<T>& S = pl.fin;
  S = SynArgs<T>{};
  S.c = c;
  S.s_in = s_in;
  S.H = n / 2;
  S.n = n;
  select(S);
  S.pos_block = pos_block;
  S.x_out = x;
  S.xh = xh;
  S.z2 = z2;
  pl.fin_fine = P.nf > 0 && fine_tiles<T>(n, kFS, kFinalFineSlots);
  const int to = pl.fin_fine ? kFS : kTO;
  pl.fgrid = dim3(cdiv(n, to), cdiv(n, to), 1);
  pl.all = P.nf == kMaxDb;
  return pl;
}

// One analysis level, one synthesis level and the final one, by the plan's kernel.
template <typename T, typename Src>
void launch_ana(const Src& src, bool fine, dim3 grid, int nz, const DbFilters<T>& f, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    if (fine) {
      launch_pdl(k_ana_fine<Src>, grid, kThr, FineAna<16>::smem, s, src, nz, f);
      return;
    }
  }
  launch_pdl(k_ana_level<T, Src>, grid, kThr, ana_smem<T>(16), s, src, nz, f);
}
template <typename T, typename Src>
void launch_syn(const Src& src, bool fine, dim3 grid, int nf, const DbFilters<T>& f, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    if (fine) {
      launch_pdl(k_syn_fine<Src>, grid, kFThr, kFineSynSmem, s, src, nf, f);
      return;
    }
  }
  launch_pdl(k_syn_level<T, Src>, grid, kThr, syn_smem<T>(16), s, src, nf, f);
}
template <typename T, typename Src>
void launch_syn_final(const Src& src, bool fine, bool all, dim3 grid, const DbFilters<T>& f, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    if (fine) {
      launch_pdl(k_syn_fine_final<Src>, grid, kFThr, kFineFinalSmem, s, src, f);
      return;
    }
  }
  if (all) launch_pdl(k_syn_final<T, true, Src>, grid, kThr, syn_smem<T>(16), s, src, f);
  else launch_pdl(k_syn_final<T, false, Src>, grid, kThr, syn_smem<T>(16), s, src, f);
}

// Runs the analysis levels; returns partial sums written (prox mode).
template <typename T>
int run_analysis(const SaraPlan<T>& P, const T* x, const CoefOut<T>& out, double* partials, cudaStream_t s) {
  const AnaPlan<T> pl = plan_analysis(P, x, out, partials);
  if (pl.dirac) k_dirac<T><<<pl.nb0, kThr, 0, s>>>(ArgVal<DiracArgs<T>>{pl.d});
  for (int l = 0; l < pl.levels; ++l) launch_ana<T>(ArgVal<AnaArgs<T>>{pl.a[l]}, pl.fine[l], pl.grid[l], pl.nz[l], P.f, s);
  return pl.np;
}

template <typename T>
void run_synthesis(const SaraPlan<T>& P, const T* c, T* x, int pos_block, const T* xh, T* z2, cudaStream_t s) {
  const SynPlan<T> pl = plan_synthesis(P, c, x, pos_block, xh, z2);
  for (int l = 0; l < pl.levels; ++l) launch_syn<T>(ArgVal<SynArgs<T>>{pl.a[l]}, pl.fine[l], pl.grid[l], P.nf, P.f, s);
  launch_syn_final<T>(ArgVal<SynArgs<T>>{pl.fin}, pl.fin_fine, pl.all, pl.fgrid, P.f, s);
}

}  // namespace

template <typename T> cudaError_t configure_sara() {
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = raise_smem_limit(k_ana_level<T, ArgVal<AnaArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_syn_level<T, ArgVal<SynArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_syn_final<T, true, ArgVal<SynArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_syn_final<T, false, ArgVal<SynArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_ana_level<T, ArgTab<AnaArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_syn_level<T, ArgTab<SynArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_syn_final<T, true, ArgTab<SynArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_syn_final<T, false, ArgTab<SynArgs<T>>>);
  if constexpr (sizeof(T) == 4) {
    if (e == cudaSuccess) e = raise_smem_limit(k_ana_fine<ArgVal<AnaArgs<T>>>);
    if (e == cudaSuccess) e = raise_smem_limit(k_ana_fine<ArgTab<AnaArgs<T>>>);
    if (e == cudaSuccess) e = raise_smem_limit(k_syn_fine<ArgVal<SynArgs<T>>>);
    if (e == cudaSuccess) e = raise_smem_limit(k_syn_fine<ArgTab<SynArgs<T>>>);
    if (e == cudaSuccess) e = raise_smem_limit(k_syn_fine_final<ArgVal<SynArgs<T>>>);
    if (e == cudaSuccess) e = raise_smem_limit(k_syn_fine_final<ArgTab<SynArgs<T>>>);
  }
  return e;
}
template cudaError_t configure_sara<float>();
template cudaError_t configure_sara<double>();

template <typename T> int sara_select(SaraPlan<T>& P, unsigned mask) {
  if (mask == 0 || (mask & ~kSaraAll)) return -1;
  P.dirac = int(mask & 1u);
  P.nf = 0;
  for (int k = 0; k < kMaxDb; ++k) {
    P.fid[k] = 0;
    if (mask & (2u << k)) P.fid[P.nf++] = k;
  }
  P.nbases = P.dirac + P.nf;
  P.scale = T(1.0 / std::sqrt(double(P.nbases)));
  return P.nbases;
}
template int sara_select<float>(SaraPlan<float>&, unsigned);
template int sara_select<double>(SaraPlan<double>&, unsigned);

int sara_partials_capacity(int n, int levels) {
  int np = (n * n + kThr - 1) / kThr;
  for (int lev = 1; lev <= levels; ++lev) {
    const int H = n >> lev;
    np += cdiv(H, kTH) * cdiv(H, kTH) * kMaxDb;
  }
  return np;
}

template <typename T> void sara_analysis(const SaraPlan<T>& P, const T* x, T* c, cudaStream_t s) {
  CoefOut<T> out{};
  out.c = c;
  out.prox = 0;
  run_analysis<T>(P, x, out, nullptr, s);
}

template <typename T> void sara_synthesis(const SaraPlan<T>& P, const T* c, T* x, cudaStream_t s) {
  run_synthesis<T>(P, c, x, 0, nullptr, nullptr, s);
}

template <typename T>
int sara_analysis_prox(const SaraPlan<T>& P, const T* xh, const L1Block<T>& b, cudaStream_t s) {
  CoefOut<T> out{};
  out.prox = 1;
  out.z1 = b.z1;
  out.w = b.w;
  out.cs = P.cs;
  out.gamma = T(b.gamma);
  return run_analysis(P, xh, out, b.partials, s);
}

template <typename T>
void sara_synthesis_pos(const SaraPlan<T>& P, const T* xh, T* z2, T* xs, cudaStream_t s) {
  run_synthesis<T>(P, P.cs, xs, 1, xh, z2, s);
}

// ---- batched SDMM blocks 1 and 2 (l1 prox on the analysis, positivity on
// the synthesis) for instances of one image side, levels and dictionary:
// every launch of the sequence covers all instances (device argument
// tables, instance in blockIdx.y / blockIdx.z).
template <typename T> struct SaraBatch {
  void* dev = nullptr;
  cudaMemPool_t pool = nullptr;  // dev from this pool (freed in stream order) when set
  cudaStream_t pool_stream = nullptr;
  int count = 0, nf = 0, levels_a = 0, levels_s = 0, nb0 = 0;
  bool dirac = false, all = false, afine[16] = {}, sfine[16] = {}, fin_fine = false;
  int anz[16] = {};
  dim3 agrid[16], sgrid[16], fgrid;
  const DiracArgs<T>* dtab = nullptr;
  const AnaArgs<T>* atab[16] = {};
  const SynArgs<T>* stab[16] = {};
  const SynArgs<T>* ftab = nullptr;
  DbFilters<T> f;
};

template <typename T>
int sara_batch_create(const std::vector<SaraBatchInst<T>>& in, SaraBatch<T>** out, int* np, cudaMemPool_t pool,
                      cudaStream_t s) {
  if (in.empty()) return PURIFY_ERR_INVALID;
  SaraBatch<T>* b = new (std::nothrow) SaraBatch<T>();
  if (!b) return PURIFY_ERR_NOMEM;
  const int count = int(in.size());
  std::vector<AnaPlan<T>> ap(count);
  std::vector<SynPlan<T>> sp(count);
  for (int i = 0; i < count; ++i) {
    const SaraBatchInst<T>& u = in[i];
    CoefOut<T> co{};
    co.prox = 1;
    co.z1 = u.z1;
    co.w = u.w;
    co.cs = u.P->cs;
    co.gamma = T(u.gamma);
    ap[i] = plan_analysis(*u.P, u.xh, co, u.partials);
    sp[i] = plan_synthesis(*u.P, u.P->cs, u.xs, 1, u.xh, u.z2);
  }
  const SaraPlan<T>& P0 = *in[0].P;
  b->count = count;
  b->nf = P0.nf;
  b->dirac = ap[0].dirac;
  b->nb0 = ap[0].nb0;
  b->levels_a = ap[0].levels;
  b->levels_s = sp[0].levels;
  b->all = sp[0].all;
  b->fin_fine = sp[0].fin_fine;
  b->f = P0.f;
  // one device buffer: Dirac table, analysis tables per level, synthesis tables per level, final table
  const size_t nd = sizeof(DiracArgs<T>) * count, na = sizeof(AnaArgs<T>) * count, ns = sizeof(SynArgs<T>) * count;
  const size_t total = nd + na * b->levels_a + ns * (b->levels_s + 1);
  std::vector<unsigned char> host(total);
  size_t off = 0;
  for (int i = 0; i < count; ++i) std::memcpy(&host[off + i * sizeof(DiracArgs<T>)], &ap[i].d, sizeof(DiracArgs<T>));
  const size_t doff = off;
  off += nd;
  size_t aoff[16], soff[16];
  for (int l = 0; l < b->levels_a; ++l, off += na) {
    aoff[l] = off;
    b->afine[l] = ap[0].fine[l];
    b->anz[l] = ap[0].nz[l];
    b->agrid[l] = dim3(ap[0].grid[l].x, ap[0].grid[l].y, ap[0].grid[l].z * count);
    for (int i = 0; i < count; ++i) std::memcpy(&host[off + i * sizeof(AnaArgs<T>)], &ap[i].a[l], sizeof(AnaArgs<T>));
  }
  for (int l = 0; l < b->levels_s; ++l, off += ns) {
    soff[l] = off;
    b->sfine[l] = sp[0].fine[l];
    b->sgrid[l] = dim3(sp[0].grid[l].x, sp[0].grid[l].y, sp[0].grid[l].z * count);
    for (int i = 0; i < count; ++i) std::memcpy(&host[off + i * sizeof(SynArgs<T>)], &sp[i].a[l], sizeof(SynArgs<T>));
  }
  const size_t foff = off;
  b->fgrid = dim3(sp[0].fgrid.x, sp[0].fgrid.y, count);
  for (int i = 0; i < count; ++i) std::memcpy(&host[off + i * sizeof(SynArgs<T>)], &sp[i].fin, sizeof(SynArgs<T>));
  b->pool = pool;
  b->pool_stream = s;
  if ((pool ? cudaMallocFromPoolAsync(&b->dev, total, pool, s) : cudaMalloc(&b->dev, total)) != cudaSuccess) {
    delete b;
    return PURIFY_ERR_NOMEM;
  }
  const cudaError_t ce = pool ? cudaMemcpyAsync(b->dev, host.data(), total, cudaMemcpyHostToDevice, s)
                              : cudaMemcpy(b->dev, host.data(), total, cudaMemcpyHostToDevice);
  if (ce != cudaSuccess || (pool && cudaStreamSynchronize(s) != cudaSuccess)) {
    sara_batch_destroy(b);
    return PURIFY_ERR_CUDA;
  }
  unsigned char* d = static_cast<unsigned char*>(b->dev);
  b->dtab = reinterpret_cast<const DiracArgs<T>*>(d + doff);
  for (int l = 0; l < b->levels_a; ++l) b->atab[l] = reinterpret_cast<const AnaArgs<T>*>(d + aoff[l]);
  for (int l = 0; l < b->levels_s; ++l) b->stab[l] = reinterpret_cast<const SynArgs<T>*>(d + soff[l]);
  b->ftab = reinterpret_cast<const SynArgs<T>*>(d + foff);
  *np = ap[0].np;
  *out = b;
  return PURIFY_OK;
}

template <typename T> void sara_batch_launch(const SaraBatch<T>* b, cudaStream_t s) {
  if (b->dirac) k_dirac<T><<<dim3(b->nb0, b->count), kThr, 0, s>>>(ArgTab<DiracArgs<T>>{b->dtab});
  for (int l = 0; l < b->levels_a; ++l)
    launch_ana<T>(ArgTab<AnaArgs<T>>{b->atab[l]}, b->afine[l], b->agrid[l], b->anz[l], b->f, s);
  for (int l = 0; l < b->levels_s; ++l)
    launch_syn<T>(ArgTab<SynArgs<T>>{b->stab[l]}, b->sfine[l], b->sgrid[l], b->nf, b->f, s);
  launch_syn_final<T>(ArgTab<SynArgs<T>>{b->ftab}, b->fin_fine, b->all, b->fgrid, b->f, s);
}

template <typename T> int sara_prox_partials(const SaraPlan<T>& P) {
  CoefOut<T> co{};
  co.prox = 1;
  double dummy = 0;
  return plan_analysis(P, static_cast<const T*>(nullptr), co, &dummy).np;
}

template <typename T> void sara_batch_destroy(SaraBatch<T>* b) {
  if (!b) return;
  if (b->dev) {
    if (b->pool) cudaFreeAsync(b->dev, b->pool_stream);
    else cudaFree(b->dev);
  }
  delete b;
}

#define INST(T)                                                                                 \
  template int sara_batch_create<T>(const std::vector<SaraBatchInst<T>>&, SaraBatch<T>**, int*,   \
                                    cudaMemPool_t, cudaStream_t);                                 \
  template void sara_batch_launch<T>(const SaraBatch<T>*, cudaStream_t);                          \
  template void sara_batch_destroy<T>(SaraBatch<T>*);                                             \
  template int sara_prox_partials<T>(const SaraPlan<T>&);                                         \
  template void sara_analysis<T>(const SaraPlan<T>&, const T*, T*, cudaStream_t);                 \
  template void sara_synthesis<T>(const SaraPlan<T>&, const T*, T*, cudaStream_t);                \
  template int sara_analysis_prox<T>(const SaraPlan<T>&, const T*, const L1Block<T>&, cudaStream_t); \
  template void sara_synthesis_pos<T>(const SaraPlan<T>&, const T*, T*, T*, cudaStream_t);
INST(float)
INST(double)
#undef INST


// ---------------------------------------------------------------------------
// Allocation-free SARA analysis.
//
// Some callers cannot call cudaMalloc once they are running: pipelines that
// reserve all device memory at start-up and must not allocate while they
// stream (an allocation can stall or fail when memory is fragmented or held
// by another framework's caching allocator), and hosts that hand this library
// only pre-sized buffers.  For them the scratch bands of the multi-level
// analysis live in one fixed file-scope device array instead of operator
// memory.  The array exists once per device that loads the library and
// stays allocated until the process exits.
constexpr int kStaticMaxN = 512;  // largest image side served from the fixed scratch
constexpr size_t kStaticBand = size_t(kMaxDb) * (kStaticMaxN / 2) * (kStaticMaxN / 2);
static __device__ __align__(256) float g_static_scratch[2 * kStaticBand];  // 4 MiB

namespace {
std::mutex g_static_mu;
float* g_static_ptr[128] = {nullptr};
DbFilters<float> g_static_filters;
bool g_static_filters_ready = false;

// Device address of the fixed scratch for the current device (host code may
// not use the symbol itself as a device address).
int static_scratch(float** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 128) {
    set_last_error("purify_sara_fwd_static: cannot query the current device");
    return PURIFY_ERR_CUDA;
  }
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!g_static_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess || !p) {
      char buf[160];
      std::snprintf(buf, sizeof(buf), "purify_sara_fwd_static: cudaGetSymbolAddress failed: %s",
                    cudaGetErrorName(e));
      set_last_error(buf);
      return PURIFY_ERR_CUDA;
    }
    g_static_ptr[dev] = static_cast<float*>(p);
  }
  if (!g_static_filters_ready) {
    for (int k = 1; k <= kMaxDb; ++k) {
      const std::vector<double>& h = daubechies_lowpass_cached(k);
      const int F = 2 * k;
      for (int m = 0; m < kMaxTaps; ++m) {
        g_static_filters.h[k - 1][m] = m < F ? float(h[m]) : 0.0f;
        g_static_filters.g[k - 1][m] = m < F ? float(((m & 1) ? -1.0 : 1.0) * h[F - 1 - m]) : 0.0f;
      }
    }
    g_static_filters_ready = true;
  }
  *out = g_static_ptr[dev];
  return PURIFY_OK;
}
}  // namespace

}  // namespace purify

extern "C" int purify_sara_fwd_static(const float* x, float* c, int n, int levels, void* stream) {
  using namespace purify;
  if (!x || !c || n < 16 || (n & (n - 1)) || levels < 1 || (n >> levels) < 2) {
    set_last_error("purify_sara_fwd_static: need non-null x and c, n a power of two >= 16, n / 2^levels >= 2");
    return PURIFY_ERR_INVALID;
  }
  if (n > kStaticMaxN) {
    char buf[160];
    std::snprintf(buf, sizeof(buf), "purify_sara_fwd_static: n = %d exceeds the fixed-scratch limit n <= %d", n,
                  kStaticMaxN);
    set_last_error(buf);
    return PURIFY_ERR_INVALID;
  }
  float* scratch = nullptr;
  const int rc = static_scratch(&scratch);
  if (rc) return rc;
  SaraPlan<float> P{};
  P.n = n;
  P.levels = levels;
  P.s0 = scratch;
  P.s1 = scratch + kStaticBand;
  P.cs = nullptr;
  P.f = g_static_filters;
  sara_select(P, kSaraAll);
  sara_analysis<float>(P, x, c, static_cast<cudaStream_t>(stream));
  const cudaError_t e = cudaPeekAtLastError();
  if (e != cudaSuccess) {
    char buf[160];
    std::snprintf(buf, sizeof(buf), "purify_sara_fwd_static: launch failed: %s", cudaGetErrorName(e));
    set_last_error(buf);
    return PURIFY_ERR_CUDA;
  }
  return PURIFY_OK;
}
