// Total-variation prior (Section 4's TV and RWTV) inside SDMM (Algorithm 1).
//
// The l1 block f_1 = gamma ||W Psi^H .||_1 is replaced by f_1 = gamma TV_w
// with L_1 = I, so the composite operator stays nu^2 Phi^H Phi + 2I.  TV_w is
// the weighted isotropic total variation with forward differences and a zero
// difference past the last row / column:
//     (grad x)_1[i, j] = x[i+1, j] - x[i, j] (0 on the last row),
//     (grad x)_2[i, j] = x[i, j+1] - x[i, j] (0 on the last column),
//     TV_w(x) = sum_ij w_ij |(grad x)[i, j]|,
// and div = -grad^T.  Its proximity operator (Eq. 7) is taken through the
// dual: prox(v) = v + div q with q minimising |v + div q|^2 / 2 over
// |q_ij| <= gamma w_ij, by projected-gradient steps
//     q <- P(q + tau grad(v + div q)),  tau = 1/8,
// a fixed number per SDMM iteration, warm-started from the previous
// iteration's q (zero at the start of each round).  A step needs its
// neighbours' previous q: large FP32 images take kTvSteps of them a launch on
// tiles with a halo as wide, in shared memory; other images one a launch
// (tv_fused).  Both ping-pong between two dual buffers from launch to launch
// and leave the dual in the first; the epilogue forms r_1 = v + div q, updates
// z_1, applies the positivity block (f_2, L_2 = I) and writes x_1 + x_2, with the
// objective's partial sums TV_w(x_hat).
#include "internal.h"
#include "solver_kernels.h"

namespace purify {

namespace {

constexpr int kTvT = 256;
constexpr int kTvSteps = 5;                    // dual steps per launch, at most
constexpr int kTvTile = 32;                    // output pixels per tile side
constexpr int kTvHalo = kTvSteps + 1;          // each step needs one more ring; the epilogue another
constexpr int kTvR = kTvTile + 2 * kTvHalo;    // tile side with its halo
constexpr int kTvPix = (kTvR * kTvR + kTvT - 1) / kTvT;  // pixels per thread

// `steps` projected-gradient steps of the dual, q <- P(q + tau grad(v + div q)),
// P the pixelwise projection onto |q_ij| <= gamma w_ij, from qi to qo (q1 plane
// first, then q2; n x n each).  first: v = x_hat + z_1 (kept in v for the
// later launches).  last: r_1 = v + div q, z_1 = v - r_1, x_1 = 2 r_1 - v; positivity
// block v_2 = x_hat + z_2, r_2 = max(v_2, 0), z_2 = v_2 - r_2; xs = x_1 + 2 r_2 - v_2;
// per-CTA partials of TV_w(x_hat).
template <typename T> struct TvArgs {
  int n, steps, first, last;
  T gamma;
  const T* xh;
  const T* w;  // may be null (w = 1)
  const T* qi;
  T* qo;
  T* v;
  T* z1;
  T* z2;
  T* xs;
  double* partials;
};
// The halo makes a tile 1.9 times its pixels' work, but a step costs two barriers
// in place of a launch and a pass over memory (the TV solve at 512^2, 20 steps an
// iteration, 5.41 -> 5.30 ms, where the ball block beside it is the longer branch).
template <typename T> __global__ void __launch_bounds__(kTvT) k_tv_steps(TvArgs<T> a) {
  __shared__ T q1[kTvR * kTvR], q2[kTvR * kTvR], ds[kTvR * kTvR];
  __shared__ double red[32];
  const int n = a.n;
  const size_t N = size_t(n) * n;
  const int i0 = int(blockIdx.y) * kTvTile - kTvHalo, j0 = int(blockIdx.x) * kTvTile - kTvHalo;
  T v[kTvPix], bound[kTvPix];
  pdl_wait();
  auto pixel = [&](int k, int& e, int& r, int& c, int& i, int& j) {  // in the image?
    e = int(threadIdx.x) + k * kTvT;
    r = e / kTvR;
    c = e - r * kTvR;
    i = i0 + r;
    j = j0 + c;
    return r < kTvR && i >= 0 && i < n && j >= 0 && j < n;
  };
  auto inner = [](int r, int c) {  // one of the tile's own pixels
    return r >= kTvHalo && r < kTvHalo + kTvTile && c >= kTvHalo && c < kTvHalo + kTvTile;
  };
  // d = v + div q at a pixel whose upper and left neighbours are in the region
  auto dval = [&](T d, int e, int i, int j) {
    if (i < n - 1) d += q1[e];
    if (i > 0) d -= q1[e - kTvR];
    if (j < n - 1) d += q2[e];
    if (j > 0) d -= q2[e - 1];
    return d;
  };
#pragma unroll
  for (int k = 0; k < kTvPix; ++k) {
    int e, r, c, i, j;
    v[k] = bound[k] = T(0);
    if (!pixel(k, e, r, c, i, j)) continue;
    const size_t at = size_t(i) * n + j;
    q1[e] = a.qi[at];
    q2[e] = a.qi[N + at];
    bound[k] = a.gamma * (a.w ? a.w[at] : T(1));
    v[k] = a.first ? a.xh[at] + a.z1[at] : a.v[at];
    if (a.first && inner(r, c)) a.v[at] = v[k];
  }
  __syncthreads();
  const T tau = T(0.125);
  for (int s = 0; s < a.steps; ++s) {
#pragma unroll
    for (int k = 0; k < kTvPix; ++k) {
      int e, r, c, i, j;
      if (pixel(k, e, r, c, i, j) && r > 0 && c > 0) ds[e] = dval(v[k], e, i, j);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kTvPix; ++k) {
      int e, r, c, i, j;
      if (!pixel(k, e, r, c, i, j) || r >= kTvR - 1 || c >= kTvR - 1) continue;
      const T d = ds[e];
      const T g1 = i < n - 1 ? ds[e + kTvR] - d : T(0);
      const T g2 = j < n - 1 ? ds[e + 1] - d : T(0);
      T x = fma(tau, g1, q1[e]), y = fma(tau, g2, q2[e]);
      const T m = sqrt(x * x + y * y);
      if (m > bound[k]) {
        const T sc = bound[k] / m;
        x *= sc;
        y *= sc;
      }
      q1[e] = x;
      q2[e] = y;
    }
    __syncthreads();
  }
  pdl_trigger();
  Acc<T> part;
#pragma unroll
  for (int k = 0; k < kTvPix; ++k) {
    int e, r, c, i, j;
    if (!pixel(k, e, r, c, i, j) || !inner(r, c)) continue;
    const size_t at = size_t(i) * n + j;
    a.qo[at] = q1[e];
    a.qo[N + at] = q2[e];
    if (!a.last) continue;
    const T r1 = dval(v[k], e, i, j);
    a.z1[at] = v[k] - r1;
    const T x0 = a.xh[at], v2 = x0 + a.z2[at];
    const T r2 = v2 > T(0) ? v2 : T(0);
    a.z2[at] = v2 - r2;
    a.xs[at] = (T(2) * r1 - v[k]) + (T(2) * r2 - v2);
    const T g1 = i < n - 1 ? a.xh[at + n] - x0 : T(0);
    const T g2 = j < n - 1 ? a.xh[at + 1] - x0 : T(0);
    part.add(sqrt(g1 * g1 + g2 * g2) * (a.w ? a.w[at] : T(1)));
  }
  if (a.last && a.partials) {
    const Acc<T> t = block_merge<kTvT>(part, red);
    if (threadIdx.x == 0) reinterpret_cast<Acc<T>*>(a.partials)[blockIdx.y * gridDim.x + blockIdx.x] = t;
  }
}

// ---- one launch per step and pixel, where that is the faster form (tv_fused)
// d = v + div q at (i, j) (q1 plane first, then q2; n x n each).
template <typename T> PD T dval(const T* __restrict__ v, const T* __restrict__ q, int n, int i, int j) {
  const size_t N = size_t(n) * n, k = size_t(i) * n + j;
  const T* q1 = q;
  const T* q2 = q + N;
  T d = v[k];
  if (i < n - 1) d += q1[k];
  if (i > 0) d -= q1[k - n];
  if (j < n - 1) d += q2[k];
  if (j > 0) d -= q2[k - 1];
  return d;
}

// One projected-gradient step of the dual per launch: qo = P(qi + tau grad(v + div qi)),
// P the pixelwise projection onto |q_ij| <= gamma w_ij.
template <typename T>
__global__ void __launch_bounds__(kTvT) k_tv_dual_step(const T* __restrict__ v, const T* __restrict__ w, T gamma,
                                                       const T* __restrict__ qi, T* __restrict__ qo, int n) {
  const size_t N = size_t(n) * n;
  const size_t k = size_t(blockIdx.x) * kTvT + threadIdx.x;
  if (k >= N) return;
  const int i = int(k / n), j = int(k - size_t(i) * n);
  const T d = dval(v, qi, n, i, j);
  const T g1 = i < n - 1 ? dval(v, qi, n, i + 1, j) - d : T(0);
  const T g2 = j < n - 1 ? dval(v, qi, n, i, j + 1) - d : T(0);
  const T tau = T(0.125);
  T a = fma(tau, g1, qi[k]), b = fma(tau, g2, qi[k + N]);
  const T bound = gamma * (w ? w[k] : T(1));
  const T m = sqrt(a * a + b * b);
  if (m > bound) {
    const T s = bound / m;
    a *= s;
    b *= s;
  }
  qo[k] = a;
  qo[k + N] = b;
}

// v_1 = x_hat + z_1 (the TV block's input).
template <typename T>
__global__ void __launch_bounds__(kTvT) k_tv_input(const T* __restrict__ xh, const T* __restrict__ z1,
                                                   T* __restrict__ v, size_t N) {
  const size_t k = size_t(blockIdx.x) * kTvT + threadIdx.x;
  if (k < N) v[k] = xh[k] + z1[k];
}

// Epilogue: r_1 = v + div q, z_1 = v - r_1, x_1 = 2 r_1 - v; positivity block
// v_2 = x_hat + z_2, r_2 = max(v_2, 0), z_2 = v_2 - r_2; xs = x_1 + 2 r_2 - v_2;
// per-CTA partials of TV_w(x_hat).  With qcopy set the final dual is also
// written back to the buffer the next iteration starts from.
template <typename T>
__global__ void __launch_bounds__(kTvT) k_tv_epilogue(const T* __restrict__ v, const T* __restrict__ q,
                                                      T* __restrict__ qcopy, const T* __restrict__ xh,
                                                      const T* __restrict__ w, T* __restrict__ z1,
                                                      T* __restrict__ z2, T* __restrict__ xs, double* partials,
                                                      int n) {
  __shared__ double red[32];
  const size_t N = size_t(n) * n;
  const size_t k = size_t(blockIdx.x) * kTvT + threadIdx.x;
  Acc<T> part;
  if (k < N) {
    const int i = int(k / n), j = int(k - size_t(i) * n);
    const T vk = v[k];
    const T r1 = dval(v, q, n, i, j);
    z1[k] = vk - r1;
    const T v2 = xh[k] + z2[k];
    const T r2 = v2 > T(0) ? v2 : T(0);
    z2[k] = v2 - r2;
    xs[k] = (T(2) * r1 - vk) + (T(2) * r2 - v2);
    if (qcopy) {
      qcopy[k] = q[k];
      qcopy[k + N] = q[k + N];
    }
    const T x0 = xh[k];
    const T g1 = i < n - 1 ? xh[k + n] - x0 : T(0);
    const T g2 = j < n - 1 ? xh[k + 1] - x0 : T(0);
    part.add(sqrt(g1 * g1 + g2 * g2) * (w ? w[k] : T(1)));
  }
  if (partials) {
    const Acc<T> t = block_merge<kTvT>(part, red);
    if (threadIdx.x == 0) reinterpret_cast<Acc<T>*>(partials)[blockIdx.x] = t;
  }
}

// |grad x| per pixel (RWTV weights and their delta).
template <typename T>
__global__ void __launch_bounds__(kTvT) k_tv_magnitude(const T* __restrict__ x, T* __restrict__ out, int n) {
  const size_t N = size_t(n) * n;
  const size_t k = size_t(blockIdx.x) * kTvT + threadIdx.x;
  if (k >= N) return;
  const int i = int(k / n), j = int(k - size_t(i) * n);
  const T x0 = x[k];
  const T g1 = i < n - 1 ? x[k + n] - x0 : T(0);
  const T g2 = j < n - 1 ? x[k + 1] - x0 : T(0);
  out[k] = sqrt(g1 * g1 + g2 * g2);
}

inline int tv_blocks(int n) { return int((size_t(n) * n + kTvT - 1) / kTvT); }
inline int tv_tiles(int n) { return (n + kTvTile - 1) / kTvTile; }
// Whether the steps go kTvSteps a launch.  The halo makes 1.9 times the work
// on tiles that are few on small images, and a launch per step costs only 1.9 us
// inside a graph; FP64 is bound by its units whatever the size.  An SDMM
// iteration with 100 dual steps, one a launch against five: FP32 64^2 293 / 376
// us, 256^2 318 / 404, 512^2 479 / 482 (20 steps 239 / 232), 1024^2 1171 / 1072,
// 2048^2 7742 / 6828; FP64 64^2 848 / 1899, 512^2 4002 / 5746.
template <typename T> constexpr bool tv_fused(int n) { return sizeof(T) == 4 && n >= 512; }

}  // namespace

int tv_partials(int n) { return tv_blocks(n) > tv_tiles(n) * tv_tiles(n) ? tv_blocks(n) : tv_tiles(n) * tv_tiles(n); }

// One launch per step: an odd number of them leaves the dual in qb, from where
// the epilogue copies it back to qa.
template <typename T> static int tv_single_steps(const TvBlock<T>& b, cudaStream_t s) {
  const int n = b.n, nb = tv_blocks(n);
  k_tv_input<T><<<nb, kTvT, 0, s>>>(b.xh, b.z1, b.v, size_t(n) * n);
  const T* qi = b.qa;
  T* qo = b.qb;
  for (int it = 0; it < b.iters; ++it) {
    k_tv_dual_step<T><<<nb, kTvT, 0, s>>>(b.v, b.w, T(b.gamma), qi, qo, n);
    const T* t = qo;
    qo = const_cast<T*>(qi);
    qi = t;
  }
  k_tv_epilogue<T><<<nb, kTvT, 0, s>>>(b.v, qi, (b.iters & 1) ? b.qa : nullptr, b.xh, b.w, b.z1, b.z2, b.xs,
                                       b.partials, n);
  return nb;
}

template <typename T> static int tv_fused_steps(const TvBlock<T>& b, cudaStream_t s) {
  const int nt = tv_tiles(b.n);
  // an even number of launches, so that the dual leaves in the buffer it came in
  const int launches = 2 * ((b.iters + 2 * kTvSteps - 1) / (2 * kTvSteps));
  TvArgs<T> a{b.n, 0, 1, 0, T(b.gamma), b.xh, b.w, b.qa, b.qb, b.v, b.z1, b.z2, b.xs, b.partials};
  for (int l = 0, done = 0; l < launches; ++l) {
    a.steps = (b.iters - done + launches - l - 1) / (launches - l);
    done += a.steps;
    a.first = l == 0;
    a.last = l == launches - 1;
    launch_pdl(k_tv_steps<T>, dim3(nt, nt), kTvT, 0, s, a);
    const T* t = a.qo;
    a.qo = const_cast<T*>(a.qi);
    a.qi = t;
  }
  return nt * nt;
}

template <typename T> int tv_block(const TvBlock<T>& b, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    if (tv_fused<T>(b.n)) return tv_fused_steps(b, s);
  }
  return tv_single_steps(b, s);
}

template <typename T> void tv_magnitude(const T* x, T* out, int n, cudaStream_t s) {
  k_tv_magnitude<T><<<tv_blocks(n), kTvT, 0, s>>>(x, out, n);
}

template int tv_block<float>(const TvBlock<float>&, cudaStream_t);
template int tv_block<double>(const TvBlock<double>&, cudaStream_t);
template void tv_magnitude<float>(const float*, float*, int, cudaStream_t);
template void tv_magnitude<double>(const double*, double*, int, cudaStream_t);

}  // namespace purify
