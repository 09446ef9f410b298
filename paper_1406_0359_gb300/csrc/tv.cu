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
// neighbours' previous q, so a launch takes kTvSteps of them on tiles with a
// halo as wide, in shared memory, ping-ponging between two dual buffers from
// launch to launch; the last launch's epilogue forms r_1 = v + div q, updates
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
// The halo makes a tile 1.9 times its pixels' work, but a step in shared memory
// costs two barriers where a launch per step cost 4.1 us (22 launches at 20 steps,
// now 4; the TV solve at 512^2 5.41 -> 5.30 ms, where the ball block beside it is
// the longer branch).
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

}  // namespace

int tv_partials(int n) { return tv_tiles(n) * tv_tiles(n); }

template <typename T>
int tv_block(const TvBlock<T>& b, cudaStream_t s) {
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

template <typename T> void tv_magnitude(const T* x, T* out, int n, cudaStream_t s) {
  k_tv_magnitude<T><<<tv_blocks(n), kTvT, 0, s>>>(x, out, n);
}

template int tv_block<float>(const TvBlock<float>&, cudaStream_t);
template int tv_block<double>(const TvBlock<double>&, cudaStream_t);
template void tv_magnitude<float>(const float*, float*, int, cudaStream_t);
template void tv_magnitude<double>(const double*, double*, int, cudaStream_t);

}  // namespace purify
