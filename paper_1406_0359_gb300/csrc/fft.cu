// Oversampled 2D FFT passes of the NUFFT (operator F of Phi = G F Z S, Section 4).
//
// All passes transform by halves (even and odd frequencies apart, see
// "half-length transforms" below); only the set-up of the PSF spectrum runs
// plain length-K transforms (K = 2n, a power of two).
//
// The image is real, so every pass works in real form: two image rows a, b
// travel as one complex row x_a + i x_b, and only the half spectra (columns
// 0..K/2 of the row transforms) are kept, n x K/2 complex values, transposed.
// Forward (Phi):   row pass over the n non-zero image rows (pairs), fused with
//                  the deapodisation S and zero-padding Z; column pass over
//                  the half-spectrum columns into the padded half grid
//                  (columns 0..n; periodic and mirrored J-wide halo) that
//                  degridding stages by TMA.
// Adjoint (Phi^H): column pass reading the padded gridding accumulator (half
//                  grid), folding its halo and taking the Hermitian part
//                  (Re of the image is all Phi^H keeps), writing only the n
//                  rows the crop Z^T keeps; row pass fused with the crop, the
//                  deapodisation and the solver epilogues.
#include <cmath>
#include <vector>

#include "internal.h"
#include "solver_kernels.h"

namespace purify {

namespace {

// Let the next pass's CTAs start.  Not in FP64 from image side 512 on (the grid's
// column passes: 256): those passes are bound by the FP64 units, and CTAs that
// start early pile up on the SMs that finish first, which then take twice as
// long while others idle (one to three CTAs an SM).  With the trigger, without,
// by plain launches: Phi^H Phi at n = 512 207, 124, 131 us, at 256 43.3, 43.9, 52;
// Phi at 512 / 131072 points 226, 194, 198, at 256 / 65536 112, 94, -.  Without it
// the next launch waits for the last CTA's end, its set-up already done; smaller
// images lose that wait (an SDMM iteration at 128^2 629 -> 638 us).
template <typename T, int LOGN, int LARGEST = 8> PD void pass_trigger() {
  if constexpr (sizeof(T) == 4 || LOGN <= LARGEST) pdl_trigger();
}

template <typename C> PD C cneg(C a) { a.x = -a.x; a.y = -a.y; return a; }

template <typename C> PD void dft2(C& a, C& b) {
  const C t = a;
  a = cadd(t, b);
  b = csub(t, b);
}

// X_k = sum_r a_r exp(dir 2 pi i r k / 4), dir = -1 forward, +1 inverse
template <typename C> PD void dft4(C& a0, C& a1, C& a2, C& a3, int dir) {
  const C s02 = cadd(a0, a2), d02 = csub(a0, a2);
  const C s13 = cadd(a1, a3), d13 = csub(a1, a3);
  C j13 = cmul_i(d13);
  if (dir < 0) j13 = cneg(j13);
  a0 = cadd(s02, s13);
  a2 = csub(s02, s13);
  a1 = cadd(d02, j13);
  a3 = csub(d02, j13);
}

// exp(dir 2 pi i m / 16) for the fixed m used by the radix-16/8 butterflies
template <typename C> PD C w16(int m, int dir) {
  typedef decltype(C().x) T;
  const T c1 = T(0.92387953251128675613), s1 = T(0.38268343236508977173);
  const T h = T(0.70710678118654752440);
  T re = 1, im = 0;
  switch (m) {
    case 1: re = c1; im = s1; break;
    case 2: re = h; im = h; break;
    case 3: re = s1; im = c1; break;
    case 4: re = 0; im = 1; break;
    case 6: re = -h; im = h; break;
    case 9: re = -c1; im = -s1; break;
    default: break;
  }
  return cmk<C>(re, dir < 0 ? -im : im);
}

// In-register DFT of a[o], a[o+st], ..., R points (Cooley-Tukey, natural order out).
template <int R, typename C> struct Dft;
template <typename C> struct Dft<2, C> {
  static PD void run(C* a, int o, int st, int) { dft2(a[o], a[o + st]); }
};
template <typename C> struct Dft<4, C> {
  static PD void run(C* a, int o, int st, int dir) { dft4(a[o], a[o + st], a[o + 2 * st], a[o + 3 * st], dir); }
};
template <typename C> struct Dft<8, C> {
  // 8 = 2 x 4: 2-point DFTs on (n2, n2+4), twiddle W8^(n2 k1), 4-point DFTs over n2
  static PD void run(C* a, int o, int st, int dir) {
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) dft2(a[o + n2 * st], a[o + (n2 + 4) * st]);
    a[o + 5 * st] = cmul(a[o + 5 * st], w16<C>(2, dir));
    a[o + 6 * st] = cmul(a[o + 6 * st], w16<C>(4, dir));
    a[o + 7 * st] = cmul(a[o + 7 * st], w16<C>(6, dir));
    dft4(a[o], a[o + st], a[o + 2 * st], a[o + 3 * st], dir);
    dft4(a[o + 4 * st], a[o + 5 * st], a[o + 6 * st], a[o + 7 * st], dir);
    C t[8];  // X[k1 + 2 k2] = a[4 k1 + k2]
#pragma unroll
    for (int k1 = 0; k1 < 2; ++k1)
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) t[k1 + 2 * k2] = a[o + (k1 * 4 + k2) * st];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[o + k * st] = t[k];
  }
};
template <typename C> struct Dft<16, C> {
  // 16 = 4 x 4: 4-point DFTs on (n2, n2+4, n2+8, n2+12), twiddle W16^(n2 k1), 4-point DFTs
  static PD void run(C* a, int o, int st, int dir) {
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2)
      dft4(a[o + n2 * st], a[o + (n2 + 4) * st], a[o + (n2 + 8) * st], a[o + (n2 + 12) * st], dir);
#pragma unroll
    for (int n2 = 1; n2 < 4; ++n2)
#pragma unroll
      for (int k1 = 1; k1 < 4; ++k1)
        a[o + (n2 + 4 * k1) * st] = cmul(a[o + (n2 + 4 * k1) * st], w16<C>(n2 * k1, dir));
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
      dft4(a[o + 4 * k1 * st], a[o + (4 * k1 + 1) * st], a[o + (4 * k1 + 2) * st], a[o + (4 * k1 + 3) * st], dir);
    C t[16];  // X[k1 + 4 k2] = a[4 k1 + k2]
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) t[k1 + 4 * k2] = a[o + (4 * k1 + k2) * st];
#pragma unroll
    for (int k = 0; k < 16; ++k) a[o + k * st] = t[k];
  }
};

// cos / sin of 2 pi m / 32 with the sign of `dir`, for the fixed m of the radix-32 butterfly
template <typename C> PD C w32(int m, int dir) {
  typedef decltype(C().x) T;
  constexpr double c[9] = {1.0,
                           0.98078528040323044913,
                           0.92387953251128675613,
                           0.83146961230254523708,
                           0.70710678118654752440,
                           0.55557023301960222474,
                           0.38268343236508977173,
                           0.19509032201612826785,
                           0.0};
  const int q = (m >> 3) & 3, f = m & 7;  // quadrant, angle within it
  const double a = c[f], b = c[8 - f];
  const T re = T(q == 0 ? a : (q == 1 ? -b : (q == 2 ? -a : b)));
  const T im = T(q == 0 ? b : (q == 1 ? a : (q == 2 ? -b : -a)));
  return cmk<C>(re, dir < 0 ? -im : im);
}
template <typename C> struct Dft<32, C> {
  // 32 = 4 x 8: 4-point DFTs on (n2, n2+8, n2+16, n2+24), twiddle W32^(n2 k1), 8-point DFTs
  static PD void run(C* a, int o, int st, int dir) {
#pragma unroll
    for (int n2 = 0; n2 < 8; ++n2)
      dft4(a[o + n2 * st], a[o + (n2 + 8) * st], a[o + (n2 + 16) * st], a[o + (n2 + 24) * st], dir);
#pragma unroll
    for (int n2 = 1; n2 < 8; ++n2)
#pragma unroll
      for (int k1 = 1; k1 < 4; ++k1)
        a[o + (n2 + 8 * k1) * st] = cmul(a[o + (n2 + 8 * k1) * st], w32<C>(n2 * k1, dir));
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) Dft<8, C>::run(a, o + 8 * k1 * st, st, dir);
    C t[32];  // X[k1 + 4 k2] = a[8 k1 + k2]
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
      for (int k2 = 0; k2 < 8; ++k2) t[k1 + 4 * k2] = a[o + (8 * k1 + k2) * st];
#pragma unroll
    for (int k = 0; k < 32; ++k) a[o + k * st] = t[k];
  }
};

PD int sidx(int e) { return e + (e >> 4); }  // padded shared index

// Compile-time plan of a length-2^LOGN transform with E (8 or 16) elements
// per thread: radix-E stages, then one radix-2^r stage for the remaining r
// bits; T = N/E threads per sequence.
template <int LOGN, int E = 16> struct Plan {
  static_assert(E == 8 || E == 16, "8 or 16 elements per thread");
  static constexpr int LE = E == 16 ? 4 : 3;
  static constexpr int N = 1 << LOGN;
  static constexpr int T = N / E;
  static constexpr int NST = (LOGN + LE - 1) / LE;
  __host__ __device__ static constexpr int radix(int st) {
    return st + 1 < NST ? E : (1 << (LOGN - LE * (NST - 1)));
  }
};

// One Stockham stage on the registers: v[m] holds element t + m T of the
// stage input.  Thread t owns butterflies j = t + q T (q < E/R); input r of
// butterfly j is element j + r N/R, i.e. register q + r E/R.  After the
// twiddles and the DFT, register q + r E/R is output (j - k) R + k + r Ns
// with k = j mod Ns; sink(position, value) receives every output.
template <int R, int N, int T, int E, typename C, typename Sink>
PD void stage(C (&v)[E], int t, int Ns, const C* __restrict__ tw, int dir, Sink sink) {
  constexpr int Q = E / R;
  const int tstride = N / (Ns * R);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = t + q * T;
    const int k = j & (Ns - 1);
    if (k) {
#pragma unroll
      for (int r = 1; r < R; ++r) {
        C w = tw[r * k * tstride];
        if (dir > 0) w.y = -w.y;
        v[q + r * Q] = cmul(v[q + r * Q], w);
      }
    }
    Dft<R, C>::run(v, q, Q, dir);
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = t + q * T;
    const int k = j & (Ns - 1);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) sink(base + r * Ns, v[q + r * Q]);
  }
}

// Shared buffers hold element q of a sequence at s[sidx(q) * ss]: ss = 1 for
// one sequence per buffer (rows), ss = cw for cw interleaved columns, so that
// the lanes that read 32 contiguous bytes of cw columns from global memory
// also touch contiguous shared words.
template <int LOGN, int ST, int E, typename C, typename Store>
PD void run_stages(C (&v)[E], int t, int Ns, C* s, int ss, const C* tw, int dir, Store store) {
  typedef Plan<LOGN, E> P;
  constexpr int R = P::radix(ST);
  if constexpr (ST + 1 == P::NST) {
    stage<R, P::N, P::T, E>(v, t, Ns, tw, dir, store);
  } else {
    stage<R, P::N, P::T, E>(v, t, Ns, tw, dir, [&](int q, C x) { s[sidx(q) * ss] = x; });
    __syncthreads();
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = s[sidx(t + m * P::T) * ss];
    __syncthreads();
    run_stages<LOGN, ST + 1, E>(v, t, Ns * R, s, ss, tw, dir, store);
  }
}

// All stages of one sequence: load(m) supplies input element t + m T,
// store(q, value) receives output q.
template <int LOGN, int E = 16, typename C, typename Load, typename Store>
PD void fft_seq(int t, C* s, int ss, const C* tw, int dir, Load load, Store store) {
  C v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = load(m);
  run_stages<LOGN, 0, E>(v, t, 1, s, ss, tw, dir, store);
}

constexpr int kRowCta = 256;  // threads per CTA of the plain row transforms

// Column passes read kColBytes contiguous bytes of each row: col_width
// interleaved columns per CTA.
constexpr int kColBytes = 32;
template <typename T> inline int col_width() { return kColBytes / int(sizeof(typename cplx_t<T>::type)); }
__host__ __device__ inline size_t padded(int N) { return size_t(N) + size_t(N) / 16 + 1; }

__host__ __device__ inline size_t align16(size_t b) { return (b + 15) & ~size_t(15); }

// ------------------------------------------------- half-length transforms
// An image row (or column) holds n values on the K = 2n grid, the rest zero,
// and only n of the inverse transform's outputs are kept.  Splitting the
// frequencies by parity turns either into two independent length-n
// transforms: with the pixel's signed position p in [-n/2, n/2) taken modulo n
// as the sequence index,
//   Z(2m)     = sum_p z_p          exp(-2 pi i m p / n),
//   Z(2m + 1) = sum_p z_p omega^p  exp(-2 pi i m p / n),  omega = exp(-2 pi i / K),
// and the inverse's output at p is E(p) + conj(omega^p) O(p) from the two
// length-n inverse transforms.  No zero is ever transformed, the two halves
// meet only once (in the sum of the inverse), and because the mirror -k of a
// frequency has k's parity, the separation of a row pair's half spectra stays
// inside each half.
//
// One half is transformed by TT = n / E threads holding E elements each
// (element j = t + TT m in register m, before and after every transform), in
// radix-E stages with shared-memory exchanges between them: at n = 1024 one
// warp, two radix-32 stages and one exchange, with no CTA barrier inside (the
// length-2048 form of four radix-8 / three radix-16 stages spent its time on
// barriers, exchanges and scattered twiddle gathers).  The twiddles of stage
// st come from a table laid out [r - 1][k], so a warp's reads are contiguous.
template <typename T, int LOGN, int E_> struct Half {
  static constexpr int E = E_;
  static constexpr int LE = E == 32 ? 5 : (E == 16 ? 4 : 3);
  static constexpr int N = 1 << LOGN;
  static constexpr int TT = N / E;
  static constexpr int NST = (LOGN + LE - 1) / LE;
  static constexpr int V = 16 / int(sizeof(T));  // reals per 16-byte vector
  // elements of one half's exchange buffer (one pad element every E: the
  // first exchange writes at a stride of E)
  static constexpr int BUF = N + N / E;
  __host__ __device__ static constexpr int radix(int st) {
    return st + 1 < NST ? E : (1 << (LOGN - LE * (NST - 1)));
  }
  // row pairs of one row-pass CTA: at least a warp of threads, and enough
  // rows to fill a 32-byte sector of a transposed column (4 rows FP32, 2 FP64)
  static constexpr int PMIN = sizeof(T) == 4 ? 2 : 1;
  static constexpr int PW = 32 / (2 * TT) > 1 ? 32 / (2 * TT) : 1;
  static constexpr int PAIRS0 = PW > PMIN ? PW : PMIN;
  static constexpr int PAIRS = PAIRS0 > N / 2 ? N / 2 : PAIRS0;
  static constexpr int ROW_THREADS = 2 * TT * PAIRS;
  // columns of one convolution CTA: at least a warp
  static constexpr int COLS = PW;
  static constexpr int COL_THREADS = 2 * TT * COLS;
  // 512 threads' worth of CTAs per SM: 128 registers per thread
  static constexpr int ROW_MINB = ROW_THREADS >= 512 ? 1 : (512 / ROW_THREADS > 16 ? 16 : 512 / ROW_THREADS);
  static constexpr int COL_MINB = COL_THREADS >= 512 ? 1 : (512 / COL_THREADS > 16 ? 16 : 512 / COL_THREADS);
};

// Elements per thread.  Small images leave most of the chip idle, so more
// threads with fewer elements win (n = 512: Phi^H Phi 11.1 us with 8 / 16
// elements in the row / column passes against 14.0 with 32); at n = 1024 the
// row passes measured the same with 16 and 32 and the column pass, whose 1024
// columns fill the chip, is faster with one exchange per transform than with
// two (22.2 against 22.8 us).  FP64 elements are twice as wide: 16 at most.
template <typename T, int LOGN> struct RowHalf : Half<T, LOGN, LOGN <= 9 ? 8 : 16> {};
template <typename T, int LOGN>
struct ColHalf : Half<T, LOGN, LOGN <= 8 ? 8 : (LOGN <= 9 || sizeof(T) == 8 ? 16 : 32)> {};

// Barrier of one half's threads: they share a warp, or are whole warps.
template <int TT> PD void half_sync(int half) {
  if constexpr (TT <= 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(half + 1), "n"(TT) : "memory");
}

// One stage: R-point DFTs over registers q + r Q (element j = t + q TT of each
// is r N/R apart), twiddled by W(r k), k = j mod Ns.
template <typename H, int R, int NS, int DIR, typename C>
PD void half_stage(C (&v)[H::E], int t, const C* __restrict__ tab) {
  constexpr int Q = H::E / R;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    if constexpr (NS > 1) {
      const int k = (t + q * H::TT) & (NS - 1);
#pragma unroll
      for (int r = 1; r < R; ++r) {
        C w = tab[(r - 1) * NS + k];
        if (DIR > 0) w.y = -w.y;
        v[q + r * Q] = cmul(v[q + r * Q], w);
      }
    }
    Dft<R, C>::run(v, q, Q, DIR);
  }
}

// All stages; s is the half's exchange buffer, free to be overwritten.  The
// last stage leaves output j = t + TT m in register m, as the input was.
template <typename H, int DIR, int ST = 0, int NS = 1, typename C>
PD void half_fft(C (&v)[H::E], int t, C* s, int half, const C* __restrict__ tab) {
  constexpr int R = H::radix(ST);
  half_stage<H, R, NS, DIR>(v, t, tab);
  if constexpr (ST + 1 < H::NST) {
    constexpr int Q = H::E / R;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int j = t + q * H::TT, k = j & (NS - 1), base = (j - k) * R + k;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int e = base + r * NS;
        s[e + (e >> H::LE)] = v[q + r * Q];
      }
    }
    half_sync<H::TT>(half);
#pragma unroll
    for (int m = 0; m < H::E; ++m) {
      const int e = t + m * H::TT;
      v[m] = s[e + (e >> H::LE)];
    }
    half_sync<H::TT>(half);
    half_fft<H, DIR, ST + 1, NS * R>(v, t, s, half, tab + (NS > 1 ? (R - 1) * NS : 0));
  }
}

// omega^p (DIR -1) or its conjugate (DIR +1) at element j = t + TT m, from the
// table tw[j] = exp(-2 pi i j / K); positions past n/2 are p = j - n: a sign.
template <typename H, int DIR, typename C> PD void half_omega(C (&v)[H::E], int t, const C* __restrict__ tw) {
#pragma unroll
  for (int m = 0; m < H::E; ++m) {
    C w = tw[t + m * H::TT];
    if (DIR > 0) w.y = -w.y;
    if (m >= H::E / 2) w = cneg(w);
    v[m] = cmul(v[m], w);
  }
}

// The sum of a column's two inverse halves into its n rows at Bc: each half
// finishes half of the rows and hands over the rest through its buffer.
template <typename H, typename C>
PD void half_join(const C (&v)[H::E], int t, int odd, C* bufs, int half, C* Bc) {
  constexpr int E = H::E, TT = H::TT;
  C* s = bufs + size_t(half) * H::BUF;
#pragma unroll
  for (int m = 0; m < E / 2; ++m) {
    if (odd) s[t + m * TT] = v[m];
    else s[t + (m + E / 2) * TT] = v[m + E / 2];
  }
  __syncthreads();
  const C* so = bufs + size_t(half ^ 1) * H::BUF;
#pragma unroll
  for (int m = 0; m < E / 2; ++m) {
    const int me = m + (odd ? E / 2 : 0);
    const C mine = odd ? v[m + E / 2] : v[m];
    Bc[t + ((me + E / 2) & (E - 1)) * TT] = cadd(mine, so[t + me * TT]);
  }
}

// 16-byte vectors of reals; `al` says the address is 16-byte aligned (a
// caller's array need not be).
template <typename T> struct V16;
template <> struct V16<float> { typedef float4 type; };
template <> struct V16<double> { typedef double2 type; };
template <typename T, int V> PD void vload(T (&d)[V], const T* p, bool al) {
  if (al) {
    const typename V16<T>::type x = *reinterpret_cast<const typename V16<T>::type*>(p);
    const T* e = reinterpret_cast<const T*>(&x);
#pragma unroll
    for (int k = 0; k < V; ++k) d[k] = e[k];
  } else {
#pragma unroll
    for (int k = 0; k < V; ++k) d[k] = p[k];
  }
}
template <typename T, int V> PD void vstore(T* p, const T (&d)[V], bool al) {
  if (al) {
    typename V16<T>::type x;
    T* e = reinterpret_cast<T*>(&x);
#pragma unroll
    for (int k = 0; k < V; ++k) e[k] = d[k];
    *reinterpret_cast<typename V16<T>::type*>(p) = x;
  } else {
#pragma unroll
    for (int k = 0; k < V; ++k) p[k] = d[k];
  }
}
PD bool aligned16(const void* p) { return (reinterpret_cast<size_t>(p) & 15) == 0; }

// V consecutive complex values in shared memory, by 16-byte accesses.
template <typename C, int V> PD void cload(C (&d)[V], const C* p) {
  constexpr int W = 16 / int(sizeof(C));
  typedef typename V16<decltype(C().x)>::type X;
#pragma unroll
  for (int k = 0; k < V; k += W) {
    const X x = *reinterpret_cast<const X*>(p + k);
    const C* e = reinterpret_cast<const C*>(&x);
#pragma unroll
    for (int q = 0; q < W; ++q) d[k + q] = e[q];
  }
}
template <typename C, int V> PD void cstore(C* p, const C (&d)[V]) {
  constexpr int W = 16 / int(sizeof(C));
  typedef typename V16<decltype(C().x)>::type X;
#pragma unroll
  for (int k = 0; k < V; k += W) {
    X x;
    C* e = reinterpret_cast<C*>(&x);
#pragma unroll
    for (int q = 0; q < W; ++q) e[q] = d[k + q];
    *reinterpret_cast<X*>(p + k) = x;
  }
}

// 32-byte global accesses (one sector): 4 complex floats or 2 complex doubles.
PD void ld32(float2 (&d)[4], const float2* p) {
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(d[0].x), "=f"(d[0].y), "=f"(d[1].x), "=f"(d[1].y), "=f"(d[2].x), "=f"(d[2].y), "=f"(d[3].x),
                 "=f"(d[3].y)
               : "l"(p));
}
PD void ld32(double2 (&d)[2], const double2* p) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(d[0].x), "=d"(d[0].y), "=d"(d[1].x), "=d"(d[1].y)
               : "l"(p));
}
PD void st32(float2* p, const float2 (&d)[4]) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(d[0].x), "f"(d[0].y),
               "f"(d[1].x), "f"(d[1].y), "f"(d[2].x), "f"(d[2].y), "f"(d[3].x), "f"(d[3].y)
               : "memory");
}
PD void st32(double2* p, const double2 (&d)[2]) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(d[0].x), "d"(d[0].y), "d"(d[1].x),
               "d"(d[1].y)
               : "memory");
}

// Element (column c, row i) of the half-spectrum buffer B: stored transposed,
// each column's n rows contiguous, the even columns before the odd ones --
// the column passes read and write whole lines, and the row passes whole
// 32-byte sectors (2 PAIRS rows of a column).
PD size_t half_at(int c, int i, int n) { return (size_t(c & 1) * (n / 2) + (c >> 1)) * n + i; }

// Row-pass epilogues (see RowEpMode): the outputs of V consecutive pixels
// from their transform values and operands (a, b: see ep_staged), and the
// mode's partial sums.
template <typename T> struct EpAcc { Acc<T> a[5]; };
template <int MODE, int V, typename T>
PD void row_ep_store(const RowEp<T>& ep, size_t idx, bool al, const T (&val)[V], const T (&a)[V], const T (&b)[V],
                     EpAcc<T>& part, Acc<T> (&sq)[V]) {
  T o[V];
#pragma unroll
  for (int k = 0; k < V; ++k) {
    if constexpr (MODE == EP_CG_AP) {
      // (A p)_i; a short run of terms is summed by plain FMAs (their rounding
      // errors are independent across the ~10^5 runs and average out) and
      // then merged compensated.
      o[k] = T(ep.nu2) * val[k] + T(2) * a[k];
      part.a[0].s = fma(a[k], o[k], part.a[0].s);
      part.a[1].s = fma(b[k], o[k], part.a[1].s);
      part.a[2].s = fma(o[k], o[k], part.a[2].s);
      part.a[3].s = fma(b[k], a[k], part.a[3].s);
      part.a[4].s = fma(b[k], b[k], part.a[4].s);
    } else if constexpr (MODE == EP_CG_R0) {
      o[k] = (a[k] - T(2) * b[k]) - T(ep.nu2) * val[k];
    } else if constexpr (MODE == EP_POWER) {
      o[k] = val[k];
      sq[k].add_prod(val[k], val[k]);
    } else if constexpr (MODE == EP_XS_ADD) {
      o[k] = a[k] + T(ep.nu) * val[k];
    } else if constexpr (MODE == EP_QX) {
      o[k] = T(ep.nu2) * val[k] + T(2) * a[k];
    } else {
      o[k] = val[k];
    }
  }
  vstore(ep.out + idx, o, al);
  if constexpr (MODE == EP_CG_R0) vstore(ep.out2 + idx, o, al);
}

// The scalars of a prologue from the sums an earlier epilogue left (one thread;
// FP64 arithmetic is slow, and its latency hides behind the loads in flight):
//   PRO_CG_STEP: from <p,Ap>, <r,Ap>, <Ap,Ap>, <r,p> and <r,r> of the step's
//             vectors the exact line search alpha = <r,p> / <p,Ap> (equal to
//             <r,r> / <p,Ap> in exact arithmetic); the next residual norm by
//             ||r - alpha Ap||^2 = <r,r> - 2 alpha <r,Ap> + alpha^2 <Ap,Ap>
//             (clamped at 0); beta = ||r_new||^2 / <r,r>.
//   PRO_SCALE: 1 / ||x||.
template <typename T> PD void pro_scalars(const RowPro<T>& pro, T* ab) {
  if (threadIdx.x == 0) {
    if (pro.mode == PRO_CG_STEP) {
      double q[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) q[k] = __ldcg(pro.acc + k);
      const double alpha = cg_alpha(q[3], q[0]);
      double rr = q[4] - 2.0 * alpha * q[1] + alpha * alpha * q[2];
      if (rr < 0.0) rr = 0.0;
      ab[0] = T(alpha);
      ab[1] = T(q[4] > 0.0 ? rr / q[4] : 0.0);
    } else {
      const double l = sqrt(__ldcg(pro.acc));
      ab[0] = T(l > 0.0 ? 1.0 / l : 0.0);
    }
  }
  __syncthreads();
}

// Forward row prologue (see RowProMode) of V consecutive pixels of U chunks
// of a row pair (pixel offsets ia of row a; row b is n further on).  All loads
// precede the CG step's stores.
template <int U, int V, typename T>
PD void row_prologue(const RowPro<T>& pro, const size_t (&ia)[U], int n, bool al, T (&va)[U][V], T (&vb)[U][V],
                     T* ab /*[2], shared*/) {
  if (pro.mode == PRO_CG_STEP) {
    // x += alpha p, r -= alpha Ap, p = r + beta p (alpha, beta of the previous step)
    T xv[2 * U][V], rv[2 * U][V], pv[2 * U][V], av[2 * U][V];
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      const size_t i = ia[u >> 1] + size_t(u & 1) * n;
      vload(xv[u], pro.xu + i, true);
      vload(rv[u], pro.r + i, true);
      vload(pv[u], pro.p + i, true);
    }
    // x, r and p come from the previous step's forward pass, which had
    // completed before its column pass let this chain go on; A p and the
    // scalars from the pass just before
    pdl_wait();
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) vload(av[u], pro.ap + ia[u >> 1] + size_t(u & 1) * n, true);
    pro_scalars(pro, ab);
    const T alpha = ab[0], beta = ab[1];
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      const size_t i = ia[u >> 1] + size_t(u & 1) * n;
      T xn[V], rn[V], pn[V];
#pragma unroll
      for (int k = 0; k < V; ++k) {
        rn[k] = fma(-alpha, av[u][k], rv[u][k]);
        xn[k] = fma(alpha, pv[u][k], xv[u][k]);
        pn[k] = fma(beta, pv[u][k], rn[k]);
        if (u & 1) vb[u >> 1][k] = pn[k];
        else va[u >> 1][k] = pn[k];
      }
      vstore(pro.xu + i, xn, true);
      vstore(pro.r + i, rn, true);
      vstore(pro.p + i, pn, true);
    }
  } else if (pro.mode == PRO_CG_START) {
    // r = b - A x_hat, p = r (b in pro.x, A x_hat in pro.ap)
    pdl_wait();
    T bv[2 * U][V], av[2 * U][V];
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      const size_t i = ia[u >> 1] + size_t(u & 1) * n;
      vload(bv[u], pro.x + i, true);
      vload(av[u], pro.ap + i, true);
    }
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      const size_t i = ia[u >> 1] + size_t(u & 1) * n;
      T rn[V];
#pragma unroll
      for (int k = 0; k < V; ++k) {
        rn[k] = bv[u][k] - av[u][k];
        if (u & 1) vb[u >> 1][k] = rn[k];
        else va[u >> 1][k] = rn[k];
      }
      vstore(pro.r + i, rn, true);
      vstore(pro.p + i, rn, true);
    }
  } else {
    pdl_wait();
    if (pro.mode == PRO_SCALE) pro_scalars(pro, ab);
    const T scl = pro.mode == PRO_SCALE ? ab[0] : T(1);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      vload(va[u], pro.x + ia[u], al);
      vload(vb[u], pro.x + ia[u] + n, al);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int k = 0; k < V; ++k) {
        va[u][k] *= scl;
        vb[u][k] *= scl;
      }
  }
}

// The epilogue's sums: each CTA's go into FP64 accumulators (ep.acc) by atomics;
// the pass that needs them reads them there (row_prologue, k_axpy), so no CTA
// waits for the others.
template <typename T> PD void row_ep_finish(const RowEp<T>& ep, EpAcc<T> part, double* red /*[5*32]*/) {
  if (!ep.acc) return;
  const int nsum = ep.mode == EP_CG_AP ? 5 : 1;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = int((blockDim.x + 31) >> 5);
  Acc<T>* st = reinterpret_cast<Acc<T>*>(red);
  for (int k = 0; k < nsum; ++k) {
    warp_merge(part.a[k]);
    if (lane == 0) st[k * 32 + w] = part.a[k];
  }
  __syncthreads();
  // one warp per sum where there are enough
  for (int k = w; k < nsum; k += nw) {
    Acc<T> b = lane < nw ? st[k * 32 + lane] : Acc<T>();
    warp_merge(b);
    if (lane == 0) atomicAdd(ep.acc + k, b.value());
  }
}

// ----------------------------------------------------------------- kernels
template <typename T, int LOGN> struct ColThreads {
  static constexpr int value = (kColBytes / int(sizeof(typename cplx_t<T>::type))) * ((1 << LOGN) / 16);
};

// The image is real, so two rows a, b travel as one complex row z = x_a + i x_b,
// whose transform Z separates as X_a(k) = (Z(k) + conj Z(-k)) / 2 and
// X_b(k) = (Z(k) - conj Z(-k)) / (2i), and only the half spectrum k in [0, K/2]
// is kept: n complex values, entry 0 carrying the two real ones,
// X(0) + i X(K/2).  They are stored transposed (half_at).

// Forward row pass of the real form: PAIRS row pairs per CTA, zero-padded to K
// columns, to their half spectra.  Per pair two halves of TT threads.  Latency
// and L1 bound (one wave, an L2-resident set; shared-memory exchanges and
// 32-byte stores): n = 1024 with the CG update as prologue 8.8 us, against
// 11.5 us for 2048-point transforms on 256 threads.
template <typename T, int LOGN, typename Src>
__global__ void __launch_bounds__(RowHalf<T, LOGN>::ROW_THREADS, RowHalf<T, LOGN>::ROW_MINB) k_row_fwd_h(Src src) {
  typedef typename cplx_t<T>::type C;
  typedef RowHalf<T, LOGN> H;
  constexpr int n = H::N, V = H::V, E = H::E, TT = H::TT, NT = H::ROW_THREADS;
  decltype(auto) a = src.get();
  const RowPro<T>& pro = a.pro;
  const T* __restrict__ deapod = a.deapod;
  C* __restrict__ B = a.B;
  const C* __restrict__ tw = a.tw;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C* zb = reinterpret_cast<C*>(sm_raw);      // [PAIRS][n]: the packed rows
  C* bufs = zb + H::PAIRS * n;               // [PAIRS][2][BUF]
  __shared__ T ab[2];
  const int r0 = int(blockIdx.x) * 2 * H::PAIRS;
  {
    constexpr int CH = H::PAIRS * n / V;     // chunks of V pixels of a row pair
    constexpr int IT = CH / NT, U = IT % 2 == 0 ? 2 : 1;
    static_assert(CH % NT == 0, "E is a multiple of 2 V");
    const bool al = aligned16(pro.x);
    for (int it = 0; it < IT; it += U) {
      size_t ia[U];
      int at[U];
      T va[U][V], vb[U][V];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int ch = int(threadIdx.x) + (it + u) * NT;
        const int pr = ch / (n / V), i = (ch - pr * (n / V)) * V;
        at[u] = pr * n + i;
        ia[u] = size_t(r0 + 2 * pr) * n + i;
      }
      row_prologue<U, V>(pro, ia, n, al, va, vb, ab);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (deapod) {  // S: deapodisation of both rows (the Phi form; the convolution form has none)
          const int row = r0 + 2 * (at[u] / n), i = at[u] & (n - 1);
          const T da = deapod[row], db = deapod[row + 1];
          T dc[V];
          vload(dc, deapod + i, true);
#pragma unroll
          for (int k = 0; k < V; ++k) {
            va[u][k] *= da * dc[k];
            vb[u][k] *= db * dc[k];
          }
        }
        C z[V];
#pragma unroll
        for (int k = 0; k < V; ++k) z[k] = cmk<C>(va[u][k], vb[u][k]);
        cstore(zb + at[u], z);
      }
    }
  }
  // (every prologue has waited by now) the accumulators of this pass's product
  if (pro.zero && blockIdx.x == 0)
    for (int k = threadIdx.x; k < pro.nzero; k += NT) pro.zero[k] = 0.0;
  __syncthreads();
  const int half = threadIdx.x / TT, t = threadIdx.x - half * TT;
  const int pr = half >> 1, odd = half & 1;
  C* s = bufs + size_t(half) * H::BUF;
  C v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = zb[pr * n + t + ((m + E / 2) & (E - 1)) * TT];  // pixel of position j mod n
  if (odd) half_omega<H, -1>(v, t, tw);
  half_fft<H, -1>(v, t, s, half, a.tws);
#pragma unroll
  for (int m = 0; m < E; ++m) s[t + m * TT] = v[m];
  __syncthreads();
  pass_trigger<T, LOGN>();
  // separate the pairs: column c = 2m + odd from elements m and -m of its half
  constexpr int PC = sizeof(T) == 4 ? 2 : 1;  // pairs per 32-byte store
  static_assert(H::PAIRS % PC == 0, "whole sectors");
  for (int w = threadIdx.x; w < n * (H::PAIRS / PC); w += NT) {
    const int cp = w & (n - 1), pc = w / n;  // column in storage order
    const int o = cp >= n / 2, m = cp - o * (n / 2), mm = o ? n - 1 - m : (n - m) & (n - 1);
    C out[2 * PC];
#pragma unroll
    for (int q = 0; q < PC; ++q) {
      const C* hs = bufs + size_t((pc * PC + q) * 2 + o) * H::BUF;
      const C zk = hs[m];
      if (cp == 0) {
        const C zh = hs[n / 2];
        out[2 * q] = cmk<C>(zk.x, zh.x);
        out[2 * q + 1] = cmk<C>(zk.y, zh.y);
      } else {
        const C zm = hs[mm];  // Z(-k)
        out[2 * q] = cmk<C>(T(0.5) * (zk.x + zm.x), T(0.5) * (zk.y - zm.y));
        out[2 * q + 1] = cmk<C>(T(0.5) * (zk.y + zm.y), T(0.5) * (zm.x - zk.x));
      }
    }
    st32(B + size_t(cp) * n + r0 + pc * 2 * PC, out);
  }
}

// Column pass of the convolution form (Section 3: Phi^H Phi precomputed): the
// forward FFT of each half-spectrum column over the K grid rows (n non-zero),
// the product with the PSF's real spectrum, and the inverse FFT's n kept rows,
// all in one thread's registers (the forward transform ends in the order in
// which the inverse begins).  Column 0 holds two real-row columns,
// c0 = X(., 0) + i X(., K/2): its transform P splits into the even part
// (P(q) + conj P(-q)) / 2 (column 0's) and (P(q) - conj P(-q)) / 2 (i times
// column K/2's), each multiplied by its own spectrum column.
// One column (two warps at n = 1024) per CTA, so that 1024 small CTAs spread
// evenly: 11.4 us against 22.3 us for 256 CTAs of four 2048-point columns.
template <typename T, int LOGN, typename Src>
__global__ void __launch_bounds__(ColHalf<T, LOGN>::COL_THREADS, ColHalf<T, LOGN>::COL_MINB) k_col_conv_h(Src src) {
  typedef typename cplx_t<T>::type C;
  typedef ColHalf<T, LOGN> H;
  constexpr int n = H::N, E = H::E, TT = H::TT;
  decltype(auto) a = src.get();
  const T* __restrict__ khat = a.khat;
  const C* __restrict__ tw = a.tw;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  pdl_wait();
  C* bufs = reinterpret_cast<C*>(sm_raw);
  const int half = threadIdx.x / TT, t = threadIdx.x - half * TT;
  const int col = int(blockIdx.x) * H::COLS + (half >> 1), odd = half & 1;
  C* s = bufs + size_t(half) * H::BUF;
  C* __restrict__ Bc = a.B + size_t(col) * n;
  C v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = Bc[t + ((m + E / 2) & (E - 1)) * TT];
  if (odd) half_omega<H, -1>(v, t, tw);
  half_fft<H, -1>(v, t, s, half, a.tws);
  const T* kc = khat + (size_t(col) * 2 + odd) * n;
  if (blockIdx.x == 0) {
#pragma unroll
    for (int m = 0; m < E; ++m) s[t + m * TT] = v[m];
    __syncthreads();
    const T* kn = a.knyq + odd * n;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int q = t + m * TT;
      const T h0 = kc[q];
      if (col == 0) {
        const T hn = kn[q];
        const C P = v[m], Pm = s[odd ? n - 1 - q : (n - q) & (n - 1)];
        const T evx = T(0.5) * (P.x + Pm.x), evy = T(0.5) * (P.y - Pm.y);
        const T odx = T(0.5) * (P.x - Pm.x), ody = T(0.5) * (P.y + Pm.y);
        v[m] = cmk<C>(h0 * evx + hn * odx, h0 * evy + hn * ody);
      } else {
        v[m] = cscale(v[m], h0);
      }
    }
    __syncthreads();
  } else {
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = cscale(v[m], kc[t + m * TT]);
  }
  half_fft<H, 1>(v, t, s, half, a.tws);
  if (odd) half_omega<H, 1>(v, t, tw);
  pass_trigger<T, LOGN>();
  half_join<H>(v, t, odd, bufs, half, Bc);
}

// Operand arrays an epilogue reads (staged in shared memory by the inverse row
// pass): CG_AP p, r; CG_R0 b, p; QX p; XS_ADD b.
template <typename T> PD int ep_staged(const RowEp<T>& ep, const T** src) {
  switch (ep.mode) {
    case EP_CG_AP: src[0] = ep.p; src[1] = ep.r; return 2;
    case EP_CG_R0: src[0] = ep.b; src[1] = ep.p; return 2;
    case EP_QX: src[0] = ep.p; return 1;
    case EP_XS_ADD: src[0] = ep.b; return 1;
    default: return 0;
  }
}
// Sum of the halves, deapodisation (S^T after the crop: the Phi^H form) and
// epilogue of the CTA's rows, V pixels of a row pair at a time; the operands
// lie in shared memory (ops[pair][k][row][n]).
template <int LOGN, int MODE, typename T>
PD EpAcc<T> row_ep_rows(const RowEp<T>& ep, const typename cplx_t<T>::type* bufs, const T* ops, const T* deapod,
                        int r0) {
  typedef typename cplx_t<T>::type C;
  typedef RowHalf<T, LOGN> H;
  constexpr int n = H::N, V = H::V, NT = H::ROW_THREADS;
  constexpr int NOP = MODE == EP_CG_AP || MODE == EP_CG_R0 ? 2 : (MODE == EP_QX || MODE == EP_XS_ADD ? 1 : 0);
  const bool al = MODE != EP_STORE || aligned16(ep.out);  // only EP_STORE writes a caller's array
  EpAcc<T> part, run;
  Acc<T> sq[V];  // compensated sums of squares, V independent chains
  int terms = 0;
  for (int ch = threadIdx.x; ch < H::PAIRS * n / V; ch += NT) {
    const int pr = ch / (n / V), i = (ch - pr * (n / V)) * V;
    const C* he = bufs + size_t(2 * pr) * H::BUF + i;
    const C* ho = he + H::BUF;
    T val[2][V];
    C ze[V], zo[V];
    cload(ze, he);
    cload(zo, ho);
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const C z = cadd(ze[k], zo[k]);
      val[0][k] = z.x;
      val[1][k] = z.y;
    }
    const int row = r0 + 2 * pr;
    if (deapod) {
      const T da = deapod[row], db = deapod[row + 1];
      T dc[V];
      vload(dc, deapod + i, true);
#pragma unroll
      for (int k = 0; k < V; ++k) {
        val[0][k] *= da * dc[k];
        val[1][k] *= db * dc[k];
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      T o0[V] = {}, o1[V] = {};
      if constexpr (NOP > 0) vload(o0, ops + (size_t(2 * pr) * 2 + r) * n + i, true);
      if constexpr (NOP > 1) vload(o1, ops + (size_t(2 * pr + 1) * 2 + r) * n + i, true);
      row_ep_store<MODE>(ep, size_t(row + r) * n + i, al, val[r], o0, o1, part, sq);
    }
    if constexpr (MODE == EP_CG_AP) {  // plain runs of 16 terms
      terms += 2 * V;
      if (terms >= 16 || V < 4) {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          run.a[k].add(part.a[k].s);
          part.a[k] = Acc<T>();
        }
        terms = 0;
      }
    }
  }
  if constexpr (MODE == EP_CG_AP) {
#pragma unroll
    for (int k = 0; k < 5; ++k) acc_merge(run.a[k], part.a[k]);
    return run;
  }
  if constexpr (MODE == EP_POWER) {
#pragma unroll
    for (int k = 0; k < V; ++k) acc_merge(part.a[0], sq[k]);
  }
  return part;
}
template <int LOGN, typename T>
PD EpAcc<T> row_ep_all(const RowEp<T>& ep, const typename cplx_t<T>::type* bufs, const T* ops, const T* deapod, int r0) {
  switch (ep.mode) {
    case EP_CG_AP: return row_ep_rows<LOGN, EP_CG_AP>(ep, bufs, ops, deapod, r0);
    case EP_CG_R0: return row_ep_rows<LOGN, EP_CG_R0>(ep, bufs, ops, deapod, r0);
    case EP_POWER: return row_ep_rows<LOGN, EP_POWER>(ep, bufs, ops, deapod, r0);
    case EP_XS_ADD: return row_ep_rows<LOGN, EP_XS_ADD>(ep, bufs, ops, deapod, r0);
    case EP_QX: return row_ep_rows<LOGN, EP_QX>(ep, bufs, ops, deapod, r0);
    default: return row_ep_rows<LOGN, EP_STORE>(ep, bufs, ops, deapod, r0);
  }
}

// Inverse row pass of the real form: the half spectra of rows a and b rebuilt
// into Z = Y_a + i Y_b over all K frequencies (Y(K - k) = conj Y(k)), one
// inverse transform by halves, Re -> row a, Im -> row b, crop and row
// epilogue.  Bound as the forward pass: n = 1024 with the CG epilogue 9.8 us,
// against 14.0 us for 2048-point transforms.
template <typename T, int LOGN, typename Src>
__global__ void __launch_bounds__(RowHalf<T, LOGN>::ROW_THREADS, RowHalf<T, LOGN>::ROW_MINB) k_row_inv_h(Src src) {
  typedef typename cplx_t<T>::type C;
  typedef RowHalf<T, LOGN> H;
  constexpr int n = H::N, E = H::E, TT = H::TT, NT = H::ROW_THREADS;
  decltype(auto) a = src.get();
  const C* __restrict__ B = a.B;
  const RowEp<T>& ep = a.ep;
  const C* __restrict__ tw = a.tw;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ double red[5 * 32];
  __shared__ __align__(8) uint64_t bar;
  C* bufs = reinterpret_cast<C*>(sm_raw);  // [PAIRS][2][BUF]
  const int r0 = int(blockIdx.x) * 2 * H::PAIRS;
  // The epilogue's operand rows (ops[pair][k][row][n]) arrive by bulk copies
  // while the transform runs.
  T* ops = reinterpret_cast<T*>(sm_raw + align16(size_t(H::PAIRS) * 2 * H::BUF * sizeof(C)));
  const T* opd[2] = {nullptr, nullptr};
  const int nop = ep_staged(ep, opd);
  // a CG step's operands p and r come from its forward pass, complete before
  // the column pass let this one start; other modes' may be the last kernel's
  if (ep.mode != EP_CG_AP) pdl_wait();
  if (nop > 0 && threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_barrier_init();
    const uint32_t pair_bytes = uint32_t(2 * n * sizeof(T));  // rows a and b are contiguous
    mbar_arrive_expect_tx(&bar, uint32_t(H::PAIRS * nop) * pair_bytes);
    for (int q = 0; q < H::PAIRS; ++q)
      for (int k = 0; k < nop; ++k)
        bulk_load(ops + (size_t(q) * 2 + k) * 2 * n, opd[k] + size_t(r0 + 2 * q) * n, pair_bytes, &bar);
  }
  if (ep.mode == EP_CG_AP) pdl_wait();
  // the halves' spectra: column c = 2m + odd gives elements m and -m of its half
  constexpr int PC = sizeof(T) == 4 ? 2 : 1;
  constexpr int LT = n * (H::PAIRS / PC) / NT, LU = LT % 4 == 0 ? 4 : (LT % 2 == 0 ? 2 : 1);  // LU loads in flight
  for (int l = 0; l < LT; l += LU) {
    C ins[LU][2 * PC];
#pragma unroll
    for (int u = 0; u < LU; ++u) {
      const int w = int(threadIdx.x) + (l + u) * NT;
      ld32(ins[u], B + size_t(w & (n - 1)) * n + r0 + (w / n) * 2 * PC);
    }
#pragma unroll
    for (int u = 0; u < LU; ++u)
#pragma unroll
    for (int q = 0; q < PC; ++q) {
      const int w = int(threadIdx.x) + (l + u) * NT;
      const int cp = w & (n - 1), pc = w / n;
      const int o = cp >= n / 2, m = cp - o * (n / 2), mm = o ? n - 1 - m : (n - m) & (n - 1);
      const C (&in)[2 * PC] = ins[u];
      C* hs = bufs + size_t((pc * PC + q) * 2 + o) * H::BUF;
      const C ya = in[2 * q], yb = in[2 * q + 1];
      if (cp == 0) {
        hs[0] = cmk<C>(ya.x, yb.x);
        hs[n / 2] = cmk<C>(ya.y, yb.y);
      } else {
        hs[m] = cmk<C>(ya.x - yb.y, ya.y + yb.x);
        hs[mm] = cmk<C>(ya.x + yb.y, yb.x - ya.y);
      }
    }
  }
  __syncthreads();
  const int half = threadIdx.x / TT, t = threadIdx.x - half * TT, odd = half & 1;
  C* s = bufs + size_t(half) * H::BUF;
  C v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = s[t + m * TT];
  half_sync<TT>(half);
  half_fft<H, 1>(v, t, s, half, a.tws);
  if (odd) half_omega<H, 1>(v, t, tw);
#pragma unroll
  for (int m = 0; m < E; ++m) s[t + ((m + E / 2) & (E - 1)) * TT] = v[m];  // at its pixel
  bool ok = true;
  if (nop > 0) ok = mbar_wait_bounded(&bar, 0, ep.err);
  __syncthreads();
  pass_trigger<T, LOGN>();
  EpAcc<T> part;
  if (ok) part = row_ep_all<LOGN>(ep, bufs, ops, a.deapod, r0);
  row_ep_finish(ep, part, red);
}

// Real-form column passes of Phi and Phi^H on the padded half grid (K + J rows,
// columns 0..n, a halo of J cells on both axes): grid cell (q, c) sits at row
// q + pad_lo, column c + pad_lo; rows near the edges also at their periodic
// image, and the halo's columns -c and 2n - c hold conj G(-q, c).  A CTA takes
// COLS columns, c = COLS u + 1 + k, so that COLS cells of a grid row start on
// a 32-byte sector; the last CTA's last column is the packed one, which holds
// columns 0 and n.
template <typename T, int LOGN>
struct GridHalf : Half<T, LOGN, LOGN <= 8 ? 8 : (LOGN <= 9 || sizeof(T) == 8 ? 16 : 32)> {
  typedef Half<T, LOGN, LOGN <= 8 ? 8 : (LOGN <= 9 || sizeof(T) == 8 ? 16 : 32)> Base;
  static constexpr int COLS = kColBytes / int(sizeof(typename cplx_t<T>::type));
  static constexpr int NT = COLS * 2 * Base::TT;
  static constexpr int MINB = NT >= 512 ? 1 : 512 / NT;
};

// Padded rows of grid row q (its periodic image too, near the edges).
PD int halo_rows(int q, int K, int pl, int (&at)[2]) {
  at[0] = q + pl;
  at[1] = q >= K - pl ? q + pl - K : q + pl + K;
  return q >= K - pl || q < kJ - pl ? 2 : 1;
}

// Phi: the column FFT of the image rows' half spectra X(., c) gives grid
// column c.  The packed column X(., 0) + i X(., n) transforms to P; column 0
// is (P(q) + conj P(-q)) / 2 and column n is -i (P(q) - conj P(-q)) / 2.
// Bound by its writes (a half grid of 17 MB at n = 1024) and latency: 15.2 us
// against 19.9 us for the whole grid by 2048-point transforms.
template <typename T, int LOGN, typename Src>
__global__ void __launch_bounds__(GridHalf<T, LOGN>::NT, GridHalf<T, LOGN>::MINB) k_col_fwd_h(Src src) {
  typedef typename cplx_t<T>::type C;
  typedef GridHalf<T, LOGN> H;
  constexpr int n = H::N, K = 2 * n, E = H::E, TT = H::TT, NC = H::COLS;
  decltype(auto) a = src.get();
  C* __restrict__ Pg = a.Pg;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C* bufs = reinterpret_cast<C*>(sm_raw);
  const int pl = a.g.pad_lo, KC = a.g.KC;
  const int half = threadIdx.x / TT, t = threadIdx.x - half * TT, odd = half & 1;
  const int c0 = NC * int(blockIdx.x) + 1;
  const bool packed = c0 + NC - 1 == n;  // this CTA's last column
  pdl_wait();
  C* s = bufs + size_t(half) * H::BUF;
  {
    const int c = c0 + (half >> 1);
    const C* __restrict__ Bc = a.B + (c == n ? size_t(0) : half_at(c, 0, n));
    C v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = Bc[t + ((m + E / 2) & (E - 1)) * TT];
    if (odd) half_omega<H, -1>(v, t, a.tw);
    half_fft<H, -1>(v, t, s, half, a.tws);
#pragma unroll
    for (int m = 0; m < E; ++m) s[t + m * TT] = v[m];
  }
  __syncthreads();
  pass_trigger<T, LOGN, 7>();
  for (int q = threadIdx.x; q < K; q += H::NT) {
    const int o = q & 1, m = q >> 1;
    C out[NC], col0 = cz<C>();
#pragma unroll
    for (int k = 0; k < NC; ++k) out[k] = bufs[size_t(2 * k + o) * H::BUF + m];
    if (packed) {
      const C P = out[NC - 1], Pm = bufs[size_t(2 * (NC - 1) + o) * H::BUF + (o ? n - 1 - m : (n - m) & (n - 1))];
      col0 = cmk<C>(T(0.5) * (P.x + Pm.x), T(0.5) * (P.y - Pm.y));
      out[NC - 1] = cmk<C>(T(0.5) * (P.y + Pm.y), T(0.5) * (Pm.x - P.x));
    }
    int at[2], am[2];
    const int nr = halo_rows(q, K, pl, at), nm = halo_rows((K - q) & (K - 1), K, pl, am);
    for (int r = 0; r < nr; ++r) {
      st32(Pg + size_t(at[r]) * KC + c0 + pl, out);
      if (packed) Pg[size_t(at[r]) * KC + pl] = col0;
    }
    if (c0 <= pl || c0 + NC > n - pl) {  // columns whose mirror image lies in the halo
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const int c = c0 + k;
        const C w = cmk<C>(out[k].x, -out[k].y);
        for (int r = 0; r < nm; ++r) {
          if (c <= pl) Pg[size_t(am[r]) * KC + pl - c] = w;
          if (c < n && c >= n - pl) Pg[size_t(am[r]) * KC + 2 * n - c + pl] = w;
        }
      }
    }
  }
}

// Phi^H: Re of the inverse transform of the gridded accumulator Q is the
// inverse transform of its Hermitian part Qh(q, c) = (Q(q, c) + conj Q(-q, -c)) / 2.
// Away from the halo's columns the second term is empty (every visibility was
// gridded in the lower half), so a column is read once, its row halo folded,
// then transformed (inverse, by halves), the n cropped rows into the
// half-spectrum rows B; the packed column is Qh(., 0) + i Qh(., n), whose
// transforms are real.  18.6 us against 34.4 us for the whole grid (n = 1024),
// where every element waited for two dependent, folded reads.
template <typename T, int LOGN, typename Src>
__global__ void __launch_bounds__(GridHalf<T, LOGN>::NT, GridHalf<T, LOGN>::MINB) k_col_inv_h(Src src) {
  typedef typename cplx_t<T>::type C;
  typedef GridHalf<T, LOGN> H;
  constexpr int n = H::N, K = 2 * n, E = H::E, TT = H::TT, NC = H::COLS;
  decltype(auto) a = src.get();
  const C* __restrict__ Q = a.Q;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C* bufs = reinterpret_cast<C*>(sm_raw);
  const int pl = a.g.pad_lo, KC = a.g.KC;
  const int half = threadIdx.x / TT, t = threadIdx.x - half * TT, odd = half & 1;
  const int c0 = NC * int(blockIdx.x) + 1;
  const bool packed = c0 + NC - 1 == n;
  auto fold = [&](int q, int c) -> C {  // one cell with its row images
    int at[2];
    const int nr = halo_rows(q & (K - 1), K, pl, at);
    C v = Q[size_t(at[0]) * KC + c + pl];
    if (nr > 1) v = cadd(v, Q[size_t(at[1]) * KC + c + pl]);
    return v;
  };
  constexpr int IT = K / H::NT, U = IT % 4 == 0 ? 4 : (IT % 2 == 0 ? 2 : 1);  // U sector loads in flight
  static_assert(K % H::NT == 0, "E is a multiple of COLS");
  pdl_wait();
  for (int it = 0; it < IT; it += U) {
    C in[U][NC];
#pragma unroll
    for (int u = 0; u < U; ++u)
      ld32(in[u], Q + size_t(int(threadIdx.x) + (it + u) * H::NT + pl) * KC + c0 + pl);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = int(threadIdx.x) + (it + u) * H::NT, o = q & 1, m = q >> 1;
      int at[2];
      if (halo_rows(q, K, pl, at) > 1) {
        C im[NC];
        ld32(im, Q + size_t(at[1]) * KC + c0 + pl);
#pragma unroll
        for (int k = 0; k < NC; ++k) in[u][k] = cadd(in[u][k], im[k]);
      }
      if (c0 <= pl || c0 + NC > n - pl) {
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          const int c = c0 + k;
          if (c <= pl || c >= n - pl) {  // the mirror image's column: -c, or 2n - c (c itself for c = n)
            const C w = fold(K - q, c <= pl ? -c : 2 * n - c);
            in[u][k] = cmk<C>(in[u][k].x + w.x, in[u][k].y - w.y);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < NC; ++k) in[u][k] = cscale(in[u][k], T(0.5));
      if (packed) {
        const C a0 = fold(q, 0), b0 = fold(K - q, 0);
        const C h0 = cmk<C>(T(0.5) * (a0.x + b0.x), T(0.5) * (a0.y - b0.y)), hn = in[u][NC - 1];
        in[u][NC - 1] = cmk<C>(h0.x - hn.y, h0.y + hn.x);  // h0 + i hn
      }
#pragma unroll
      for (int k = 0; k < NC; ++k) bufs[size_t(2 * k + o) * H::BUF + m] = in[u][k];
    }
  }
  __syncthreads();
  C* s = bufs + size_t(half) * H::BUF;
  C v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = s[t + m * TT];
  half_sync<TT>(half);
  half_fft<H, 1>(v, t, s, half, a.tws);
  if (odd) half_omega<H, 1>(v, t, a.tw);
  pass_trigger<T, LOGN, 7>();
  const int c = c0 + (half >> 1);
  half_join<H>(v, t, odd, bufs, half, a.B + (c == n ? size_t(0) : half_at(c, 0, n)));
}

// Plain in-place transforms of a K x K complex array (set-up of the PSF spectrum).
template <typename T, int LOGN>
__global__ void __launch_bounds__(kRowCta) k_rows_plain(typename cplx_t<T>::type* __restrict__ X,
                                                        const typename cplx_t<T>::type* __restrict__ tw, int nseq,
                                                        int dir) {
  typedef typename cplx_t<T>::type C;
  constexpr int TT = Plan<LOGN>::T, K = Plan<LOGN>::N;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int seq = threadIdx.x / TT, t = threadIdx.x - seq * TT;
  C* row = X + size_t(blockIdx.x * nseq + seq) * K;
  C* s = reinterpret_cast<C*>(sm_raw) + seq * padded(K);
  auto load = [&](int m) -> C { return row[t + m * TT]; };
  C out[16];
  int qs[16];
  int cnt = 0;
  auto store = [&](int q, C v) { out[cnt] = v; qs[cnt] = q; ++cnt; };
  fft_seq<LOGN>(t, s, 1, tw, dir, load, store);
  __syncthreads();
#pragma unroll
  for (int m = 0; m < 16; ++m) row[qs[m]] = out[m];
}

template <typename T, int LOGN>
__global__ void __launch_bounds__(ColThreads<T, LOGN>::value) k_cols_plain(typename cplx_t<T>::type* __restrict__ X,
                                                                         const typename cplx_t<T>::type* __restrict__ tw,
                                                                         int cw, int dir) {
  typedef typename cplx_t<T>::type C;
  constexpr int TT = Plan<LOGN>::T, K = Plan<LOGN>::N;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int cc = threadIdx.x % cw, t = threadIdx.x / cw;
  const int c = blockIdx.x * cw + cc;
  C* s = reinterpret_cast<C*>(sm_raw) + cc;  // cw interleaved columns
  auto load = [&](int m) -> C { return X[size_t(t + m * TT) * K + c]; };
  C out[16];
  int qs[16];
  int cnt = 0;
  auto store = [&](int q, C v) { out[cnt] = v; qs[cnt] = q; ++cnt; };
  fft_seq<LOGN>(t, s, cw, tw, dir, load, store);
  __syncthreads();
#pragma unroll
  for (int m = 0; m < 16; ++m) X[size_t(qs[m]) * K + c] = out[m];
}

}  // namespace


#define PURIFY_LOGN_SWITCH(K, BODY)     \
  switch (K) {                          \
    case 32: { constexpr int L = 5; BODY; } break;   \
    case 64: { constexpr int L = 6; BODY; } break;   \
    case 128: { constexpr int L = 7; BODY; } break;  \
    case 256: { constexpr int L = 8; BODY; } break;  \
    case 512: { constexpr int L = 9; BODY; } break;  \
    case 1024: { constexpr int L = 10; BODY; } break; \
    case 2048: { constexpr int L = 11; BODY; } break; \
    default: { constexpr int L = 12; BODY; } break;  \
  }

// Grid sides of the batched passes (image sides 64..1024).
#define PURIFY_LOGN_SWITCH_BATCH(K, BODY)                 \
  switch (K) {                                            \
    case 128: { constexpr int L = 7; BODY; } break;       \
    case 256: { constexpr int L = 8; BODY; } break;       \
    case 512: { constexpr int L = 9; BODY; } break;       \
    case 1024: { constexpr int L = 10; BODY; } break;     \
    case 2048: { constexpr int L = 11; BODY; } break;     \
    default: break;                                       \
  }

// L = log2 K; the passes of half transforms are templated on log2 n = L - 1
template <typename T, int L> cudaError_t configure_one() {
  cudaError_t e = raise_smem_limit(k_row_fwd_h<T, L - 1, ArgVal<RowFwdArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_col_conv_h<T, L - 1, ArgVal<ColConvArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_col_fwd_h<T, L - 1, ArgVal<ColFwdArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_col_inv_h<T, L - 1, ArgVal<ColInvArgs<T>>>);
  if (e == cudaSuccess) e = raise_smem_limit(k_row_inv_h<T, L - 1, ArgVal<RowInvArgs<T>>>);
  if constexpr (L >= 7 && L <= 11) {
    if (e == cudaSuccess) e = raise_smem_limit(k_row_fwd_h<T, L - 1, ArgTab<RowFwdArgs<T>>>);
    if (e == cudaSuccess) e = raise_smem_limit(k_col_conv_h<T, L - 1, ArgTab<ColConvArgs<T>>>);
    if (e == cudaSuccess) e = raise_smem_limit(k_col_fwd_h<T, L - 1, ArgTab<ColFwdArgs<T>>>);
    if (e == cudaSuccess) e = raise_smem_limit(k_col_inv_h<T, L - 1, ArgTab<ColInvArgs<T>>>);
    if (e == cudaSuccess) e = raise_smem_limit(k_row_inv_h<T, L - 1, ArgTab<RowInvArgs<T>>>);
  }
  if (e == cudaSuccess) e = raise_smem_limit(k_rows_plain<T, L>);
  if (e == cudaSuccess) e = raise_smem_limit(k_cols_plain<T, L>);
  return e;
}

template <typename T> cudaError_t configure_fft() {
  cudaError_t e = cudaSuccess;
  for (int K = 32; K <= 4096 && e == cudaSuccess; K *= 2) {
    PURIFY_LOGN_SWITCH(K, e = (configure_one<T, L>()));
  }
  return e;
}
template cudaError_t configure_fft<float>();
template cudaError_t configure_fft<double>();

cudaError_t set_wait_spins_fft(uint32_t spins) { return set_module_wait_spins(spins); }

template <typename T>
__global__ void k_embed_psf(const T* __restrict__ psf, int n, typename cplx_t<T>::type* __restrict__ X) {
  typedef typename cplx_t<T>::type C;
  const int K = 2 * n;
  const size_t idx = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= size_t(K) * K) return;
  const int q1 = int(idx / K), q2 = int(idx % K);
  // kernel offset d = q - K for q >= n; the PSF image holds offsets [-n, n)
  const int i1 = (q1 + n) & (K - 1), i2 = (q2 + n) & (K - 1);
  X[idx] = cmk<C>(psf[size_t(i1) * K + i2], T(0));
}

// Real part of the spectrum in launch_col_conv_h's layout: per column (storage
// order of half_at) its even grid rows, then its odd ones; column K/2 after them.
template <typename T>
__global__ void k_spectrum_layout(const typename cplx_t<T>::type* __restrict__ X, int K, double scale,
                                  T* __restrict__ khat) {
  const size_t idx = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= size_t(K) * K) return;
  const int q = int(idx / K), c = int(idx % K), n = K / 2;
  if (c > n) return;
  const size_t col = c == n ? size_t(n) : size_t(c & 1) * (n / 2) + (c >> 1);
  khat[(col * 2 + (q & 1)) * n + (q >> 1)] = T(double(X[idx].x) * scale);
}

template <typename T>
void build_psf_spectrum(const T* psf, int n, T* khat, typename cplx_t<T>::type* X, const typename cplx_t<T>::type* tw,
                        cudaStream_t s) {
  const int K = 2 * n;
  const size_t tot = size_t(K) * K;
  const int tb = 256;
  k_embed_psf<T><<<int((tot + tb - 1) / tb), tb, 0, s>>>(psf, n, X);
  launch_fft2_plain<T>(K, X, tw, -1, s);
  k_spectrum_layout<T><<<int((tot + tb - 1) / tb), tb, 0, s>>>(X, K, 1.0 / (double(K) * K), khat);
}

// Launch shapes of the passes of half transforms.
template <typename T, int LOGN> struct HalfShape {
  typedef RowHalf<T, LOGN> H;
  typedef ColHalf<T, LOGN> HC;
  typedef typename cplx_t<T>::type C;
  static constexpr int row_ctas = H::N / 2 / H::PAIRS;
  static constexpr int col_ctas = HC::N / HC::COLS;
  static size_t fwd_smem() { return size_t(H::PAIRS) * (H::N + 2 * H::BUF) * sizeof(C); }
  static size_t inv_smem(bool operands) {
    return align16(size_t(H::PAIRS) * 2 * H::BUF * sizeof(C)) + (operands ? size_t(H::PAIRS) * 4 * H::N * sizeof(T) : 0);
  }
  typedef GridHalf<T, LOGN> HG;
  static constexpr int grid_ctas = H::N / HG::COLS;
  static size_t grid_smem() { return size_t(HG::COLS) * 2 * HG::BUF * sizeof(C); }
  static size_t conv_smem() { return size_t(HC::COLS) * 2 * HC::BUF * sizeof(C); }
};
// Twiddles of the half transforms of length n: per stage after the first,
// W(r k) = exp(-2 pi i r k / (Ns R)) as [r - 1][k], k < Ns; the row passes'
// table, then the column passes' from element *col_at on.
template <typename H, typename C> static void half_twiddles_of(std::vector<C>& out) {
  int ns = H::radix(0);
  for (int st = 1; st < H::NST; ++st) {
    const int R = H::radix(st);
    for (int r = 1; r < R; ++r)
      for (int k = 0; k < ns; ++k) {
        const double a = -2.0 * M_PI * double(r) * k / (double(ns) * R);
        C w;
        w.x = decltype(w.x)(std::cos(a));
        w.y = decltype(w.y)(std::sin(a));
        out.push_back(w);
      }
    ns *= R;
  }
}
template <typename T> void half_twiddles(int n, std::vector<typename cplx_t<T>::type>& out, size_t* col_at) {
  out.clear();
  PURIFY_LOGN_SWITCH(2 * n, (half_twiddles_of<RowHalf<T, L - 1>>(out)));
  *col_at = out.size();
  PURIFY_LOGN_SWITCH(2 * n, (half_twiddles_of<ColHalf<T, L - 1>>(out)));
}
template void half_twiddles<float>(int, std::vector<float2>&, size_t*);
template void half_twiddles<double>(int, std::vector<double2>&, size_t*);
template <typename T> void launch_row_fwd_h(const RowFwdArgs<T>& a, cudaStream_t s) {
  ArgVal<RowFwdArgs<T>> src{a};
  PURIFY_LOGN_SWITCH(a.g.K, (launch_pdl(k_row_fwd_h<T, L - 1, ArgVal<RowFwdArgs<T>>>, HalfShape<T, L - 1>::row_ctas,
                                           RowHalf<T, L - 1>::ROW_THREADS, HalfShape<T, L - 1>::fwd_smem(), s, src)));
}

template <typename T> void launch_col_conv_h(const ColConvArgs<T>& a, cudaStream_t s) {
  ArgVal<ColConvArgs<T>> src{a};
  PURIFY_LOGN_SWITCH(a.g.K, (launch_pdl(k_col_conv_h<T, L - 1, ArgVal<ColConvArgs<T>>>, HalfShape<T, L - 1>::col_ctas,
                                           ColHalf<T, L - 1>::COL_THREADS, HalfShape<T, L - 1>::conv_smem(), s, src)));
}

template <typename T> void launch_col_fwd_h(const ColFwdArgs<T>& a, cudaStream_t s) {
  ArgVal<ColFwdArgs<T>> src{a};
  PURIFY_LOGN_SWITCH(a.g.K, (launch_pdl(k_col_fwd_h<T, L - 1, ArgVal<ColFwdArgs<T>>>, HalfShape<T, L - 1>::grid_ctas,
                                           GridHalf<T, L - 1>::NT, HalfShape<T, L - 1>::grid_smem(), s, src)));
}

template <typename T> void launch_col_inv_h(const ColInvArgs<T>& a, cudaStream_t s) {
  ArgVal<ColInvArgs<T>> src{a};
  PURIFY_LOGN_SWITCH(a.g.K, (launch_pdl(k_col_inv_h<T, L - 1, ArgVal<ColInvArgs<T>>>, HalfShape<T, L - 1>::grid_ctas,
                                           GridHalf<T, L - 1>::NT, HalfShape<T, L - 1>::grid_smem(), s, src)));
}

template <typename T> void launch_row_inv_h(const RowInvArgs<T>& a, cudaStream_t s) {
  ArgVal<RowInvArgs<T>> src{a};
  const bool operands = a.ep.mode != EP_STORE && a.ep.mode != EP_POWER;
  PURIFY_LOGN_SWITCH(a.g.K, (launch_pdl(k_row_inv_h<T, L - 1, ArgVal<RowInvArgs<T>>>, HalfShape<T, L - 1>::row_ctas,
                                           RowHalf<T, L - 1>::ROW_THREADS, HalfShape<T, L - 1>::inv_smem(operands), s,
                                           src)));
}

// Batched passes: `count` instances of one grid side (g gives the shared
// shape), arguments in a device table, instance = blockIdx.y.
template <typename T>
void launch_row_fwd_h_batch(const Geometry& g, const RowFwdArgs<T>* tab, int count, cudaStream_t s) {
  ArgTab<RowFwdArgs<T>> src{tab};
  PURIFY_LOGN_SWITCH_BATCH(g.K, (k_row_fwd_h<T, L - 1><<<dim3(HalfShape<T, L - 1>::row_ctas, count),
                                                         RowHalf<T, L - 1>::ROW_THREADS, HalfShape<T, L - 1>::fwd_smem(),
                                                         s>>>(src)));
}
template <typename T>
void launch_col_conv_h_batch(const Geometry& g, const ColConvArgs<T>* tab, int count, cudaStream_t s) {
  ArgTab<ColConvArgs<T>> src{tab};
  PURIFY_LOGN_SWITCH_BATCH(g.K, (k_col_conv_h<T, L - 1><<<dim3(HalfShape<T, L - 1>::col_ctas, count),
                                                          ColHalf<T, L - 1>::COL_THREADS,
                                                          HalfShape<T, L - 1>::conv_smem(), s>>>(src)));
}
template <typename T>
void launch_col_fwd_h_batch(const Geometry& g, const ColFwdArgs<T>* tab, int count, cudaStream_t s) {
  ArgTab<ColFwdArgs<T>> src{tab};
  PURIFY_LOGN_SWITCH_BATCH(g.K, (k_col_fwd_h<T, L - 1><<<dim3(HalfShape<T, L - 1>::grid_ctas, count),
                                                         GridHalf<T, L - 1>::NT, HalfShape<T, L - 1>::grid_smem(),
                                                         s>>>(src)));
}
template <typename T>
void launch_col_inv_h_batch(const Geometry& g, const ColInvArgs<T>* tab, int count, cudaStream_t s) {
  ArgTab<ColInvArgs<T>> src{tab};
  PURIFY_LOGN_SWITCH_BATCH(g.K, (k_col_inv_h<T, L - 1><<<dim3(HalfShape<T, L - 1>::grid_ctas, count),
                                                         GridHalf<T, L - 1>::NT, HalfShape<T, L - 1>::grid_smem(),
                                                         s>>>(src)));
}
template <typename T>
void launch_row_inv_h_batch(const Geometry& g, const RowInvArgs<T>* tab, int count, cudaStream_t s) {
  ArgTab<RowInvArgs<T>> src{tab};
  PURIFY_LOGN_SWITCH_BATCH(g.K, (k_row_inv_h<T, L - 1><<<dim3(HalfShape<T, L - 1>::row_ctas, count),
                                                         RowHalf<T, L - 1>::ROW_THREADS,
                                                         HalfShape<T, L - 1>::inv_smem(true), s>>>(src)));
}

template <typename T>
void launch_fft2_plain(int K, typename cplx_t<T>::type* X, const typename cplx_t<T>::type* tw, int dir,
                       cudaStream_t s) {
  typedef typename cplx_t<T>::type C;
  const int cw = col_width<T>();
  int nseq = kRowCta / (K / 16);
  if (nseq < 1) nseq = 1;
  if (nseq > K) nseq = K;
  const size_t smr = nseq * padded(K) * sizeof(C);
  const size_t smc = cw * padded(K) * sizeof(C);
  PURIFY_LOGN_SWITCH(K, (k_rows_plain<T, L><<<K / nseq, nseq * Plan<L>::T, smr, s>>>(X, tw, nseq, dir)));
  PURIFY_LOGN_SWITCH(K, (k_cols_plain<T, L><<<K / cw, cw * Plan<L>::T, smc, s>>>(X, tw, cw, dir)));
}

#define INST(T)                                                                                              \
  template void launch_row_fwd_h<T>(const RowFwdArgs<T>&, cudaStream_t);                                     \
  template void launch_col_conv_h<T>(const ColConvArgs<T>&, cudaStream_t);                                   \
  template void launch_row_inv_h<T>(const RowInvArgs<T>&, cudaStream_t);                                     \
  template void launch_fft2_plain<T>(int, cplx_t<T>::type*, const cplx_t<T>::type*, int, cudaStream_t);     \
  template void launch_col_fwd_h<T>(const ColFwdArgs<T>&, cudaStream_t);                                     \
  template void launch_col_inv_h<T>(const ColInvArgs<T>&, cudaStream_t);                                     \
  template void build_psf_spectrum<T>(const T*, int, T*, cplx_t<T>::type*, const cplx_t<T>::type*, cudaStream_t); \
  template void launch_row_fwd_h_batch<T>(const Geometry&, const RowFwdArgs<T>*, int, cudaStream_t);         \
  template void launch_col_conv_h_batch<T>(const Geometry&, const ColConvArgs<T>*, int, cudaStream_t);       \
  template void launch_col_fwd_h_batch<T>(const Geometry&, const ColFwdArgs<T>*, int, cudaStream_t);         \
  template void launch_col_inv_h_batch<T>(const Geometry&, const ColInvArgs<T>*, int, cudaStream_t);         \
  template void launch_row_inv_h_batch<T>(const Geometry&, const RowInvArgs<T>*, int, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace purify
