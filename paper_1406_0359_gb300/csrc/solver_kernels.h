// Vector kernels and device scalars of the SDMM solver.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "common.cuh"

namespace purify {

// Device scalar slots (double[kNumScalars]).
enum ScalarSlot : int {
  S_BALLSCALE = 0, S_RESID, S_OBJ, S_MEAN, S_STD, S_MAXABS, S_FEAS,
  // sums of the row passes' epilogues, accumulated across CTAs; two sets taken
  // in turn, each zeroed by the forward pass of the step that fills it
  S_CG0,                // a CG step's five inner products
  S_POW0 = S_CG0 + 10,  // a power iteration's squared norm
  kNumScalars = S_POW0 + 2
};
enum FinOp : int { FIN_OBJ = 0, FIN_MEAN, FIN_VAR };
enum RedOp : int { RED_SQ = 0, RED_SUM, RED_VAR, RED_MAXABS };

int vec_blocks(size_t N);
// The step length of a CG step from its sums <r,p> and <p,Ap> (0 when the latter is).
__host__ __device__ inline double cg_alpha(double rp, double pap) { return pap > 0.0 ? rp / pap : 0.0; }
// The last CG step's x += alpha p, alpha from its sums; N a multiple of 4, both
// arrays 16-byte aligned.
template <typename T> void launch_axpy(T* x, const T* p, const double* acc, size_t N, cudaStream_t s);
// Merge na partials (Acc<T> values in double-sized slots) and apply `op`.
template <typename T> void launch_finalize(const double* pa, int na, int op, double arg, double* sc, cudaStream_t s);
template <typename T>
int launch_reduce(const T* v, size_t N, int op, const double* sc, double* partials, cudaStream_t s);
void launch_max_partials(const double* p, int np, double* sc, cudaStream_t s);
// Ball scalars per visibility block from the work items' partials; items_as_int
// points at the WorkItem array (four ints per item, the block in the fourth).
template <typename T>
void launch_finalize_blocks(const double* part0, const double* part1, const int* items_as_int, int n_items, int R,
                            double nu, const double* eps_b, double* scale_b, double* sc, cudaStream_t s);
// The same scalars for one block (R = 1) from kBallAcc accumulator pairs, which
// are left at zero.
struct Ball1Args {
  double* acc;
  double nu;
  const double* eps_b;
  double* scale_b;
  double* sc;
};
void launch_finalize_ball1(const Ball1Args& a, cudaStream_t s);
template <typename T> void launch_reweight(T* w, size_t N, double delta, cudaStream_t s);
template <typename T> void launch_fill(T* v, size_t N, T val, cudaStream_t s);
template <typename T> void launch_scale(T* v, size_t N, const double* sc, int idx, double mul, cudaStream_t s);
// Into and out of the operator's sorted order (perm_index, perm_value).
template <typename C> void launch_scatter(const C* src, const int* perm, size_t M, C* dst, cudaStream_t s);
template <typename C> void launch_gather(const C* src, const int* perm, size_t M, C* dst, cudaStream_t s);
// Batched vector steps of instances of one size (argument tables in device
// memory; instance = blockIdx.y, one grid for all).
template <typename T> struct AxpyArgs { T* x; const T* p; const double* acc; size_t N; };
template <typename T> void launch_axpy_batch(const AxpyArgs<T>* tab, int count, size_t N, cudaStream_t s);
struct FinArgs { const double* pa; int na; int op; double arg; double* sc; };
template <typename T> void launch_finalize_batch(const FinArgs* tab, int count, cudaStream_t s);
void launch_finalize_ball1_batch(const Ball1Args* tab, int count, cudaStream_t s);
struct ZeroArgs { void* p; size_t bytes; };  // bytes a multiple of 16
void launch_zero_batch(const ZeroArgs* tab, int count, size_t max_bytes, cudaStream_t s);

// Device flag set when any of the n values is not finite (NaN or infinity).
template <typename T> void launch_check_finite(const T* v, size_t n, int* flag, cudaStream_t s);

}  // namespace purify
