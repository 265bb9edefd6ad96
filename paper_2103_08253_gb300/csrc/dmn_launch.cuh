// Launch parameters shared by the translation units of the DMN library (csrc/dmn.cu, the C ABI and
// the thread-per-point kernels; csrc/dmn_warp.cu, the warp organisation): the trees of a handle,
// the Newton kernels' parameters, and the warp organisation's scratch and launch.
#pragma once
#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>

#include "../../include/dmn.h"
#include "dmn_device.cuh"

namespace dmn {

// All trees of a handle, passed by value to the kernels.
struct Forest {
  TreeDev t[DMN_MAX_TREES];
  int n;
};

// point handled by thread/work item i and its tree (n_trees = invalid)
__device__ __forceinline__ void point_of(const int64_t* perm, const int32_t* tid, int n_trees, int64_t i,
                                         int64_t& p, int& tree) {
  p = perm ? perm[i] : i;
  const int t = tid ? tid[p] : 0;
  tree = (t >= 0 && t < n_trees) ? t : n_trees;
}

template <typename T>
struct NewtonParams {
  Forest F;
  int64_t n, nslots;
  int N_max;
  const int32_t* tid;
  const int64_t* perm;
  const double* state_in;
  double *state_out, *stress, *tangent;
  int32_t *iters, *status;
  const double* nbuf;
  double* scr_d;
  T* scr_t;
  unsigned long long* counter;
  double tol;
  int max_iter;
  int write_outputs;  // no final sweep: stress and tangent (local frame) come from the converged Newton pass
  int predictor;      // extrapolated start; the state carries the last jump change and strain increment
  const double* dE;   // [n][6] strain increments (global frame), read with the extrapolated start
  const double* a_start;  // the jumps to start from (state layout), or NULL for those of state_in; with the
                          // first stage these are its jumps in state_out, and iters holds its corrections
  unsigned long long* passes;  // profiling: tree passes of all points added here, or NULL
  int min_corr;       // corrections before the criterion may end the iteration (1 for the FP64 form after
                      // the first stage: one quadratic step from the FP32 iterate, so that the accepted
                      // iterate is as far inside the criterion as in the plain FP64 iteration)
  const unsigned long long* n_list = nullptr;  // the points are perm[0 .. *n_list) instead of all n
};

// Status of a point that k_newton_block leaves to the all-FP64 kernels; never returned to a caller.
constexpr int32_t STATUS_RETRY = -1;

// number of points a launch works through (lists hold points of the FP64 form only)
template <typename T>
__device__ __forceinline__ unsigned long long n_work(const NewtonParams<T>& P) {
  return sizeof(T) == 8 && P.n_list ? *P.n_list : (unsigned long long)P.n;
}

// Small calls: one point per group of G lanes of a warp (G = 32, 16 or 8; the paper's start; heap
// trees or compressed ones), the group's lanes sharing each level of the tree (warp_tree_pass).
// The Newton loop is k_newton's.  The warp's groups run their passes side by side: every iteration
// of the warp's loop is one pass of every group that holds a point, so the groups' lanes stay
// together (the pass's instructions are the same for every point); a group whose point is done
// writes it out and takes the next one from the work counter.  Each group owns a block of scratch
// (warp_slot_doubles<T>(N) doubles) holding its point's jumps, g, H, level hand-over and subtree
// results, in two buffers where the line search needs them.
template <typename T>
__host__ __device__ inline size_t warp_slot_doubles(int N) {
  // jumps 2 x 3N, ein 6N, sb 6N, normals 3N, leaf-child strains 6N (FP64); g, H 2 x 21N, dein 6N,
  // ds + C 27N (T); FP32 normals 3N
  const size_t d = (size_t)27 * N, tt = (size_t)75 * N * sizeof(T), f = (size_t)3 * N * sizeof(float);
  return d + (tt + f + sizeof(double) - 1) / sizeof(double);
}
constexpr int WARP_CTAS_PER_SM = 2;   // 128-thread CTAs: 8 warps per SM
constexpr int WARP_MIN_LANES = 8;     // the smallest group: the scratch holds 32 / 8 = 4 slots per warp

// k_newton_warp<T, LS, lanes, CMP> on `grid` CTAs of 128 threads (csrc/dmn_warp.cu); `scr` holds
// grid * 128 / lanes slots of warp_slot_doubles<T>(P.N_max) doubles
template <typename T, bool CMP>
void launch_warp(const NewtonParams<T>& P, bool ls, int lanes, unsigned grid, double* scr, cudaStream_t s);
// the points on P.n_list in this organisation, 32 lanes each if there are at most `few`, else 8
template <bool CMP>
void launch_list(const NewtonParams<double>& P, bool ls, int64_t few, unsigned grid, double* scr, cudaStream_t s);
// The CTA organisation of the FP64 form (csrc/dmn_block.cu).  counter: [1..9] points per tree and
// [10..18] their ends in perm (several trees), [21..28] work counters per tree, [29] points on the list.
constexpr int BLOCK_THREADS = 256;
constexpr int BLOCK_CTAS_PER_SM = 2;
constexpr int BLOCK_TOKENS = 256;   // counters [32 ..]: an SM's FP64 phase is taken
struct BlockParams {
  Forest F;
  int64_t n;
  int N_max, n_sm, leaf_slots;   // leaf_slots: leaves with a state in a subtree of 8 (4, or 8 with two inelastic phases)
  const int32_t* tid;
  const int64_t* perm;
  const double* state_in;
  double *state_out, *stress, *tangent;
  int32_t *iters, *status;
  const double* nbuf;
  char* scratch;           // block_scratch_bytes per CTA
  unsigned long long* counter;
  int64_t* list;           // points left to the all-FP64 kernels
  double tol;
  int max_iter;
  unsigned long long* passes;
};
// per thread, for 8 laminates: jumps (two buffers with the line search) and normals (FP64), H, Kn^-1, g, step
// and residual (FP32: 36 fields); per leaf its state (FP64: 6) and tangent (FP32: 16)
__host__ __device__ inline size_t block_scratch_bytes(int threads, int leaf_slots, bool line_search) {
  return (size_t)threads * (sizeof(double) * (8 * (line_search ? 9 : 6) + 6 * leaf_slots) +
                                  sizeof(float) * (8 * 36 + 16 * leaf_slots));
}
__device__ __forceinline__ void block_bad_tree(const BlockParams& P, int64_t pt) {
  const double qnan = __longlong_as_double(0x7ff8000000000000LL);
  P.iters[pt] = 0;
  P.status[pt] = DMN_STATUS_BAD_TREE;
  for (int I = 0; I < 6; ++I) P.stress[6 * pt + I] = qnan;
  for (int I = 0; I < 36; ++I) P.tangent[36 * pt + I] = qnan;
}
__device__ __forceinline__ void block_retry(const BlockParams& P, int64_t pt) {
  P.status[pt] = STATUS_RETRY;
  P.list[atomicAdd(P.counter + 29, 1ull)] = pt;
}
// The FP64 sweep in the same organisation (k_sweep_block): stress, tangent and, on request, leaf states at the
// jumps in state_out, of every point whose status is not RETRY.  counter: as above, [1..9] and [10..18].
constexpr int SWEEP_THREADS = 128;
constexpr int SWEEP_CTAS_PER_SM = 2;
struct SweepParams {
  Forest F;
  int64_t n;
  int N_max;
  const int32_t* tid;
  const int64_t* perm;
  const double *Q, *state_in;
  double *state_out, *stress, *tangent;
  const int32_t* status;
  const double* nbuf;
  const unsigned long long* counter;
};
cudaError_t launch_sweep_block(const SweepParams& P, bool cmp, bool states, unsigned grid, cudaStream_t s);
// K: the depth of the handle's deepest tree; scratch for BLOCK_CTAS_PER_SM CTAs of BLOCK_THREADS per SM
cudaError_t launch_block(const BlockParams& P, int K, bool ls, bool cmp, cudaStream_t s);

// The adjoints in the CTA organisation (csrc/dmn_grad.cu): one chunk of nc points from n0 on.  work, field-major
// over the chunk: normals [3 N], sin(alpha), cos(beta), sin(beta) [3 N], dL/d alpha [N], dL/d beta [N], dL/dw [L],
// shape-function values [6].
constexpr int GRAD_SCRATCH_DOUBLES = 320;   // per thread of a CTA
struct GradWork {
  TreeDev t;
  int64_t n, n0, nc;
  const double *lam, *Q, *En, *dE, *state_in, *state_out, *g_stress, *g_tangent;
  double* g_E;
  double* work;
  double* scratch;
  __host__ __device__ int gab() const { return 6 * t.N; }
  __host__ __device__ int gw() const { return 8 * t.N; }
  __host__ __device__ int ph() const { return 8 * t.N + t.L; }
  __host__ __device__ int fields() const { return 8 * t.N + t.L + 6; }
};
cudaError_t launch_grad_normals(const GradWork& G, unsigned split, cudaStream_t s);
cudaError_t launch_grad_block(const GradWork& G, bool cmp, bool tangent, unsigned grid, cudaStream_t s);

}  // namespace dmn
