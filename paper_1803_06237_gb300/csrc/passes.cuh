// Shared by the operator's pass kernels (matvec.cu, any_x.cuh, any_b.cuh): the
// per-problem pointers of a launch, the plane geometry, and the launchers of
// the passes for sizes without a compiled kernel of their own.
#pragma once

#include <cuda_pipeline.h>

#include "vie_internal.cuh"

namespace vie {

template <typename V> __device__ __forceinline__ V zero_c();
template <> __device__ __forceinline__ float2 zero_c<float2>() { return make_float2(0.f, 0.f); }
template <> __device__ __forceinline__ double2 zero_c<double2>() { return make_double2(0.0, 0.0); }

// Per-problem pointers of one launch: blockIdx.y selects the problem.  All
// problems of a launch share the grid and circulant sizes (and twiddles).
constexpr int kMaxBatch = 16;
template <typename V>
struct PassPtrs {
  const V* x[kMaxBatch];
  V* y[kMaxBatch];
  V* work[kMaxBatch];
  const V* ghat[kMaxBatch];
  const V* M[kMaxBatch];
  V* work2[kMaxBatch];        // y-pass buffer of the split pass B (or null)
  const int* live[kMaxBatch]; // per problem: null, or a device flag; 0 skips the problem (its blocks return)
};

// The wait for the kernel before, then whether the problem is skipped: one
// whose live flag is 0 is, by every block of every pass (blockIdx.y is the
// problem in all grouped launches).  Every pass waits, skipped or not, and
// reads the flag behind its wait.  A grid whose blocks leave without waiting
// can complete before the one it was launched behind does; a kernel after it
// that waits for it alone would then read vectors still being written (several
// shapes in one call, the last of them skipped).  The copies of plan data that
// a pass starts ahead of the wait have landed before its blocks leave.
template <typename V>
__device__ __forceinline__ bool skip_after_wait(const PassPtrs<V>& pp) {
  const int* f = pp.live[blockIdx.y];   // a kernel parameter
  pdl_wait();
  if (f == nullptr || *(const volatile int*)f != 0) return false;
  __pipeline_commit();
  __pipeline_wait_prior(0);
  return true;
}

struct PassBGeom {
  int ny, nz, NL, Mx, My, Mz, Ky, Kz;
};

// Whether pass B may start while the x pass before it still runs.  Blocks that
// start early crowd onto the SMs the x pass leaves idle; complex128 planes are
// bound by the SM's FP64 rate, so where most of the grid is resident at once
// that costs more than the overlap gives: up to two planes an SM (73 x 11 x 9,
// 150 planes: 151 us an application against 83), and up to four small ones
// (191 x 23 x 7, 384 planes of 45 x 15: 254 against 209; 180 x 27 x 9, 360 of
// 54 x 18: 260 against 263).
template <typename V> inline bool b_starts_early(const PassBGeom& g, int count) {
  const long planes = (long)g.Mx * count;
  return sizeof(V) == sizeof(float2) || !(planes <= 2 * kSMs || (planes <= 4 * kSMs && g.My * g.Mz < 800));
}

// x pass (or the split pass B's y passes) for lines of n values and length
// len, with register butterflies of run-time radices.  nyz: voxels of the
// cross-section (the contrast row of a line is line % nyz); gsz: lines of a
// group of the transposed side.  *done = false where len has no split into
// three of the radices or the lines do not fit shared memory.
template <typename V>
vie_status launch_x_any(bool forward, const PassPtrs<V>& pp, int count, int n, int nyz, int NL, int len, const V* tw,
                        int mode, cudaStream_t s, int gsz, bool* done);

// Pass B on one CTA per kx with run-time radices: nc = 3 (J-VIE) or 6
// (JM-VIE: pp.work[0], pp.ghat[0], chat and kappa, one problem).  *done =
// false where a length has no compiled split or the plane does not fit.
template <typename V>
vie_status launch_b_any(const PassPtrs<V>& pp, int count, const PassBGeom& g, int nc, const V* chat, double kappa,
                        const V* twy, cudaStream_t s, bool* done);

}  // namespace vie
