// Operator passes for sizes without a compiled kernel of their own: any
// 5-smooth circulant sizes, so grids of every length and cross-section that
// fit a CTA take register butterflies.
//
// A transform of length L = r1 r2 r3 runs as three in-place stages of r-point
// register DFTs (radices up to 25, chosen on the host, selected by a
// block-uniform switch); every butterfly reads and writes the same places, so
// a line needs one shared buffer and one barrier per stage, against two
// buffers, a radix of at most 5 and five or six round trips in the Stockham
// kernels these replace.  The first stage of a pass takes its operands from
// global memory and the last one stores its results there, so a line makes
// two round trips through shared memory.
#pragma once

#include <cuda_pipeline.h>
#include <string.h>

#include "fft.cuh"
#include "passes.cuh"
#include "regfft.cuh"
#include "vie_internal.cuh"

namespace vie {

template <int N> using IC = std::integral_constant<int, N>;

// f(IC<r>{}) for the radix r <= TOP of a stage.  TOP bounds a kernel's
// registers: the largest radix sets them for every length it serves.
#define VIE_RADICES(X) X(1) X(2) X(3) X(4) X(5) X(6) X(8) X(9) X(10) X(12) X(15) X(16) X(20) X(25)
template <int TOP, typename F>
__device__ __forceinline__ void with_radix(int r, F&& f) {
  switch (r) {
#define VIE_X(a) case a: if constexpr (a <= TOP) f(IC<a>{}); break;
    VIE_RADICES(VIE_X)
#undef VIE_X
    default: break;
  }
}
static const int kRadices[] = {
#define VIE_X(a) a,
    VIE_RADICES(VIE_X)
#undef VIE_X
};

// a / d for a, d < 2^16 from m = ceil(2^32 / d) (d = 1: m = 0)
__device__ __forceinline__ int div_by(int a, unsigned m) { return m ? (int)__umulhi((unsigned)a, m) : a; }
static unsigned div_magic(int d) { return d == 1 ? 0u : (unsigned)((0x100000000ull + d - 1) / d); }

// ---------------------------------------------------------------------------
// x passes.  Indices: n = n' + M2 n1, n' = n'' + r3 n2, M2 = r2 r3; frequency
// k = k1 + r1 (k2 + r2 k3).
//   1: over n1 (stride M2), twiddle w_L^(n' k1);
//   2: over n2 (stride r3), twiddle w_M2^(n'' k2);
//   3: over n''.
// The inverse runs 3, 2, 1 with conjugate twiddles.  Shared place of (k1 or
// n1, n2, n''): lpb (n'' + p3 (n2 + r2 k1)) + line, p3 = r3 | 1: lanes run
// fastest over the block's lpb lines, then over n'' (stages 1, 2) or over
// rows of the odd pitch p3 (stage 3), so no stage has bank conflicts beyond
// two.
// ---------------------------------------------------------------------------
struct XAny {
  int L, r1, r2, r3, M2, p3;
  int lpb, row, blk;              // lines per block; lpb p3, lpb p3 r2
  unsigned mr2, mr3, ml;          // division by r2, r3, lpb
};

// most threads of a block: 64 registers a thread in the small complex64 class,
// 128 otherwise
template <typename V, int TOP> __host__ __device__ constexpr int x_any_threads() { return TOP <= 16 && sizeof(V) == sizeof(float2) ? 1024 : 512; }

template <typename V, int TOP>
__global__ void __launch_bounds__(x_any_threads<V, TOP>(), 1) pass_a_any_kernel(const __grid_constant__ PassPtrs<V> pp, XAny g, int nx,
                                                         int NL, const V* __restrict__ tw, int gsz) {
  pdl_launch_dependents();
  if (skip_after_wait(pp)) return;
  extern __shared__ unsigned char smem_raw[];
  V* S = reinterpret_cast<V*>(smem_raw);
  const int lpb = g.lpb, t0 = div_by(threadIdx.x, g.ml), l = threadIdx.x - t0 * lpb, step = div_by(blockDim.x, g.ml);
  const int line = blockIdx.x * lpb + l;
  const int first = t0 < step ? t0 : g.L;   // threads beyond a whole row of lines take no item
  const bool on = line < NL;
  {
    const V* __restrict__ src = pp.x[blockIdx.y] + (size_t)(on ? line : 0) * nx;
    with_radix<TOP>(g.r1, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int np = first; np < g.M2; np += step) {
        V a[R];
#pragma unroll
        for (int n1 = 0; n1 < R; ++n1) {
          const int n = np + g.M2 * n1;
          // nx <= (L + 1) / 2: the upper half of the inputs is padding
          a[n1] = (n1 < (R + 1) / 2 && on && n < nx) ? src[n] : zero_c<V>();
        }
        reg_fft<V, false, R, (R + 1) / 2>(a, nullptr);
        V* d = S + (np + (g.p3 - g.r3) * div_by(np, g.mr3)) * lpb + l;
        d[0] = a[0];
#pragma unroll
        for (int k1 = 1; k1 < R; ++k1) d[g.blk * k1] = mul(a[k1], tw[np * k1]);
      }
    });
  }
  __syncthreads();
  if (g.r2 > 1) {
    with_radix<TOP>(g.r2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int it = first; it < g.r1 * g.r3; it += step) {
        const int k1 = div_by(it, g.mr3), n3 = it - k1 * g.r3;
        V* d = S + n3 * lpb + g.blk * k1 + l;
        V a[R];
#pragma unroll
        for (int n2 = 0; n2 < R; ++n2) a[n2] = d[g.row * n2];
        reg_fft<V, false, R>(a, nullptr);
        d[0] = a[0];
#pragma unroll
        for (int k2 = 1; k2 < R; ++k2) d[g.row * k2] = mul(a[k2], tw[n3 * k2 * g.r1]);
      }
    });
    __syncthreads();
  }
  {
    const int grp = line / gsz;
    V* __restrict__ dst = pp.work[blockIdx.y] + (size_t)grp * g.L * gsz + (line - grp * gsz);
    with_radix<TOP>(g.r3, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int it = first; it < g.r1 * g.r2; it += step) {
        const int k1 = div_by(it, g.mr2), k2 = it - k1 * g.r2;
        const V* d = S + g.row * it + l;
        V a[R];
#pragma unroll
        for (int n3 = 0; n3 < R; ++n3) a[n3] = d[n3 * lpb];
        reg_fft<V, false, R>(a, nullptr);
        if (on) {
          V* o = dst + (size_t)(k1 + g.r1 * k2) * gsz;
          const size_t st = (size_t)g.r1 * g.r2 * gsz;
#pragma unroll
          for (int k3 = 0; k3 < R; ++k3) o[k3 * st] = a[k3];
        }
      }
    });
  }
}

template <typename V, int TOP>
__global__ void __launch_bounds__(x_any_threads<V, TOP>(), 1) pass_c_any_kernel(const __grid_constant__ PassPtrs<V> pp, XAny g, int nx,
                                                         int nyz, int NL, const V* __restrict__ tw, int mode,
                                                         int gsz) {
  pdl_launch_dependents();
  if (skip_after_wait(pp)) return;
  extern __shared__ unsigned char smem_raw[];
  V* S = reinterpret_cast<V*>(smem_raw);
  const int lpb = g.lpb, t0 = div_by(threadIdx.x, g.ml), l = threadIdx.x - t0 * lpb, step = div_by(blockDim.x, g.ml);
  const int line = blockIdx.x * lpb + l;
  const int first = t0 < step ? t0 : g.L;   // threads beyond a whole row of lines take no item
  const bool on = line < NL;
  {
    const int ln = on ? line : 0, grp = ln / gsz;
    const V* __restrict__ src = pp.work[blockIdx.y] + (size_t)grp * g.L * gsz + (ln - grp * gsz);
    const size_t st = (size_t)g.r1 * g.r2 * gsz;
    with_radix<TOP>(g.r3, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int it = first; it < g.r1 * g.r2; it += step) {
        const int k1 = div_by(it, g.mr2), k2 = it - k1 * g.r2;
        const V* i = src + (size_t)(k1 + g.r1 * k2) * gsz;
        V a[R];
#pragma unroll
        for (int k3 = 0; k3 < R; ++k3) a[k3] = i[k3 * st];
        reg_fft<V, true, R>(a, nullptr);
        V* d = S + g.row * it + l;
        const int e = g.r2 > 1 ? k2 * g.r1 : k1;   // two-stage lengths: the outer twiddle here
        d[0] = a[0];
#pragma unroll
        for (int n3 = 1; n3 < R; ++n3) d[n3 * lpb] = mulc(a[n3], tw[n3 * e]);
      }
    });
  }
  __syncthreads();
  if (g.r2 > 1) {
    with_radix<TOP>(g.r2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int it = first; it < g.r1 * g.r3; it += step) {
        const int k1 = div_by(it, g.mr3), n3 = it - k1 * g.r3;
        V* d = S + n3 * lpb + g.blk * k1 + l;
        V a[R];
#pragma unroll
        for (int k2 = 0; k2 < R; ++k2) a[k2] = d[g.row * k2];
        reg_fft<V, true, R>(a, nullptr);
#pragma unroll
        for (int n2 = 0; n2 < R; ++n2) d[g.row * n2] = mulc(a[n2], tw[(n3 + g.r3 * n2) * k1]);
      }
    });
    __syncthreads();
  }
  {
    const int ln = on ? line : 0;
    const size_t g0 = (size_t)ln * nx;
    V* __restrict__ y = pp.y[blockIdx.y] + g0;
    const V* __restrict__ x = pp.x[blockIdx.y] + g0;
    const V* __restrict__ Mc = pp.M[blockIdx.y] + (size_t)(ln % nyz) * nx;
    with_radix<TOP>(g.r1, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      constexpr int H = (R + 1) / 2;   // outputs that can lie below nx <= (L + 1) / 2
      for (int np = first; np < g.M2; np += step) {
        const V* d = S + (np + (g.p3 - g.r3) * div_by(np, g.mr3)) * lpb + l;
        V a[R];
#pragma unroll
        for (int k1 = 0; k1 < R; ++k1) a[k1] = d[g.blk * k1];
        reg_fft<V, true, R>(a, nullptr);
        if (!on) continue;
        if (mode == MODE_PLAIN) {
#pragma unroll
          for (int n1 = 0; n1 < H; ++n1)
            if (np + g.M2 * n1 < nx) y[np + g.M2 * n1] = a[n1];
          continue;
        }
        V w[H], m[H];
#pragma unroll
        for (int n1 = 0; n1 < H; ++n1) {
          const int n = np + g.M2 * n1;
          w[n1] = n < nx ? x[n] : zero_c<V>();
          m[n1] = n < nx ? Mc[n] : zero_c<V>();
        }
#pragma unroll
        for (int n1 = 0; n1 < H; ++n1) {
          const int n = np + g.M2 * n1;
          if (n < nx) y[n] = (mode == MODE_OPERATOR) ? sub(w[n1], mul(m[n1], a[n1])) : mul(m[n1], sub(a[n1], w[n1]));
        }
      }
    });
  }
}

// Split of len into at most three radices (within the small class TOP = 16
// where possible, then the fewest stages, the smallest largest radix, the
// smallest sum; the outer radix the largest): false where there is none.
// small (complex128): the smallest largest radix before the fewest stages, as
// more butterflies keep the FP64 pipes of more warps busy on short lines (73 x
// 11 x 9: 65 us an application against 78).
static bool x_any_split(int len, bool small, XAny* g) {
  long best = -1;
  for (int r1 : kRadices) {
    if (len % r1) continue;
    for (int r3 : kRadices) {
      if (r3 > r1 || (len / r1) % r3 || (r3 == 1 && len > 1)) continue;
      const int r2 = len / (r1 * r3);
      if (r2 > r1) continue;
      bool known = false;
      for (int r : kRadices) known |= r == r2;
      if (!known) continue;
      // a last radix of 4, without multiplications, beside larger even ones
      // counts as 2 (200 x 200 x 11, 400 = 10 10 4: 103 us an application, 10
      // 8 5: 115); beside odd ones it does not pay (162 x 162 x 11, 324 = 9 9 4:
      // 97, 9 6 6: 75)
      const int sum = r1 + r2 + (r3 == 4 && r2 > 1 && r1 % 2 == 0 && r2 % 2 == 0 ? 2 : r3);
      const long cost = (r1 > 16 ? 1000000L : 0) + (r2 > 1 && !small ? 10000L : 0) + r1 * 100L + sum;
      if (best >= 0 && cost >= best) continue;
      best = cost;
      *g = XAny{len, r1, r2, r3, r2 * r3, r3 | 1, 0, 0, 0, div_magic(r2), div_magic(r3), 0};
    }
  }
  return best >= 0 && len < 65536;
}

// Lines per block: the fewest lines on the busiest SM; rows of the transposed
// side that are no multiple of 32 bytes cost a tenth more (measured: 600 x 23
// x 11, 759 lines, 5 lines 33 us against 36 with 4; JM-VIE 396 x 30 x 12,
// 2160 lines, 8 lines 58 us against 62 with 4 and 65 with 5 and 6).  *per:
// blocks of the busiest SM.
static int x_any_lines(long NL, int count, size_t line_bytes, int* per) {
  static const int lines[] = {4, 8, 6, 5, 3, 2, 1};
  int best = 0;
  double least = 0.0;
  for (int lpb : lines) {
    if (lpb * line_bytes > 220 * 1024) continue;
    const long blocks = (NL + lpb - 1) / lpb * count, p = (blocks + kSMs - 1) / kSMs;
    const double cost = (double)(p * lpb) * (lpb % 4 == 0 ? 1.0 : lpb > 2 ? 1.1 : lpb == 2 ? 1.2 : 1.5);
    if (best && cost >= least) continue;
    best = lpb;
    least = cost;
    *per = (int)p;
  }
  return best;
}

template <typename V, int TOP>
static vie_status launch_x_any_top(bool forward, const PassPtrs<V>& pp, int count, const XAny& g, int per, int n,
                                   int nyz, int NL, const V* tw, int mode, cudaStream_t s, int gsz) {
  const size_t smem = (size_t)g.r1 * g.blk * sizeof(V);
  int items = g.M2 > g.r1 * g.r3 ? g.M2 : g.r1 * g.r3;
  if (g.r1 * g.r2 > items) items = g.r1 * g.r2;
  items *= g.lpb;
  // few blocks on an SM: as many threads as there are items, so that a block's
  // loads are all in flight; many blocks hide each other's latency (800 x 600
  // x 11: 1250 us with 384 threads, 1356 with 512, 1476 with 768)
  const int want = per == 1 ? 1024 : per == 2 ? 512 : 384;
  const int most = want < x_any_threads<V, TOP>() ? want : x_any_threads<V, TOP>();
  const int turns = (items + most - 1) / most;
  const int threads = ((items + turns - 1) / turns + 31) / 32 * 32;
  const dim3 blocks((unsigned)((NL + g.lpb - 1) / g.lpb), (unsigned)count);
  if (forward) {
    VIE_CUDA_TRY(allow_shared(pass_a_any_kernel<V, TOP>, smem));
    VIE_CUDA_TRY(launch_pdl(pass_a_any_kernel<V, TOP>, blocks, dim3(threads), smem, s, pp, g, n, NL, tw, gsz));
  } else {
    VIE_CUDA_TRY(allow_shared(pass_c_any_kernel<V, TOP>, smem));
    VIE_CUDA_TRY(launch_pdl(pass_c_any_kernel<V, TOP>, blocks, dim3(threads), smem, s, pp, g, n, nyz, NL, tw, mode, gsz));
  }
  return VIE_OK;
}

template <typename V>
vie_status launch_x_any(bool forward, const PassPtrs<V>& pp, int count, int n, int nyz, int NL, int len, const V* tw,
                        int mode, cudaStream_t s, int gsz, bool* done) {
  *done = false;
  XAny g;
  if (!x_any_split(len, sizeof(V) == sizeof(double2), &g)) return VIE_OK;
  int per = 1;
  const int lpb = x_any_lines(NL, count, (size_t)g.r1 * g.r2 * g.p3 * sizeof(V), &per);
  if (!lpb) return VIE_OK;
  g.lpb = lpb;
  g.row = lpb * g.p3;
  g.blk = g.row * g.r2;
  g.ml = div_magic(lpb);
  *done = true;
  if (g.r1 <= 16) return launch_x_any_top<V, 16>(forward, pp, count, g, per, n, nyz, NL, tw, mode, s, gsz);
  return launch_x_any_top<V, 25>(forward, pp, count, g, per, n, nyz, NL, tw, mode, s, gsz);
}

}  // namespace vie
