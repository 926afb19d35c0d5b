// Pass B for any cross-section whose plane fits one CTA: register butterflies
// of run-time radices.
#pragma once

#include <cuda_pipeline.h>

#include "any_x.cuh"

namespace vie {

// ---------------------------------------------------------------------------
// pass B, one CTA per kx.  z lines (Mz <= 32) in registers: half of a z
// line's inputs are padding and half of its outputs are cropped, so for even
// Mz the radix-2 step falls apart into two transforms of Mz / 2 points, even
// and odd frequencies, by two neighbouring lanes (complex64; the half step's
// twiddles cost FP64, which binds complex128, 5 % more); y
// lines My = r1 r2 in two in-place stages, n = n2 + r2 n1, ky = k1 + r1 k2.
// The second forward stage, the spectral product and the first inverse stage
// need the same (kz, k1) group of r2 values of every component, so one thread
// takes them through all three without leaving its registers: the plane makes
// four round trips through shared memory instead of a dozen.
// Place of (c, kz; n1 or k1, n2): (c Mz + kz) py + p2 k1 + n2, p2 = r2 | 1,
// py = r1 p2: rows of stage items and of fused items fall on distinct banks.
// ---------------------------------------------------------------------------
// Row pitch py = r1 p2 + pad with the fewest bank conflicts of the two patterns
// that cross rows: stage items (row py + n2) and fused items (kz py + p2 k1).
// An element is 8 or 16 bytes and a shared-memory phase serves 128, i.e. 16
// or 8 lanes.  Without it the 54 x 24 planes of the Bragg grating spent half
// of their shared-memory cycles on conflicts.
constexpr int b_pad(int r1, int r2, int lanes) {
  int best = 1 << 30, at = 0;
  for (int pad = 0; pad < lanes; ++pad) {
    const int p2 = r2 | 1, py = r1 * p2 + pad;
    int cost = pad;   // ties: the smaller plane
    for (int warp = 0; warp < 96; warp += lanes) {
      int n1[16] = {0}, n2[16] = {0};
      for (int i = warp; i < warp + lanes; ++i) {
        ++n1[(i / r2 * py + i % r2) % lanes];
        ++n2[(i / r1 * py + i % r1 * p2) % lanes];
      }
      for (int k = 0; k < lanes; ++k) cost += 16 * (n1[k] * n1[k] + n2[k] * n2[k]);
    }
    if (cost < best) { best = cost; at = pad; }
  }
  return at;
}

// Transform lengths known at compile time: the same kernel (complex64) with its
// divisions by them, its strides and its switches folded; the cross-section
// stays a run-time value (21 to 24 x 11 or 12 voxels meet in 45 or 48 x 24; with
// 23 x 11 compiled in too, that one took 30.1 us instead of 30.3 and the others
// stayed behind by 5 to 20 %).  Zeros: all at run time.
template <int R1_, int R2_, int MZ_>
struct BFix {
  static constexpr int R1 = R1_, R2 = R2_, MZ = MZ_, P2 = R2_ | 1;
  static constexpr bool on = R1_ > 0;
  // voxels that every cross-section of the plane has: all but the last one of z,
  // all rows of r2 but the last one of y (taken only where they are there)
  static constexpr int min_z = MZ_ / 2 - 1, min_y = R2_ * ((R1_ + 1) / 2 - 1);
  static __device__ __forceinline__ bool full_z(int z) { return on && z < min_z; }
  static __device__ __forceinline__ bool full_y(int n1) { return on && R2_ * (n1 + 1) <= min_y; }
  static constexpr int PY = on ? R1_ * P2 + b_pad(on ? R1_ : 1, on ? R2_ : 1, 16) : 0;
};
typedef BFix<0, 0, 0> BFree;

#define VIE_Z_LENGTHS(X) \
  X(1) X(2) X(3) X(4) X(5) X(6) X(8) X(9) X(10) X(12) X(15) X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32)
template <int TOP, typename FIX, typename F>
__device__ __forceinline__ void with_z(int mz, F&& f) {
  if constexpr (FIX::on) {
    f(IC<FIX::MZ>{});
    return;
  }
  switch (mz) {
#define VIE_X(a) case a: if constexpr (a <= TOP) f(IC<a>{}); break;
    VIE_Z_LENGTHS(VIE_X)
#undef VIE_X
    default: break;
  }
}
static bool z_length_any(int mz) {
#define VIE_X(a) if (mz == a) return true;
  VIE_Z_LENGTHS(VIE_X)
#undef VIE_X
  return false;
}

struct BAny {
  int r1, r2, p2, py;
  unsigned mny, mr1, mr2;   // division by ny, r1, r2
};

#define VIE_R1(X) X(1) X(2) X(3) X(4) X(5) X(6) X(8) X(9) X(10) X(12) X(15) X(16)
template <int TOP, typename FIX, typename F>
__device__ __forceinline__ void with_r1(int r, F&& f) {
  if constexpr (FIX::on) {
    f(IC<FIX::R1>{});
    return;
  }
  switch (r) {
#define VIE_X(a) case a: if constexpr (a <= TOP) f(IC<a>{}); break;
    VIE_R1(VIE_X)
#undef VIE_X
    default: break;
  }
}
// largest fused radix: the group of nc r2 complex values lives in registers
template <typename V, int NC> __host__ __device__ constexpr int fused_max() { return sizeof(V) * NC <= 24 ? 10 : 6; }
template <int TOP, typename FIX, typename F>
__device__ __forceinline__ void with_r2(int r, F&& f) {
  if constexpr (FIX::on) {
    f(IC<FIX::R2>{});
    return;
  }
  switch (r) {
    case 1: f(IC<1>{}); break;
    case 2: f(IC<2>{}); break;
    case 3: f(IC<3>{}); break;
    case 4: f(IC<4>{}); break;
    case 5: f(IC<5>{}); break;
    case 6: f(IC<6>{}); break;
    case 8: if constexpr (TOP >= 8) f(IC<8>{}); break;
    case 9: if constexpr (TOP >= 9) f(IC<9>{}); break;
    case 10: if constexpr (TOP >= 10) f(IC<10>{}); break;
    default: break;
  }
}

template <typename V, int NC, bool STAGE, bool SMALL, typename FIX>
__global__ void __launch_bounds__(256, sizeof(V) == sizeof(float2) ? (SMALL && NC == 3 ? 3 : 2) : 1) pass_b_any_kernel(
    const __grid_constant__ PassPtrs<V> pp, const V* __restrict__ chat, double kappa, PassBGeom g, BAny q,
    const V* __restrict__ twy) {
  typedef typename real_of<V>::type R;
  constexpr int ZTOP = SMALL ? 24 : 32, R1TOP = SMALL ? 10 : 16, R2TOP = SMALL ? 6 : fused_max<V, NC>();
  extern __shared__ unsigned char smem_raw[];
  V* S = reinterpret_cast<V*>(smem_raw);
  const int kx = blockIdx.x, tid = threadIdx.x, nth = blockDim.x;
  const int ny = g.ny, nz = g.nz, Mz = FIX::on ? FIX::MZ : g.Mz;
  const int r1 = FIX::on ? FIX::R1 : q.r1, r2 = FIX::on ? FIX::R2 : q.r2;
  const int p2 = FIX::on ? FIX::P2 : q.p2, py = FIX::on ? FIX::PY : q.py;
  const int My = FIX::on ? FIX::R1 * FIX::R2 : g.My, Ky = FIX::on ? My / 2 + 1 : g.Ky;
  auto by_ny = [&](int v) { return FIX::on ? (int)__umulhi((unsigned)v, q.mny) : div_by(v, q.mny); };
  auto by_r1 = [&](int v) { return FIX::on ? v / (FIX::on ? FIX::R1 : 1) : div_by(v, q.mr1); };
  auto by_r2 = [&](int v) { return FIX::on ? v / (FIX::on ? FIX::R2 : 1) : div_by(v, q.mr2); };
  const bool fx = kx > g.Mx - kx;
  const int kxf = fx ? g.Mx - kx : kx;
  const int cs = FIX::on ? (Mz / 2 + 1) * Ky : g.Kz * g.Ky;
  const V* G = pp.ghat[blockIdx.y] + (size_t)kxf * 6 * cs;
  const V* Cc = NC == 6 ? chat + (size_t)kxf * 3 * cs : nullptr;
  pdl_launch_dependents();
  if (STAGE) {
    V* Gs = S + (size_t)NC * Mz * py;
    for (int i = tid; i < 6 * cs; i += nth) __pipeline_memcpy_async(Gs + i, G + i, sizeof(V));
    if (NC == 6)
      for (int i = tid; i < 3 * cs; i += nth) __pipeline_memcpy_async(Gs + 6 * cs + i, Cc + i, sizeof(V));
    __pipeline_commit();
    G = Gs;
    Cc = Gs + 6 * cs;
  }
  if (skip_after_wait(pp)) return;
  V* slab = pp.work[blockIdx.y] + (size_t)kx * g.NL;
  with_z<ZTOP, FIX>(Mz, [&](auto zc) {
    constexpr int MZ = decltype(zc)::value;
    if constexpr (MZ % 2 == 0 && sizeof(V) == sizeof(float2)) {
      constexpr int M = MZ / 2;
      for (int it = tid; it < 2 * NC * ny; it += nth) {
        const int line = it >> 1, odd = it & 1;
        const int c = by_ny(line), y = line - c * ny;
        const V* src = slab + c * nz * ny + y;
        V a[M];
#pragma unroll
        for (int z = 0; z < M; ++z, src += ny) a[z] = (FIX::full_z(z) || z < nz) ? *src : zero_c<V>();
        if (odd) half_twiddle<V, false, MZ>(a);
        reg_fft<V, false, M>(a, nullptr);
        V* d = S + (c * MZ + odd) * py + y + (p2 - r2) * by_r2(y);
#pragma unroll
        for (int k = 0; k < M; ++k) d[2 * k * py] = a[k];
      }
    } else {
      for (int line = tid; line < NC * ny; line += nth) {
        const int c = by_ny(line), y = line - c * ny;
        V a[MZ];
#pragma unroll
        for (int z = 0; z < MZ; ++z) a[z] = (z < (MZ + 1) / 2 && z < nz) ? slab[(c * nz + z) * ny + y] : zero_c<V>();
        reg_fft<V, false, MZ, (MZ + 1) / 2>(a, nullptr);
        V* d = S + c * MZ * py + y + (p2 - r2) * by_r2(y);
#pragma unroll
        for (int kz = 0; kz < MZ; ++kz) d[kz * py] = a[kz];
      }
    }
  });
  __syncthreads();
  with_r1<R1TOP, FIX>(r1, [&](auto rc) {
    constexpr int R1 = decltype(rc)::value;
    for (int it = tid; it < NC * Mz * r2; it += nth) {
      const int row = by_r2(it), n2 = it - row * r2;
      V* d = S + row * py + n2;
      V a[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1)
        a[n1] = (n1 < (R1 + 1) / 2 && (FIX::full_y(n1) || n2 + r2 * n1 < ny)) ? d[n1 * p2] : zero_c<V>();
      reg_fft<V, false, R1, (R1 + 1) / 2>(a, nullptr);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) d[k1 * p2] = a[k1];
    }
  });
  if (STAGE) __pipeline_wait_prior(0);
  __syncthreads();
  with_r2<R2TOP, FIX>(r2, [&](auto rc) {
    constexpr int R2 = decltype(rc)::value;
    for (int it = tid; it < Mz * r1; it += nth) {
      const int kz = by_r1(it), k1 = it - kz * r1;
      V* d = S + kz * py + k1 * p2;
      const int stride = Mz * py;
      V u[NC][R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) {
        const V w = n2 ? twy[n2 * k1] : V{};
#pragma unroll
        for (int c = 0; c < NC; ++c) u[c][n2] = n2 ? mul(d[c * stride + n2], w) : d[c * stride];
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) reg_fft<V, false, R2>(u[c], nullptr);
      const bool fz = kz > Mz - kz;
      const V* Gz = G + (fz ? Mz - kz : kz) * Ky;
      const V* Cz = NC == 6 ? Cc + (fz ? Mz - kz : kz) * Ky : nullptr;
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) {
        const int ky = k1 + r1 * k2;
        const bool fy = ky > My - ky;
        const int o = fy ? My - ky : ky;
        const V gxx = Gz[o], gyy = Gz[cs + o], gzz = Gz[2 * cs + o];
        V gxy = Gz[3 * cs + o], gxz = Gz[4 * cs + o], gyz = Gz[5 * cs + o];
        if (fx ^ fy) gxy = scale(gxy, (R)-1);
        if (fx ^ fz) gxz = scale(gxz, (R)-1);
        if (fy ^ fz) gyz = scale(gyz, (R)-1);
        V t[NC];
#pragma unroll
        for (int c = 0; c < NC; c += 3) {
          const V wx = u[c][k2], wy = u[c + 1][k2], wz = u[c + 2][k2];
          t[c] = add(add(mul(gxx, wx), mul(gxy, wy)), mul(gxz, wz));
          t[c + 1] = add(add(mul(gxy, wx), mul(gyy, wy)), mul(gyz, wz));
          t[c + 2] = add(add(mul(gxz, wx), mul(gyz, wy)), mul(gzz, wz));
        }
        if constexpr (NC == 6) {
          // j kappa C_a with the fold signs; v_e -= (jkC) x u_m, v_m += (jkC) x u_e
          const R kap = (R)kappa;
          const V cx = scale(mul_pi(Cz[o]), fx ? -kap : kap);
          const V cy = scale(mul_pi(Cz[cs + o]), fy ? -kap : kap);
          const V cz = scale(mul_pi(Cz[2 * cs + o]), fz ? -kap : kap);
          const V e0 = u[0][k2], e1 = u[1][k2], e2 = u[2][k2], m0 = u[3][k2], m1 = u[4][k2], m2 = u[5][k2];
          t[0] = sub(t[0], sub(mul(cy, m2), mul(cz, m1)));
          t[1] = sub(t[1], sub(mul(cz, m0), mul(cx, m2)));
          t[2] = sub(t[2], sub(mul(cx, m1), mul(cy, m0)));
          t[3] = add(t[3], sub(mul(cy, e2), mul(cz, e1)));
          t[4] = add(t[4], sub(mul(cz, e0), mul(cx, e2)));
          t[5] = add(t[5], sub(mul(cx, e1), mul(cy, e0)));
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) u[c][k2] = t[c];
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) reg_fft<V, true, R2>(u[c], nullptr);
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) {
        const V w = n2 ? twy[n2 * k1] : V{};
#pragma unroll
        for (int c = 0; c < NC; ++c) d[c * stride + n2] = n2 ? mulc(u[c][n2], w) : u[c][0];
      }
    }
  });
  __syncthreads();
  with_r1<R1TOP, FIX>(r1, [&](auto rc) {
    constexpr int R1 = decltype(rc)::value;
    for (int it = tid; it < NC * Mz * r2; it += nth) {
      const int row = by_r2(it), n2 = it - row * r2;
      V* d = S + row * py + n2;
      V a[R1];
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) a[k1] = d[k1 * p2];
      reg_fft<V, true, R1>(a, nullptr);
#pragma unroll
      for (int n1 = 0; n1 < (R1 + 1) / 2; ++n1)
        if (FIX::full_y(n1) || n2 + r2 * n1 < ny) d[n1 * p2] = a[n1];
    }
  });
  __syncthreads();
  with_z<ZTOP, FIX>(Mz, [&](auto zc) {
    constexpr int MZ = decltype(zc)::value;
    if constexpr (MZ % 2 == 0 && sizeof(V) == sizeof(float2)) {
      // even and odd frequencies by lanes 2 l, 2 l + 1: x[z] = E[z] + w^-z O[z];
      // each lane finishes half of the outputs
      constexpr int M = MZ / 2, H = (M + 1) / 2;
      const int total = 2 * NC * ny, turns = (total + nth - 1) / nth;
      for (int turn = 0, it = tid; turn < turns; ++turn, it += nth) {   // every lane takes every turn (shuffles)
        const bool in = it < total;
        const int line = in ? it >> 1 : 0, odd = it & 1;
        const int c = by_ny(line), y = line - c * ny;
        const V* d = S + (c * MZ + odd) * py + y + (p2 - r2) * by_r2(y);
        V a[M];
#pragma unroll
        for (int k = 0; k < M; ++k) a[k] = d[2 * k * py];
        reg_fft<V, true, M>(a, nullptr);
        if (odd) half_twiddle<V, true, MZ>(a);
        V* o = slab + (c * nz) * ny + y;
#pragma unroll
        for (int h = 0; h < H; ++h) {
          // even lane: z = h (gives E[z'] of the other half), odd lane: z' = h + H
          V give = odd ? a[h] : (h + H < M ? a[h + H] : zero_c<V>());
          V got;
          got.x = __shfl_xor_sync(0xffffffffu, give.x, 1);
          got.y = __shfl_xor_sync(0xffffffffu, give.y, 1);
          const int z = odd ? h + H : h;
          const V mine = odd ? (h + H < M ? a[h + H] : zero_c<V>()) : a[h];
          if (in && (FIX::full_z(z) || z < nz)) o[z * ny] = add(mine, got);
        }
      }
    } else {
      for (int line = tid; line < NC * ny; line += nth) {
        const int c = by_ny(line), y = line - c * ny;
        const V* d = S + c * MZ * py + y + (p2 - r2) * by_r2(y);
        V a[MZ];
#pragma unroll
        for (int kz = 0; kz < MZ; ++kz) a[kz] = d[kz * py];
        reg_fft<V, true, MZ>(a, nullptr);
#pragma unroll
        for (int z = 0; z < (MZ + 1) / 2; ++z)
          if (z < nz) slab[(c * nz + z) * ny + y] = a[z];
      }
    }
  });
}

// b_pad of every split
struct BPads {
  unsigned char pad[17][11];
};
static BPads b_pads(int lanes) {
  BPads t;
  for (int r1 = 1; r1 <= 16; ++r1)
    for (int r2 = 1; r2 <= 10; ++r2) t.pad[r1][r2] = (unsigned char)b_pad(r1, r2, lanes);
  return t;
}

// My = r1 r2, the radices as close as they come, within the kernel's small
// class (r1 <= 10, r2 <= 6) where possible.
template <typename V, int NC>
static bool b_any_split(int ny, int my, BAny* q) {
  static const BPads pads = b_pads(128 / (int)sizeof(V));
  int best = -1;
  const int r1s[] = {
#define VIE_X(a) a,
      VIE_R1(VIE_X)
#undef VIE_X
  };
  const int r2s[] = {1, 2, 3, 4, 5, 6, 8, 9, 10};
  for (int r1 : r1s)
    for (int r2 : r2s) {
      if (r1 * r2 != my || r2 > fused_max<V, NC>()) continue;
      const int cost = (r1 > r2 ? r1 - r2 : r2 - r1) + (r2 > 6 || r1 > 10 ? 1000 : 0);
      if (best >= 0 && cost >= best) continue;
      best = cost;
      *q = BAny{r1, r2, r2 | 1, r1 * (r2 | 1) + pads.pad[r1][r2], div_magic(ny), div_magic(r1), div_magic(r2)};
    }
  return best >= 0;
}

template <typename V, int NC>
static vie_status launch_b_any_nc(const PassPtrs<V>& pp, int count, const PassBGeom& g, const V* chat, double kappa,
                                  const V* twy, cudaStream_t s, bool* done) {
  *done = false;
  // small complex128 planes, at most one an SM, or three where one warp holds
  // all z lines: the generic pass spreads them over more warps (20 x 9 x 6: 44
  // us an application against 55; 152 x 9 x 14: 156 against 169)
  if (sizeof(V) == sizeof(double2) && (((long)g.Mx * count <= kSMs && g.My * g.Mz < 500) ||
                                       (NC * g.ny <= 32 && (long)g.Mx * count <= 3 * kSMs)))
    return VIE_OK;
  BAny q;
  if (!z_length_any(g.Mz) || !b_any_split<V, NC>(g.ny, g.My, &q)) return VIE_OK;
  const size_t plane = (size_t)NC * g.Mz * q.py * sizeof(V);
  const size_t spec = (size_t)(NC == 6 ? 9 : 6) * g.Kz * g.Ky * sizeof(V);
  if (plane > 220 * 1024) return VIE_OK;
  // spectrum staged where two blocks with it still fit an SM
  const bool stage = plane + spec <= 110 * 1024;
  const size_t smem = plane + (stage ? spec : 0);
  // one item per thread in the z and the fused phase, or a fraction of them;
  // complex128 keeps to four warps (200 registers a thread: more blocks)
  const int most = sizeof(V) == sizeof(float2) ? 256 : 128;
  int lines = NC * g.ny;
  if (g.Mz * q.r1 > lines) lines = g.Mz * q.r1;
  const int turns = (lines + most - 1) / most;
  const int threads = ((lines + turns - 1) / turns + 31) / 32 * 32;
  const dim3 grid((unsigned)g.Mx, (unsigned)count);
  const bool small = g.Mz <= 24 && q.r1 <= 10 && q.r2 <= 6;
  auto run = [&](auto kernel, int threads) -> vie_status {
    VIE_CUDA_TRY(allow_shared(kernel, smem));
    VIE_CUDA_TRY(launch_pdl_if(b_starts_early<V>(g, count), kernel, grid, dim3(threads), smem, s, pp, chat, kappa, g, q, twy));
    return VIE_OK;
  };
  vie_status st;
  if constexpr (sizeof(V) == sizeof(float2)) {
    typedef BFix<9, 5, 24> F45;
    typedef BFix<8, 6, 24> F48;
    auto is = [&](auto fix) {
      typedef decltype(fix) F;
      return q.r1 == F::R1 && q.r2 == F::R2 && g.Mz == F::MZ && g.nz >= F::min_z && g.ny >= F::min_y;
    };
    if (stage && (is(F45{}) || is(F48{}))) {
      // Compiled with their radices these planes take 8 to 20 % less than with
      // run-time ones (600 x 23 x 11: 30.3 us an application against 34.4; 600 x
      // 24 x 12: 35.7 against 39.1; 250 x 22 x 12: 19.3 against 24.3; JM 600 x 22 x
      // 11: 67.9 against 75.9).  Three components: five warps, one turn of the z
      // phase, two of the fused phase and three of the first y stage (600 x 23 x
      // 11: 30.5 with five, 32.0 with seven; 250 x 21 x 11: 20.2, 21.3 with seven,
      // 22.7 with four; 600 x 24 x 12: 35.9, 35.7 with six).
      const int t = NC == 3 ? 160 : threads;
      st = is(F45{}) ? run(pass_b_any_kernel<V, NC, true, true, F45>, t) : run(pass_b_any_kernel<V, NC, true, true, F48>, t);
      if (st != VIE_OK) return st;
      *done = true;
      return VIE_OK;
    }
  }
  if (stage) st = small ? run(pass_b_any_kernel<V, NC, true, true, BFree>, threads) : run(pass_b_any_kernel<V, NC, true, false, BFree>, threads);
  else st = small ? run(pass_b_any_kernel<V, NC, false, true, BFree>, threads) : run(pass_b_any_kernel<V, NC, false, false, BFree>, threads);
  if (st != VIE_OK) return st;
  *done = true;
  return VIE_OK;
}

template <typename V>
vie_status launch_b_any(const PassPtrs<V>& pp, int count, const PassBGeom& g, int nc, const V* chat, double kappa,
                        const V* twy, cudaStream_t s, bool* done) {
  return nc == 6 ? launch_b_any_nc<V, 6>(pp, count, g, chat, kappa, twy, s, done)
                 : launch_b_any_nc<V, 3>(pp, count, g, chat, kappa, twy, s, done);
}
}  // namespace vie
