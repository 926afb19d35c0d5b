// Block-circulant preconditioner of Sec. 5.4: the Frobenius-nearest matrix W
// to A = I - M N that is circulant in x, with dense (3 ny nz)^2 blocks.
//
// View A as nx x nx blocks A[i][j] (rows and columns ordered (p, z, y)):
// A[i][j] = delta_ij I - M_i T(i - j).  The nearest block-circulant matrix
// has the blocks c_k = (1/nx) sum_i A[i][(i - k) mod nx], i.e.
//   c_k = delta_k0 I - S+_k T(k) - S-_k T(k - nx),
//   S+_k = (1/nx) sum_{i >= k} M_i,  S-_k = (1/nx) sum_{i < k} M_i
// (row scalings by the x-averaged contrast).  The DFT along x
// block-diagonalises W: W_hat(w) = sum_k c_k exp(-2 pi i w k / nx).
//
// Setup (once per plan and contrast):
//   1. prefix sums of M along x (FP64),
//   2. W_hat: the blocks c_k of up to 16 entries at a time are formed in
//      shared memory and transformed along k by a Stockham FFT (radices 2-5
//      as butterflies, larger prime factors such as 7, 11, 13 summed
//      directly), so the blocks c_k are never stored,
//   3. LU with partial pivoting of the nx blocks W_hat(w): outer blocks of 64
//      columns in left-looking panels of 16 held in registers, row swaps, one
//      triangular solve for the block's rows and one update A22 -= L21 U12 of
//      the trailing matrix per outer block, in FP32.
// Application z = W^{-1} v (complex64):
//   V_hat = FFT along x of the 3 ny nz lines, one pivoted forward and
//   backward substitution per frequency (one CTA each, the factor streamed
//   once from HBM), then z = inverse FFT / nx.  The vectors' planar layout
//   [p][z][y][x] is already the (3B) x nx matrix the transforms need.
#include <cuda_fp16.h>
#include <cuda_pipeline.h>
#include <math.h>
#include <stdio.h>

#include <chrono>

#include "fft.cuh"
#include "vie_internal.cuh"

struct vie_circulant {
  int device = 0;
  const vie_plan* plan = nullptr;
  int gen = 0;                 // contrast generation the factors were built from
  int nx = 0, ny = 0, nz = 0, B = 0, R = 0;
  float2* W = nullptr;         // nx x R x R: LU factors (unit L below, U on and above the diagonal)
  __half2* W16 = nullptr;      // the same in complex half precision, as tiles (VIE_CIRC_FP16_FACTORS; W is then freed)
  bool fp16 = false;
  int* perm = nullptr;         // nx x R: row r of P b is b[perm[r]]
  float2* vh = nullptr;        // nx x R scratch (row-major [w][r])
  float2* v32 = nullptr;       // 3N scratch for complex128 callers
  float2* z32 = nullptr;
  int* flag = nullptr;         // 1: a zero pivot was met
  float2* tw = nullptr;        // nx twiddles exp(-2 pi i k / nx)
  vie::Radices rd;             //   and the radices of nx for the FFTs along x
  double build_ms = 0.0;
};

namespace vie {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 csub_mul(float2 acc, float2 a, float2 b) {
  // acc - a b
  return make_float2(acc.x - (a.x * b.x - a.y * b.y), acc.y - (a.x * b.y + a.y * b.x));
}

// ---------------------------------------------------------------------------
// setup kernels
// ---------------------------------------------------------------------------
// S+[zy][k] = (1/nx) sum_{i >= k} M[zy][i], S-[zy][k] = (1/nx) sum_{i < k} M[zy][i]
__global__ void prefix_kernel(const double2* __restrict__ M, int nx, int B, float2* __restrict__ Sp,
                              float2* __restrict__ Sm) {
  const int zy = blockIdx.x * blockDim.x + threadIdx.x;
  if (zy >= B) return;
  const double2* row = M + (size_t)zy * nx;
  double tx = 0.0, ty = 0.0;
  for (int i = 0; i < nx; ++i) {
    tx += row[i].x;
    ty += row[i].y;
  }
  double lx = 0.0, ly = 0.0;   // sum over i < k
  const double inv = 1.0 / nx;
  for (int k = 0; k < nx; ++k) {
    Sm[(size_t)zy * nx + k] = make_float2((float)(lx * inv), (float)(ly * inv));
    Sp[(size_t)zy * nx + k] = make_float2((float)((tx - lx) * inv), (float)((ty - ly) * inv));
    lx += row[k].x;
    ly += row[k].y;
  }
}

// Component index of (p, q) in the Toeplitz table order xx, yy, zz, xy, xz, yz.
__device__ __forceinline__ int comp_of(int p, int q) {
  if (p == q) return p;
  const int a = min(p, q), b = max(p, q);
  return a == 0 ? (b == 1 ? 3 : 4) : 5;
}

// T_pq(dx, dy, dz) for signed offsets from the octant table; an
// off-diagonal component is odd in each of its two axes.
__device__ __forceinline__ float2 toeplitz_at(const double2* __restrict__ T, int nx, int ny, int nz, int p, int q,
                                             int dx, int dy, int dz) {
  const int c = comp_of(p, q);
  const double2 t = T[(((size_t)c * nz + abs(dz)) * ny + abs(dy)) * nx + abs(dx)];
  float sgn = 1.f;
  if (p != q) {
    const int d[3] = {dx, dy, dz};
    if (d[p] < 0) sgn = -sgn;
    if (d[q] < 0) sgn = -sgn;
  }
  return make_float2(sgn * (float)t.x, sgn * (float)t.y);
}

// W_hat[w][e] for tl (<= kTL) consecutive entries e = r R + s at once:
// c_k[e] for every k is formed in shared memory and transformed along k by
// the Stockham FFT, so the blocks c_k are never stored.  tw = exp(-2 pi i k
// / nx).  tl is chosen so that the 2 tl lines of nx + 1 values fit in shared
// memory.
constexpr int kTL = 16;
constexpr int kBuildShared = kTL * (int)(sizeof(void*) + 4 * sizeof(int));   // static shared memory
__global__ void __launch_bounds__(256) build_fft_kernel(const double2* __restrict__ T, const float2* __restrict__ Sp,
                                                        const float2* __restrict__ Sm, int nx, int ny, int nz, int tl,
                                                        Radices rd, const float2* __restrict__ twg,
                                                        float2* __restrict__ What) {
  extern __shared__ float2 sb[];
  __shared__ const double2* tline[kTL];
  __shared__ float sgn_yz[kTL], sgn_neg[kTL];
  __shared__ int zyrow[kTL], diag[kTL];
  const int B = ny * nz, R = 3 * B;
  const long long RR = (long long)R * R;
  const int pitch = nx + 1;
  float2* tw = sb;
  float2* A = tw + nx;
  float2* Bf = A + tl * pitch;
  const long long e0 = (long long)blockIdx.x * tl;
  const int nl = (int)min((long long)tl, RR - e0);
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int i = tid; i < nx; i += nth) tw[i] = twg[i];
  if (tid < nl) {
    const long long e = e0 + tid;
    const int r = (int)(e / R), s2 = (int)(e % R);
    const int p = r / B, zy = r % B, z = zy / ny, y = zy % ny;
    const int q = s2 / B, zy2 = s2 % B, z2 = zy2 / ny, y2 = zy2 % ny;
    const int dy = y - y2, dz = z - z2;
    const int c = comp_of(p, q);
    float sg = 1.f, sx = 1.f;
    if (p != q) {
      // odd in the axes of both components: y (1) and z (2) here, x (0) for the negative offsets k - nx
      if ((p == 1 || q == 1) && dy < 0) sg = -sg;
      if ((p == 2 || q == 2) && dz < 0) sg = -sg;
      if (p == 0 || q == 0) sx = -1.f;
    }
    tline[tid] = T + (((size_t)c * nz + abs(dz)) * ny + abs(dy)) * nx;
    sgn_yz[tid] = sg;
    sgn_neg[tid] = sg * sx;
    zyrow[tid] = zy;
    diag[tid] = (r == s2);
  }
  __syncthreads();
  for (int idx = tid; idx < nl * nx; idx += nth) {
    const int l = idx / nx, k = idx - l * nx;
    const double2* tl = tline[l];
    const double2 tp = tl[k];
    float2 out = make_float2((k == 0 && diag[l]) ? 1.f : 0.f, 0.f);
    const float2 sp = Sp[(size_t)zyrow[l] * nx + k];
    out = csub_mul(out, sp, make_float2(sgn_yz[l] * (float)tp.x, sgn_yz[l] * (float)tp.y));
    if (k > 0) {
      const double2 tn = tl[nx - k];
      const float2 sm = Sm[(size_t)zyrow[l] * nx + k];
      out = csub_mul(out, sm, make_float2(sgn_neg[l] * (float)tn.x, sgn_neg[l] * (float)tn.y));
    }
    A[l * pitch + k] = out;
  }
  for (int idx = nl * nx + tid; idx < tl * nx; idx += nth) A[(idx / nx) * pitch + idx % nx] = make_float2(0.f, 0.f);
  __syncthreads();
  const float2* res = fft_lines<float2, false, true>(A, Bf, rd, pitch, tl, tw, tid, nth);
  for (int idx = tid; idx < nx * tl; idx += nth) {
    const int w = idx / tl, l = idx - w * tl;
    if (l < nl) What[(size_t)w * RR + e0 + l] = res[l * pitch + w];
  }
}

__global__ void twiddle_kernel(int nx, float2* __restrict__ tw) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nx) return;
  double sn, cs;
  sincospi(2.0 * (double)k / (double)nx, &sn, &cs);
  tw[k] = make_float2((float)cs, (float)-sn);
}

// DFTs along x of the application as FFTs, kLines rows per block.  Forward: vh[w][r] = sum_x v[r][x] exp(-2 pi i w x /
// nx); inverse: z[r][x] = (1/nx) sum_w vh[w][r] exp(+2 pi i w x / nx).
constexpr int kLines = 4;
template <bool INV>
__global__ void __launch_bounds__(256) lines_fft_kernel(const float2* __restrict__ in, float2* __restrict__ out, int R,
                                                        int nx, Radices rd, const float2* __restrict__ twg) {
  extern __shared__ float2 sb[];
  const int pitch = nx + 1;
  float2* tw = sb;
  float2* A = tw + nx;
  float2* Bf = A + kLines * pitch;
  const int r0 = blockIdx.x * kLines, nl = min(kLines, R - r0);
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int i = tid; i < nx; i += nth) tw[i] = twg[i];
  for (int idx = tid; idx < kLines * nx; idx += nth) {
    int l, k;
    if (INV) { k = idx / kLines; l = idx - k * kLines; } else { l = idx / nx; k = idx - l * nx; }
    float2 v = make_float2(0.f, 0.f);
    if (l < nl) v = INV ? in[(size_t)k * R + r0 + l] : in[(size_t)(r0 + l) * nx + k];
    A[l * pitch + k] = v;
  }
  __syncthreads();
  const float2* res = fft_lines<float2, INV, true>(A, Bf, rd, pitch, kLines, tw, tid, nth);
  const float inv = 1.f / (float)nx;
  for (int idx = tid; idx < kLines * nx; idx += nth) {
    int l, k;
    if (INV) { l = idx / nx; k = idx - l * nx; } else { k = idx / kLines; l = idx - k * kLines; }
    if (l >= nl) continue;
    const float2 v = res[l * pitch + k];
    if (INV) out[(size_t)(r0 + l) * nx + k] = make_float2(v.x * inv, v.y * inv);
    else out[(size_t)k * R + r0 + l] = v;
  }
}

// ---------------------------------------------------------------------------
// batched LU with partial pivoting (row-major blocks, one matrix per CTA)
// ---------------------------------------------------------------------------
// An outer block of kOuter columns is factored in panels of kPanel, looking to
// the left: a panel first takes up the products of the block's panels before
// it, so that no column of the block is rewritten by them.
constexpr int kOuter = 64;
constexpr int kPanel = 16;
constexpr int kMaxUnknowns = 1656;      // of a cross-section
constexpr int kPanelRows = 7 * 256;     // a panel's rows in registers: up to 7 a thread
static_assert(kMaxUnknowns <= kPanelRows, "the largest panel has no kernel");

// acc - a b, four multiply-adds
__device__ __forceinline__ void fnma(float2& acc, float2 a, float2 b) {
  acc.x = fmaf(-a.x, b.x, fmaf(a.y, b.y, acc.x));
  acc.y = fmaf(-a.x, b.y, fmaf(-a.y, b.x, acc.y));
}

// Panel j0 .. j0 + nbe - 1 of every matrix, rows j0 .. R - 1, one CTA a
// matrix: the block's earlier panels J .. j0 - 1 are applied, then per column
// the largest |a| below the diagonal is the pivot (lowest row on ties), rows
// are swapped inside the panel, the column is scaled by the pivot's inverse
// and the rest of the panel gets the rank-1 update.  piv[j] = the row swapped
// with row j.  A thread keeps rows tid + 256 k of the panel in registers (RP
// of them): a column costs two barriers, eight candidates and one broadcast
// row.  Bound by those and by one CTA an SM; with the panel in shared memory
// and its products with later columns as launches of their own, panels, those
// products and triangular solves took 8.5 ms for 160 blocks of 1080 unknowns,
// here 6.1 (396 blocks, the whole setup: 67 -> 58.5 ms).
template <int RP>
__global__ void __launch_bounds__(256, RP == 1 ? 3 : RP == 2 ? 2 : 1) lu_panel_kernel(
    float2* __restrict__ W, int R, int J, int j0, int nbe, int* __restrict__ piv, int* __restrict__ flag) {
  constexpr int NB = kPanel, NL = kOuter - kPanel;
  __shared__ float2 Lb[NL][NL + 1];                // rows and columns J .. j0 - 1: unit lower triangle
  __shared__ __align__(16) float2 U[NL][NB];       // rows J .. j0 - 1 of the panel's columns
  __shared__ __align__(16) float2 prow[2][NB], srow[2][NB];
  __shared__ float bval[2][8];
  __shared__ int bidx[2][8];
  float2* A = W + (size_t)blockIdx.x * R * R;
  const int rows = R - j0, k0 = j0 - J;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  float2 a[RP][NB];
#pragma unroll
  for (int k = 0; k < RP; ++k) {
    const int i = tid + 256 * k;
    const float2* src = A + (size_t)(j0 + i) * R + j0;
#pragma unroll
    for (int c = 0; c < NB; ++c) a[k][c] = i < rows && c < nbe ? src[c] : make_float2(0.f, 0.f);
  }
  if (k0 > 0) {
    for (int e = tid; e < k0 * k0; e += 256) {
      const int i = e / k0, t = e - i * k0;
      Lb[i][t] = A[(size_t)(J + i) * R + J + t];
    }
    for (int e = tid; e < k0 * NB; e += 256) {
      const int i = e / NB, c = e - i * NB;
      U[i][c] = c < nbe ? A[(size_t)(J + i) * R + j0 + c] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    // unit lower solve, two columns a warp, a lane per row of 16
    const int c = 2 * wid + (lane >> 4), r = lane & 15;
    for (int q = 0; q < k0; q += 16) {
      float2 x = U[q + r][c];
      for (int t = 0; t < q; ++t) fnma(x, Lb[q + r][t], U[t][c]);
#pragma unroll
      for (int t = 0; t < 15; ++t) {
        const float2 xt = make_float2(__shfl_sync(0xffffffffu, x.x, t, 16), __shfl_sync(0xffffffffu, x.y, t, 16));
        if (r > t) fnma(x, Lb[q + r][q + t], xt);
      }
      U[q + r][c] = x;
      __syncwarp();
    }
    __syncthreads();
    for (int e = tid; e < k0 * NB; e += 256) {
      const int i = e / NB, c2 = e - i * NB;
      if (c2 < nbe) A[(size_t)(J + i) * R + j0 + c2] = U[i][c2];
    }
    const float2* L[RP];
#pragma unroll
    for (int k = 0; k < RP; ++k) L[k] = A + (size_t)(j0 + min(tid + 256 * k, rows - 1)) * R + J;
#pragma unroll 2
    for (int t = 0; t < k0; ++t) {
      float2 l[RP];
#pragma unroll
      for (int k = 0; k < RP; ++k) l[k] = L[k][t];
#pragma unroll
      for (int c2 = 0; c2 < NB; c2 += 2) {
        const float4 u = *reinterpret_cast<const float4*>(&U[t][c2]);
#pragma unroll
        for (int k = 0; k < RP; ++k) {
          fnma(a[k][c2], l[k], make_float2(u.x, u.y));
          fnma(a[k][c2 + 1], l[k], make_float2(u.z, u.w));
        }
      }
    }
  }
#pragma unroll
  for (int jj = 0; jj < NB; ++jj) {
    if (jj >= nbe) break;
    const int s = jj & 1;
    // pivot: rows jj .. rows - 1 of column jj, the lowest row on ties
    float best = -1.f;
    int ip = rows;
#pragma unroll
    for (int k = 0; k < RP; ++k) {
      const int i = tid + 256 * k;
      const float m = a[k][jj].x * a[k][jj].x + a[k][jj].y * a[k][jj].y;
      if (i >= jj && i < rows && m > best) { best = m; ip = i; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ob = __shfl_down_sync(0xffffffffu, best, o);
      const int oi = __shfl_down_sync(0xffffffffu, ip, o);
      if (ob > best || (ob == best && oi < ip)) { best = ob; ip = oi; }
    }
    if (lane == 0) { bval[s][wid] = best; bidx[s][wid] = ip; }
    __syncthreads();
    best = bval[s][0];
    ip = bidx[s][0];
#pragma unroll
    for (int w = 1; w < 8; ++w) {
      const float ob = bval[s][w];
      const int oi = bidx[s][w];
      if (ob > best || (ob == best && oi < ip)) { best = ob; ip = oi; }
    }
    if (!(best > 0.f)) {
      ip = jj;
      if (tid == 0) atomicExch(flag, 1);
    }
    if (tid == 0) piv[(size_t)blockIdx.x * R + j0 + jj] = j0 + ip;
#pragma unroll
    for (int k = 0; k < RP; ++k)
      if (tid + 256 * k == ip) {
#pragma unroll
        for (int c = 0; c < NB; ++c) prow[s][c] = a[k][c];
      }
    if (tid == jj) {
#pragma unroll
      for (int c = 0; c < NB; ++c) srow[s][c] = a[0][c];
    }
    __syncthreads();
    // the other buffers of s are written again two columns on, behind the next column's barriers
    if (ip != jj) {
#pragma unroll
      for (int k = 0; k < RP; ++k)
        if (tid + 256 * k == ip) {
#pragma unroll
          for (int c = 0; c < NB; ++c) a[k][c] = srow[s][c];
        }
      if (tid == jj) {
#pragma unroll
        for (int c = 0; c < NB; ++c) a[0][c] = prow[s][c];
      }
    }
    const float2 d = prow[s][jj];
    const float dd = d.x * d.x + d.y * d.y;
    const float2 inv = dd > 0.f ? make_float2(d.x / dd, -d.y / dd) : make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < RP; ++k) {
      if (tid + 256 * k <= jj) continue;
      const float2 l = cmul(a[k][jj], inv);
      a[k][jj] = l;
#pragma unroll
      for (int c = jj + 1; c < NB; ++c) fnma(a[k][c], l, prow[s][c]);
    }
  }
#pragma unroll
  for (int k = 0; k < RP; ++k) {
    const int i = tid + 256 * k;
    if (i >= rows) continue;
    float2* dst = A + (size_t)(j0 + i) * R + j0;
#pragma unroll
    for (int c = 0; c < NB; ++c)
      if (c < nbe) dst[c] = a[k][c];
  }
}

// The panel's row swaps applied to every column outside it (the L columns
// to its left included, as in the usual packed LU).  One thread per column.
__global__ void __launch_bounds__(256) lu_swap_kernel(float2* __restrict__ W, int R, int j0, int nbe,
                                                      const int* __restrict__ piv) {
  const int c = blockIdx.y * blockDim.x + threadIdx.x;
  if (c >= R || (c >= j0 && c < j0 + nbe)) return;
  float2* A = W + (size_t)blockIdx.x * R * R;
  const int* pv = piv + (size_t)blockIdx.x * R;
  for (int jj = 0; jj < nbe; ++jj) {
    const int r1 = j0 + jj, r2 = pv[r1];
    if (r2 != r1) {
      const float2 t = A[(size_t)r1 * R + c];
      A[(size_t)r1 * R + c] = A[(size_t)r2 * R + c];
      A[(size_t)r2 * R + c] = t;
    }
  }
}

// U12 = L11^{-1} A12 of an outer block: rows J .. J + kOuter - 1, the columns
// right of the block; L11 is the block's unit lower triangle.  One thread per
// column, 16 rows at a time in registers, the rows solved before in shared
// memory.  (A launch per panel read and wrote the rows four times.)
constexpr int kTrsmCols = 128;
constexpr size_t kTrsmSmem = (kOuter * kOuter + (kOuter - 16) * kTrsmCols) * sizeof(float2);
__global__ void __launch_bounds__(kTrsmCols) lu_trsm_kernel(float2* __restrict__ W, int R, int J) {
  extern __shared__ __align__(16) float2 ts[];
  float2* Lt = ts;                          // [t][i]
  float2* xs = Lt + kOuter * kOuter;        // [t][column]
  float2* A = W + (size_t)blockIdx.x * R * R;
  const int tid = threadIdx.x;
  for (int e = tid; e < kOuter * kOuter; e += kTrsmCols) {
    const int i = e / kOuter, t = e - i * kOuter;
    Lt[t * kOuter + i] = A[(size_t)(J + i) * R + J + t];
  }
  __syncthreads();
  const int c = J + kOuter + blockIdx.y * kTrsmCols + tid;
  if (c >= R) return;
#pragma unroll 1
  for (int q = 0; q < kOuter; q += 16) {
    float2 x[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) x[r] = A[(size_t)(J + q + r) * R + c];
#pragma unroll 2
    for (int t = 0; t < q; ++t) {
      const float2 xt = xs[t * kTrsmCols + tid];
#pragma unroll
      for (int r = 0; r < 16; r += 2) {
        const float4 l = *reinterpret_cast<const float4*>(Lt + t * kOuter + q + r);
        fnma(x[r], make_float2(l.x, l.y), xt);
        fnma(x[r + 1], make_float2(l.z, l.w), xt);
      }
    }
#pragma unroll
    for (int i = 1; i < 16; ++i)
#pragma unroll
      for (int t = 0; t < i; ++t) fnma(x[i], Lt[(q + t) * kOuter + q + i], x[t]);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      A[(size_t)(J + q + r) * R + c] = x[r];
      if (q + 16 < kOuter) xs[(q + r) * kTrsmCols + tid] = x[r];
    }
  }
}

// Trailing update of an outer block, A22 -= L21 U12 with L21 = A[j1 .. R)[j0 ..
// j1), U12 = A[j0 .. j1)[j1 .. R), j1 = j0 + kOuter.  FP32-bound: with the
// rank of one panel every tile of A22 went through memory once per 16
// products, as long as the products took; with 64 the products dominate.  128
// x 64 tiles, 8 x 4 complex accumulators a thread, all 64 products' operands
// on their way into shared memory at once (four groups, summed as they
// arrive), the left ones transposed so that a thread's eight come in four
// 16-byte loads.  160 blocks of 1080 unknowns: 13.8 ms, 36 TFLOP/s; 15.1 with
// operands staged through registers 16 products ahead (three different
// register operands hold FP32 multiply-adds to 50 TFLOP/s on this chip).
constexpr int kUpdK = 16;
constexpr int kUpdPitch = 130;
constexpr size_t kTrailSmem = (size_t)kOuter * (kUpdPitch + 64) * sizeof(float2);
__global__ void __launch_bounds__(256, 2) lu_trailing_kernel(float2* __restrict__ W, int R, int j0) {
  extern __shared__ __align__(16) float2 us[];
  float2* As = us;                          // [k][row]
  float2* Bs = As + kOuter * kUpdPitch;     // [k][column]
  float2* A = W + (size_t)blockIdx.z * R * R;
  const int j1 = j0 + kOuter;
  const int i0 = j1 + blockIdx.y * 128, c0 = j1 + blockIdx.x * 64;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  // past the matrix's edge: zeros (bytes not copied are filled with zeros)
#pragma unroll
  for (int g = 0; g < kOuter; g += kUpdK) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int r = i0 + ty + 16 * u;
      __pipeline_memcpy_async(As + (g + tx) * kUpdPitch + ty + 16 * u, A + (size_t)min(r, R - 1) * R + j0 + g + tx,
                              sizeof(float2), r < R ? 0 : sizeof(float2));
    }
    const int c = c0 + (tid & 63);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = g + (tid >> 6) + 4 * u;
      __pipeline_memcpy_async(Bs + k * 64 + (tid & 63), A + (size_t)(j0 + k) * R + min(c, R - 1), sizeof(float2),
                              c < R ? 0 : sizeof(float2));
    }
    __pipeline_commit();
  }
  // thread: rows 2 ty + 32 a + {0, 1}, columns tx + 16 b
  float2 acc[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int g = 0; g < kOuter; g += kUpdK) {
    if (g == 0) __pipeline_wait_prior(3);
    else if (g == kUpdK) __pipeline_wait_prior(2);
    else if (g == 2 * kUpdK) __pipeline_wait_prior(1);
    else __pipeline_wait_prior(0);
    __syncthreads();
#pragma unroll 4
    for (int k = g; k < g + kUpdK; ++k) {
      float2 av[8], bv[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float4 t = *reinterpret_cast<const float4*>(As + k * kUpdPitch + 2 * ty + 32 * a);
        av[2 * a] = make_float2(t.x, t.y);
        av[2 * a + 1] = make_float2(t.z, t.w);
      }
#pragma unroll
      for (int b = 0; b < 4; ++b) bv[b] = Bs[k * 64 + tx + 16 * b];
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          acc[a][b].x = fmaf(av[a].x, bv[b].x, fmaf(-av[a].y, bv[b].y, acc[a][b].x));
          acc[a][b].y = fmaf(av[a].x, bv[b].y, fmaf(av[a].y, bv[b].x, acc[a][b].y));
        }
    }
  }
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int r = i0 + 2 * ty + 32 * (a >> 1) + (a & 1);
    if (r >= R) continue;
    float2* row = A + (size_t)r * R;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int c = c0 + tx + 16 * b;
      if (c < R) {
        float2 v = row[c];
        v.x -= acc[a][b].x;
        v.y -= acc[a][b].y;
        row[c] = v;
      }
    }
  }
}

// perm[w][r]: the swaps piv[w][0 .. R) applied in order to the identity, so
// that (P b)[r] = b[perm[r]].  One thread per matrix.
__global__ void perm_kernel(const int* __restrict__ piv, int R, int nmat, int* __restrict__ perm) {
  const int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= nmat) return;
  int* pm = perm + (size_t)w * R;
  const int* pv = piv + (size_t)w * R;
  for (int r = 0; r < R; ++r) pm[r] = r;
  for (int r = 0; r < R; ++r) {
    const int o = pv[r];
    if (o != r) {
      const int t = pm[r];
      pm[r] = pm[o];
      pm[o] = t;
    }
  }
}

// ---------------------------------------------------------------------------
// application: one CTA per frequency solves W_hat(w) z = b in place
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 cdiv(float2 a, float2 b) {
  const float d = b.x * b.x + b.y * b.y;
  return make_float2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}

// Streamer part of the pipelined substitution: 224 threads (warps 1-7),
// seven per row of a 32-row block row.  Thread (row, sub) sums
// A[j0 + row][t] x[t] over t = c0 + sub + 7 u < c1 with 16 loads in flight and
// leaves the sum in red[row][sub].
__device__ __forceinline__ void stream_partial(const float2* __restrict__ A, int R, int j0, int nr, int c0, int c1,
                                               const float2* __restrict__ x, float2 (*red)[8], int st) {
  const int row = st / 7, sub = st - row * 7;
  float sx = 0.f, sy = 0.f;
  if (row < nr) {
    constexpr int U = 16;
    const float2* rp = A + (size_t)(j0 + row) * R;
    int t = c0 + sub;
    for (; t + 7 * (U - 1) < c1; t += 7 * U) {
      float2 l[U];
#pragma unroll
      for (int u = 0; u < U; ++u) l[u] = rp[t + 7 * u];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float2 xt = x[t + 7 * u];
        sx += l[u].x * xt.x - l[u].y * xt.y;
        sy += l[u].x * xt.y + l[u].y * xt.x;
      }
    }
    for (; t < c1; t += 7) {
      const float2 l = rp[t], xt = x[t];
      sx += l.x * xt.x - l.y * xt.y;
      sy += l.x * xt.y + l.y * xt.x;
    }
  }
  red[row][sub] = make_float2(sx, sy);
}

// x = P b (gather), then L y = x and U z = y in blocks of 32 rows, pipelined:
// while warp 0 solves block k (its rows minus the streamed partial and the
// coupling to the block solved just before, then the 32 x 32 diagonal block
// with shuffles), warps 1-7 stream block k+1's products with every column
// that is already final and prefetch block k+1's diagonal block and its
// coupling block into the other half of double-buffered shared memory.  One
// barrier per block.  256 threads.
constexpr int kSolveShared = (2 * 2 * 32 * 33 + 2 * 32 * 8) * (int)sizeof(float2);   // static shared memory
__global__ void __launch_bounds__(256, 4) circ_solve_kernel(const float2* __restrict__ W, const int* __restrict__ perm,
                                                         float2* __restrict__ vh, int R) {
  extern __shared__ float2 x[];
  __shared__ float2 D[2][32][33];   // diagonal block
  __shared__ float2 E[2][32][33];   // coupling to the previously solved block
  __shared__ float2 red[2][32][8];  // streamed partial sums, 7 per row
  const float2* A = W + (size_t)blockIdx.x * R * R;
  const int* pm = perm + (size_t)blockIdx.x * R;
  float2* b = vh + (size_t)blockIdx.x * R;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, st = tid - 32;
  const int nblk = (R + 31) / 32;
  auto nrows = [&](int k) { return min(32, R - 32 * k); };
  for (int r = tid; r < R; r += blockDim.x) x[r] = b[pm[r]];
  // ---------------- forward: unit lower L ----------------
  {
    const int nr = nrows(0);
    for (int e = tid; e < 32 * 32; e += blockDim.x) {
      const int a = e >> 5, t = e & 31;
      D[0][a][t] = (a < nr && t < nr) ? A[(size_t)a * R + t] : make_float2(0.f, 0.f);
      if (t < 8) red[0][a][t] = make_float2(0.f, 0.f);
    }
  }
  __syncthreads();
  for (int k = 0; k < nblk; ++k) {
    const int cur = k & 1, nxt = cur ^ 1, i0 = 32 * k, nr = nrows(k);
    if (wid == 0) {
      float2 xi = lane < nr ? x[i0 + lane] : make_float2(0.f, 0.f);
      if (lane < nr) {
#pragma unroll
        for (int q = 0; q < 7; ++q) xi = make_float2(xi.x - red[cur][lane][q].x, xi.y - red[cur][lane][q].y);
        if (k > 0)
          for (int t = 0; t < 32; ++t) xi = csub_mul(xi, E[cur][lane][t], x[i0 - 32 + t]);
      }
      for (int t = 0; t < nr; ++t) {
        const float2 xt = make_float2(__shfl_sync(0xffffffffu, xi.x, t), __shfl_sync(0xffffffffu, xi.y, t));
        if (lane > t && lane < nr) xi = csub_mul(xi, D[cur][lane][t], xt);
      }
      if (lane < nr) x[i0 + lane] = xi;
    } else if (k + 1 < nblk) {
      const int j0 = i0 + 32, nr1 = nrows(k + 1);
      stream_partial(A, R, j0, nr1, 0, i0, x, red[nxt], st);
      for (int e = st; e < 32 * 32; e += blockDim.x - 32) {
        const int a = e >> 5, t = e & 31;
        const bool in = a < nr1;
        D[nxt][a][t] = (in && t < nr1) ? A[(size_t)(j0 + a) * R + j0 + t] : make_float2(0.f, 0.f);
        E[nxt][a][t] = in ? A[(size_t)(j0 + a) * R + i0 + t] : make_float2(0.f, 0.f);
      }
    }
    __syncthreads();
  }
  // ---------------- backward: upper U with its diagonal ----------------
  {
    const int kl = nblk - 1, i0 = 32 * kl, nr = nrows(kl);
    for (int e = tid; e < 32 * 32; e += blockDim.x) {
      const int a = e >> 5, t = e & 31;
      D[0][a][t] = (a < nr && t < nr) ? A[(size_t)(i0 + a) * R + i0 + t] : make_float2(0.f, 0.f);
      if (t < 8) red[0][a][t] = make_float2(0.f, 0.f);
    }
  }
  __syncthreads();
  for (int it = 0; it < nblk; ++it) {
    const int k = nblk - 1 - it, cur = it & 1, nxt = cur ^ 1;
    const int i0 = 32 * k, nr = nrows(k), i1 = i0 + nr;
    if (wid == 0) {
      float2 xi = lane < nr ? x[i0 + lane] : make_float2(0.f, 0.f);
      if (lane < nr) {
#pragma unroll
        for (int q = 0; q < 7; ++q) xi = make_float2(xi.x - red[cur][lane][q].x, xi.y - red[cur][lane][q].y);
        if (k + 1 < nblk) {
          const int nrn = nrows(k + 1);
          for (int t = 0; t < nrn; ++t) xi = csub_mul(xi, E[cur][lane][t], x[i1 + t]);
        }
      }
      for (int t = nr - 1; t >= 0; --t) {
        if (lane == t) xi = cdiv(xi, D[cur][t][t]);
        const float2 xt = make_float2(__shfl_sync(0xffffffffu, xi.x, t), __shfl_sync(0xffffffffu, xi.y, t));
        if (lane < t) xi = csub_mul(xi, D[cur][lane][t], xt);
      }
      if (lane < nr) x[i0 + lane] = xi;
    } else if (k > 0) {
      const int j0 = i0 - 32;      // block k - 1 has 32 rows
      stream_partial(A, R, j0, 32, i1, R, x, red[nxt], st);
      for (int e = st; e < 32 * 32; e += blockDim.x - 32) {
        const int a = e >> 5, t = e & 31;
        D[nxt][a][t] = A[(size_t)(j0 + a) * R + j0 + t];
        E[nxt][a][t] = t < nr ? A[(size_t)(j0 + a) * R + i0 + t] : make_float2(0.f, 0.f);
      }
    }
    __syncthreads();
  }
  for (int r = tid; r < R; r += blockDim.x) b[r] = x[r];
}

// ---------------------------------------------------------------------------
// complex-half factors: 32 x 32 tiles in the order the substitutions read them
// ---------------------------------------------------------------------------
// Of each matrix (nb block rows): forward, block row k = 0 .. nb - 1: L tiles
// (k, 0) .. (k, k - 1), then the diagonal tile; backward, k = nb - 1 .. 0: U
// tiles (k, k + 1) .. (k, nb - 1), then the diagonal tile again.  One linear
// stream of nb (nb + 1) tiles of 4 KB per frequency, which is what lets the
// substitution keep its loads 16 bytes wide and far ahead.  Off-diagonal tiles
// are row-major; diagonal ones column-major (the solve walks columns, a lane
// per row), with the identity beyond row R.
constexpr int kTile = 32;
constexpr int kTileElems = kTile * kTile;

__global__ void __launch_bounds__(256) to_tiles_kernel(const float2* __restrict__ W, __half2* __restrict__ F, int R,
                                                       int nb) {
  const float2* A = W + (size_t)blockIdx.y * R * R;
  const int t = blockIdx.x, half = nb * (nb + 1) / 2;
  __half2* out = F + ((size_t)blockIdx.y * 2 * half + t) * kTileElems;
  // block row and position of tile t of a direction: rows have 1, 2, .. nb tiles
  const int u = t < half ? t : t - half;
  int k = (int)((sqrtf(8.f * u + 1.f) - 1.f) * 0.5f);
  while (k * (k + 1) / 2 > u) --k;
  while ((k + 1) * (k + 2) / 2 <= u) ++k;
  const int i = u - k * (k + 1) / 2;               // i == k: the diagonal tile
  const int row = t < half ? k : nb - 1 - k;
  const int col = i == k ? row : (t < half ? i : row + 1 + i);
  __shared__ __half2 D[kTile][kTile + 1];
  for (int e = threadIdx.x; e < kTileElems; e += 256) {
    const int r = e >> 5, c = e & 31, gr = row * kTile + r, gc = col * kTile + c;
    float2 v = make_float2(i == k && gr == gc ? 1.f : 0.f, 0.f);
    if (gr < R && gc < R) v = A[(size_t)gr * R + gc];
    if (i == k) D[c][r] = __float22half2_rn(v);
    else out[e] = __float22half2_rn(v);
  }
  if (i != k) return;
  __syncthreads();
  for (int e = threadIdx.x; e < kTileElems; e += 256) out[e] = D[e >> 5][e & 31];
}

// x = P b, then L y = x and U z = y from the tile stream, one CTA per
// frequency.  HBM-bound: the factors are read once.  A stage is up to four
// tiles of one block row (16 KB); two stages, 32 KB a CTA, are in flight
// (asynchronous copies) while one is used.  48 KB of stages and the vector: four
// CTAs an SM up to 992 unknowns, three beyond.  Warp w sums rows
// 4 w .. 4 w + 3 of a tile, a lane per column; at the end of a block row the
// sums meet in shared memory and warp 0 solves the diagonal tile.  The rows
// used to be read by seven threads each, 4 bytes at a time: 599 us for 396
// frequencies of 1080 unknowns.
constexpr int kStageTiles = 4;
constexpr int kSolveStages = 3;

struct TileRow {   // position in the stream: direction, block row, next tile of the row
  int dir, k, i;
  __device__ __forceinline__ int count() const { return min(kStageTiles, k + 1 - i); }
  __device__ __forceinline__ void next(int nb) {
    i += kStageTiles;
    if (i > k) {
      i = 0;
      if (++k == nb) { k = 0; ++dir; }
    }
  }
};

__global__ void __launch_bounds__(256, 4) circ_solve_tiles_kernel(const __half2* __restrict__ F,
                                                                  const int* __restrict__ perm,
                                                                  float2* __restrict__ vh, int R, int nb) {
  extern __shared__ __align__(16) unsigned char circ_smem[];
  __half2* ring = reinterpret_cast<__half2*>(circ_smem);                                  // [stage][tile][1024]
  float2* x = reinterpret_cast<float2*>(ring + kSolveStages * kStageTiles * kTileElems);  // nb kTile
  __shared__ float psum[2 * kTile];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const __half2* src = F + (size_t)blockIdx.x * nb * (nb + 1) * kTileElems;
  const int* pm = perm + (size_t)blockIdx.x * R;
  float2* b = vh + (size_t)blockIdx.x * R;
  TileRow ahead{0, 0, 0}, at{0, 0, 0};
  auto issue = [&](int slot) {   // the next stage's copies into a slot (an empty group past the end)
    if (ahead.dir < 2) {
      const int n = ahead.count();
      for (int t = 0; t < n; ++t)
        __pipeline_memcpy_async(ring + (slot * kStageTiles + t) * kTileElems + tid * 4,
                                src + (size_t)t * kTileElems + tid * 4, 16);
      src += (size_t)n * kTileElems;
      ahead.next(nb);
    }
    __pipeline_commit();
  };
  issue(0);
  issue(1);
  for (int r = tid; r < nb * kTile; r += 256) x[r] = r < R ? b[pm[r]] : make_float2(0.f, 0.f);
  float acc[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) acc[u] = 0.f;
  for (int slot = 0; at.dir < 2; slot = slot == kSolveStages - 1 ? 0 : slot + 1) {
    __pipeline_wait_prior(kSolveStages - 2);
    __syncthreads();   // the stage has landed for every thread; the slot of the one before is free
    issue(slot == 0 ? kSolveStages - 1 : slot - 1);
    const int n = at.count();
    const bool last = at.i + n > at.k;                      // the row's diagonal tile is the stage's last
    const int row = at.dir == 0 ? at.k : nb - 1 - at.k;
    const __half2* tile = ring + slot * kStageTiles * kTileElems;
    for (int t = 0; t < n - (last ? 1 : 0); ++t) {
      const int col = at.dir == 0 ? at.i + t : row + 1 + at.i + t;
      const float2 xt = x[col * kTile + lane];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float2 l = __half22float2(tile[t * kTileElems + (4 * warp + u) * kTile + lane]);
        acc[2 * u] += l.x * xt.x - l.y * xt.y;
        acc[2 * u + 1] += l.x * xt.y + l.y * xt.x;
      }
    }
    if (last) {
      // eight sums a lane over the warp: after three exchanges a lane holds one
#pragma unroll
      for (int o = 16, k = 4; k >= 1; o >>= 1, k >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int u = 0; u < k; ++u) {
          const float keep = up ? acc[u + k] : acc[u], give = up ? acc[u] : acc[u + k];
          acc[u] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
      }
      acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
      acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
      if ((lane & 3) == 0) psum[8 * warp + (lane >> 2)] = acc[0];   // lane bits 4, 3, 2: the value's index
#pragma unroll
      for (int u = 0; u < 8; ++u) acc[u] = 0.f;
      __syncthreads();
      if (warp == 0) {
        const __half2* D = tile + (n - 1) * kTileElems;     // column-major
        float2 xi = x[row * kTile + lane];
        xi.x -= psum[2 * lane];
        xi.y -= psum[2 * lane + 1];
        if (at.dir == 0) {
#pragma unroll 8
          for (int t = 0; t < kTile - 1; ++t) {
            const float2 l = __half22float2(D[t * kTile + lane]);
            const float2 xt = make_float2(__shfl_sync(0xffffffffu, xi.x, t), __shfl_sync(0xffffffffu, xi.y, t));
            if (lane > t) xi = csub_mul(xi, l, xt);
          }
        } else {
          const float2 inv = cdiv(make_float2(1.f, 0.f), __half22float2(D[lane * kTile + lane]));
#pragma unroll 8
          for (int t = kTile - 1; t >= 0; --t) {
            const float2 l = __half22float2(D[t * kTile + lane]);
            if (lane == t) xi = cmul(xi, inv);
            const float2 xt = make_float2(__shfl_sync(0xffffffffu, xi.x, t), __shfl_sync(0xffffffffu, xi.y, t));
            if (lane < t) xi = csub_mul(xi, l, xt);
          }
        }
        x[row * kTile + lane] = xi;
      }
    }
    at.next(nb);
  }
  __syncthreads();
  for (int r = tid; r < R; r += 256) b[r] = x[r];
}

__global__ void to_c64_kernel(const double2* __restrict__ a, float2* __restrict__ b, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    b[i] = make_float2((float)a[i].x, (float)a[i].y);
}
__global__ void to_c128_kernel(const float2* __restrict__ a, double2* __restrict__ b, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    b[i] = make_double2((double)a[i].x, (double)a[i].y);
}

static unsigned blocks_for(size_t n) {
  const size_t b = (n + 255) / 256;
  return (unsigned)(b < 152 * 16 ? (b ? b : 1) : 152 * 16);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static void circ_free(vie_circulant* c) {
  if (!c) return;
  cudaFree(c->W); cudaFree(c->W16); cudaFree(c->tw); cudaFree(c->perm); cudaFree(c->vh);
  cudaFree(c->v32); cudaFree(c->z32); cudaFree(c->flag);
  delete c;
}

// Lines per block of the fused build (blocks formed and transformed along x
// in shared memory): the largest of 16, 8, 4, 2, 1 whose two buffers of
// nx + 1 values and the twiddle table fit in `smem_max` bytes, or 0.
static int build_lines(int nx, size_t smem_max) {
  for (int tl = kTL; tl >= 1; tl >>= 1)
    if ((size_t)nx * sizeof(float2) + (size_t)2 * tl * (nx + 1) * sizeof(float2) <= smem_max) return tl;
  return 0;
}

static vie_status circ_build(vie_circulant* c, cudaStream_t s, size_t smem_max) {
  const vie_plan* p = c->plan;
  const int nx = c->nx, ny = c->ny, nz = c->nz, B = c->B, R = c->R;
  const size_t RR = (size_t)R * R, N3 = (size_t)3 * B * nx;
  float2 *Sp = nullptr, *Sm = nullptr;
  int* piv = nullptr;
  vie_status st = VIE_OK;
  auto fail = [&](vie_status e) { cudaFree(Sp); cudaFree(Sm); cudaFree(piv); return e; };
#define CIRC_TRY(expr)                                                                         \
  do {                                                                                         \
    cudaError_t e__ = (expr);                                                                  \
    if (e__ != cudaSuccess) {                                                                  \
      set_error("%s:%d: %s failed: %s", __FILE__, __LINE__, #expr, cudaGetErrorString(e__));   \
      return fail(e__ == cudaErrorMemoryAllocation ? VIE_ERR_OOM : VIE_ERR_CUDA);             \
    }                                                                                          \
  } while (0)
  CIRC_TRY(cudaMalloc((void**)&Sp, (size_t)nx * B * sizeof(float2)));
  CIRC_TRY(cudaMalloc((void**)&Sm, (size_t)nx * B * sizeof(float2)));
  CIRC_TRY(cudaMalloc((void**)&piv, (size_t)nx * R * sizeof(int)));
  CIRC_TRY(cudaMalloc((void**)&c->W, (size_t)nx * RR * sizeof(float2)));
  CIRC_TRY(cudaMalloc((void**)&c->perm, (size_t)nx * R * sizeof(int)));
  CIRC_TRY(cudaMalloc((void**)&c->vh, (size_t)nx * R * sizeof(float2)));
  CIRC_TRY(cudaMalloc((void**)&c->v32, N3 * sizeof(float2)));
  CIRC_TRY(cudaMalloc((void**)&c->z32, N3 * sizeof(float2)));
  CIRC_TRY(cudaMalloc((void**)&c->flag, sizeof(int)));
  CIRC_TRY(cudaMalloc((void**)&c->tw, (size_t)nx * sizeof(float2)));
  CIRC_TRY(cudaMemsetAsync(c->flag, 0, sizeof(int), s));

  prefix_kernel<<<(B + 127) / 128, 128, 0, s>>>(p->M64, nx, B, Sp, Sm);
  twiddle_kernel<<<(nx + 127) / 128, 128, 0, s>>>(nx, c->tw);
  CIRC_TRY(cudaGetLastError());
  // W_hat: blocks formed and transformed along x in shared memory
  const int tl = build_lines(nx, smem_max);
  const size_t fft_smem = (size_t)nx * sizeof(float2) + (size_t)2 * tl * (nx + 1) * sizeof(float2);
  CIRC_TRY(allow_shared(build_fft_kernel, fft_smem, kBuildShared));
  build_fft_kernel<<<(unsigned)((RR + tl - 1) / tl), 256, fft_smem, s>>>(p->toeplitz, Sp, Sm, nx, ny, nz, tl, c->rd,
                                                                        c->tw, c->W);
  CIRC_TRY(cudaGetLastError());
  // LU of the nx blocks: within an outer block of kOuter columns the panels
  // look to the left; the rows right of the block and the trailing matrix are
  // updated once per outer block
  CIRC_TRY(cudaFuncSetAttribute(lu_trsm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrsmSmem));
  CIRC_TRY(cudaFuncSetAttribute(lu_trailing_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrailSmem));
  for (int J = 0; J < R; J += kOuter) {
    const int JE = min(J + kOuter, R);
    for (int j0 = J; j0 < JE; j0 += kPanel) {
      const int nbe = min(kPanel, R - j0);
      switch ((R - j0 + 255) / 256) {
        case 1: lu_panel_kernel<1><<<nx, 256, 0, s>>>(c->W, R, J, j0, nbe, piv, c->flag); break;
        case 2: lu_panel_kernel<2><<<nx, 256, 0, s>>>(c->W, R, J, j0, nbe, piv, c->flag); break;
        case 3: lu_panel_kernel<3><<<nx, 256, 0, s>>>(c->W, R, J, j0, nbe, piv, c->flag); break;
        case 4: lu_panel_kernel<4><<<nx, 256, 0, s>>>(c->W, R, J, j0, nbe, piv, c->flag); break;
        case 5: lu_panel_kernel<5><<<nx, 256, 0, s>>>(c->W, R, J, j0, nbe, piv, c->flag); break;
        default: lu_panel_kernel<kPanelRows / 256><<<nx, 256, 0, s>>>(c->W, R, J, j0, nbe, piv, c->flag); break;
      }
      lu_swap_kernel<<<dim3(nx, (R + 255) / 256), 256, 0, s>>>(c->W, R, j0, nbe, piv);
    }
    CIRC_TRY(cudaGetLastError());
    if (JE < R) {
      const int n = R - JE;
      lu_trsm_kernel<<<dim3((unsigned)nx, (unsigned)((n + kTrsmCols - 1) / kTrsmCols)), kTrsmCols, kTrsmSmem, s>>>(c->W, R, J);
      lu_trailing_kernel<<<dim3((unsigned)((n + 63) / 64), (unsigned)((n + 127) / 128), (unsigned)nx), 256, kTrailSmem,
                           s>>>(c->W, R, J);
      CIRC_TRY(cudaGetLastError());
    }
  }
  perm_kernel<<<(nx + 127) / 128, 128, 0, s>>>(piv, R, nx, c->perm);
  CIRC_TRY(cudaGetLastError());
  CIRC_TRY(cudaStreamSynchronize(s));
  int flag = 0;
  CIRC_TRY(cudaMemcpy(&flag, c->flag, sizeof(int), cudaMemcpyDeviceToHost));
  fail(VIE_OK);
  Sp = Sm = nullptr;
  piv = nullptr;
  if (flag) {
    set_error("block-circulant preconditioner: a diagonal block is singular");
    st = VIE_ERR_NONFINITE;
  }
#undef CIRC_TRY
  return st;
}

const vie_plan* circulant_plan(const vie_circulant* c) { return c->plan; }

vie_status circulant_apply(vie_circulant* c, int dtype, const void* v, void* z, cudaStream_t s) {
  if (c->gen != c->plan->contrast_gen) {
    set_error("block-circulant preconditioner is stale: the plan's contrast changed after it was built");
    return VIE_ERR_INVALID;
  }
  const int nx = c->nx, R = c->R;
  const size_t N3 = (size_t)R * nx;
  const float2* vin = (const float2*)v;
  float2* zout = (float2*)z;
  if (dtype == VIE_C128) {
    to_c64_kernel<<<blocks_for(N3), 256, 0, s>>>((const double2*)v, c->v32, N3);
    VIE_LAUNCH_CHECK();
    vin = c->v32;
    zout = c->z32;
  }
  const size_t fft_smem = (size_t)nx * sizeof(float2) + (size_t)2 * kLines * (nx + 1) * sizeof(float2);
  VIE_CUDA_TRY(allow_shared(lines_fft_kernel<false>, fft_smem));
  VIE_CUDA_TRY(allow_shared(lines_fft_kernel<true>, fft_smem));
  // V_hat[w][r] = sum_x exp(-2 pi i w x / nx) v[r][x]
  lines_fft_kernel<false><<<(R + kLines - 1) / kLines, 256, fft_smem, s>>>(vin, c->vh, R, nx, c->rd, c->tw);
  VIE_LAUNCH_CHECK();
  if (c->fp16) {
    const int nb = (R + kTile - 1) / kTile;
    const size_t smem = (size_t)kSolveStages * kStageTiles * kTileElems * sizeof(__half2) + (size_t)nb * kTile * sizeof(float2);
    VIE_CUDA_TRY(allow_shared(circ_solve_tiles_kernel, smem, 2 * kTile * sizeof(float)));
    circ_solve_tiles_kernel<<<nx, 256, smem, s>>>(c->W16, c->perm, c->vh, R, nb);
  } else {
    // the vector and 37 KB of tiles: past 48 KB from 1409 unknowns on
    VIE_CUDA_TRY(allow_shared(circ_solve_kernel, R * sizeof(float2), kSolveShared));
    circ_solve_kernel<<<nx, 256, (size_t)R * sizeof(float2), s>>>(c->W, c->perm, c->vh, R);
  }
  VIE_LAUNCH_CHECK();
  // z[r][x] = (1/nx) sum_w exp(+2 pi i w x / nx) Z_hat[w][r]
  lines_fft_kernel<true><<<(R + kLines - 1) / kLines, 256, fft_smem, s>>>(c->vh, zout, R, nx, c->rd, c->tw);
  VIE_LAUNCH_CHECK();
  if (dtype == VIE_C128) {
    to_c128_kernel<<<blocks_for(N3), 256, 0, s>>>(c->z32, (double2*)z, N3);
    VIE_LAUNCH_CHECK();
  }
  return VIE_OK;
}

}  // namespace vie

using namespace vie;

extern "C" {

vie_status vie_circulant_create(vie_plan* plan, int flags, vie_circulant** out, void* stream) {
  clear_error();
  if (!plan || !out) { set_error("null argument"); return VIE_ERR_INVALID; }
  if (flags & ~VIE_CIRC_FP16_FACTORS) { set_error("unknown flags 0x%x", flags); return VIE_ERR_INVALID; }
  *out = nullptr;
  if (!plan->M64) { set_error("set the plan's contrast before building its circulant preconditioner"); return VIE_ERR_INVALID; }
  const auto t0 = std::chrono::steady_clock::now();
  vie_circulant* c = new vie_circulant();
  c->plan = plan;
  c->gen = plan->contrast_gen;
  c->nx = plan->n[0];
  c->ny = plan->n[1];
  c->nz = plan->n[2];
  c->B = c->ny * c->nz;
  c->R = 3 * c->B;
  if (c->R > kMaxUnknowns) {
    set_error("cross-section of %d unknowns is too large for the block-circulant preconditioner", c->R);
    delete c;
    return VIE_ERR_INVALID;
  }
  if ((size_t)c->R * c->R > (size_t)0x7fffffff) {
    set_error("cross-section too large for the block-circulant preconditioner");
    delete c;
    return VIE_ERR_INVALID;
  }
  VIE_CUDA_TRY(cudaGetDevice(&c->device));
  int smem_optin = 0;
  VIE_CUDA_TRY(cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device));
  // the FFTs along x: radices of nx (any prime factors) and shared memory for
  // the application's kLines lines and at least one line of the build
  AxisPlan ax;
  if (!factor_length_any(c->nx, &ax) ||
      (size_t)c->nx * sizeof(float2) + (size_t)2 * kLines * (c->nx + 1) * sizeof(float2) > (size_t)smem_optin ||
      build_lines(c->nx, (size_t)smem_optin) == 0) {
    set_error("nx = %d is too long for the block-circulant preconditioner's FFTs along x", c->nx);
    delete c;
    return VIE_ERR_INVALID;
  }
  c->rd = radices_of(ax);
  vie_status st = circ_build(c, (cudaStream_t)stream, (size_t)smem_optin);
  if (st == VIE_OK && (flags & VIE_CIRC_FP16_FACTORS)) {
    // keep only a complex-half copy of the factors
    const int nb = (c->R + kTile - 1) / kTile, tiles = nb * (nb + 1);
    cudaError_t e = cudaMalloc((void**)&c->W16, (size_t)c->nx * tiles * kTileElems * sizeof(__half2));
    if (e == cudaSuccess) {
      to_tiles_kernel<<<dim3((unsigned)tiles, (unsigned)c->nx), 256, 0, (cudaStream_t)stream>>>(c->W, c->W16, c->R, nb);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize((cudaStream_t)stream);
    if (e != cudaSuccess) {
      set_error("half-precision factors: %s", cudaGetErrorString(e));
      st = e == cudaErrorMemoryAllocation ? VIE_ERR_OOM : VIE_ERR_CUDA;
    } else {
      cudaFree(c->W);
      c->W = nullptr;
      c->fp16 = true;
    }
  }
  if (st != VIE_OK) {
    circ_free(c);
    return st;
  }
  c->build_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  *out = c;
  return VIE_OK;
}

vie_status vie_circulant_apply(vie_circulant* c, const void* v_dev, void* z_dev, int dtype, void* stream) {
  clear_error();
  if (!c || !v_dev || !z_dev) { set_error("null argument"); return VIE_ERR_INVALID; }
  if (dtype != VIE_C64 && dtype != VIE_C128) { set_error("dtype must be VIE_C64 or VIE_C128"); return VIE_ERR_INVALID; }
  return circulant_apply(c, dtype, v_dev, z_dev, (cudaStream_t)stream);
}

vie_status vie_circulant_info(const vie_circulant* c, double* build_ms, size_t* device_bytes) {
  clear_error();
  if (!c) { set_error("null argument"); return VIE_ERR_INVALID; }
  if (build_ms) *build_ms = c->build_ms;
  const size_t nb = (size_t)(c->R + kTile - 1) / kTile;
  if (device_bytes)
    *device_bytes = (c->fp16 ? (size_t)c->nx * nb * (nb + 1) * kTileElems * sizeof(__half2)
                             : (size_t)c->nx * c->R * c->R * sizeof(float2)) +
                    (size_t)c->nx * c->R * (sizeof(int) + sizeof(float2)) + (size_t)c->nx * sizeof(float2) +
                    (size_t)2 * c->nx * c->R * sizeof(float2);
  return VIE_OK;
}

vie_status vie_circulant_destroy(vie_circulant* c) {
  circ_free(c);
  return VIE_OK;
}

}  // extern "C"
