// Setup on the device, in FP64: Galerkin Toeplitz entries of N and the
// spectra of their circulant embedding.
//
// Paper (arXiv:1803.06237): N f = curl curl S f with G = exp(-j k r)/(4 pi r)
// (Sec. 3); N_ij = <N P_j, P_i> with P_i = h^(-3/2) on voxel i (Sec. 3.1);
// N is block-Toeplitz with six unique tensor components and its product is
// computed with FFTs (Sec. 5.4).
//
// With h as the unit of length and kappa = k h, (lap + k^2) G = -delta gives
// N = k^2 S + grad div S + I, and the entry for offset D and components p, q is
//   T_pq(D) = delta_pq delta_D0 + int L_D(v) (kappa^2 delta_pq + d_p d_q) g(v) dv,
// L_D(v) = prod_a max(0, 1 - |v_a - D_a|) (the overlap of two unit voxels),
// g(v) = exp(-j kappa |v|)/(4 pi |v|), the derivatives taken in the sense of
// distributions.  Two routes are used:
//   * |D|_inf >= 2: the support of L_D misses v = 0, so the derivatives act on g
//     (closed-form dyadic kernel) and the tent-weighted integral is done with
//     the tensor Gauss rule of the tent weight itself, one rule across the
//     whole support (the integrand is analytic there, the tent is not).
//   * |D|_inf <= 1: the derivatives act on L_D.  The off-diagonal part becomes
//     int g sign(v_p - D_p) sign(v_q - D_q) L(v_r - D_r) dv, the diagonal part a
//     second difference of plane integrals F_p(t) = int int g L L over the
//     planes v_p = D_p - 1, D_p, D_p + 1.  Unit cells that have the origin as
//     a corner use the Duffy map (pyramids / triangles, Jacobian t^2 / t).
#include <math.h>
#include <stdio.h>

#include <mutex>
#include <vector>

#include "fft.cuh"
#include "vie_internal.cuh"

namespace vie {

// ---------------------------------------------------------------------------
// Gauss-Legendre nodes on [0, 1] for orders 1..kMaxGL (host Newton iteration
// on the three-term Legendre recurrence), stored at offset q (q - 1) / 2.
// ---------------------------------------------------------------------------
constexpr int kMaxGL = 24;
__constant__ double c_gl_x[kMaxGL * (kMaxGL + 1) / 2];
__constant__ double c_gl_w[kMaxGL * (kMaxGL + 1) / 2];

static void legendre_nodes(int q, double* x01, double* w01) {
  for (int i = 0; i < q; ++i) {
    double x = cos(M_PI * (i + 0.75) / (q + 0.5));
    double dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = x;
      for (int k = 2; k <= q; ++k) {
        double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      if (q == 1) { p1 = x; p0 = 1.0; }
      dp = q * (x * p1 - p0) / (x * x - 1.0);
      double dx = p1 / dp;
      x -= dx;
      if (fabs(dx) < 1e-17) break;
    }
    // recompute the derivative at the converged node
    double p0 = 1.0, p1 = x;
    for (int k = 2; k <= q; ++k) {
      double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
      p0 = p1;
      p1 = p2;
    }
    if (q == 1) { p1 = x; p0 = 1.0; }
    dp = q * (x * p1 - p0) / (x * x - 1.0);
    x01[i] = 0.5 * (1.0 - x);
    w01[i] = 1.0 / ((1.0 - x * x) * dp * dp);   // (2/((1-x^2) P'^2)) / 2
  }
}

// Gauss rules of the weight 1 - |t| on [-1, 1], orders 1..kMaxGL, stored at
// offset q (q - 1) / 2: c_tg_x nodes, c_tg_w weights (sum 1).
__constant__ double c_tg_x[kMaxGL * (kMaxGL + 1) / 2];
__constant__ double c_tg_w[kMaxGL * (kMaxGL + 1) / 2];

// The recurrence p_{k+1} = t p_k - b_k p_{k-1} of the weight's orthogonal
// polynomials (Stieltjes; the weight is even, so there is no other term) with
// inner products by a Gauss-Legendre rule of degree 2 kMaxGL + 1 on each half,
// where the weight is linear; then the nodes of each order by bisection
// between the nodes of the order below and Newton steps, and the weights
// 1 / sum_k p_k^2 / |p_k|^2.  In long double, so that nodes and weights are
// double-precision exact: an error there enters every entry.
static void tent_gauss_rules(double* xs, double* ws) {
  typedef long double L;
  constexpr int G = kMaxGL + 2;
  L gx[G], gw[G];
  for (int i = 0; i < G; ++i) {
    L x = cosl(M_PI * ((L)i + 0.75L) / (G + 0.5L)), dp = 1.0L;
    for (int it = 0; it < 60; ++it) {
      L p0 = 1.0L, p1 = x;
      for (int k = 2; k <= G; ++k) {
        const L p2 = ((2.0L * k - 1.0L) * x * p1 - (k - 1.0L) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = G * (x * p1 - p0) / (x * x - 1.0L);
      x -= p1 / dp;
    }
    L p0 = 1.0L, p1 = x;
    for (int k = 2; k <= G; ++k) {
      const L p2 = ((2.0L * k - 1.0L) * x * p1 - (k - 1.0L) * p0) / k;
      p0 = p1;
      p1 = p2;
    }
    dp = G * (x * p1 - p0) / (x * x - 1.0L);
    gx[i] = 0.5L * (1.0L - x);
    gw[i] = 1.0L / ((1.0L - x * x) * dp * dp);
  }
  L t[2 * G], w[2 * G], pm[2 * G], pk[2 * G], b[kMaxGL + 1], nk[kMaxGL + 1];
  for (int i = 0; i < G; ++i) {
    t[i] = gx[i];
    t[G + i] = -gx[i];
    w[i] = w[G + i] = gw[i] * (1.0L - gx[i]);
  }
  for (int i = 0; i < 2 * G; ++i) { pm[i] = 0.0L; pk[i] = 1.0L; }
  for (int k = 0; k <= kMaxGL; ++k) {
    L n = 0.0L;
    for (int i = 0; i < 2 * G; ++i) n += w[i] * pk[i] * pk[i];
    nk[k] = n;
    b[k] = k > 0 ? n / nk[k - 1] : 0.0L;
    for (int i = 0; i < 2 * G; ++i) {
      const L q = t[i] * pk[i] - b[k] * pm[i];
      pm[i] = pk[i];
      pk[i] = q;
    }
  }
  std::vector<L> prev, cur;   // nodes of the order below, of this order
  for (int q = 1; q <= kMaxGL; ++q) {
    auto eval = [&](L x, L* d) {   // p_q(x) and its derivative
      L p0 = 0.0L, p1 = 1.0L, d0 = 0.0L, d1 = 0.0L;
      for (int k = 0; k < q; ++k) {
        const L p2 = x * p1 - b[k] * p0, d2 = p1 + x * d1 - b[k] * d0;
        p0 = p1; p1 = p2;
        d0 = d1; d1 = d2;
      }
      *d = d1;
      return p1;
    };
    cur.clear();
    for (int i = 0; i < q; ++i) {
      L lo = i == 0 ? -1.0L : prev[i - 1], hi = i == q - 1 ? 1.0L : prev[i], d;
      const L slo = eval(lo, &d);
      for (int it = 0; it < 20; ++it) {
        const L mid = 0.5L * (lo + hi);
        if ((eval(mid, &d) > 0.0L) == (slo > 0.0L)) lo = mid; else hi = mid;
      }
      L x = 0.5L * (lo + hi);
      for (int it = 0; it < 6; ++it) { const L p = eval(x, &d); x -= p / d; }
      cur.push_back(x);
    }
    for (int i = 0; i < q; ++i) {
      L p0 = 0.0L, p1 = 1.0L, sum = 0.0L;
      for (int k = 0; k < q; ++k) {
        sum += p1 * p1 / nk[k];
        const L p2 = cur[i] * p1 - b[k] * p0;
        p0 = p1;
        p1 = p2;
      }
      xs[q * (q - 1) / 2 + i] = (double)cur[i];
      ws[q * (q - 1) / 2 + i] = (double)(1.0L / sum);
    }
    prev = cur;
  }
}

static vie_status upload_gl_tables() {
  static std::mutex lock;
  static bool done[64] = {false};
  int dev = 0;
  VIE_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> hold(lock);
  if (dev < 64 && done[dev]) return VIE_OK;
  std::vector<double> xs(kMaxGL * (kMaxGL + 1) / 2), ws(xs.size()), xt(xs.size()), wt(xs.size());
  for (int q = 1; q <= kMaxGL; ++q) legendre_nodes(q, &xs[q * (q - 1) / 2], &ws[q * (q - 1) / 2]);
  tent_gauss_rules(xt.data(), wt.data());
  VIE_CUDA_TRY(cudaMemcpyToSymbol(c_gl_x, xs.data(), xs.size() * sizeof(double)));
  VIE_CUDA_TRY(cudaMemcpyToSymbol(c_gl_w, ws.data(), ws.size() * sizeof(double)));
  VIE_CUDA_TRY(cudaMemcpyToSymbol(c_tg_x, xt.data(), xt.size() * sizeof(double)));
  VIE_CUDA_TRY(cudaMemcpyToSymbol(c_tg_w, wt.data(), wt.size() * sizeof(double)));
  VIE_CUDA_TRY(cudaDeviceSynchronize());
  if (dev < 64) done[dev] = true;
  return VIE_OK;
}

// Order of the tent rule for an offset at Chebyshev distance `cheb`: the
// larger of two lower limits.  (1) The kernel's pole: the error falls like
// rho^(-2q) with rho about 2 (cheb - 1); the table is the smallest order
// whose error against a 20-point split rule in extended precision is below
// 2e-16 of the largest component (checked on axis, face, diagonal and skew
// offsets).  (2) The oscillation exp(-j kappa t): about kappa^(2q) / ((2q)!
// 2^(2q-1)), kept below 1e-16 (q_osc, set on the host, at most 16, where a
// voxel is longer than a wavelength).  The previous rule, Gauss-Legendre on
// each of the 8 unit cells, took 8 x 6^3 = 1728 points where this one takes
// 5^3 = 125.
__host__ __device__ inline int tent_order(int cheb, int q_osc) {
  const int q = cheb <= 2 ? 21 : cheb == 3 ? 14 : cheb == 4 ? 12 : cheb == 5 ? 10 : cheb <= 7 ? 9
              : cheb <= 9 ? 8 : cheb <= 13 ? 7 : cheb <= 29 ? 6 : 5;
  return q > q_osc ? q : q_osc;
}

static int oscillation_order(double kappa) {
  double term = 2.0;   // kappa^(2q) / ((2q)! 2^(2q-1)) at q = 0
  for (int q = 1; q <= 16; ++q) {
    term *= kappa * kappa / (4.0 * (2.0 * q - 1.0) * (2.0 * q));
    if (term <= 1e-16) return q;
  }
  return 16;
}

constexpr int kQNear = 16;

__device__ __forceinline__ double tent(double t) { return fmax(0.0, 1.0 - fabs(t)); }
__device__ __forceinline__ double sgn1(double t) { return fabs(t) < 1.0 ? (t > 0.0 ? 1.0 : (t < 0.0 ? -1.0 : 0.0)) : 0.0; }

// g(r) * w as (re, im)
__device__ __forceinline__ double2 green_w(double r, double kappa, double w) {
  double s, c;
  sincos(kappa * r, &s, &c);
  const double f = w / (4.0 * M_PI * r);
  return make_double2(c * f, -s * f);
}

// ---------------------------------------------------------------------------
// near offsets: one block per D in {0,1}^3
// ---------------------------------------------------------------------------
// accumulator slots: 0 V, 1 xy, 2 xz, 3 yz, 4 + 3p + (dt+1) F_p(D_p + dt)
constexpr int kNearAcc = 13;

__device__ void block_reduce_acc(double2* acc, double* red, int tid, int nth) {
  // warp reduce then shared reduce; red has (nth/32) * 2 * kNearAcc doubles
  const int lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
  for (int k = 0; k < kNearAcc; ++k) {
    double re = acc[k].x, im = acc[k].y;
    for (int o = 16; o > 0; o >>= 1) {
      re += __shfl_down_sync(0xffffffffu, re, o);
      im += __shfl_down_sync(0xffffffffu, im, o);
    }
    if (lane == 0) { red[(warp * kNearAcc + k) * 2] = re; red[(warp * kNearAcc + k) * 2 + 1] = im; }
  }
  __syncthreads();
  if (tid < kNearAcc) {
    double re = 0.0, im = 0.0;
    for (int w = 0; w < nw; ++w) { re += red[(w * kNearAcc + tid) * 2]; im += red[(w * kNearAcc + tid) * 2 + 1]; }
    red[(nw * kNearAcc + tid) * 2] = re;
    red[(nw * kNearAcc + tid) * 2 + 1] = im;
  }
  __syncthreads();
}

// Grid (8, kNearParts): block (D, part) sums part `part` of the integrals of
// offset D = (b & 1, (b >> 1) & 1, (b >> 2) & 1) into partial[D][part][slot].
// Parts 0 .. 8 kNearChunks - 1: one unit cell of the volume and one node of
// the first coordinate each; the rest: the nine planes.  CURL: the three
// volume integrals of C_a instead (no planes).  FP64-bound (an SM retires
// about two FP64 operations a clock), so the work is spread over all SMs:
// with one block per D this took 2.7 ms, 8 SMs busy; now 0.22 ms.
constexpr int kNearChunks = kQNear;
constexpr int kNearParts = 8 * kNearChunks + 9;

template <bool CURL>
__global__ void __launch_bounds__(128) near_part_kernel(double2* __restrict__ partial, int nx, int ny, int nz,
                                                        double kappa) {
  const int b = blockIdx.x, part = blockIdx.y;
  const int D[3] = {b & 1, (b >> 1) & 1, (b >> 2) & 1};
  if (D[0] >= nx || D[1] >= ny || D[2] >= nz) return;
  const int tid = threadIdx.x, nth = blockDim.x;
  constexpr int q = kQNear, q2 = q * q;
  const double* X = c_gl_x + q * (q - 1) / 2;
  const double* W = c_gl_w + q * (q - 1) / 2;
  double2 acc[kNearAcc];
#pragma unroll
  for (int k = 0; k < kNearAcc; ++k) acc[k] = make_double2(0.0, 0.0);
  if (part < 8 * kNearChunks) {
    // ---- one of the 8 unit cells covering [D-1, D+1]^3, first node i
    const int cell = part / kNearChunks, i = part - cell * kNearChunks;
    const int c0[3] = {D[0] - 1 + (cell & 1), D[1] - 1 + ((cell >> 1) & 1), D[2] - 1 + ((cell >> 2) & 1)};
    const bool duffy = (c0[0] == 0 || c0[0] == -1) && (c0[1] == 0 || c0[1] == -1) && (c0[2] == 0 || c0[2] == -1);
    const int npts = duffy ? 3 * q2 : q2;
    for (int pt = tid; pt < npts; pt += nth) {
      const int a = pt / q2, rest = pt - a * q2;
      const int j = rest / q, k = rest - j * q;
      double v[3], w;
      if (duffy) {
        const double t = X[i], uj = t * X[j], uk = t * X[k];
        const double u0 = a == 0 ? t : a == 1 ? uk : uj;      // u[a] = t, u[a + 1] = t X_j, u[a + 2] = t X_k
        const double u1 = a == 0 ? uj : a == 1 ? t : uk;
        const double u2 = a == 0 ? uk : a == 1 ? uj : t;
        v[0] = (c0[0] == -1) ? -u0 : u0;
        v[1] = (c0[1] == -1) ? -u1 : u1;
        v[2] = (c0[2] == -1) ? -u2 : u2;
        w = W[i] * W[j] * W[k] * t * t;
      } else {
        v[0] = c0[0] + X[i]; v[1] = c0[1] + X[j]; v[2] = c0[2] + X[k];
        w = W[i] * W[j] * W[k];
      }
      const double r = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
      const double2 g = green_w(r, kappa, w);
      const double rx = v[0] - D[0], ry = v[1] - D[1], rz = v[2] - D[2];
      const double Lx = tent(rx), Ly = tent(ry), Lz = tent(rz);
      const double Sx = sgn1(rx), Sy = sgn1(ry), Sz = sgn1(rz);
      const double f[4] = {CURL ? Sx * Ly * Lz : Lx * Ly * Lz, CURL ? Lx * Sy * Lz : Sx * Sy * Lz,
                           CURL ? Lx * Ly * Sz : Sx * Sz * Ly, CURL ? 0.0 : Sy * Sz * Lx};
#pragma unroll
      for (int s = 0; s < 4; ++s) { acc[s].x += g.x * f[s]; acc[s].y += g.y * f[s]; }
    }
  } else if (!CURL) {
    // ---- plane integral F_p(D_p + dt) over 4 unit squares
    const int pl = part - 8 * kNearChunks, p = pl / 3, dt = pl - 3 * p - 1;
    const int a = (p + 1) % 3, bb = (p + 2) % 3;
    const int tp = D[p] + dt;
    double2 sum = make_double2(0.0, 0.0);
    for (int sq = 0; sq < 4; ++sq) {
      const int ca = D[a] - 1 + (sq & 1), cb = D[bb] - 1 + ((sq >> 1) & 1);
      const bool duffy = (tp == 0) && (ca == 0 || ca == -1) && (cb == 0 || cb == -1);
      const int npts = duffy ? 2 * q2 : q2;
      for (int pt = tid; pt < npts; pt += nth) {
        const int tri = pt / q2, rest = pt - tri * q2;
        const int i = rest / q, j = rest - i * q;
        double va, vb, w;
        if (duffy) {
          const double t = X[i];
          double u0 = tri == 0 ? t : t * X[j];
          double u1 = tri == 0 ? t * X[j] : t;
          va = (ca == -1) ? -u0 : u0;
          vb = (cb == -1) ? -u1 : u1;
          w = W[i] * W[j] * t;
        } else {
          va = ca + X[i];
          vb = cb + X[j];
          w = W[i] * W[j];
        }
        const double r = sqrt((double)tp * tp + va * va + vb * vb);
        const double2 g = green_w(r, kappa, w * tent(va - D[a]) * tent(vb - D[bb]));
        sum.x += g.x;
        sum.y += g.y;
      }
    }
#pragma unroll
    for (int s = 4; s < kNearAcc; ++s)
      if (s == 4 + pl) acc[s] = sum;
  }
  extern __shared__ double red[];
  block_reduce_acc(acc, red, tid, nth);
  if (tid < kNearAcc)
    partial[((size_t)b * kNearParts + part) * kNearAcc + tid] =
        make_double2(red[((nth >> 5) * kNearAcc + tid) * 2], red[((nth >> 5) * kNearAcc + tid) * 2 + 1]);
}

// Sum of the parts (fixed order) and the entries of the eight near offsets.
template <bool CURL>
__global__ void near_finish_kernel(const double2* __restrict__ partial, double2* __restrict__ T, int nx, int ny,
                                   int nz, double kappa) {
  const int b = blockIdx.x;
  const int D[3] = {b & 1, (b >> 1) & 1, (b >> 2) & 1};
  if (D[0] >= nx || D[1] >= ny || D[2] >= nz) return;
  __shared__ double2 R[kNearAcc];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < kNearAcc) {
    double re = 0.0, im = 0.0;
    for (int k = lane; k < kNearParts; k += 32) {
      const double2 v = partial[((size_t)b * kNearParts + k) * kNearAcc + warp];
      re += v.x;
      im += v.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
      re += __shfl_down_sync(0xffffffffu, re, o);
      im += __shfl_down_sync(0xffffffffu, im, o);
    }
    if (lane == 0) R[warp] = make_double2(re, im);
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  const size_t N = (size_t)nx * ny * nz;
  const size_t vox = ((size_t)D[2] * ny + D[1]) * nx + D[0];
  const bool self = b == 0;
  if (CURL) {
    for (int a = 0; a < 3; ++a) T[a * N + vox] = self ? make_double2(0.0, 0.0) : R[a];
    return;
  }
  const double2 V = R[0];
  const double k2 = kappa * kappa;
  for (int p = 0; p < 3; ++p) {
    const double2* F = R + 4 + 3 * p;
    T[p * N + vox] = make_double2((self ? 1.0 : 0.0) + k2 * V.x + F[2].x - 2.0 * F[1].x + F[0].x,
                                  k2 * V.y + F[2].y - 2.0 * F[1].y + F[0].y);
  }
  for (int c = 0; c < 3; ++c) T[(3 + c) * N + vox] = R[1 + c];
}

// ---------------------------------------------------------------------------
// far offsets, |D|_inf >= 2: tensor tent rule of the closed-form kernels
//   T: e^{-j kr} / (4 pi r^3) [ (k^2 r^2 - 1 - j kr) d_pq + (3 + 3 j kr - k^2 r^2) v_p v_q / r^2 ]
//   C: -(1 + j kr) e^{-j kr} v_a / (4 pi r^3)
// The phase at the offset itself is taken out, e^{-j kr} = e^{-j kr0}
// e^{-j k (r - r0)} with |r - r0| <= sqrt 3, so that for k sqrt 3 <= 1/4 the
// points need only the Taylor series of sine and cosine on [-1/4, 1/4] (next
// terms 3e-18 and 4e-20); larger k calls sincos.
// ---------------------------------------------------------------------------
template <bool SMALLK>
__device__ __forceinline__ void phase(double d, double* s, double* c) {
  if (SMALLK) {
    const double x = d * d;
    *s = d * fma(x, fma(x, fma(x, fma(x, fma(x, -1.0 / 39916800.0, 1.0 / 362880.0), -1.0 / 5040.0), 1.0 / 120.0),
                        -1.0 / 6.0), 1.0);
    *c = fma(x, fma(x, fma(x, fma(x, fma(x, fma(x, 1.0 / 479001600.0, -1.0 / 3628800.0), 1.0 / 40320.0),
                                  -1.0 / 720.0), 1.0 / 24.0), -0.5), 1.0);
  } else {
    sincos(d, s, c);
  }
}

// One z line of the rule: the moments over z of the kernel's two factors.
// T: P (delta part) and Q v_z^m, m = 0..2; C: G v_z^m, m = 0, 1.
struct FarLine {
  double p0x, p0y, q0x, q0y, q1x, q1y, q2x, q2y;
};
template <bool SMALLK, bool CURL>
__device__ __forceinline__ void far_point(FarLine& L, double rho2, double vz, double w, double kappa, double kr0) {
  const double r2 = fma(vz, vz, rho2);
  const double ri = rsqrt(r2);
  const double kr = kappa * (r2 * ri);
  double s, c;
  phase<SMALLK>(kr - kr0, &s, &c);
  const double ri2 = ri * ri;
  const double f = w * (ri2 * ri);
  const double er = c * f, ei = -s * f;
  if (CURL) {
    const double gx = fma(kr, ei, -er), gy = -fma(kr, er, ei);   // -(1 + j kr)(er + j ei)
    L.q0x += gx;
    L.q0y += gy;
    L.q1x = fma(gx, vz, L.q1x);
    L.q1y = fma(gy, vz, L.q1y);
  } else {
    const double k2r2 = kr * kr, ar = k2r2 - 1.0, br = 3.0 - k2r2, bi = 3.0 * kr;
    L.p0x += fma(ar, er, kr * ei);          // (ar - j kr)(er + j ei)
    L.p0y += fma(ar, ei, -kr * er);
    const double qx = fma(br, er, -bi * ei) * ri2, qy = fma(br, ei, bi * er) * ri2;
    L.q0x += qx;
    L.q0y += qy;
    const double q1x = qx * vz, q1y = qy * vz;
    L.q1x += q1x;
    L.q1y += q1y;
    L.q2x = fma(q1x, vz, L.q2x);
    L.q2y = fma(q1y, vz, L.q2y);
  }
}

// acc += wxy * (a line's moments combined with v_x, v_y); T: xx yy zz xy xz yz, C: x y z
template <bool CURL>
__device__ __forceinline__ void far_line_add(double2 (&acc)[6], const FarLine& L, double vx, double vy, double wxy) {
  auto put = [&](int k, double x, double y) { acc[k].x = fma(wxy, x, acc[k].x); acc[k].y = fma(wxy, y, acc[k].y); };
  if (CURL) {
    put(0, vx * L.q0x, vx * L.q0y);
    put(1, vy * L.q0x, vy * L.q0y);
    put(2, L.q1x, L.q1y);
  } else {
    const double xx = vx * vx, yy = vy * vy, xy = vx * vy;
    put(0, fma(xx, L.q0x, L.p0x), fma(xx, L.q0y, L.p0y));
    put(1, fma(yy, L.q0x, L.p0x), fma(yy, L.q0y, L.p0y));
    put(2, L.q2x + L.p0x, L.q2y + L.p0y);
    put(3, xy * L.q0x, xy * L.q0y);
    put(4, vx * L.q1x, vx * L.q1y);
    put(5, vy * L.q1x, vy * L.q1y);
  }
}

// acc times e^{-j kr0} / (4 pi) to the table
template <bool CURL>
__device__ __forceinline__ void far_store(const double2 (&acc)[6], double kr0, double2* __restrict__ T, size_t N,
                                          size_t vox) {
  double s, c;
  sincos(kr0, &s, &c);
  c *= 1.0 / (4.0 * M_PI);
  s *= 1.0 / (4.0 * M_PI);
#pragma unroll
  for (int k = 0; k < (CURL ? 3 : 6); ++k)
    T[k * N + vox] = make_double2(fma(acc[k].x, c, acc[k].y * s), fma(acc[k].y, c, -acc[k].x * s));
}

// Offsets below kFarThread: high orders and few offsets, one block each, the
// (x, y) lines of the rule over its threads.  From kFarThread on: one thread
// per offset, no reduction, nodes read uniformly from constant memory.
constexpr int kFarThread = 10;

template <bool SMALLK, bool CURL>
__global__ void __launch_bounds__(128) far_block_kernel(double2* __restrict__ T, int nx, int ny, int nz, int bx,
                                                        int by, double kappa, int q_osc) {
  const int dx = blockIdx.x % bx, dy = (blockIdx.x / bx) % by, dz = blockIdx.x / (bx * by);
  const int cheb = max(dx, max(dy, dz));
  if (cheb <= 1) return;
  const int q = tent_order(cheb, q_osc);
  const double* X = c_tg_x + q * (q - 1) / 2;
  const double* W = c_tg_w + q * (q - 1) / 2;
  const double kr0 = kappa * sqrt((double)(dx * dx + dy * dy + dz * dz));
  double2 acc[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) acc[k] = make_double2(0.0, 0.0);
  for (int l = threadIdx.x; l < q * q; l += blockDim.x) {
    const int i = l / q, j = l - i * q;
    const double vx = dx + X[i], vy = dy + X[j], rho2 = fma(vx, vx, vy * vy);
    FarLine L = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int k = 0; k < q; ++k) far_point<SMALLK, CURL>(L, rho2, dz + X[k], W[k], kappa, kr0);
    far_line_add<CURL>(acc, L, vx, vy, W[i] * W[j]);
  }
  __shared__ double2 red[4][6];
#pragma unroll
  for (int k = 0; k < (CURL ? 3 : 6); ++k) {
    for (int o = 16; o > 0; o >>= 1) {
      acc[k].x += __shfl_down_sync(0xffffffffu, acc[k].x, o);
      acc[k].y += __shfl_down_sync(0xffffffffu, acc[k].y, o);
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][k] = acc[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      acc[k] = make_double2(0.0, 0.0);
      if (k < (CURL ? 3 : 6))
        for (int w = 0; w < 4; ++w) { acc[k].x += red[w][k].x; acc[k].y += red[w][k].y; }
    }
    far_store<CURL>(acc, kr0, T, (size_t)nx * ny * nz, ((size_t)dz * ny + dy) * nx + dx);
  }
}

// FP64-bound: about 58 operations a point.  600 x 23 x 11 offsets at kappa =
// 0.117: 2.9 ms (before, one warp per offset over 8 cells: 67.7 ms).
template <bool SMALLK, bool CURL>
__global__ void __launch_bounds__(128) far_thread_kernel(double2* __restrict__ T, int nx, int ny, int nz,
                                                         double kappa, int q_osc) {
  const size_t N = (size_t)nx * ny * nz;
  const size_t vox = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (vox >= N) return;
  const int dx = (int)(vox % nx), dy = (int)((vox / nx) % ny), dz = (int)(vox / ((size_t)nx * ny));
  const int cheb = max(dx, max(dy, dz));
  if (cheb < kFarThread) return;
  const int q = tent_order(cheb, q_osc);
  const double* X = c_tg_x + q * (q - 1) / 2;
  const double* W = c_tg_w + q * (q - 1) / 2;
  const double kr0 = kappa * sqrt((double)dx * dx + (double)dy * dy + (double)dz * dz);
  double2 acc[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) acc[k] = make_double2(0.0, 0.0);
  for (int i = 0; i < q; ++i) {
    const double vx = dx + X[i];
    for (int j = 0; j < q; ++j) {
      const double vy = dy + X[j], rho2 = fma(vx, vx, vy * vy);
      FarLine L = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
      for (int k = 0; k < q; ++k) far_point<SMALLK, CURL>(L, rho2, dz + X[k], W[k], kappa, kr0);
      far_line_add<CURL>(acc, L, vx, vy, W[i] * W[j]);
    }
  }
  far_store<CURL>(acc, kr0, T, N, vox);
}

template <bool SMALLK, bool CURL>
static vie_status launch_far(double2* T, const int n[3], double kappa, cudaStream_t s) {
  const size_t N = (size_t)n[0] * n[1] * n[2];
  const int q_osc = oscillation_order(kappa);
  const int bx = n[0] < kFarThread ? n[0] : kFarThread, by = n[1] < kFarThread ? n[1] : kFarThread;
  const int bz = n[2] < kFarThread ? n[2] : kFarThread;
  far_block_kernel<SMALLK, CURL><<<bx * by * bz, 128, 0, s>>>(T, n[0], n[1], n[2], bx, by, kappa, q_osc);
  VIE_LAUNCH_CHECK();
  if (n[0] > kFarThread || n[1] > kFarThread || n[2] > kFarThread) {
    far_thread_kernel<SMALLK, CURL><<<(unsigned)((N + 127) / 128), 128, 0, s>>>(T, n[0], n[1], n[2], kappa, q_osc);
    VIE_LAUNCH_CHECK();
  }
  return VIE_OK;
}

// Every entry of T (six tables) or C (three) on stream s.
template <bool CURL>
static vie_status launch_entries(double2* T, const int n[3], double kappa, cudaStream_t s) {
  vie_status st = kappa * 1.7320508075688772 <= 0.25 ? launch_far<true, CURL>(T, n, kappa, s)
                                                     : launch_far<false, CURL>(T, n, kappa, s);
  if (st != VIE_OK) return st;
  double2* partial = nullptr;
  VIE_CUDA_TRY(cudaMallocAsync((void**)&partial, (size_t)8 * kNearParts * kNearAcc * sizeof(double2), s));
  const size_t smem = (size_t)(128 / 32 + 1) * kNearAcc * 2 * sizeof(double);
  near_part_kernel<CURL><<<dim3(8, kNearParts), 128, smem, s>>>(partial, n[0], n[1], n[2], kappa);
  near_finish_kernel<CURL><<<8, 32 * kNearAcc, 0, s>>>(partial, T, n[0], n[1], n[2], kappa);
  const cudaError_t launch = cudaGetLastError();
  const cudaError_t freed = cudaFreeAsync(partial, s);
  VIE_CUDA_TRY(launch);
  VIE_CUDA_TRY(freed);
  return VIE_OK;
}

// ---------------------------------------------------------------------------
// Spectra of the circulant embedding.  Along each axis the embedded table is
// even or odd (index m holds Delta = m for m < n and the mirrored value for
// m > M - n; the gap is zero), so its transform is too, and the transforms of
// the other axes act line by line: only the octant is ever formed.  Three
// passes, each embedding its own axis in shared memory:
//   x: lines (c, z, y) of nx entries       -> F1[c][z][y][kx], kx <= Mx / 2
//   y: lines (c, z, kx) of ny values       -> F2[c][kx][z][ky], ky <= My / 2
//   z: lines (c, kx, ky) of nz values      -> spectrum [kx][c][kz][ky], kz <= Mz / 2,
//      scaled by 1 / (Mx My Mz), in complex128 and complex64
// A quarter of the FP64 transforms that the whole embedding takes, and no
// buffer of its 6 Mx My Mz values (600 x 23 x 11: 1.73 -> 0.38 ms).
// ---------------------------------------------------------------------------
struct SpecGeom {
  int n[3], m[3], k[3];
  int ncomp;
  unsigned odd[3];   // per axis: bit c set when component c is odd along it
};

// value of index m of an embedded line of n values
__device__ __forceinline__ double2 embedded(const double2* __restrict__ v, long long stride, int m, int n, int M,
                                            bool odd) {
  if (m < n) return v[m * stride];
  if (m <= M - n) return make_double2(0.0, 0.0);
  const double2 t = v[(M - m) * stride];
  return odd ? make_double2(-t.x, -t.y) : t;
}

// AXIS 0: block = tl lines of the n2 n1 ncomp x lines.  AXIS 1: block = tl
// consecutive kx of one (c, z).  AXIS 2: block = tl consecutive ky of one
// (c, kx).
template <int AXIS>
__global__ void __launch_bounds__(256) spectrum_axis_kernel(const double2* __restrict__ in, double2* __restrict__ out,
                                                            double2* __restrict__ g64, float2* __restrict__ g32,
                                                            SpecGeom g, Radices rd, const double2* __restrict__ twg,
                                                            int tl, double scale_) {
  extern __shared__ double2 sm64[];
  const int L = rd.len, pitch = L + 1, K = g.k[AXIS], n = g.n[AXIS];
  double2* tw = sm64;
  double2* A = tw + L;
  double2* B = A + (size_t)tl * pitch;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int per = AXIS == 0 ? g.ncomp * g.n[1] * g.n[2] : AXIS == 1 ? g.k[0] : g.k[1];   // lines of one group
  const int blocks_per = (per + tl - 1) / tl;
  const int grp = blockIdx.x / blocks_per;          // AXIS 1: c nz + z; AXIS 2: c Kx + kx
  const int l0 = (blockIdx.x - grp * blocks_per) * tl;
  const int nl = min(tl, per - l0);
  for (int i = tid; i < L; i += nth) tw[i] = twg[i];
  for (int e = tid; e < nl * L; e += nth) {
    int l, m;
    double2 v;
    if (AXIS == 0) {
      l = e / L;
      m = e - l * L;
      const int c = (l0 + l) / (g.n[1] * g.n[2]);
      v = embedded(in + (size_t)(l0 + l) * n, 1, m, n, L, g.odd[0] >> c & 1);
    } else if (AXIS == 1) {
      m = e / nl;
      l = e - m * nl;
      const int c = grp / g.n[2];
      v = embedded(in + (size_t)grp * g.n[1] * g.k[0] + l0 + l, g.k[0], m, n, L, g.odd[1] >> c & 1);
    } else {
      m = e / nl;
      l = e - m * nl;
      const int c = grp / g.k[0];
      v = embedded(in + (size_t)grp * g.n[2] * g.k[1] + l0 + l, g.k[1], m, n, L, g.odd[2] >> c & 1);
    }
    A[l * pitch + m] = v;
  }
  __syncthreads();
  const double2* res = fft_lines<double2, false>(A, B, rd, pitch, nl, tw, tid, nth);
  for (int e = tid; e < nl * K; e += nth) {
    if (AXIS == 0) {
      const int l = e / K, k = e - l * K;
      out[(size_t)(l0 + l) * K + k] = res[l * pitch + k];
    } else if (AXIS == 1) {
      const int l = e / K, k = e - l * K;
      const int c = grp / g.n[2], z = grp - c * g.n[2];
      out[(((size_t)c * g.k[0] + l0 + l) * g.n[2] + z) * K + k] = res[l * pitch + k];
    } else {
      const int k = e / nl, l = e - k * nl;
      const int c = grp / g.k[0], kx = grp - c * g.k[0];
      double2 v = res[l * pitch + k];
      v.x *= scale_;
      v.y *= scale_;
      const size_t o = (((size_t)kx * g.ncomp + c) * K + k) * g.k[1] + l0 + l;
      g64[o] = v;
      g32[o] = make_float2((float)v.x, (float)v.y);
    }
  }
}

template <int AXIS>
static vie_status launch_spectrum_axis(const double2* in, double2* out, double2* g64, float2* g32, const SpecGeom& g,
                                       const AxisPlan& ax, double scale_, cudaStream_t s) {
  const int L = ax.len;
  const size_t per_line = (size_t)2 * (L + 1) * sizeof(double2);
  const size_t tw_bytes = (size_t)L * sizeof(double2);
  const size_t budget = 200 * 1024;
  if (tw_bytes + per_line > budget) {
    set_error("FFT length %d too large for the setup transform", L);
    return VIE_ERR_INVALID;
  }
  const int per = AXIS == 0 ? g.ncomp * g.n[1] * g.n[2] : AXIS == 1 ? g.k[0] : g.k[1];
  const long long groups = AXIS == 0 ? 1 : AXIS == 1 ? (long long)g.ncomp * g.n[2] : (long long)g.ncomp * g.k[0];
  // lines per block: up to 16 while two blocks fit an SM (FP64-bound, so
  // occupancy beyond that buys nothing), at least one
  int tl = 16;
  while (tl > 1 && tw_bytes + (size_t)tl * per_line > 100 * 1024) tl >>= 1;
  const size_t smem = tw_bytes + (size_t)tl * per_line;
  VIE_CUDA_TRY(allow_shared(spectrum_axis_kernel<AXIS>, smem));
  const long long blocks = groups * ((per + tl - 1) / tl);
  spectrum_axis_kernel<AXIS><<<(unsigned)blocks, 256, smem, s>>>(in, out, g64, g32, g, radices_of(ax), ax.tw64, tl,
                                                               scale_);
  VIE_LAUNCH_CHECK();
  return VIE_OK;
}

static vie_status folded_spectra(const vie_plan* p, const double2* table, int ncomp, const unsigned odd[3],
                                 double2* g64, float2* g32, cudaStream_t s) {
  SpecGeom g;
  for (int a = 0; a < 3; ++a) {
    g.n[a] = p->n[a];
    g.m[a] = p->m[a];
    g.k[a] = p->kf[a];
    g.odd[a] = odd[a];
  }
  g.ncomp = ncomp;
  const size_t f1 = (size_t)ncomp * g.n[2] * g.n[1] * g.k[0], f2 = (size_t)ncomp * g.k[0] * g.n[2] * g.k[1];
  double2* buf = nullptr;
  VIE_CUDA_TRY(cudaMallocAsync((void**)&buf, (f1 + f2) * sizeof(double2), s));
  const double scale_ = 1.0 / ((double)g.m[0] * g.m[1] * g.m[2]);
  vie_status st = launch_spectrum_axis<0>(table, buf, nullptr, nullptr, g, p->ax[0], 1.0, s);
  if (st == VIE_OK) st = launch_spectrum_axis<1>(buf, buf + f1, nullptr, nullptr, g, p->ax[1], 1.0, s);
  if (st == VIE_OK) st = launch_spectrum_axis<2>(buf + f1, nullptr, g64, g32, g, p->ax[2], scale_, s);
  const cudaError_t e = cudaFreeAsync(buf, s);
  if (st == VIE_OK && e != cudaSuccess) { set_error("cudaFreeAsync: %s", cudaGetErrorString(e)); st = VIE_ERR_CUDA; }
  return st;
}

// ---------------------------------------------------------------------------
// host drivers
// ---------------------------------------------------------------------------
vie_status compute_toeplitz(vie_plan* p, cudaStream_t s) {
  vie_status st = upload_gl_tables();
  if (st != VIE_OK) return st;
  return launch_entries<false>(p->toeplitz, p->n, p->kappa, s);
}

vie_status compute_spectrum(vie_plan* p, cudaStream_t s) {
  // xy is odd in x and y, xz in x and z, yz in y and z
  const unsigned odd[3] = {1u << 3 | 1u << 4, 1u << 3 | 1u << 5, 1u << 4 | 1u << 5};
  return folded_spectra(p, p->toeplitz, 6, odd, p->ghat64, p->ghat32, s);
}

// ---------------------------------------------------------------------------
// JM-VIE (Sec. 3): Galerkin entries of the scalar derivatives of S, in units
// of h, C_a(D) = <P_i, d_a S P_j> / h = int (d_a g)(v) L_D(v) dv; the curl
// operator K = curl S has K_pq(D) = h eps_paq C_a(D).  C_a is odd in D_a and
// even in the other two offsets, C_a(0) = 0.  As for T:
//   * |D|_inf >= 2: d_a g in closed form, -g (1 + j kappa r) v_a / r^2, by the
//     tent rule;
//   * |D|_inf = 1: by parts on the tent, C_a = int g sign(v_a - D_a)
//     L(v_b - D_b) L(v_c - D_c) dv, Duffy cells where the origin is a corner.
// Stored like T: octant [a][z][y][x] for D in [0, n); spectra folded to the
// octant [kx'][a][kz'][ky'].
// ---------------------------------------------------------------------------
vie_status compute_curl(vie_plan* p, cudaStream_t s) {
  vie_status st = upload_gl_tables();
  if (st == VIE_OK) st = launch_entries<true>(p->curl, p->n, p->kappa, s);
  const unsigned odd[3] = {1u, 2u, 4u};
  if (st == VIE_OK) st = folded_spectra(p, p->curl, 3, odd, p->chat64, p->chat32, s);
  return st;
}

}  // namespace vie
