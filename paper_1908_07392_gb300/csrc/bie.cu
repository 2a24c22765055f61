// Boundary integral equation of the homogeneous modified Stokes problem and its GMRES solver.
//
// Sec. 2.2 (Eqs. uH_dbl, dbl_lyr_pot, dbl_lyr_ker, BIE): u^H = D[mu] with the double-layer kernel
// D_ij(x, y) = -T_jik(x - y) n_k(y), n the unit normal pointing into the domain, and the density
// solves 1/2 mu + D[mu] + W[mu] = g on the boundary, W[mu](x) = n(x) / |boundary| * int mu.n ds.
// The stresslet T is the closed form of App. B (Eq. app_stresslet with T1, T2, T3), evaluated by the
// power series of App. C for small alpha r; the stokeslet S (Eq. app_stokeslet) gives exact solutions
// for tests. Discretisation (Sec. 3.2, Eq. BIE_quad): the boundary is a star r(t) = R + A cos(k t + phi),
// split into n_panels equal parameter panels with 16 Gauss-Legendre nodes each (Nystrom). Entries
// for source panels adjacent to (or containing) the target use a locally graded quadrature: the
// panel is cut at the target (self panel) or toward the nearer end (neighbours) into geometrically
// shrinking pieces with 12-point Gauss-Legendre each, the density interpolated by the panel's
// Lagrange basis; this integrates the r log r terms of the kernel (which make plain Gauss-Legendre
// converge slowly, Sec. 4.1) to full precision. The coincident-point limit of the kernel is
// kappa t t / (2 pi) (Sec. 4.2).
// The dense FP64 system (2N x 2N) is solved by GMRES with classical Gram-Schmidt applied twice.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <memory>
#include <new>
#include <vector>

#include "special.cuh"
#include "stokes.cuh"
#include "vp_internal.h"
#include "../../include/bie.h"

namespace vp {
namespace {

#define TRY(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { set_last_cuda(e_); return e_ == cudaErrorMemoryAllocation ? VP_ERR_OOM : VP_ERR_CUDA; } } while (0)

constexpr int kPP = 16;        // nodes per panel
constexpr int kGradeN = 12;    // nodes per graded piece
constexpr int kGradeLevels = 36;

__constant__ double c_glx16[kPP], c_glw16[kPP], c_glx12[kGradeN], c_glw12[kGradeN], c_bw16[kPP];

struct Star { double R, A, phase; int k; };

__device__ inline void star_geom(const Star& s, double t, double& x, double& y, double& dx, double& dy,
                                 double& ddx, double& ddy) {
  const double c = cos(t), sn = sin(t);
  const double r = s.R + s.A * cos(s.k * t + s.phase);
  const double dr = -s.A * s.k * sin(s.k * t + s.phase);
  const double d2r = -s.A * s.k * s.k * cos(s.k * t + s.phase);
  x = r * c; y = r * sn;
  dx = dr * c - r * sn; dy = dr * sn + r * c;
  ddx = d2r * c - 2.0 * dr * sn - r * c;
  ddy = d2r * sn + 2.0 * dr * c - r * sn;
}

__device__ inline double lag16(double tau, int j) {
  double num = 0.0, den = 0.0;
  for (int m = 0; m < kPP; ++m) {
    const double d = tau - c_glx16[m];
    if (d == 0.0) return m == j ? 1.0 : 0.0;
    const double w = c_bw16[m] / d;
    den += w;
    if (m == j) num = w;
  }
  return num / den;
}

struct Nodes {
  double *x, *y, *nx, *ny, *w, *kappa, *tx, *ty, *theta;
};

__global__ void k_nodes(Star s, int np, Nodes nd) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= np * kPP) return;
  const int p = j / kPP, q = j % kPP;
  const double h = 2.0 * kPi / np;
  const double t = (p + 0.5) * h + 0.5 * h * c_glx16[q];
  double x, y, dx, dy, ddx, ddy;
  star_geom(s, t, x, y, dx, dy, ddx, ddy);
  const double sp = sqrt(dx * dx + dy * dy);
  nd.x[j] = x; nd.y[j] = y;
  nd.tx[j] = dx / sp; nd.ty[j] = dy / sp;
  nd.nx[j] = -dy / sp; nd.ny[j] = dx / sp;  // counter-clockwise curve: left normal points inside
  nd.w[j] = sp * 0.5 * h * c_glw16[q];
  nd.kappa[j] = (dx * ddy - dy * ddx) / (sp * sp * sp);
  nd.theta[j] = t;
}

// Plain Nystrom entries (row-major [2N][2N]) with the W term and the coincident-point limit.
__global__ void k_matrix_plain(int N, double alpha, double Lb, Nodes nd, double* A) {
  const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= (long long)N * N) return;
  const int i = (int)(idx / N), j = (int)(idx % N);
  double D[4];
  if (i == j) {
    const double c = nd.kappa[j] / (2.0 * kPi);
    D[0] = c * nd.tx[j] * nd.tx[j]; D[1] = c * nd.tx[j] * nd.ty[j];
    D[2] = D[1]; D[3] = c * nd.ty[j] * nd.ty[j];
  } else {
    dl_kernel(alpha, nd.x[i] - nd.x[j], nd.y[i] - nd.y[j], nd.nx[j], nd.ny[j], D);
  }
  const double w = nd.w[j];
  const double ni[2] = {nd.nx[i], nd.ny[i]}, nj[2] = {nd.nx[j], nd.ny[j]};
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 2; ++b)
      A[(size_t)(2 * i + a) * (2 * N) + 2 * j + b] =
          (i == j && a == b ? 0.5 : 0.0) + D[2 * a + b] * w + ni[a] * nj[b] * w / Lb;
}

// Graded local quadrature: for target i and source panels p-1, p, p+1, the exact (to quadrature
// precision) integral of the kernel against each Lagrange basis function of the source panel.
__global__ void __launch_bounds__(128) k_matrix_local(int np, double alpha, double Lb, Star s, Nodes nd, double* A) {
  const int i = blockIdx.x;
  const int N = np * kPP;
  const int pi = i / kPP;
  const double h = 2.0 * kPi / np;
  const double ti = nd.theta[i];
  const double xi = nd.x[i], yi = nd.y[i];
  // accumulators: 3 panels x 16 basis x 4 components
  __shared__ double acc[3 * kPP * 4];
  for (int e = threadIdx.x; e < 3 * kPP * 4; e += blockDim.x) acc[e] = 0.0;
  __syncthreads();
  // pieces: for each of the 3 panels, 2 sides x (levels + 1) pieces, 12 nodes each
  const int pieces_per_side = kGradeLevels + 1;
  const int npts = 3 * 2 * pieces_per_side * kGradeN;
  for (int e = threadIdx.x; e < npts; e += blockDim.x) {
    const int pn = e / (2 * pieces_per_side * kGradeN);
    int rem = e % (2 * pieces_per_side * kGradeN);
    const int side = rem / (pieces_per_side * kGradeN);
    rem %= pieces_per_side * kGradeN;
    const int lev = rem / kGradeN, q = rem % kGradeN;
    const int p = (pi + pn - 1 + np) % np;
    // panel parameter interval, unwrapped next to the target's panel
    const double ta = (pi + pn - 1) * h, tb = ta + h;
    // grading point: the target (self panel) or the panel end nearest to it (neighbours)
    const double tc = (pn == 1) ? ti : (pn == 0 ? tb : ta);
    const double lo_end = side == 0 ? ta : tc, hi_end = side == 0 ? tc : tb;
    const double len = hi_end - lo_end;
    if (len <= 0.0) continue;
    // geometric pieces toward tc: side 0 grades toward hi_end = tc, side 1 toward lo_end = tc
    double u0, u1;  // fractions of len measured from tc
    if (lev == kGradeLevels) { u0 = 0.0; u1 = ldexp(1.0, -kGradeLevels); }
    else { u0 = ldexp(1.0, -lev - 1); u1 = ldexp(1.0, -lev); }
    const double fa = 0.5 * (u0 + u1) + 0.5 * (u1 - u0) * c_glx12[q];
    const double wq = 0.5 * (u1 - u0) * c_glw12[q] * len;
    const double t = (side == 0) ? (tc - fa * len) : (tc + fa * len);
    if (!(t > ta && t < tb) && !(t == ta || t == tb)) continue;
    double x, y, dx, dy, ddx, ddy;
    star_geom(s, t, x, y, dx, dy, ddx, ddy);
    const double sp = sqrt(dx * dx + dy * dy);
    const double nxq = -dy / sp, nyq = dx / sp;
    // x_i - y(t) from the parameter offset, free of cancellation:
    // z(ti) - z(t) = e^{i ti} [ (r(ti) - r(t)) + r(t) (1 - e^{i d}) ],  d = t - ti,
    // r(ti) - r(t) = 2 A sin(k (ti + t)/2 + phase) sin(k d / 2),  1 - e^{i d} = 2 sin^2(d/2) - i sin d
    const double d = (tc - ti) + ((side == 0) ? -fa * len : fa * len);
    const double rt = s.R + s.A * cos(s.k * t + s.phase);
    const double dR = 2.0 * s.A * sin(0.5 * s.k * (ti + t) + s.phase) * sin(0.5 * s.k * d);
    const double sh = sin(0.5 * d);
    const double re = dR + rt * 2.0 * sh * sh, im = -rt * sin(d);
    const double ct = cos(ti), st = sin(ti);
    const double rx = ct * re - st * im, ry = st * re + ct * im;
    if (rx == 0.0 && ry == 0.0) continue;
    (void)x; (void)y; (void)xi; (void)yi;
    double D[4];
    dl_kernel(alpha, rx, ry, nxq, nyq, D);
    const double tau = 2.0 * (t - ta) / h - 1.0;  // reference coordinate on the source panel
    for (int j = 0; j < kPP; ++j) {
      const double l = lag16(tau, j) * wq * sp;
      for (int c = 0; c < 4; ++c) atomicAdd(&acc[(pn * kPP + j) * 4 + c], D[c] * l);
    }
    (void)p;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 3 * kPP; e += blockDim.x) {
    const int pn = e / kPP, jj = e % kPP;
    const int p = (pi + pn - 1 + np) % np;
    const int j = p * kPP + jj;
    const double ni[2] = {nd.nx[i], nd.ny[i]}, nj[2] = {nd.nx[j], nd.ny[j]};
    for (int a = 0; a < 2; ++a)
      for (int b = 0; b < 2; ++b)
        A[(size_t)(2 * i + a) * (2 * N) + 2 * j + b] =
            (i == j && a == b ? 0.5 : 0.0) + acc[(pn * kPP + jj) * 4 + 2 * a + b] + ni[a] * nj[b] * nd.w[j] / Lb;
  }
}

// GMRES state on the device; every Krylov kernel returns at once when `done` is set, so the host
// can queue several iterations ahead and look at the state only once per group.
struct GmresCtl {
  double bnorm, res, hn;
  int done, it;
};

__device__ inline bool gm_done(const GmresCtl* c) { return c && *(volatile const int*)&c->done; }

// ------------------------------------------------------------------ y = A x in fixed point
//
// An FP64 multiply-add per entry takes longer than reading the entry: 67 M of them at 2 per clock and SM are 107 us
// for the 8192 x 8192 operator, whose 537 MB stream in 79 us at the measured copy rate. So the operator is kept as
// 63-bit integers (two balanced 32-bit digits in the 8 bytes of an entry, one exponent per row) and the vector is
// taken as 72-bit integers (three balanced 24-bit digits, one exponent): an entry takes five widening 32-bit
// multiply-adds into 64-bit sums, of which 128 stay below 2^62. The diagonal, 1/2 and far above the other
// entries, is kept in FP64 beside them. An entry down to 2^-9 of its row's largest, and a component down to 2^-18 of
// the vector's, keep all 53 bits; the error of an apply against extended precision is about half of the FP64
// form's (random, smooth, constant, wide-ranged and spiked vectors, 256 to 2560 unknowns, alpha 5 to 400).
// Measured (8192 unknowns): 83 us an apply = 6.4 TB/s, 0.95 of the measured copy rate; 127 us in FP64.

constexpr int kNotFinite = 1 << 28;  // exponent of a row or vector with an infinity or a NaN in it

__device__ inline int exponent_field(double x) {
  const int e = (int)((unsigned long long)__double_as_longlong(x) >> 52) & 0x7ff;
  return e ? e : 1;
}

__device__ inline unsigned long long mantissa(double x, int& ex) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  unsigned long long m = b & ((1ull << 52) - 1);
  ex = (int)((b >> 52) & 0x7ff);
  if (ex) m |= 1ull << 52;
  else ex = 1;
  return m;
}

__device__ inline unsigned long long shift_right_rn(unsigned long long m, int d) {
  return d <= 0 ? m : (d > 63 ? 0ull : (m >> d) + ((m >> (d - 1)) & 1ull));
}

// An entry as digits (low, high) in units of 2^(emax - 1084), emax the largest exponent field of the row.
__device__ inline int2 entry_digits(double x, int emax) {
  int ex;
  const unsigned long long m = mantissa(x, ex) << 9;
  const long long v = (long long)shift_right_rn(m, emax - ex), w = __double_as_longlong(x) < 0 ? -v : v;
  return make_int2((int)w, (int)(w >> 32) + (int)((unsigned)w >> 31));
}

// A component as digits (high, middle, low) in units of 2^(emax - 1093).
__device__ inline int3 component_digits(double x, int emax) {
  int ex;
  const unsigned long long m = mantissa(x, ex);
  const int sh = 18 - (emax - ex);
  const unsigned long long r = sh >= 0 ? m << sh : shift_right_rn(m, -sh);  // low 64 bits of the shifted value
  const int low = (int)(r & 0xffffff);
  long long up = (long long)(sh >= 0 ? m >> (24 - sh) : r >> 24);
  const int d2 = low - ((low & 0x800000) << 1);
  up += low >> 23;
  const int mid = (int)(up & 0xffffff), d1 = mid - ((mid & 0x800000) << 1);
  const int d0 = (int)(up >> 24) + (mid >> 23);
  return __double_as_longlong(x) < 0 ? make_int3(-d0, -d1, -d2) : make_int3(d0, d1, d2);
}

template <int OP_THREADS>
__device__ inline int block_max(int v, int* red) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  return __reduce_max_sync(0xffffffffu, lane < OP_THREADS / 32 ? red[lane] : red[0]);
}

// Row blockIdx.x of A in place: diagonal to diag, the rest to digits, the row's exponent to re.
__global__ void __launch_bounds__(256) k_matrix_digits(int n, double* A, double* diag, int* re) {
  __shared__ int red[8];
  const int row = blockIdx.x;
  double* a = A + (size_t)row * n;
  int e = 1;
  for (int k = threadIdx.x; k < n; k += 256)
    if (k != row) e = max(e, exponent_field(a[k]));
  const int emax = block_max<256>(e, red);
  for (int k = threadIdx.x; k < n; k += 256) {
    const double x = a[k];
    if (k == row) diag[row] = x;
    reinterpret_cast<int2*>(a)[k] = k == row ? make_int2(0, 0) : entry_digits(x, emax);
  }
  if (threadIdx.x == 0) re[row] = emax == 0x7ff ? kNotFinite : emax - 1084;
}

// y = A x, one CTA per SM, each with ceil(n / gridDim.x) rows: the CTA finds the exponent of x, puts the digits of
// a segment of it in shared memory (about 3 us, a small part of the stream; no state is shared between calls) and
// its warps stream quarters of rows past L1, four 16-byte loads in flight per lane. Quarters even out the warps: at
// 8192 unknowns 54 rows are 216 units for 32 warps.
constexpr int kGemvThreads = 1024, kGemvParts = 4, kGemvSeg = 8192;
constexpr int kMaxUnknowns = 2 * 4096 * kPP;

size_t gemv_smem(int n, int rows) {
  return (size_t)std::min(n, kGemvSeg) * 3 * sizeof(int) + (size_t)rows * kGemvParts * sizeof(double);
}

__global__ void __launch_bounds__(kGemvThreads, 1)
    k_gemv(int n, int rows, const double* __restrict__ A, const double* __restrict__ diag, const int* __restrict__ re,
           const double* __restrict__ x, double* __restrict__ y, const GmresCtl* ctl = nullptr) {
  if (gm_done(ctl)) return;
  extern __shared__ __align__(16) unsigned char gemv_sm[];
  double* acc = reinterpret_cast<double*>(gemv_sm);           // [rows][kGemvParts]
  const int seg = min(n, kGemvSeg);
  int2* xu = reinterpret_cast<int2*>(acc + rows * kGemvParts);  // digits of a segment of x: high and middle,
  int* xl = reinterpret_cast<int*>(xu + seg);                   // low
  __shared__ int red[kGemvThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = blockIdx.x * rows, nr = min(rows, n - r0);
  int e = 1;
  for (int k = tid; k < n; k += kGemvThreads) e = max(e, exponent_field(x[k]));
  const int emax = block_max<kGemvThreads>(e, red);
  for (int k0 = 0; k0 < n; k0 += kGemvSeg) {
    const int len = min(kGemvSeg, n - k0), len2 = len >> 1, q = (len2 + kGemvParts - 1) / kGemvParts;
    __syncthreads();
    for (int k = tid; k < len; k += kGemvThreads) {
      const int3 d = component_digits(x[k0 + k], emax);
      xu[k] = make_int2(d.x, d.y);
      xl[k] = d.z;
    }
    __syncthreads();
    const int4* xv = reinterpret_cast<const int4*>(xu);
    const int2* xw = reinterpret_cast<const int2*>(xl);
    for (int u = warp; u < nr * kGemvParts; u += kGemvThreads / 32) {
      const int4* a = reinterpret_cast<const int4*>(A + (size_t)(r0 + u / kGemvParts) * n + k0);
      const int part = u % kGemvParts, end = min(len2, (part + 1) * q);
      double s = 0.0;
      for (int kb = part * q; kb < end; kb += 32 * 64) {  // 128 entries per lane
        // sums of products of weight 2^80, 2^56, 2^48, 2^32, 2^24 (high x high .. low x middle)
        long long h0 = 0, h1 = 0, l0 = 0, h2 = 0, l1 = 0;
        auto mac = [&](int4 p, int i) {
          const int4 v = xv[i];
          const int2 w = xw[i];
          h0 += (long long)p.y * v.x; h1 += (long long)p.y * v.y; h2 += (long long)p.y * w.x;
          l0 += (long long)p.x * v.x; l1 += (long long)p.x * v.y;
          h0 += (long long)p.w * v.z; h1 += (long long)p.w * v.w; h2 += (long long)p.w * w.y;
          l0 += (long long)p.z * v.z; l1 += (long long)p.z * v.w;
        };
        const int k1 = min(end, kb + 32 * 64);
        int k = kb + lane;
        for (; k + 96 < k1; k += 128) {
          const int4 a0 = __ldcs(a + k), a1 = __ldcs(a + k + 32), a2 = __ldcs(a + k + 64), a3 = __ldcs(a + k + 96);
          mac(a0, k);
          mac(a1, k + 32);
          mac(a2, k + 64);
          mac(a3, k + 96);
        }
        for (; k < k1; k += 32) mac(__ldcs(a + k), k);
        // in units of 2^56: what the shifts drop is below 2^-80 of the largest products
        s += (double)h0 * (double)(1 << 24) + (double)(h1 + (l0 >> 8) + (h2 >> 24) + (l1 >> 32));
      }
      for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) acc[u] = k0 ? acc[u] + s : s;
    }
  }
  __syncthreads();
  for (int r = tid; r < nr; r += kGemvThreads) {
    const double* p = acc + r * kGemvParts;
    const double s = (p[0] + p[1]) + (p[2] + p[3]);
    const int er = re[r0 + r], ex = emax == 0x7ff ? kNotFinite : emax - 1093;
    const double d = diag[r0 + r] * x[r0 + r];
    y[r0 + r] = er == kNotFinite || ex == kNotFinite ? __longlong_as_double(0x7ff8000000000000ll)
                                                     : d + ldexp(s, er + ex + 56);
  }
}

// h[c] = sum_k V[c][k] w[k] for c < ncols (V row-major [ncols][n]): one block per column.
__global__ void k_dots(int n, int ncols, const double* __restrict__ V, const double* __restrict__ w, double* h,
                       const GmresCtl* ctl = nullptr) {
  if (gm_done(ctl)) return;
  const int c = blockIdx.x;
  if (c >= ncols) return;
  __shared__ double red[32];
  double s = 0.0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) s += V[(size_t)c * n + k] * w[k];
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) h[c] = s;
  }
}

// w -= sum_c h[c] V[c]
__global__ void k_sub_proj(int n, int ncols, const double* __restrict__ V, const double* __restrict__ h, double* w,
                           const GmresCtl* ctl = nullptr) {
  if (gm_done(ctl)) return;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  double s = w[k];
  for (int c = 0; c < ncols; ++c) s -= h[c] * V[(size_t)c * n + k];
  w[k] = s;
}

__global__ void k_axpby(int n, double a, const double* x, double b, double* y) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) y[k] = a * x[k] + b * y[k];
}

// x += sum_{c < it} y[c] V[c], it the iteration count in the GMRES state
__global__ void k_add_comb(int n, const GmresCtl* ctl, const double* __restrict__ V, const double* __restrict__ coef,
                           double* x) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int ncols = ctl->it;
  double s = x[k];
  for (int c = 0; c < ncols; ++c) s += coef[c] * V[(size_t)c * n + k];
  x[k] = s;
}

// Start of GMRES (one thread): norms from the dot products gr = (g.g, r.r).
__global__ void k_gm_init(GmresCtl* ctl, const double* gr, double tol, double* gv) {
  const double bnorm = gr[0] > 0.0 ? sqrt(gr[0]) : 1.0, beta = sqrt(fmax(gr[1], 0.0));
  ctl->bnorm = bnorm;
  ctl->res = beta / bnorm;
  ctl->hn = beta;
  ctl->it = 0;
  ctl->done = (beta / bnorm <= tol || beta == 0.0) ? 1 : 0;
  gv[0] = beta;
}

// y = x / ctl->hn (the next Krylov vector), skipped once converged.
__global__ void k_gm_scale(int n, const GmresCtl* ctl, const double* __restrict__ x, double* __restrict__ y) {
  if (gm_done(ctl)) return;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) y[k] = x[k] / ctl->hn;
}

// Arnoldi step j (one thread): Hessenberg column j from the two Gram-Schmidt passes hv0, hv1 and
// |w|^2, earlier Givens rotations applied, new rotation, residual estimate |gv[j+1]| / |g|.
__global__ void k_gm_step(int j, int m, double tol, GmresCtl* ctl, double* H, double* cs, double* sn, double* gv,
                          const double* hv0, const double* hv1, const double* wn2) {
  if (ctl->done) return;
  for (int i = 0; i <= j; ++i) H[(size_t)i * m + j] = hv0[i] + hv1[i];
  const double hn = sqrt(fmax(*wn2, 0.0));
  H[(size_t)(j + 1) * m + j] = hn;
  for (int i = 0; i < j; ++i) {
    const double a = H[(size_t)i * m + j], c = H[(size_t)(i + 1) * m + j];
    H[(size_t)i * m + j] = cs[i] * a + sn[i] * c;
    H[(size_t)(i + 1) * m + j] = -sn[i] * a + cs[i] * c;
  }
  const double a = H[(size_t)j * m + j], c = H[(size_t)(j + 1) * m + j];
  const double d = hypot(a, c);
  cs[j] = d > 0.0 ? a / d : 1.0;
  sn[j] = d > 0.0 ? c / d : 0.0;
  H[(size_t)j * m + j] = d;
  H[(size_t)(j + 1) * m + j] = 0.0;
  gv[j + 1] = -sn[j] * gv[j];
  gv[j] = cs[j] * gv[j];
  ctl->it = j + 1;
  ctl->hn = hn;
  ctl->res = fabs(gv[j + 1]) / ctl->bnorm;
  if (ctl->res <= tol || hn == 0.0) ctl->done = 1;
}

// One Arnoldi step after w = A v_j in one launch: classical Gram-Schmidt applied twice, the Hessenberg column and its
// rotations (as k_gm_step) and v_(j+1) = w / |w|; with `ac` first the projection w -= (ac . w) ac, whose
// coefficient goes to abv[j]. A cluster of 16 CTAs holds w in shared memory, a sixteenth each; dot products meet in
// distributed shared memory, added in the order of the ranks. The separate kernels (k_dots ... k_gm_scale) take
// seven launches a step, each a few microseconds on a vector of 64 KB; they stay for devices that cannot hold the
// cluster, and for vectors and subspaces beyond kArnN and kArnCols, where more than 16 SMs' worth of FP64 pays. Measured at 8192 unknowns, 17 steps:
// 22 us a step beside the operator, 87 with the separate kernels; a cold solve 3.64 -> 2.24 ms with k_gemv.
constexpr int kArnCtas = 16, kArnThreads = 512, kArnN = 32768, kArnCols = 64;

__global__ void __cluster_dims__(kArnCtas, 1, 1) __launch_bounds__(kArnThreads)
    k_arnoldi(int n, int j, int m, double tol, GmresCtl* ctl, double* H, double* cs, double* sn, double* gv,
              const double* __restrict__ w, double* V, const double* __restrict__ ac, double* abv) {
  if (gm_done(ctl)) return;  // the same for all CTAs: written only by earlier launches, or after the barriers below
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ double ws[kArnN / kArnCtas], part[2][kArnCols], tail[2], h[2][kArnCols], rot[2][kArnCols];
  __shared__ double red[kArnThreads / 32];
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = n / kArnCtas, k0 = rank * per;
  for (int i = tid; i < per; i += kArnThreads) ws[i] = w[k0 + i];
  if (tid < j) { rot[0][tid] = cs[tid]; rot[1][tid] = sn[tid]; }
  __syncthreads();
  auto block_sum = [&](double v, double* sum) {  // in warp order
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (tid == 0) {
      v = 0.0;
      for (int q = 0; q < kArnThreads / 32; ++q) v += red[q];
      *sum = v;
    }
    __syncthreads();
  };
  auto over_ranks = [&](double* p) {
    double v = 0.0;
    for (int r = 0; r < kArnCtas; ++r) v += *cl.map_shared_rank(p, r);
    return v;
  };
  if (ac) {
    double v = 0.0;
    for (int i = tid; i < per; i += kArnThreads) v = fma(ac[k0 + i], ws[i], v);
    block_sum(v, &tail[1]);
    cl.sync();
    const double b = over_ranks(&tail[1]);
    if (rank == 0 && tid == 0) abv[j] = b;
    for (int i = tid; i < per; i += kArnThreads) ws[i] -= b * ac[k0 + i];
    __syncthreads();
  }
  for (int pass = 0; pass < 2; ++pass) {
    for (int c = warp; c <= j; c += kArnThreads / 32) {
      const double* v = V + (size_t)c * n + k0;
      double s = 0.0;
#pragma unroll 4
      for (int i = lane; i < per; i += 32) s = fma(v[i], ws[i], s);
      for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) part[pass][c] = s;
    }
    cl.sync();
    if (tid <= j) h[pass][tid] = over_ranks(&part[pass][tid]);
    __syncthreads();
    for (int i = tid; i < per; i += kArnThreads) {
      double s = ws[i];
      const double* v = V + k0 + i;
#pragma unroll 4
      for (int c = 0; c <= j; ++c) s -= h[pass][c] * v[(size_t)c * n];
      ws[i] = s;
    }
    __syncthreads();
  }
  double v = 0.0;
  for (int i = tid; i < per; i += kArnThreads) v = fma(ws[i], ws[i], v);
  block_sum(v, &tail[0]);
  cl.sync();
  const double hn = sqrt(fmax(over_ranks(&tail[0]), 0.0));
  for (int i = tid; i < per; i += kArnThreads) V[(size_t)(j + 1) * n + k0 + i] = ws[i] / hn;
  if (rank == 0 && tid == 0) {
    double a = h[0][0] + h[1][0];
    for (int i = 0; i < j; ++i) {
      const double c = h[0][i + 1] + h[1][i + 1];
      H[(size_t)i * m + j] = rot[0][i] * a + rot[1][i] * c;
      a = -rot[1][i] * a + rot[0][i] * c;
    }
    const double d = hypot(a, hn), c = d > 0.0 ? a / d : 1.0, sj = d > 0.0 ? hn / d : 0.0;
    cs[j] = c;
    sn[j] = sj;
    H[(size_t)j * m + j] = d;
    H[(size_t)(j + 1) * m + j] = 0.0;
    const double g = gv[j], res = fabs(sj * g) / ctl->bnorm;
    gv[j + 1] = -sj * g;
    gv[j] = c * g;
    ctl->it = j + 1;
    ctl->hn = hn;
    ctl->res = res;
    if (res <= tol || hn == 0.0) ctl->done = 1;
  }
  cl.sync();  // no CTA ends while another reads its shared memory
}

// Whether the current device can hold a cluster of k_arnoldi, which is larger than the portable size; otherwise the
// separate kernels take every step.
bool arnoldi_cluster_fits() {
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(kArnCtas);
  c.blockDim = dim3(kArnThreads);
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = kArnCtas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  c.attrs = &at;
  c.numAttrs = 1;
  int clusters = 0;
  const bool ok = cudaFuncSetAttribute(k_arnoldi, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                  cudaOccupancyMaxActiveClusters(&clusters, k_arnoldi, &c) == cudaSuccess;
  cudaGetLastError();  // not an error of the caller's
  return ok && clusters > 0;
}

// Augmentation by a direction d (w = A d on entry): with s = (w.r)/(w.w), mu += s d, r -= s w
// (the least-squares step along d), c = w/|w|, u = d/|w|; nothing when w = 0.
__global__ void k_aug_setup(int n, const double* ww_wr, const double* w, const double* d, double* r, double* mu,
                            double* c, double* u) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const double ww = ww_wr[0], wr = ww_wr[1];
  if (!(ww > 0.0)) {
    c[k] = 0.0;
    u[k] = 0.0;
    return;
  }
  const double nrm = sqrt(ww), st = wr / ww;
  mu[k] += st * d[k];
  r[k] -= st * w[k];
  c[k] = w[k] / nrm;
  u[k] = d[k] / nrm;
}

// w -= beta c, beta = *bj (the component of A v_j along c, removed from the Krylov operator).
__global__ void k_aug_project(int n, const GmresCtl* ctl, const double* bj, const double* c, double* w) {
  if (gm_done(ctl)) return;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) w[k] -= *bj * c[k];
}

// mu -= (sum_{j < it} b_j y_j) u: the update V y moved A mu by the removed components c b.y.
__global__ void k_aug_final(int n, const GmresCtl* ctl, const double* bv, const double* y, const double* u,
                            double* mu) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  double sdot = 0.0;
  for (int j = 0; j < ctl->it; ++j) sdot += bv[j] * y[j];
  mu[k] -= sdot * u[k];
}

// Least-squares solution of the rotated Hessenberg system by columns: y_i, then its column taken off the others
// (one block; the right-hand side in shared memory, kMaxKrylov of it).
constexpr int kMaxKrylov = 1000;
__global__ void __launch_bounds__(256) k_gm_backsub(int m, const GmresCtl* ctl, const double* H, const double* gv, double* y) {
  __shared__ double t[kMaxKrylov];
  const int it = ctl->it;
  for (int i = threadIdx.x; i < it; i += 256) t[i] = gv[i];
  for (int i = it - 1; i >= 0; --i) {
    __syncthreads();
    const double yi = t[i] / H[(size_t)i * m + i];
    if (threadIdx.x == 0) y[i] = yi;
    for (int k = threadIdx.x; k < i; k += 256) t[k] -= H[(size_t)k * m + i] * yi;
  }
}

// u(x_t) = sum_j D(x_t, y_j) mu_j w_j (targets away from the boundary), NT targets per block.
//
// FP64 bounds it. For alpha r >= kFarZ the terms of T1, T2, T3 with K0 and K1 are below 2^-54 of the algebraic
// ones (z^3 e^-z sqrt(pi / 2z) < 5e-18 against 4), so adding them changes nothing and only the algebraic part is
// formed: with q = 1 / r^2, c = 2 q^2 / (pi alpha^2), m = mu w,
//   D m = -c (n (r.m) + r (n.m) + m (r.n)) + 4 c q r (r.n)(r.m) + q / (2 pi) r (n.m),
// about 35 FP64 operations and no transcendental function. Measured: 2000 targets, 4096 nodes, alpha = 316: 576 us
// (5,754 us with the Bessel functions for every pair).
constexpr double kFarZ = 50.0;

template <int NT>
__global__ void __launch_bounds__(256) k_eval_dl(int N, double alpha, Nodes nd, const double* mu, int M,
                                                 const double* txy, double* u) {
  const int t0 = blockIdx.x * NT;
  const double far2 = kFarZ / alpha * (kFarZ / alpha), ca = 2.0 / (kPi * alpha * alpha);
  double x[NT], y[NT], s[NT][2] = {};
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    const int k = min(t0 + t, M - 1);
    x[t] = txy[k];
    y[t] = txy[M + k];
  }
  for (int j = threadIdx.x; j < N; j += 256) {
    const double xj = nd.x[j], yj = nd.y[j], nx = nd.nx[j], ny = nd.ny[j], w = nd.w[j];
    const double mx = mu[2 * j] * w, my = mu[2 * j + 1] * w, nm = nx * mx + ny * my;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const double rx = x[t] - xj, ry = y[t] - yj, r2 = rx * rx + ry * ry;
      if (r2 >= far2) {
        const double q = 1.0 / r2, c = ca * q * q;
        const double rn = rx * nx + ry * ny, cm = c * (rx * mx + ry * my), cr = c * rn;
        const double f = fma(4.0 * q * rn, cm, nm * (0.5 / kPi * q - c));
        s[t][0] += f * rx - cm * nx - cr * mx;
        s[t][1] += f * ry - cm * ny - cr * my;
      } else {
        double D[4];
        dl_kernel(alpha, rx, ry, nx, ny, D);
        s[t][0] += D[0] * mx + D[1] * my;
        s[t][1] += D[2] * mx + D[3] * my;
      }
    }
  }
  __shared__ double red[8][2 * NT];
#pragma unroll
  for (int t = 0; t < NT; ++t)
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      double v = s[t][a];
      for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][2 * t + a] = v;
    }
  __syncthreads();
  if (threadIdx.x < 2 * NT) {
    const int t = threadIdx.x >> 1, a = threadIdx.x & 1;
    double v = 0.0;
    for (int q = 0; q < 8; ++q) v += red[q][threadIdx.x];
    if (t0 + t < M) u[(size_t)a * M + t0 + t] = v;
  }
}

// Stokeslet sum at points: u_a(x) = sum_k S_ab(x - s_k) f_kb.
__global__ void k_stokeslets(double alpha, int K, const double* src, const double* f, int M, const double* xy,
                             double* u) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= M) return;
  double u0 = 0.0, u1 = 0.0;
  for (int k = 0; k < K; ++k) {
    const double rx = xy[t] - src[2 * k], ry = xy[M + t] - src[2 * k + 1];
    const double r = sqrt(rx * rx + ry * ry);
    double T1, T2, T3, S1, S2;
    stress_funcs(alpha * r, T1, T2, T3, S1, S2);
    const double a2 = alpha * alpha;
    u0 += (S1 + a2 * S2 * rx * rx) * f[2 * k] + a2 * S2 * rx * ry * f[2 * k + 1];
    u1 += a2 * S2 * rx * ry * f[2 * k] + (S1 + a2 * S2 * ry * ry) * f[2 * k + 1];
  }
  u[t] = u0;
  u[M + t] = u1;
}

// Kernel scalars at given z (for tests): out[5][n] = T1, T2, T3, S1, S2.
__global__ void k_stress_funcs(int n, const double* z, double* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  double T1, T2, T3, S1, S2;
  stress_funcs(z[t], T1, T2, T3, S1, S2);
  out[t] = T1; out[n + t] = T2; out[2 * n + t] = T3; out[3 * n + t] = S1; out[4 * n + t] = S2;
}

void gl_host(int n, double* x, double* w) { gauss_legendre_host(n, x, w); }

}  // namespace
}  // namespace vp

struct bie_s {
  int np = 0, N = 0, n2 = 0;
  double alpha = 0.0, Lb = 0.0;
  vp::Star star{};
  vp::Nodes nd{};
  std::vector<void*> allocs;
  double* A = nullptr;
  // GMRES work space
  int m = 0;
  double *V = nullptr, *w = nullptr, *r = nullptr;
  double* diag = nullptr;        // the operator's diagonal; A holds the rest as digits (k_matrix_digits)
  int* re = nullptr;             // row exponents
  int sms = 0;
  bool cluster = false;          // the device can hold a cluster of k_arnoldi
  int ctas = 0, rows = 0;        // launch of k_gemv: one CTA per SM, rows of each
  double* gm = nullptr;          // H [(m+1) m], cs [m], sn [m], gv [m+2], y [m], hv [2(m+1)], scalars [8]
  double *ac = nullptr, *au = nullptr, *abv = nullptr;  // augmentation: c, u [2N], b [m]
  vp::GmresCtl* ctl = nullptr;   // device
  vp::GmresCtl* hctl = nullptr;  // pinned host copies (two groups of iterations)
  cudaEvent_t ev[2] = {nullptr, nullptr};
};

using namespace vp;

namespace {
template <class T>
int dalloc(bie_s* b, T** p, size_t n) {
  void* q = nullptr;
  TRY(cudaMalloc(&q, std::max<size_t>(1, n) * sizeof(T)));
  b->allocs.push_back(q);
  *p = static_cast<T*>(q);
  return VP_OK;
}
}  // namespace

extern "C" void bie_free(bie b) {
  if (!b) return;
  if (b->hctl) cudaFreeHost(b->hctl);
  for (cudaEvent_t e : b->ev)
    if (e) cudaEventDestroy(e);
  for (void* p : b->allocs) cudaFree(p);
  delete b;
}

extern "C" int bie_create(double alpha, double R, double A, int k, double phase, int n_panels, int max_krylov,
                          void* stream, bie* out) {
  if (!out) return VP_ERR_ARG;
  *out = nullptr;
  if (!(alpha > 0.0) || !(R > 0.0) || !(A >= 0.0) || A >= R || k < 0 || n_panels < 4 || n_panels > 4096 ||
      max_krylov < 1 || max_krylov > kMaxKrylov)
    return VP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  std::unique_ptr<bie_s> B(new (std::nothrow) bie_s());
  if (!B) return VP_ERR_OOM;
  B->np = n_panels; B->N = n_panels * kPP; B->n2 = 2 * B->N; B->alpha = alpha;
  B->star = {R, A, phase, k};
  B->m = max_krylov;
  {
    double x16[kPP], w16[kPP], x12[kGradeN], w12[kGradeN], bw[kPP];
    gl_host(kPP, x16, w16);
    gl_host(kGradeN, x12, w12);
    for (int i = 0; i < kPP; ++i) {
      double prod = 1.0;
      for (int j = 0; j < kPP; ++j) if (j != i) prod *= x16[i] - x16[j];
      bw[i] = 1.0 / prod;
    }
    TRY(cudaMemcpyToSymbolAsync(c_glx16, x16, sizeof(x16), 0, cudaMemcpyHostToDevice, s));
    TRY(cudaMemcpyToSymbolAsync(c_glw16, w16, sizeof(w16), 0, cudaMemcpyHostToDevice, s));
    TRY(cudaMemcpyToSymbolAsync(c_glx12, x12, sizeof(x12), 0, cudaMemcpyHostToDevice, s));
    TRY(cudaMemcpyToSymbolAsync(c_glw12, w12, sizeof(w12), 0, cudaMemcpyHostToDevice, s));
    TRY(cudaMemcpyToSymbolAsync(c_bw16, bw, sizeof(bw), 0, cudaMemcpyHostToDevice, s));
  }
  int rc, dev = 0;
  TRY(cudaGetDevice(&dev));
  TRY(cudaDeviceGetAttribute(&B->sms, cudaDevAttrMultiProcessorCount, dev));
  B->rows = (B->n2 + B->sms - 1) / B->sms;
  B->ctas = (B->n2 + B->rows - 1) / B->rows;
  const int N = B->N;
  Nodes& nd = B->nd;
  for (double** p : {&nd.x, &nd.y, &nd.nx, &nd.ny, &nd.w, &nd.kappa, &nd.tx, &nd.ty, &nd.theta})
    if ((rc = dalloc(B.get(), p, N))) { bie_free(B.release()); return rc; }
  if ((rc = dalloc(B.get(), &B->A, (size_t)B->n2 * B->n2))) { bie_free(B.release()); return rc; }
  if ((rc = dalloc(B.get(), &B->V, (size_t)(B->m + 1) * B->n2)) || (rc = dalloc(B.get(), &B->w, B->n2)) ||
      (rc = dalloc(B.get(), &B->r, B->n2)) ||
      (rc = dalloc(B.get(), &B->gm, (size_t)(B->m + 1) * B->m + 6 * (size_t)B->m + 12)) ||
      (rc = dalloc(B.get(), &B->ctl, 1)) || (rc = dalloc(B.get(), &B->ac, B->n2)) ||
      (rc = dalloc(B.get(), &B->au, B->n2)) || (rc = dalloc(B.get(), &B->abv, B->m)) ||
      (rc = dalloc(B.get(), &B->diag, B->n2)) || (rc = dalloc(B.get(), &B->re, B->n2))) {
    bie_free(B.release());
    return rc;
  }
  if (cudaHostAlloc(&B->hctl, 2 * sizeof(GmresCtl), cudaHostAllocDefault) != cudaSuccess ||
      cudaEventCreateWithFlags(&B->ev[0], cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&B->ev[1], cudaEventDisableTiming) != cudaSuccess) {
    bie_free(B.release());
    return VP_ERR_OOM;
  }
  k_nodes<<<(N + 127) / 128, 128, 0, s>>>(B->star, B->np, nd);
  // boundary length
  std::vector<double> w(N);
  if (cudaMemcpyAsync(w.data(), nd.w, N * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    bie_free(B.release());
    return VP_ERR_CUDA;
  }
  double L = 0.0;
  for (double v : w) L += v;
  B->Lb = L;
  const long long NN = (long long)N * N;
  k_matrix_plain<<<(unsigned)((NN + 255) / 256), 256, 0, s>>>(N, alpha, L, nd, B->A);
  k_matrix_local<<<N, 128, 0, s>>>(B->np, alpha, L, B->star, nd, B->A);
  k_matrix_digits<<<B->n2, 256, 0, s>>>(B->n2, B->A, B->diag, B->re);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess ||
      cudaFuncSetAttribute(k_gemv, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)gemv_smem(kMaxUnknowns, (kMaxUnknowns + B->ctas - 1) / B->ctas)) != cudaSuccess) {
    bie_free(B.release());
    return VP_ERR_CUDA;
  }
  B->cluster = arnoldi_cluster_fits();
  *out = B.release();
  return VP_OK;
}

extern "C" int bie_size(bie b, int* n_nodes, double* boundary_length) {
  if (!b) return VP_ERR_ARG;
  if (n_nodes) *n_nodes = b->N;
  if (boundary_length) *boundary_length = b->Lb;
  return VP_OK;
}

extern "C" int bie_nodes(bie b, double* out, void* stream) {
  if (!b || !out) return VP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int N = b->N;
  const double* src[7] = {b->nd.x, b->nd.y, b->nd.nx, b->nd.ny, b->nd.w, b->nd.kappa, b->nd.theta};
  for (int k = 0; k < 7; ++k)
    TRY(cudaMemcpyAsync(out + (size_t)k * N, src[k], N * sizeof(double), cudaMemcpyDeviceToDevice, s));
  return VP_OK;
}

namespace {
void apply_operator(const bie_s* b, const double* x, double* y, cudaStream_t s, const GmresCtl* ctl = nullptr) {
  k_gemv<<<b->ctas, kGemvThreads, gemv_smem(b->n2, b->rows), s>>>(b->n2, b->rows, b->A, b->diag, b->re, x, y, ctl);
}
}  // namespace

extern "C" int bie_apply(bie b, const double* mu, double* out, void* stream) {
  if (!b || !mu || !out || (reinterpret_cast<uintptr_t>(mu) & 15)) return VP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  apply_operator(b, mu, out, s);
  TRY(cudaGetLastError());
  return VP_OK;
}

extern "C" int bie_solve_aug(bie b, const double* g, double* mu, const double* d, double tol, int max_iter,
                             int* iters, double* relres, void* stream) {
  if (!b || !g || !mu || !(tol > 0.0) || max_iter < 1 || (reinterpret_cast<uintptr_t>(mu) & 15) ||
      (reinterpret_cast<uintptr_t>(d) & 15))
    return VP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int n = b->n2, M = b->m;
  const int m = std::min(max_iter, M);
  const int T = 256, G = (n + T - 1) / T;
  double* H = b->gm;
  double* cs = H + (size_t)(M + 1) * M;
  double* sn = cs + M;
  double* gv = sn + M;
  double* y = gv + M + 2;
  double* hv = y + M;
  double* wn2 = hv + 2 * (M + 1);
  GmresCtl* ctl = b->ctl;
  // r = g - A mu, norms, V0 = r / |r|
  apply_operator(b, mu, b->r, s);
  k_axpby<<<G, T, 0, s>>>(n, 1.0, g, -1.0, b->r);
  if (d) {
    // least-squares step along d, then GMRES on (I - c c^T) A so that direction stays removed
    apply_operator(b, d, b->w, s);
    k_dots<<<1, 256, 0, s>>>(n, 1, b->w, b->w, wn2 + 4);
    k_dots<<<1, 256, 0, s>>>(n, 1, b->w, b->r, wn2 + 5);
    k_aug_setup<<<G, T, 0, s>>>(n, wn2 + 4, b->w, d, b->r, mu, b->ac, b->au);
  }
  k_dots<<<1, 256, 0, s>>>(n, 1, g, g, wn2);
  k_dots<<<1, 256, 0, s>>>(n, 1, b->r, b->r, wn2 + 1);
  k_gm_init<<<1, 1, 0, s>>>(ctl, wn2, tol, gv);
  k_gm_scale<<<G, T, 0, s>>>(n, ctl, b->r, b->V);
  // Arnoldi with classical Gram-Schmidt applied twice; the host queues kGroup iterations at a time and looks at
  // the state of a group only once the next one is queued, so the device does not wait for it (iterations past
  // convergence are no-ops).
  constexpr int kGroup = 4;
  int slot = 0;
  for (int j = 0; j < m; slot ^= 1) {
    const int jend = std::min(m, j + kGroup);
    for (; j < jend; ++j) {
      const double* vj = b->V + (size_t)j * n;
      apply_operator(b, vj, b->w, s, ctl);
      if (b->cluster && n <= kArnN && j < kArnCols) {
        k_arnoldi<<<kArnCtas, kArnThreads, 0, s>>>(n, j, M, tol, ctl, H, cs, sn, gv, b->w, b->V,
                                                   d ? b->ac : nullptr, b->abv);
        continue;
      }
      if (d) {
        k_dots<<<1, 256, 0, s>>>(n, 1, b->ac, b->w, b->abv + j, ctl);
        k_aug_project<<<G, T, 0, s>>>(n, ctl, b->abv + j, b->ac, b->w);
      }
      for (int pass = 0; pass < 2; ++pass) {
        k_dots<<<j + 1, 256, 0, s>>>(n, j + 1, b->V, b->w, hv + pass * (M + 1), ctl);
        k_sub_proj<<<G, T, 0, s>>>(n, j + 1, b->V, hv + pass * (M + 1), b->w, ctl);
      }
      k_dots<<<1, 256, 0, s>>>(n, 1, b->w, b->w, wn2 + 2, ctl);
      k_gm_step<<<1, 1, 0, s>>>(j, M, tol, ctl, H, cs, sn, gv, hv, hv + M + 1, wn2 + 2);
      k_gm_scale<<<G, T, 0, s>>>(n, ctl, b->w, b->V + (size_t)(j + 1) * n);
    }
    TRY(cudaGetLastError());  // a refused launch would leave `done` unset for every step to come
    TRY(cudaMemcpyAsync(b->hctl + slot, ctl, sizeof(GmresCtl), cudaMemcpyDeviceToHost, s));
    TRY(cudaEventRecord(b->ev[slot], s));
    if (jend > kGroup) {  // the group before this one
      TRY(cudaEventSynchronize(b->ev[slot ^ 1]));
      if (b->hctl[slot ^ 1].done) break;
    }
  }
  // update and the true residual
  k_gm_backsub<<<1, 256, 0, s>>>(M, ctl, H, gv, y);
  k_add_comb<<<G, T, 0, s>>>(n, ctl, b->V, y, mu);
  if (d) k_aug_final<<<G, T, 0, s>>>(n, ctl, b->abv, y, b->au, mu);
  apply_operator(b, mu, b->r, s);
  k_axpby<<<G, T, 0, s>>>(n, 1.0, g, -1.0, b->r);
  k_dots<<<1, 256, 0, s>>>(n, 1, b->r, b->r, wn2 + 3);
  double rr[2] = {0.0, 0.0};
  TRY(cudaMemcpyAsync(b->hctl, ctl, sizeof(GmresCtl), cudaMemcpyDeviceToHost, s));
  TRY(cudaMemcpyAsync(rr, wn2 + 3, sizeof(double), cudaMemcpyDeviceToHost, s));
  TRY(cudaStreamSynchronize(s));
  if (iters) *iters = b->hctl->it;
  if (relres) *relres = std::sqrt(std::max(rr[0], 0.0)) / b->hctl->bnorm;
  TRY(cudaGetLastError());
  return VP_OK;
}

extern "C" int bie_solve(bie b, const double* g, double* mu, double tol, int max_iter, int* iters, double* relres,
                         void* stream) {
  return bie_solve_aug(b, g, mu, nullptr, tol, max_iter, iters, relres, stream);
}

extern "C" int bie_eval(bie b, const double* mu, int n_targets, const double* txy, double* u, void* stream) {
  if (!b || !mu || !txy || !u || n_targets < 0) return VP_ERR_ARG;
  if (n_targets == 0) return VP_OK;
  // Two targets per block share the nodes' loads (5 % of the algebraic form), where that takes no more rounds over the
  // SMs: time goes in steps of a target per SM. Measured with one / two on 152 SMs, 4096 nodes, alpha = 30 (Bessel pairs):
  // 100 targets 977 / 1,865 us, 400 2,790 / 3,660, 600 3,724 / 3,748, 2000 12,457 / 12,541; alpha = 316: 100 targets 60 / 99,
  // 400 144 / 178, 600 187 / 179, 2000 605 / 576.
  const int rounds = (n_targets + b->sms - 1) / b->sms;
  const bool two = n_targets >= 2 * b->sms && rounds % 2 == 0;
  const auto eval = two ? k_eval_dl<2> : k_eval_dl<1>;
  eval<<<two ? (n_targets + 1) / 2 : n_targets, 256, 0, static_cast<cudaStream_t>(stream)>>>(b->N, b->alpha, b->nd, mu,
                                                                                         n_targets, txy, u);
  TRY(cudaGetLastError());
  return VP_OK;
}

extern "C" int bie_stokeslets(double alpha, int n_sources, const double* src, const double* f, int n_points,
                              const double* xy, double* u, void* stream) {
  if (!(alpha > 0.0) || n_sources < 0 || n_points < 0 || !src || !f || !xy || !u) return VP_ERR_ARG;
  if (n_points == 0) return VP_OK;
  k_stokeslets<<<(n_points + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(alpha, n_sources, src, f,
                                                                                       n_points, xy, u);
  TRY(cudaGetLastError());
  return VP_OK;
}

extern "C" int bie_kernel_scalars(int n, const double* z, double* out, void* stream) {
  if (n < 0 || !z || !out) return VP_ERR_ARG;
  if (n == 0) return VP_OK;
  k_stress_funcs<<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(n, z, out);
  TRY(cudaGetLastError());
  return VP_OK;
}
