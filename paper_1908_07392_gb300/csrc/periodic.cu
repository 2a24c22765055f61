// Periodic particular solution by FFT (Sec. 2.1, Eqs. uhat, periodic_stokeslet, uP_Fourier,
// uP_Fourier_deriv; Sec. 3.1.2): on a uniform n x n grid of the periodic box of side L, the velocity
// of the modified Stokes equations (alpha^2 - Laplacian) u + grad p = F, div u = 0 is
//   u_hat(k) = S_hat(k) F_hat(k),  S_hat = (I - k k^T / |k|^2) / (alpha^2 + |k|^2),  S_hat(0) = I / alpha^2,
// and its gradient is i k_m u_hat. This is the paper's own route to the particular solution (the
// force extended by PUX, which stays out of scope here; the caller supplies the periodic force).
//
// Three launches:
//   k_rows_forward  row y: transform along x of F_x + i F_y, stored transposed ([kx][y]);
//   k_columns       column kx = 0 .. n/2: the spectra of F_x and F_y along x (by the symmetry of a real
//                   row), their transforms along y, the multiplier, and the inverse transforms along y
//                   of u_x, u_y, k_y u_x, k_y u_y; stored as rows ([y][kx]) of A = u_x + i u_y and
//                   D = k_y (u_x + i u_y) (k_y the wavenumber, 2 pi / L times an integer);
//   k_rows_inverse  row y: inverse transforms along x of A (the velocity), k_x A and D (the gradient).
// The derivative along x is taken after the inverse transform along y, so a solution takes 7 n length-n
// transforms (8 n when every output field has its own 2-D transform) and 160 bytes per point.
//
// Arithmetic: block floating point on 64-bit integers. This GPU issues 2 FP64 operations per clock
// and SM and 64 32-bit integer ones, and a transform is additions and multiplications by constants
// below one: a complex addition is 4 instructions, a complex multiplication by a twiddle 12 widening
// 32-bit multiply-adds (balanced 32-bit digits, no carries). Each length-n transform keeps one
// exponent; after every radix-8 stage the largest bit in use is found over the row and the row is
// shifted to just below the stage's headroom (58 to 59 bits used), so the rounding of a stage is about
// 2^-59 of the row's largest value, below the 2^-53 of each FP64 operation. Twiddles carry 62 bits.
// The multiplier is applied in FP64.
// Measured per solution: 4096^2 2.70 ms (15.0 ms with FP64 radix-4 rows, transposes and a separate spectral
// pass), 2048^2 0.564 ms (3.6), 512^2 56 us (about 250). The error against long double is 0.2 to 0.9 of the
// FP64 form's in the 2-norm (32^2 .. 2048^2; white noise, few modes, point forces). What bounds it: 2048^2 runs
// at 2 to 2.4 instructions per clock and SM of 4, the integer pipe half busy, the rest latency (about 330
// instructions per point and transform), 4096^2 at 1.4 with one CTA of k_columns per SM (registers, of which it
// spills some); 160 bytes per point at the copy rate would take 0.10 ms at 2048^2, 0.40 at 4096^2.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <new>
#include <vector>

#include "special.cuh"
#include "vp_internal.h"

struct vp_periodic_s {
  double alpha = 0.0, side = 0.0;
  int n = 0, logn = 0;
  int4* tw = nullptr;       // stage twiddles
  int4* wave = nullptr;     // k_x: mantissa digits, exponent
  double* mult = nullptr;   // [n/2 + 1][n/2 + 1]: 2^-mult_exp / ((i^2 + j^2)(alpha^2 + |k|^2)), and 2^-mult_exp / alpha^2
                            // at (0, 0)
  int mult_exp = 0;         // 128 where 1 / alpha^2 may be large: it meets spectra that are integers of up to 62 bits
  longlong2* z = nullptr;   // [kx][y] spectra along x, and two more columns of work space
  longlong2* a = nullptr;   // [y][kx] rows of A and D
  longlong2* d = nullptr;
  int2* ez = nullptr;       // per row y of z, per column kx of a and d: exponent, and exponent + bits in use
  int* ea = nullptr;
  int* ed = nullptr;
};

namespace vp {
namespace {

#define TRY(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { set_last_cuda(e_); return e_ == cudaErrorMemoryAllocation ? VP_ERR_OOM : VP_ERR_CUDA; } } while (0)

constexpr int kMinLog = 5, kMaxLog = 12;
constexpr int kMaxN = 1 << kMaxLog;
constexpr int kTopBits = 59;              // bits in use before a radix-8 stage (sums of 8 stay below 2^62.5)
constexpr int kZeroTop = -(1 << 28);      // "bits in use" of a block of zeros
constexpr int kNanTop = 1 << 28;          // ... of a block with an infinity or a NaN in it

typedef longlong2 c64;

// ------------------------------------------------------------------ fixed-point arithmetic

// a = h 2^32 + l with l in [-2^31, 2^31).
__device__ inline void digits(long long a, int& h, int& l) {
  l = (int)a;
  h = (int)(a >> 32) + (int)((unsigned)l >> 31);
}

// a (kh 2^32 + kl) / 2^64, rounded (the product of the low digits, at most a quarter of the last bit, is
// left out).
__device__ inline long long mul_hi(long long a, int kh, int kl) {
  int h, l;
  digits(a, h, l);
  const long long mid = (long long)h * kl + (long long)l * kh + 0x80000000ll;
  return (long long)h * kh + (mid >> 32);
}

// a sqrt(1/2) = a - a (1 - sqrt(1/2)).
__device__ inline long long mul_sqrt_half(long long a) {
  constexpr unsigned long long k = 5402926248376769404ull;  // (1 - sqrt(1/2)) 2^64
  constexpr int kl = (int)(unsigned)(k & 0xffffffffull);
  constexpr int kh = (int)((k >> 32) + ((k >> 31) & 1));
  return a - mul_hi(a, kh, kl);
}

// v w / 4 (DIR 1) or v conj(w) / 4 (DIR -1) for a twiddle w = (cos, sin) in units of 2^-62, given as balanced
// digits (ch, cl, sh, sl).
template <int DIR>
__device__ inline c64 mul_twiddle(c64 v, int4 w) {
  int ah, al, bh, bl;
  digits(v.x, ah, al);
  digits(v.y, bh, bl);
  const int sh = DIR > 0 ? w.z : -w.z, sl = DIR > 0 ? w.w : -w.w, nsh = -sh, nsl = -sl;
  const long long mr = (long long)ah * w.y + (long long)al * w.x + (long long)bh * nsl + (long long)bl * nsh + 0x80000000ll;
  const long long mi = (long long)ah * sl + (long long)al * sh + (long long)bh * w.y + (long long)bl * w.x + 0x80000000ll;
  c64 r;
  r.x = (long long)ah * w.x + (long long)bh * nsh + (mr >> 32);
  r.y = (long long)ah * sh + (long long)bh * w.x + (mi >> 32);
  return r;
}

__device__ inline c64 operator+(c64 a, c64 b) { return {a.x + b.x, a.y + b.y}; }
__device__ inline c64 operator-(c64 a, c64 b) { return {a.x - b.x, a.y - b.y}; }
// (DIR i) a
template <int DIR>
__device__ inline c64 rot(c64 a) {
  c64 r;
  if (DIR > 0) { r.x = -a.y; r.y = a.x; }
  else { r.x = a.y; r.y = -a.x; }
  return r;
}

// x 2^-s, rounded to nearest even for s > 0 (ties rounded one way add up coherently over a transform
// and show in its lowest modes).
__device__ inline long long shift_rn(long long x, int s) {
  if (s <= 0) return x << (-s > 63 ? 63 : -s);
  if (s > 61) return 0;
  return (x + (((x >> s) & 1) + ((1ll << (s - 1)) - 1))) >> s;
}

// The high words of the magnitudes, or'ed into `bits`.
__device__ inline void high_bits(unsigned& bits, c64 v) {
  bits |= (unsigned)abs((int)(v.x >> 32)) | (unsigned)abs((int)(v.y >> 32));
}

// The fixed-point value of x in units of 2^(emax - 1081), emax the largest exponent field in the block
// (fields 0 and 1 have the same unit): |result| < 2^59.
__device__ inline long long from_double(double x, int emax) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  int ex = (int)((b >> 52) & 0x7ff);
  unsigned long long m = b & ((1ull << 52) - 1);
  if (ex) m |= 1ull << 52;
  else ex = 1;
  m <<= 6;
  const int d = emax - ex;
  // halves away from zero: no bias, the values come with both signs
  m = d <= 0 ? m : (d > 63 ? 0ull : (m >> d) + ((m >> (d - 1)) & 1ull));
  return (long long)b < 0 ? -(long long)m : (long long)m;
}

__device__ inline int exponent_field(double x) {
  const int e = (int)((unsigned long long)__double_as_longlong(x) >> 52) & 0x7ff;
  return e ? e : 1;
}

// x 2^e for an integer x converted from 64 bits and |e| <= 900: an integer addition to the exponent field (the
// FP64 pipe is the scarce one).
__device__ inline double times_pow2(double x, int e) {
  const int hi = __double2hiint(x);
  return __hiloint2double(hi ? hi + e * (1 << 20) : 0, __double2loint(x));
}

// ------------------------------------------------------------------ one transform by n / 8 threads

// A row of n = 2^LOGN points is held by NT = n / 8 threads, thread i holding points i + q n / 8; a CTA
// holds as many rows as 64 threads need.
template <int LOGN>
struct Shape {
  static constexpr int n = 1 << LOGN, NT = n / 8, S8 = LOGN / 3, R = LOGN % 3;
  static constexpr int rows = NT >= 64 ? 1 : 64 / NT, threads = NT * rows;
  static constexpr int warps = NT >= 32 ? NT / 32 : 1;
};

// Threads of a column CTA, and the derivatives d = 0, 1 of u that each of its groups of n / 8 threads
// takes in turn: a group per component and derivative (the groups of d = 1 repeat the forward
// transform) where a column is short and the chain of transforms bounds the kernel (64^2: 36 -> 33 us), a group
// per component otherwise (1024^2: 219 -> 172 us).
template <int LOGN>
struct Columns {
  static constexpr int turns = LOGN <= 8 ? 1 : 2, groups = 4 / turns;
  static constexpr int cols = Shape<LOGN>::NT * groups >= 64 ? 1 : 64 / (Shape<LOGN>::NT * groups);
  static constexpr int threads = Shape<LOGN>::NT * groups * cols;
};

// CTAs per SM the compiler leaves registers for: 64 a thread where CTAs are large and throughput counts, 128
// where they are small and a thread's own speed does (512^2: 64, 80 and 128 registers 64.5, 58.4 and 56.3
// us; at 1024^2 more than 64 are slower, 189 against 172 us). k_columns spills 460 to 604 bytes a thread at 64 registers
// (1024^2 and up) and 20 at 512^2; the row kernels and the smaller columns spill nothing.
constexpr int resident(int threads) { return (threads >= 256 ? 1024 : 512) / threads; }

enum { RED_OR, RED_MAX };

// OR or maximum over the threads of a row; ends with a CTA barrier (and begins a phase in which `red`, one
// word per warp, is free).
template <int LOGN, int OP>
__device__ inline int row_reduce(int v, int* red) {
  constexpr int NT = Shape<LOGN>::NT, NW = Shape<LOGN>::warps;
  if (NT < 32) {
#pragma unroll
    for (int o = NT / 2; o; o >>= 1) {
      const int w = __shfl_xor_sync(0xffffffffu, v, o);
      v = OP == RED_OR ? (v | w) : max(v, w);
    }
    __syncthreads();
    return v;
  }
  v = OP == RED_OR ? (int)__reduce_or_sync(0xffffffffu, (unsigned)v) : __reduce_max_sync(0xffffffffu, v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, first = warp / NW * NW;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  const int w = red[first + (lane & (NW - 1))];
  return OP == RED_OR ? (int)__reduce_or_sync(0xffffffffu, (unsigned)w) : __reduce_max_sync(0xffffffffu, w);
}

template <int DIR>
__device__ inline void dft4(c64& a0, c64& a1, c64& a2, c64& a3) {
  const c64 s02 = a0 + a2, d02 = a0 - a2, s13 = a1 + a3, d13 = rot<DIR>(a1 - a3);
  a0 = s02 + s13;
  a1 = d02 + d13;
  a2 = s02 - s13;
  a3 = d02 - d13;
}

// b_p = sum_q a_q e^(DIR 2 pi i p q / 8), in place.
template <int DIR>
__device__ inline void dft8(c64 (&v)[8]) {
  c64 s0 = v[0] + v[4], s1 = v[1] + v[5], s2 = v[2] + v[6], s3 = v[3] + v[7];
  c64 d0 = v[0] - v[4], d1 = v[1] - v[5], d2 = v[2] - v[6], d3 = v[3] - v[7];
  // d1 e^(DIR i pi / 4) and d3 e^(DIR 3 i pi / 4)
  const c64 r1 = d1 + rot<DIR>(d1), r3 = rot<DIR>(d3) - d3;
  d1 = {mul_sqrt_half(r1.x), mul_sqrt_half(r1.y)};
  d2 = rot<DIR>(d2);
  d3 = {mul_sqrt_half(r3.x), mul_sqrt_half(r3.y)};
  dft4<DIR>(s0, s1, s2, s3);
  dft4<DIR>(d0, d1, d2, d3);
  v[0] = s0; v[2] = s1; v[4] = s2; v[6] = s3;
  v[1] = d0; v[3] = d1; v[5] = d2; v[7] = d3;
}

// Unnormalised transform of the row (sign DIR in the exponent), natural order in and out: Stockham
// autosort, radix 8 (a last stage of radix 4 or 2 where log2 n is no multiple of 3), the stages
// exchanging through shared memory `buf` (16-byte points, the low three index bits xored with the next
// three, so the stride-8 stores of the first stage and all unit-stride loads are free of bank
// conflicts). In: |components| < 2^59, values v 2^E. Out: |components| < 2^62.5, E updated. A stage of
// radix 8 with m points combined (l = n / 8 m) maps, for j < l and k < m, inputs a_q = x[k + (j + q l) m] to
// x[k + (8 j + p) m] = e^(DIR 2 pi i p j m / n) b_p.
template <int LOGN, int DIR>
__device__ inline void fft(c64 (&v)[8], int& E, int i, c64* buf, int* red, const int4* __restrict__ tw) {
  using S = Shape<LOGN>;
#pragma unroll
  for (int st = 0; st < S::S8; ++st) {
    const int lg_m = 3 * st, m = 1 << lg_m, l = S::n >> (lg_m + 3);
    dft8<DIR>(v);
    if (l == 1) break;  // the last stage has no twiddles (and no stage follows)
    const int k = i & (m - 1), j = i >> lg_m;
    // v[0] / 4, and below the shift of all points, round halves up or down by a bit of the thread's own:
    // unbiased over the row, two instructions cheaper per word than halves to even
    const long long tie = (i * 2654435761u) >> (31 - st) & 1;
    v[0] = {(v[0].x + 2 - tie) >> 2, (v[0].y + 2 - tie) >> 2};
#pragma unroll
    for (int p = 1; p < 8; ++p) v[p] = mul_twiddle<DIR>(v[p], __ldg(tw + (p - 1) * l + j));
    tw += 7 * l;
    unsigned bits = 0;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      high_bits(bits, v[p]);
      const int pos = k + (8 * j + p) * m;
      buf[pos ^ ((pos >> 3) & 7)] = v[p];
    }
    // bits in use now -> 59 (a row of zeros, or below 2^32: as if 32 were in use)
    const int s = 64 - __clz(row_reduce<LOGN, RED_OR>((int)bits, red)) - kTopBits;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int pos = i + q * S::NT;
      v[q] = buf[pos ^ ((pos >> 3) & 7)];
    }
    if (s > 0) {
      const long long c = (1ll << (s - 1)) - tie;
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = {(v[q].x + c) >> s, (v[q].y + c) >> s};
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = {v[q].x << -s, v[q].y << -s};
    }
    E += s + 2;
    __syncthreads();
  }
  if (S::R == 2) {
    dft4<DIR>(v[0], v[2], v[4], v[6]);
    dft4<DIR>(v[1], v[3], v[5], v[7]);
  } else if (S::R == 1) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const c64 a = v[q], b = v[q + 4];
      v[q] = a + b;
      v[q + 4] = a - b;
    }
  }
}

// Bits in use over the row (kZeroTop if it is zero).
template <int LOGN>
__device__ inline int row_bits(const c64 (&v)[8], int* red) {
  unsigned hi = 0, any = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    high_bits(hi, v[q]);
    any |= (unsigned)(v[q].x != 0 || v[q].y != 0);
  }
  const int r = row_reduce<LOGN, RED_OR>((int)(hi | any), red);  // any: as 33 bits when only low words are in use
  __syncthreads();
  return r ? 64 - __clz(r) : kZeroTop;
}

template <int LOGN>
__global__ void __launch_bounds__(Shape<LOGN>::threads, resident(Shape<LOGN>::threads))
    k_rows_forward(const double* __restrict__ F, c64* __restrict__ Z, int2* __restrict__ ez,
                   const int4* __restrict__ tw) {
  using S = Shape<LOGN>;
  extern __shared__ c64 fsm[];
  __shared__ int red[S::threads / 32];
  const int g = threadIdx.x / S::NT, i = threadIdx.x % S::NT;
  const int row = blockIdx.x * S::rows + g;
  const double* fx = F + (size_t)row * S::n;
  const double* fy = fx + (size_t)S::n * S::n;
  double x[8], y[8];
  int e = 1;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    x[q] = fx[i + q * S::NT];
    y[q] = fy[i + q * S::NT];
    e = max(e, max(exponent_field(x[q]), exponent_field(y[q])));
  }
  const int emax = row_reduce<LOGN, RED_MAX>(e, red);
  __syncthreads();
  c64 v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = {from_double(x[q], emax), from_double(y[q], emax)};
  int E = emax - 1081;
  fft<LOGN, -1>(v, E, i, fsm + (size_t)g * S::n, red, tw);
#pragma unroll
  for (int p = 0; p < 8; ++p) Z[(size_t)(i + p * S::NT) * S::n + row] = v[p];
  int top = row_bits<LOGN>(v, red);
  if (top != kZeroTop) top += E;
  if (emax == 0x7ff) top = kNanTop;
  if (i == 0) ez[row] = make_int2(E, top);
}

// Column kx: see the head of the file. A group of threads per component c (and derivative d, see Columns);
// the spectra, and later the inverse transforms, of the two components meet in shared memory. With two
// turns per group the spectrum of the group's component waits in the CTA's own columns of Z (columns n and
// n + 1 in place of the second one at kx = 0 and n / 2), every thread reading back what it wrote.
template <int LOGN>
__global__ void __launch_bounds__(Columns<LOGN>::threads, resident(Columns<LOGN>::threads))
    k_columns(double two_pi_over_L, const double* __restrict__ mult, int mult_exp, c64* Z, const int2* __restrict__ ez, c64* __restrict__ A,
              c64* __restrict__ D, int* __restrict__ ea, int* __restrict__ ed, const int4* __restrict__ tw) {
  using S = Shape<LOGN>;
  using C = Columns<LOGN>;
  constexpr int n = S::n, half = n / 2;
  extern __shared__ c64 fsm[];
  __shared__ int red[(C::threads + 31) / 32];
  __shared__ int2 ex[C::cols * C::groups];
  const int grp = threadIdx.x / S::NT, i = threadIdx.x % S::NT;
  const int c = grp & 1;
  const int kx = blockIdx.x * C::cols + grp / C::groups;
  const bool live = kx <= half;
  const int col = live ? kx : half, mir = (n - col) & (n - 1);
  c64* buf = fsm + (size_t)grp * n;
  c64* other = fsm + (size_t)(grp ^ 1) * n;
  double2* park = reinterpret_cast<double2*>(Z + (size_t)(c == 0 ? col : (mir != col ? mir : n + (col != 0))) * n);

  int top = kZeroTop;
  int er[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int2 e = ez[i + q * S::NT];
    er[q] = e.x;
    top = max(top, e.y);
  }
  top = row_reduce<LOGN, RED_MAX>(top, red);
  bool poison = top == kNanTop;
  const int E0 = top - (kTopBits - 1);  // |z| < 2^58 in this unit

  // spectrum along y of F_x or F_y: 2 F_x = z(kx) + conj z(-kx), 2 i F_y = z(kx) - conj z(-kx)
  c64 v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int y = i + q * S::NT, s = E0 - er[q];
    const c64 zp = Z[(size_t)col * n + y], zm = Z[(size_t)mir * n + y];
    const c64 p = {shift_rn(zp.x, s), shift_rn(zp.y, s)}, m = {shift_rn(zm.x, s), shift_rn(zm.y, s)};
    v[q] = c == 0 ? c64{p.x + m.x, p.y - m.y} : c64{p.y + m.y, m.x - p.x};
  }
  int E = E0 - 1;
  __syncthreads();
  fft<LOGN, -1>(v, E, i, buf, red, tw);
  double2 w[8];
  double2* mine = reinterpret_cast<double2*>(buf);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    w[q] = make_double2((double)v[q].x, (double)v[q].y);
    mine[q * S::NT + i] = w[q];
  }
  if (i == 0) ex[grp].x = E;
  __syncthreads();

  // the multiplier: u = k_perp (k_perp . F) mult, in units of 2^E
  const int de = max(-900, min(900, ex[grp ^ 1].x - E));
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int iy = i + q * S::NT, ky = iy <= half ? iy : iy - n;
    const double2 o = reinterpret_cast<const double2*>(other)[q * S::NT + i];
    const double m = __ldg(mult + (size_t)col * (half + 1) + (ky < 0 ? -ky : ky));
    const double2 fs = w[q];                                                // own component
    const double2 fo = make_double2(times_pow2(o.x, de), times_pow2(o.y, de));  // the other
    const double ko = c == 0 ? ky : col, ks = c == 0 ? col : ky;
    if (col == 0 && iy == 0) {
      w[q] = make_double2(m * fs.x, m * fs.y);
    } else if ((col == half) != (iy == half)) {
      // on the Nyquist row or column (not the corner) the wavenumber n/2 stands for +n/2 and -n/2 alike,
      // and the cross term, odd in it, averages to zero: the multiplier of a real field stays even
      w[q] = make_double2(m * ko * ko * fs.x, m * ko * ko * fs.y);
    } else {
      const double mk = m * ko;
      w[q] = make_double2(mk * (ko * fs.x - ks * fo.x), mk * (ko * fs.y - ks * fo.y));
    }
    if (C::turns == 2 && live) park[i + q * S::NT] = w[q];
  }
  const int E1 = E + mult_exp;

  // inverse transforms along y of u (d = 0) and k_y u (d = 1; the derivative is i times this, and the
  // Nyquist wavenumber carries none: its sine mode vanishes on the grid)
#pragma unroll 1
  for (int t = 0; t < C::turns; ++t) {
    const int d = C::turns == 2 ? t : (grp >> 1) & 1;
    if (t && live) {
#pragma unroll
      for (int q = 0; q < 8; ++q) w[q] = park[i + q * S::NT];
    }
    int e = 1;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int iy = i + q * S::NT;
      const double dk = two_pi_over_L * (iy < half ? iy : (iy == half ? 0 : iy - n));
      if (d) w[q] = make_double2(w[q].x * dk, w[q].y * dk);
      e = max(e, max(exponent_field(w[q].x), exponent_field(w[q].y)));
    }
    const int emax = row_reduce<LOGN, RED_MAX>(e, red);
    poison |= emax == 0x7ff;  // the multiplier overflowed
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = {from_double(w[q].x, emax), from_double(w[q].y, emax)};
    E = emax - 1081 + E1;
    __syncthreads();
    fft<LOGN, 1>(v, E, i, buf, red, tw);
    int own = row_bits<LOGN>(v, red);
    if (own != kZeroTop) own += E;
    if (poison) own = kNanTop;
#pragma unroll
    for (int q = 0; q < 8; ++q) buf[q * S::NT + i] = v[q];
    if (i == 0) ex[grp] = make_int2(E, own);
    __syncthreads();
    // one unit for both components: |u| < 2^60. Group 0 stores u_x + i u_y at kx, group 1 the same of the
    // conjugates at -kx (times -1 for k_y u: i k_y u is the real field)
    const int2 eo = ex[grp ^ 1];
    const int tm = max(own, eo.y), Eo = tm - 60, s0 = Eo - E, s1 = Eo - eo.x;
    c64* out = d ? D : A;
    if (live && (c == 0 || mir != col)) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const c64 o = other[q * S::NT + i];
        const c64 a = {shift_rn(v[q].x, s0), shift_rn(v[q].y, s0)}, b = {shift_rn(o.x, s1), shift_rn(o.y, s1)};
        c64 r;  // c = 0: a + i b; c = 1 (a = u_y, b = u_x): conj b + i conj a, negated for d = 1
        if (c == 0) r = {a.x - b.y, a.y + b.x};
        else if (d == 0) r = {b.x + a.y, a.x - b.y};
        else r = {-b.x - a.y, b.y - a.x};
        out[(size_t)(i + q * S::NT) * n + (c == 0 ? col : mir)] = r;
      }
      if (i == 0) (d ? ed : ea)[c == 0 ? col : mir] = tm == kNanTop || tm == kZeroTop ? tm : Eo;
    }
    __syncthreads();
  }
}

// Row y, field 0: A -> u; 1: k_x A -> d u / dx; 2: D -> d u / dy (the last two times i).
template <int LOGN>
__global__ void __launch_bounds__(Shape<LOGN>::threads, resident(Shape<LOGN>::threads))
    k_rows_inverse(const int4* __restrict__ wave, const c64* __restrict__ A, const c64* __restrict__ D,
                   const int* __restrict__ ea, const int* __restrict__ ed, double* __restrict__ u,
                   double* __restrict__ gradu, const int4* __restrict__ tw) {
  using S = Shape<LOGN>;
  constexpr int n = S::n;
  extern __shared__ c64 fsm[];
  __shared__ int red[S::threads / 32];
  const int g = threadIdx.x / S::NT, i = threadIdx.x % S::NT;
  const int field = blockIdx.x % 3, row = blockIdx.x / 3 * S::rows + g;
  const c64* in = (field == 2 ? D : A) + (size_t)row * n;
  const int* ee = field == 2 ? ed : ea;
  c64 v[8];
  int er[8], top = kZeroTop;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    v[q] = in[i + q * S::NT];
    er[q] = ee[i + q * S::NT];
  }
  if (field == 1) {
    // k_x as a mantissa and an exponent, so the element keeps its relative precision; none at 0 and n / 2
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int4 k = __ldg(wave + i + q * S::NT);
      v[q] = {mul_hi(v[q].x, k.x, k.y), mul_hi(v[q].y, k.x, k.y)};  // v k / 4, |.| < 2^59
      if (er[q] != kNanTop) er[q] = er[q] == kZeroTop || k.z == kZeroTop ? kZeroTop : er[q] + k.z;
    }
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) top = max(top, er[q]);
  top = row_reduce<LOGN, RED_MAX>(top, red);
  __syncthreads();
  const bool poison = top == kNanTop;
  const int up = field == 1 ? 0 : 2;  // |A|, |D| < 2^61 -> 2^59
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = {shift_rn(v[q].x, top - er[q] + up), shift_rn(v[q].y, top - er[q] + up)};
  int E = top == kZeroTop || poison ? 0 : top + up;
  fft<LOGN, 1>(v, E, i, fsm + (size_t)g * n, red, tw);
  E -= 2 * LOGN;  // 1 / n^2
  const size_t nn = (size_t)n * n, o = (size_t)row * n;
  double* re = (field == 0 ? u : gradu + (field == 1 ? 2 : 3) * nn) + o;       // field 0: u_x; else d u_y
  double* im = (field == 0 ? u + nn : gradu + (field == 1 ? 0 : 1) * nn) + o;  // field 0: u_y; else -d u_x
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int ix = i + q * S::NT;
    double a = (double)v[q].x, b = (double)(field == 0 ? v[q].y : -v[q].y);
    if (E > -900 && E < 900) {
      a = times_pow2(a, E);
      b = times_pow2(b, E);
    } else {
      a = ldexp(a, E);
      b = ldexp(b, E);
    }
    if (poison) a = b = __longlong_as_double(0x7ff8000000000000ll);
    re[ix] = a;
    im[ix] = b;
  }
}

__global__ void k_multiplier(int half, double alpha, double two_pi_over_L, double unit, double* mult) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int w = half + 1;
  if (e >= (long long)w * w) return;
  const double i = (double)(e / w), j = (double)(e % w);
  const double r2 = i * i + j * j, k2 = two_pi_over_L * two_pi_over_L * r2;
  mult[e] = r2 == 0.0 ? unit / (alpha * alpha) : unit / (r2 * (alpha * alpha + k2));
}

// ------------------------------------------------------------------ twiddles (host)

// cos and sin of 2 pi / 2^b in units of 2^-62, by the half-angle formulas on 128-bit integers.
struct Root { int64_t c, s; };

uint64_t isqrt128(unsigned __int128 x) {
  unsigned __int128 r = 0;
  for (int b = 63; b >= 0; --b) {
    const unsigned __int128 t = r | ((unsigned __int128)1 << b);
    if (t * t <= x) r = t;
  }
  return (uint64_t)r;
}

Root mul_root(Root a, Root b) {
  auto rnd = [](__int128 x) { return (int64_t)((x + ((__int128)1 << 61)) >> 62); };
  return {rnd((__int128)a.c * b.c - (__int128)a.s * b.s), rnd((__int128)a.c * b.s + (__int128)a.s * b.c)};
}

int4 to_digits(Root r) {
  auto split = [](int64_t v, int& h, int& l) {
    l = (int32_t)(uint32_t)(uint64_t)v;
    h = (int32_t)((v - l) >> 32);
    if (l == INT32_MIN) ++l;  // keeps -l representable (one unit of 2^-62)
  };
  int4 d;
  split(r.c, d.x, d.y);
  split(r.s, d.z, d.w);
  return d;
}

// Stage by stage (m = 1, 8, ..), [p = 1 .. 7][j < l]: e^(2 pi i p j m / n).
void make_twiddles(int logn, std::vector<int4>& out) {
  const int n = 1 << logn;
  const int64_t one = (int64_t)1 << 62;
  std::vector<Root> w(n);
  w[0] = {one, 0};
  Root r{-one, 0};  // e^(2 pi i / 2^b), b = 1
  for (int b = 1; b <= logn; ++b) {
    if (b == 2) {
      r = {0, one};
    } else if (b > 2) {
      const int64_t c = (int64_t)isqrt128((unsigned __int128)(uint64_t)((one + r.c) >> 1) << 62);
      r = {c, (int64_t)((((__int128)r.s << 61) + c / 2) / c)};
    }
    // the points at odd multiples of n / 2^b
    for (int q = n >> b; q < n; q += 2 * (n >> b)) w[q] = mul_root(w[q - (n >> b)], r);
  }
  out.clear();
  for (int m = 1; n / (8 * m) > 1; m *= 8) {
    const int l = n / (8 * m);
    for (int p = 1; p < 8; ++p)
      for (int j = 0; j < l; ++j) out.push_back(to_digits(w[(int64_t)p * j * m % n]));
  }
}

// k_x of a derivative along x, zero at n/2: 2^e m with m in units of 2^-62 given as balanced digits; (mh, ml, e + 2)
// so that mul_hi(v, mh, ml) 2^(e + 2) is v k_x.
void make_wave(int n, double two_pi_over_L, std::vector<int4>& out) {
  out.resize(n);
  for (int q = 0; q < n; ++q) {
    const int k = q < n / 2 ? q : (q == n / 2 ? 0 : q - n);
    int e = 0;
    const double m = std::frexp(two_pi_over_L * k, &e);
    const int4 d = to_digits({(int64_t)std::ldexp(m, 62), 0});
    out[q] = int4{d.x, d.y, k ? e + 2 : kZeroTop, 0};
  }
}

// ------------------------------------------------------------------ launches by size

template <int LOGN>
size_t smem_rows() { return (size_t)Shape<LOGN>::rows * Shape<LOGN>::n * sizeof(c64); }

template <int LOGN>
size_t smem_columns() { return (size_t)Columns<LOGN>::cols * Columns<LOGN>::groups * Shape<LOGN>::n * sizeof(c64); }

template <int LOGN>
int prepare_size() {
  TRY(cudaFuncSetAttribute(k_rows_forward<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_rows<LOGN>()));
  TRY(cudaFuncSetAttribute(k_columns<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_columns<LOGN>()));
  TRY(cudaFuncSetAttribute(k_rows_inverse<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_rows<LOGN>()));
  return VP_OK;
}

template <int LOGN>
int eval_size(const vp_periodic_s* P, const double* F, double* u, double* gradu, cudaStream_t s) {
  using S = Shape<LOGN>;
  using C = Columns<LOGN>;
  k_rows_forward<LOGN><<<S::n / S::rows, S::threads, smem_rows<LOGN>(), s>>>(F, P->z, P->ez, P->tw);
  TRY(cudaGetLastError());
  k_columns<LOGN><<<(S::n / 2 + C::cols) / C::cols, C::threads, smem_columns<LOGN>(), s>>>(
      2.0 * kPi / P->side, P->mult, P->mult_exp, P->z, P->ez, P->a, P->d, P->ea, P->ed, P->tw);
  TRY(cudaGetLastError());
  k_rows_inverse<LOGN><<<3 * (S::n / S::rows), S::threads, smem_rows<LOGN>(), s>>>(P->wave, P->a, P->d, P->ea, P->ed,
                                                                                    u, gradu, P->tw);
  TRY(cudaGetLastError());
  return VP_OK;
}

}  // namespace
}  // namespace vp

using namespace vp;

#define VP_BY_SIZE(logn, call)        \
  switch (logn) {                     \
    case 5: return call<5>;           \
    case 6: return call<6>;           \
    case 7: return call<7>;           \
    case 8: return call<8>;           \
    case 9: return call<9>;           \
    case 10: return call<10>;         \
    case 11: return call<11>;         \
    default: return call<12>;         \
  }

namespace {
typedef int (*prepare_fn)();
typedef int (*eval_fn)(const vp_periodic_s*, const double*, double*, double*, cudaStream_t);
prepare_fn prepare_of(int logn) { VP_BY_SIZE(logn, prepare_size) }
eval_fn eval_of(int logn) { VP_BY_SIZE(logn, eval_size) }
}  // namespace

extern "C" int vp_periodic_create(double alpha, int n, double side, void* stream, vp_periodic* out) {
  if (!out) return VP_ERR_ARG;
  *out = nullptr;
  if (!(alpha > 0.0) || !(side > 0.0) || n < (1 << kMinLog) || n > kMaxN || (n & (n - 1))) return VP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  vp_periodic_s* P = new (std::nothrow) vp_periodic_s();
  if (!P) return VP_ERR_OOM;
  P->alpha = alpha; P->side = side; P->n = n;
  while ((1 << P->logn) < n) ++P->logn;
  auto fail = [&](int code) { vp_periodic_free(P); return code; };
  auto alloc = [&](auto** p, size_t count) {
    if (cudaMalloc(p, count * sizeof(**p)) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
  };
  const size_t nn = (size_t)n * n, hw = (size_t)n / 2 + 1;
  std::vector<int4> tw, wave;
  make_twiddles(P->logn, tw);
  make_wave(n, 2.0 * kPi / side, wave);
  if (!alloc(&P->z, nn + 2 * (size_t)n) || !alloc(&P->a, nn) || !alloc(&P->d, nn) || !alloc(&P->ez, n) || !alloc(&P->ea, n) ||
      !alloc(&P->ed, n) || !alloc(&P->mult, hw * hw) || !alloc(&P->wave, n) || !alloc(&P->tw, tw.size()))
    return fail(VP_ERR_OOM);
  const int rc = prepare_of(P->logn)();
  if (rc) return fail(rc);
  P->mult_exp = alpha < 1.0 ? 128 : 0;
  k_multiplier<<<(unsigned)((hw * hw + 255) / 256), 256, 0, s>>>(n / 2, alpha, 2.0 * kPi / side, std::ldexp(1.0, -P->mult_exp),
                                                                 P->mult);
  if (cudaMemcpyAsync(P->tw, tw.data(), tw.size() * sizeof(int4), cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(P->wave, wave.data(), wave.size() * sizeof(int4), cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    set_last_cuda(cudaGetLastError());
    return fail(VP_ERR_CUDA);
  }
  *out = P;
  return VP_OK;
}

extern "C" int vp_periodic_eval(vp_periodic P, const double* F, double* u, double* gradu, void* stream) {
  if (!P || !F || !u || !gradu) return VP_ERR_ARG;
  return eval_of(P->logn)(P, F, u, gradu, static_cast<cudaStream_t>(stream));
}

extern "C" void vp_periodic_free(vp_periodic P) {
  if (!P) return;
  for (void* p : {(void*)P->z, (void*)P->a, (void*)P->d, (void*)P->ez, (void*)P->ea, (void*)P->ed, (void*)P->mult,
                  (void*)P->wave, (void*)P->tw})
    if (p) cudaFree(p);
  delete P;
}
