// Learned warm start for the boundary integral equation: a circular 1D convolutional network over
// the boundary nodes with hand-written FP32 forward, backward and Adam kernels.
//
// Layers l = 0..L-1 map C_l -> C_{l+1} channels (C_0 = in_ch, C_L = out_ch, width in between):
//   z_{l+1}[b][o][x] = bias_l[o] + sum_{c,k} W_l[o][c][k] a_l[b][c][(x + k - K/2) mod n],
//   a_{l+1} = relu(z_{l+1}) for l < L-1, output y = z_L.
// Loss mean((y - t)^2); backward: dW_l[o][c][k] = sum_{b,x} dz[b][o][x] a_l[b][c][x + k - K/2],
// dbias_l[o] = sum dz, and da_l = the same convolution of dz with the weights transposed in (o, c)
// and reversed in k; relu masks by a > 0. Adam (Kingma & Ba) with bias correction.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <memory>
#include <new>
#include <vector>

#include "vp_internal.h"
#include "../../include/bie.h"

namespace vp {
namespace {

#define TRY(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { set_last_cuda(e_); return e_ == cudaErrorMemoryAllocation ? VP_ERR_OOM : VP_ERR_CUDA; } } while (0)

constexpr int kMaxK = 15;
constexpr int kTC = 8;      // input channels per shared chunk
constexpr int kTO = 64;     // output channels per block at most
constexpr int kWPitch = kTO + 4;

// Positions of halo kept on each side of a tile, a whole number of 16-byte groups.
__host__ __device__ constexpr int halo(int K) { return (K / 2 + 3) / 4 * 4; }

__device__ inline void cp_async16(float* smem, const float* gmem, bool valid) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  const int bytes = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(bytes) : "memory");
}
__device__ inline void cp_async4(float* smem, const float* gmem, bool valid) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  const int bytes = valid ? 4 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sa), "l"(gmem), "r"(bytes) : "memory");
}

// Rows r < rows of sm (pitch P) = src[r][(x0 + xx) mod n] for 0 <= xx < LEN (x0 >= -n), zeros for r >= have and for
// x0 + xx >= lim. vec: src 16-byte aligned, n and x0 multiples of 4, so whole groups of 4 wrap together.
template <int LEN, int P>
__device__ inline void load_rows(float* sm, const float* src, int rows, int have, int n, int x0, int lim, bool vec,
                                 int tid, int nt) {
  static_assert(LEN % 4 == 0 && P % 4 == 0, "whole groups");
  if (vec) {
    for (int e = tid; e < rows * (LEN / 4); e += nt) {
      const int r = e / (LEN / 4), x = (e - r * (LEN / 4)) * 4;
      int gx = x0 + x;
      const bool ok = r < have && gx < lim;
      gx = gx < 0 ? gx + n : (gx >= n ? gx - n : gx);
      cp_async16(sm + r * P + x, ok ? src + (size_t)r * n + gx : src, ok);
    }
  } else {
    for (int e = tid; e < rows * LEN; e += nt) {
      const int r = e / LEN, x = e - r * LEN;
      int gx = x0 + x;
      const bool ok = r < have && gx < lim && gx >= -n;
      gx = gx < 0 ? gx + n : (gx >= n ? gx - n : gx);
      cp_async4(sm + r * P + x, ok ? src + (size_t)r * n + gx : src, ok);
    }
  }
}

__host__ __device__ inline int pad4(int c) { return (c + 3) & ~3; }

// out[b][o][x] = (bias ? bias[o] : 0) + sum_{c,k} w(o, c, k) in[b][c][(x + k - K/2) mod n], the weights laid out as
// W[c][k][pad4(Cout)] (Layer); relu: max(., 0); mask (an array like out): 0 where mask is not positive.
//
// A thread holds OT output channels x XT groups of 4 positions in registers (the groups XG * 4 apart, so that
// the 16-byte reads of the window are free of bank conflicts). Per input channel it reads the window of
// K + 3 positions of each group once and, per tap, OT weights by broadcast: with 8 x 8 outputs and K = 9, 24
// shared reads of 16 bytes for 576 multiply-adds, so the FP32 pipe bounds it and not shared memory (one
// output per position read took 17 reads per 16 multiply-adds). Chunks of kTC channels are copied one ahead
// by 16-byte cp.async (scalar loads of the parameter order cost as many instructions as the multiply-adds).
// Every output is summed in the order of the definition, channel after channel, tap after tap.
template <int K, int OT, int XT, int XG>
__global__ void __launch_bounds__(256) k_conv(int n, int Cin, int Cout, const float* __restrict__ W,
                                              const float* __restrict__ bias, const float* __restrict__ in,
                                              float* __restrict__ out, int relu, const float* __restrict__ mask,
                                              int vec) {
  constexpr int TX = XG * 4 * XT, PAD = halo(K), TP = TX + 2 * PAD;  // positions of a block; row of the input tile
  constexpr int half = K / 2, off = PAD - half;                    // first tap of a group's window
  constexpr int NW = (off + K + 6) / 4;                            // 16-byte reads per window
  extern __shared__ __align__(16) float conv_sm[];  // [2][input tile [kTC][TP], weights [kTC][K][kWPitch]]
  constexpr int kBuf = kTC * (TP + K * kWPitch);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int xg = tid % XG, og = tid / XG;
  const int x0 = blockIdx.x * TX, o0 = blockIdx.y * kTO, b = blockIdx.z;
  const int ldw = pad4(Cout), wq = min(kTO, ldw - o0) / 4;  // weight row; groups of 4 of it in this block
  float acc[OT][XT][4];
#pragma unroll
  for (int r = 0; r < OT; ++r) {
    const int o = o0 + og * OT + r;
    const float v = (bias && o < Cout) ? bias[o] : 0.f;
#pragma unroll
    for (int j = 0; j < XT; ++j)
#pragma unroll
      for (int t = 0; t < 4; ++t) acc[r][j][t] = v;
  }
  auto load = [&](int c0, float* sm) {
    // positions past the last output's window are not used
    load_rows<TP, TP>(sm, in + ((size_t)b * Cin + c0) * n, kTC, Cin - c0, n, x0 - PAD, n + half, vec, tid, nt);
    float* ws = sm + kTC * TP;
    const int rows = min(kTC, Cin - c0) * K;
    for (int e = tid; e < kTC * K * wq; e += nt) {
      const int row = e / wq, q = (e - row * wq) * 4;
      const bool ok = row < rows;
      cp_async16(ws + row * kWPitch + q, ok ? W + (size_t)(c0 * K + row) * ldw + o0 + q : W, ok);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  load(0, conv_sm);
  for (int c0 = 0, st = 0; c0 < Cin; c0 += kTC, st ^= 1) {
    if (c0 + kTC < Cin) {
      load(c0 + kTC, conv_sm + (st ^ 1) * kBuf);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    const float* tile = conv_sm + st * kBuf;
    const float* wsh = tile + kTC * TP;
#pragma unroll 1
    for (int c = 0; c < kTC; ++c) {
      float win[XT][NW * 4];
#pragma unroll
      for (int j = 0; j < XT; ++j)
#pragma unroll
        for (int q = 0; q < NW; ++q) {
          const float4 v = *reinterpret_cast<const float4*>(tile + c * TP + (j * XG + xg + q) * 4);
          win[j][4 * q] = v.x; win[j][4 * q + 1] = v.y; win[j][4 * q + 2] = v.z; win[j][4 * q + 3] = v.w;
        }
#pragma unroll
      for (int k = 0; k < K; ++k) {
        float w[OT];
        if constexpr (OT >= 4) {
#pragma unroll
          for (int r = 0; r < OT; r += 4) {
            const float4 v = *reinterpret_cast<const float4*>(wsh + (c * K + k) * kWPitch + og * OT + r);
            w[r] = v.x; w[r + 1] = v.y; w[r + 2] = v.z; w[r + 3] = v.w;
          }
        } else {
#pragma unroll
          for (int r = 0; r < OT; ++r) w[r] = wsh[(c * K + k) * kWPitch + og * OT + r];
        }
#pragma unroll
        for (int r = 0; r < OT; ++r)
#pragma unroll
          for (int j = 0; j < XT; ++j)
#pragma unroll
            for (int t = 0; t < 4; ++t) acc[r][j][t] = fmaf(w[r], win[j][off + k + t], acc[r][j][t]);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < OT; ++r) {
    const int o = o0 + og * OT + r;
    if (o >= Cout) break;
    float* y = out + ((size_t)b * Cout + o) * n;
    const float* m = mask ? mask + ((size_t)b * Cout + o) * n : nullptr;
#pragma unroll
    for (int j = 0; j < XT; ++j) {
      const int x = x0 + (j * XG + xg) * 4;
      float v[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        v[t] = relu ? fmaxf(acc[r][j][t], 0.f) : acc[r][j][t];
        if (m && x + t < n && !(m[x + t] > 0.f)) v[t] = 0.f;
      }
      if (vec) {
        if (x < n) *reinterpret_cast<float4*>(y + x) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (x + t < n) y[x + t] = v[t];
      }
    }
  }
}

template <int K, int XT, int XG>
constexpr size_t conv_smem() { return (size_t)2 * kTC * (XG * 4 * XT + 2 * halo(K) + K * kWPitch) * sizeof(float); }

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

template <int K, int OT, int XT, int XG>
int launch_conv(int n, int B, int Cin, int Cout, const float* W, const float* bias, const float* in, float* out,
                int relu, const float* mask, cudaStream_t s) {
  constexpr int TX = XG * 4 * XT;
  const int co = std::min(Cout, kTO), vec = n % 4 == 0 && aligned16(in) && aligned16(out);
  k_conv<K, OT, XT, XG><<<dim3((n + TX - 1) / TX, (Cout + kTO - 1) / kTO, B), (co + OT - 1) / OT * XG,
                          conv_smem<K, XT, XG>(), s>>>(n, Cin, Cout, W, bias, in, out, relu, mask, vec);
  TRY(cudaGetLastError());
  return VP_OK;
}

// 8 x 8 outputs a thread where that gives every SM two blocks (304 on 152 SMs); 4 x 4 where it does not (four
// times the threads); one output channel a thread for at most two of them, which would leave most of an 8 x 8
// tile empty. Measured (64 -> 64 channels, K = 9, n = 4096): batch 32 204 us = 47 TFLOP/s, FP32 pipe 67 % busy (389 us
// with one position per thread); batch 1, 4 x 4 tiles, the whole network of four layers 66 us (243).
template <int K>
int launch_conv_k(int n, int B, int Cin, int Cout, const float* W, const float* bias, const float* in, float* out,
                  int relu, const float* mask, cudaStream_t s) {
  const long long blocks = (long long)((n + 127) / 128) * ((Cout + kTO - 1) / kTO) * B;
  const auto f = Cout <= 2 ? launch_conv<K, 1, 1, 16> : (blocks >= 304 ? launch_conv<K, 8, 2, 16> : launch_conv<K, 4, 1, 8>);
  return f(n, B, Cin, Cout, W, bias, in, out, relu, mask, s);
}

// The weights of a layer ([out][in][k] at woff in the parameters, the bias at boff) as k_conv reads them:
// wf[in][k][pad4(out)] for the forward pass, and wb[out][k][pad4(in)], reversed in k, for the transposed convolution of
// the backward pass. The padding is zero from the allocation on.
struct Layer {
  size_t woff, boff;
  int Cin, Cout;
  float *wf, *wb;
};

// Parameter e, now v, into its layer's layouts.
__device__ inline void store_layouts(const Layer* __restrict__ layers, int L, int K, size_t e, float v) {
  int l = 0;
  for (int hi = L - 1; l < hi;) {
    const int mid = (l + hi + 1) / 2;
    if (layers[mid].woff <= e) l = mid;
    else hi = mid - 1;
  }
  const Layer y = layers[l];
  if (e >= y.boff) return;  // a bias
  e -= y.woff;              // layers of 2^31 weights and more are accepted
  const int c = (int)(e / K % y.Cin), k = (int)(e % K);
  const size_t o = e / K / y.Cin;
  y.wf[((size_t)c * K + k) * pad4(y.Cout) + o] = v;
  y.wb[(o * K + K - 1 - k) * pad4(y.Cin) + c] = v;
}

__global__ void k_layouts(const Layer* __restrict__ layers, int L, int K, size_t m, const float* __restrict__ p) {
  const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (e < m) store_layouts(layers, L, K, e, p[e]);
}

// Part sums of dW[o][c][k] = sum_{b,x} dz[b][o][x] a[b][c][(x + k - K/2) mod n] and dbias[o] = sum dz over a
// segment of the positions: block (seg, pair) takes every gridDim.x-th chunk of kWX positions for the pair0 + pair-th
// pair of an output and an input channel tile.
// A thread holds OT output channels x 2 input channels x K taps in registers and walks along x four positions at a
// time, so an input position is read once for its K taps: with OT = 4 and K = 9, 10 shared reads of 16 bytes for
// 288 multiply-adds (one (o, c) pair per block read 10 values from L1 per 10 multiply-adds). Chunks are copied
// to shared memory one ahead (cp.async). Row pitches of 4 mod 32 words and channels dealt out row by row keep
// the reads free of bank conflicts. part[seg][pair][output][input channel][tap], then [output] for the bias, is summed
// by k_sum_parts, so the result does not depend on the order in which blocks run.
// SHORT: eight products are added up before they enter a running sum, which keeps its chain to 8 and its error to that of
// one term per thread and a tree over the threads; it costs an eighth more instructions (batch 32, n = 4096: 1,806 instead
// of 1,666 us for the gradient), so longer sums, whose single chains of B n / 304 products stay below
// the B n / 256 of 256 threads, do without.
// Measured (64 x 64 channels, K = 9, n = 4096, batch 32): 227 us = 43 TFLOP/s, FP32 pipe 58 % busy, 13 us for the
// sum (about 3.3 ms with a block per (o, c) pair).
constexpr int kWX = 64;                   // positions per chunk
constexpr int kWPitchZ = kWX + 4;         // row of the dz chunk
constexpr int kWPitchA = kWX + 20;        // row of the activation chunk (halos of at most 8 on each side)

// Output channels held by a thread (at most 72 sums) and of a tile; the tiles of a layer and their share of a segment's
// part sums.
__host__ __device__ constexpr int wgrad_ot(int K) { return K <= 9 ? 4 : 2; }
struct WgradTiles {
  int no, nc, pairs_c, pairs;  // channels of a tile (the layer's, if fewer), input tiles, pairs of tiles
  size_t ld;                   // part sums of a pair
};
WgradTiles wgrad_tiles(int Cin, int Cout, int K) {
  const int ot = 16 * wgrad_ot(K);
  WgradTiles t;
  t.no = std::min(Cout, ot);
  t.nc = std::min(Cin, kTO);
  t.pairs_c = (Cin + kTO - 1) / kTO;
  t.pairs = (Cout + ot - 1) / ot * t.pairs_c;
  t.ld = (size_t)t.no * t.nc * K + t.no;
  return t;
}

template <int K, bool SHORT>
__global__ void __launch_bounds__(512) k_conv_wgrad(int n, int B, int Cin, int Cout, const float* __restrict__ dz,
                                                    const float* __restrict__ a, float* __restrict__ part,
                                                    WgradTiles tl, int pair0, int vec) {
  extern __shared__ __align__(16) float wg_sm[];
  constexpr int OT = wgrad_ot(K), half = K / 2, PAD = halo(K), off = PAD - half;
  constexpr int kStep = SHORT ? 8 : 4, NW = (off + K + kStep + 2) / 4;  // positions of a step; 16-byte reads per window
  constexpr int kOTile = 16 * OT;
  const int ot = (pair0 + (int)blockIdx.y) / tl.pairs_c, ct = (pair0 + (int)blockIdx.y) - ot * tl.pairs_c;
  const int o0 = ot * kOTile, c0 = ct * kTO;
  const int no = min(kOTile, Cout - o0), nc = min(kTO, Cin - c0);
  const int nog = (no + OT - 1) / OT, ncg = (nc + 1) / 2;
  const int zrows = nog * OT, arows = ncg * 2;
  const int buf = zrows * kWPitchZ + arows * kWPitchA;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int cg = tid % ncg, og = tid / ncg;
  const bool live = og < nog;
  const int nx = (n + kWX - 1) / kWX, chunks = B * nx;

  auto load = [&](int ch, float* sm) {
    const int b = ch / nx, x0 = (ch - b * nx) * kWX;
    load_rows<kWX, kWPitchZ>(sm, dz + ((size_t)b * Cout + o0) * n, zrows, no, n, x0, n, vec, tid, nt);
    load_rows<kWX + 2 * PAD, kWPitchA>(sm + zrows * kWPitchZ, a + ((size_t)b * Cin + c0) * n, arows, nc, n, x0 - PAD,
                                      n + half, vec, tid, nt);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };

  float acc[OT][2][K];
#pragma unroll
  for (int r = 0; r < OT; ++r)
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int k = 0; k < K; ++k) acc[r][q][k] = 0.f;
  float bsum = 0.f;
  int ch = blockIdx.x, st = 0;
  if (ch < chunks) load(ch, wg_sm);
  for (; ch < chunks; ch += gridDim.x, st ^= 1) {
    const int next = ch + gridDim.x;
    if (next < chunks) {
      load(next, wg_sm + (st ^ 1) * buf);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    const float* sz = wg_sm + st * buf;
    const float* sa = sz + zrows * kWPitchZ;
    if (live) {
#pragma unroll 1
      for (int x = 0; x < kWX; x += kStep) {
        float w[2][NW * 4];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int t = 0; t < NW; ++t) {
            const float4 v = *reinterpret_cast<const float4*>(sa + (cg + q * ncg) * kWPitchA + x + 4 * t);
            w[q][4 * t] = v.x; w[q][4 * t + 1] = v.y; w[q][4 * t + 2] = v.z; w[q][4 * t + 3] = v.w;
          }
#pragma unroll
        for (int r = 0; r < OT; ++r) {
          float d[kStep];
#pragma unroll
          for (int t = 0; t < kStep; t += 4) {
            const float4 v = *reinterpret_cast<const float4*>(sz + (og + r * nog) * kWPitchZ + x + t);
            d[t] = v.x; d[t + 1] = v.y; d[t + 2] = v.z; d[t + 3] = v.w;
          }
#pragma unroll
          for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int k = 0; k < K; ++k) {
              float s = SHORT ? 0.f : acc[r][q][k];
#pragma unroll
              for (int t = 0; t < kStep; ++t) s = fmaf(d[t], w[q][off + t + k], s);
              acc[r][q][k] = SHORT ? acc[r][q][k] + s : s;
            }
        }
      }
    }
    if (ct == 0 && tid < no) {
      for (int x = 0; x < kWX; x += 8) {
        const float4 y = *reinterpret_cast<const float4*>(sz + tid * kWPitchZ + x);
        const float4 z = *reinterpret_cast<const float4*>(sz + tid * kWPitchZ + x + 4);
        bsum += ((y.x + y.y) + (y.z + y.w)) + ((z.x + z.y) + (z.z + z.w));
      }
    }
    __syncthreads();
  }
  float* pw = part + ((size_t)blockIdx.x * gridDim.y + blockIdx.y) * tl.ld;
  if (live) {
#pragma unroll
    for (int r = 0; r < OT; ++r)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int o = og + r * nog, c = cg + q * ncg;
        if (o < no && c < nc)
#pragma unroll
          for (int k = 0; k < K; ++k) pw[((size_t)o * tl.nc + c) * K + k] = acc[r][q][k];
      }
  }
  if (ct == 0 && tid < no) pw[(size_t)tl.no * tl.nc * K + tid] = bsum;
}

size_t wgrad_smem(int zrows, int arows) { return (size_t)2 * (zrows * kWPitchZ + arows * kWPitchA) * sizeof(float); }

// Pairs pair0 .. pair0 + pairs - 1 of the layer's tiles.
template <int K>
int launch_wgrad_k(int n, int B, int Cin, int Cout, const float* dz, const float* a, float* part, int segs,
                   const WgradTiles& tl, int pair0, int pairs, cudaStream_t s) {
  constexpr int OT = wgrad_ot(K);
  const int nog = (tl.no + OT - 1) / OT, ncg = (tl.nc + 1) / 2;
  const int threads = std::max(64, (nog * ncg + 31) / 32 * 32);  // a thread per output channel for the bias sums
  const bool one_chunk = (long long)B * ((n + kWX - 1) / kWX) == segs;
  (one_chunk ? k_conv_wgrad<K, true> : k_conv_wgrad<K, false>)<<<dim3(segs, pairs), threads, wgrad_smem(nog * OT, ncg * 2), s>>>(
      n, B, Cin, Cout, dz, a, part, tl, pair0, n % 4 == 0 && aligned16(dz) && aligned16(a));
  TRY(cudaGetLastError());
  return VP_OK;
}

template <int K>
int prepare_k() {
  for (auto f : {k_conv_wgrad<K, true>, k_conv_wgrad<K, false>})
    TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wgrad_smem(kTO, kTO)));
  TRY(cudaFuncSetAttribute(k_conv<K, 1, 1, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)conv_smem<K, 1, 16>()));
  TRY(cudaFuncSetAttribute(k_conv<K, 8, 2, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)conv_smem<K, 2, 16>()));
  TRY(cudaFuncSetAttribute(k_conv<K, 4, 1, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)conv_smem<K, 1, 8>()));
  return VP_OK;
}

// Kernel sizes are odd and at most kMaxK.
#define WS_BY_K(k, call)                 \
  switch (k) {                           \
    case 1: return call<1>;              \
    case 3: return call<3>;              \
    case 5: return call<5>;              \
    case 7: return call<7>;              \
    case 9: return call<9>;              \
    case 11: return call<11>;            \
    case 13: return call<13>;            \
    default: return call<15>;            \
  }
auto conv_of(int k) -> decltype(&launch_conv_k<1>) { WS_BY_K(k, launch_conv_k) }
auto wgrad_of(int k) -> decltype(&launch_wgrad_k<1>) { WS_BY_K(k, launch_wgrad_k) }
auto prepare_of(int k) -> decltype(&prepare_k<1>) { WS_BY_K(k, prepare_k) }

// Segments of a weight gradient: two blocks per SM of the 152 (an uneven last wave costs less, and the running sums are
// half as long as with one), whatever the layer's width: tiles beyond kPartBytes of part sums take their turns
// (one pair of tiles takes 45 MB at most). Fewer segments for wider layers made the sums longer: at 512 x 512 channels,
// K = 15, 2048 positions the gradient's error was 1.08e-7 with 8 segments and single running sums, 6.2e-8 with a tree
// over 256 threads, 4.6e-8 now.
// No more segments than chunks: the sums over empty ones cost a network of 4 channels 73 -> 85 us a gradient.
constexpr int kMaxSegs = 304;
int wgrad_segs(int n, int B) { return (int)std::min<long long>(kMaxSegs, (long long)B * ((n + kWX - 1) / kWX)); }
constexpr size_t kPartBytes = (size_t)128 << 20;
size_t part_floats(const WgradTiles& tl, int segs) {
  const size_t one = segs * tl.ld;
  return one * std::max<size_t>(1, std::min<size_t>(tl.pairs, kPartBytes / sizeof(float) / one));
}

// Sums over the segments of part[seg][m], compensated, into the layer's gradient g (weights [output][input][tap], then
// the bias): 32 part sums per block, warp w taking the segments w mod 8, the eight sums added in their order.
__global__ void __launch_bounds__(256) k_sum_parts(size_t m, int segs, const float* __restrict__ part, WgradTiles tl,
                                                   int pair0, int Cin, int Cout, int K, float* __restrict__ g) {
  __shared__ float2 sh[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const size_t p = blockIdx.x * (size_t)32 + lane;
  float s = 0.f, e = 0.f;
  auto add = [&](float v) {
    const float t = s + v, bb = t - s;
    e += (s - (t - bb)) + (v - bb);
    s = t;
  };
  if (p < m) {
#pragma unroll 8
    for (int q = w; q < segs; q += 8) add(part[q * m + p]);
  }
  sh[w][lane] = make_float2(s, e);
  __syncthreads();
  if (w || p >= m) return;
  for (int q = 1; q < 8; ++q) {
    add(sh[q][lane].x);
    e += sh[q][lane].y;
  }
  const int pair = pair0 + (int)(p / tl.ld), ot = pair / tl.pairs_c, ct = pair - ot * tl.pairs_c;
  int r = (int)(p % tl.ld);
  const int weights = tl.no * tl.nc * K, o = ot * 16 * wgrad_ot(K) + (r < weights ? r / (tl.nc * K) : r - weights);
  if (o >= Cout) return;
  if (r < weights) {
    r %= tl.nc * K;
    const int c = ct * kTO + r / K;
    if (c < Cin) g[((size_t)o * Cin + c) * K + r % K] = s + e;
  } else if (ct == 0) {
    g[(size_t)Cout * Cin * K + o] = s + e;
  }
}

// g = 2 (y - t) / m and partial sums of (y - t)^2 (one per block, into part[blockIdx.x]).
__global__ void k_mse(size_t m, const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ g,
                      double* __restrict__ part) {
  __shared__ double red[32];
  double s = 0.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < m; i += (size_t)gridDim.x * blockDim.x) {
    const float d = y[i] - t[i];
    g[i] = 2.f * d / (float)m;
    s += (double)d * d;
  }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
  }
}

// Adam, and the layouts of the new weights (a launch per layer for them took a step of three small layers from 93 to
// 110 us).
__global__ void k_adam(size_t m, float* __restrict__ p, const float* __restrict__ g, float* __restrict__ mo,
                       float* __restrict__ ve, float lr, float b1, float b2, float eps, float c1, float c2,
                       const Layer* __restrict__ layers, int L, int K) {
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= m) return;
  const float gi = g[i];
  const float mi = b1 * mo[i] + (1.f - b1) * gi;
  const float vi = b2 * ve[i] + (1.f - b2) * gi * gi;
  mo[i] = mi;
  ve[i] = vi;
  const float v = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  p[i] = v;
  store_layouts(layers, L, K, i, v);
}

}  // namespace
}  // namespace vp

struct ws_s {
  int in_ch = 0, width = 0, out_ch = 0, L = 0, K = 0, n = 0, max_batch = 0;
  std::vector<int> C;                       // channels per activation, size L+1
  std::vector<size_t> woff, boff;           // parameter offsets
  size_t nparams = 0;
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
  std::vector<float*> wf, wb;               // per layer: the weights as k_conv reads them (Layer)
  vp::Layer* layers = nullptr;                  // the same on the device
  std::vector<float*> act;                  // activations a_0..a_{L-1}, z_L (size L+1), max_batch each
  float *d0 = nullptr, *d1 = nullptr;       // gradient work buffers
  double* part = nullptr;
  float* wparts = nullptr;                  // part sums of a layer's weight gradient, or of some of its tiles
  size_t part_count = 0;                    // elements of wparts
  long long step = 0;
  std::vector<void*> allocs;
};

using namespace vp;

namespace {

int walloc(ws_s* w, float** p, size_t n) {
  void* q = nullptr;
  TRY(cudaMalloc(&q, std::max<size_t>(1, n) * sizeof(float)));
  w->allocs.push_back(q);
  *p = static_cast<float*>(q);
  return VP_OK;
}

// splitmix64 (Steele, Lea and Flood 2014): counter-based seeded uniform numbers for initialisation.
inline uint64_t splitmix64(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// The convolution layouts of the weights, after the parameters have been replaced.
int layout(ws_s* w, cudaStream_t s) {
  k_layouts<<<(unsigned)((w->nparams + 255) / 256), 256, 0, s>>>(w->layers, w->L, w->K, w->nparams, w->p);
  TRY(cudaGetLastError());
  return VP_OK;
}

// y: destination of the last layer.
int forward(ws_s* w, const float* x, int B, float* y, cudaStream_t s) {
  const float* in = x;
  for (int l = 0; l < w->L; ++l) {
    float* out = l == w->L - 1 ? y : w->act[l + 1];
    const int rc = conv_of(w->K)(w->n, B, w->C[l], w->C[l + 1], w->wf[l], w->p + w->boff[l], in, out,
                                 l < w->L - 1 ? 1 : 0, nullptr, s);
    if (rc) return rc;
    in = out;
  }
  return VP_OK;
}

int grad(ws_s* w, const float* x, const float* t, int B, float* loss, cudaStream_t s) {
  if (B < 1 || B > w->max_batch) return VP_ERR_ARG;
  // keep the input as a_0 (read only; the caller's buffer)
  int rc = forward(w, x, B, w->act[w->L], s);
  if (rc) return rc;
  const size_t mout = (size_t)B * w->out_ch * w->n;
  const int nb = 256;
  k_mse<<<nb, 256, 0, s>>>(mout, w->act[w->L], t, w->d0, w->part);
  TRY(cudaGetLastError());
  float* dz = w->d0;
  float* da = w->d1;
  for (int l = w->L - 1; l >= 0; --l) {
    const int Cin = w->C[l], Cout = w->C[l + 1];
    const float* a = (l == 0) ? x : w->act[l];
    const WgradTiles tl = wgrad_tiles(Cin, Cout, w->K);
    const int segs = wgrad_segs(w->n, B);
    const bool direct = segs == 1 && tl.pairs == 1;  // the one tile's part sums are the gradient, in its order
    const int group = (int)std::min<size_t>({(size_t)tl.pairs, w->part_count / (segs * tl.ld), 65535});
    float* g = w->g + w->woff[l];
    for (int pair0 = 0; pair0 < tl.pairs; pair0 += group) {
      const int pairs = std::min(group, tl.pairs - pair0);
      if ((rc = wgrad_of(w->K)(w->n, B, Cin, Cout, dz, a, direct ? g : w->wparts, segs, tl, pair0, pairs, s))) return rc;
      if (direct) break;
      const size_t m = pairs * tl.ld;
      k_sum_parts<<<(unsigned)((m + 31) / 32), 256, 0, s>>>(m, segs, w->wparts, tl, pair0, Cin, Cout, w->K, g);
      TRY(cudaGetLastError());
    }
    if (l > 0) {
      // da masked by the activation of the layer
      if ((rc = conv_of(w->K)(w->n, B, Cout, Cin, w->wb[l], nullptr, dz, da, 0, w->act[l], s))) return rc;
      std::swap(dz, da);
    }
  }
  std::vector<double> part(nb);
  TRY(cudaMemcpyAsync(part.data(), w->part, nb * sizeof(double), cudaMemcpyDeviceToHost, s));
  TRY(cudaStreamSynchronize(s));
  double tot = 0.0;
  for (double v : part) tot += v;
  if (loss) *loss = (float)(tot / (double)mout);
  return VP_OK;
}

}  // namespace

extern "C" void ws_free(ws_net net) {
  if (!net) return;
  for (void* p : net->allocs) cudaFree(p);
  delete net;
}

extern "C" int ws_create(int in_ch, int width, int out_ch, int n_layers, int ksize, int n, int max_batch,
                         uint64_t seed, void* stream, ws_net* out) {
  if (!out) return VP_ERR_ARG;
  *out = nullptr;
  if (in_ch < 1 || width < 1 || out_ch < 1 || n_layers < 1 || ksize < 1 || ksize > kMaxK || (ksize % 2) == 0 ||
      n < ksize || max_batch < 1)
    return VP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  std::unique_ptr<ws_s> w(new (std::nothrow) ws_s());
  if (!w) return VP_ERR_OOM;
  w->in_ch = in_ch; w->width = width; w->out_ch = out_ch; w->L = n_layers; w->K = ksize; w->n = n;
  w->max_batch = max_batch;
  w->C.assign(n_layers + 1, width);
  w->C[0] = in_ch;
  w->C[n_layers] = out_ch;
  size_t off = 0;
  for (int l = 0; l < n_layers; ++l) {
    w->woff.push_back(off);
    off += (size_t)w->C[l + 1] * w->C[l] * ksize;
    w->boff.push_back(off);
    off += w->C[l + 1];
  }
  w->nparams = off;
  int rc;
  auto fail = [&](int code) { ws_free(w.release()); return code; };
  if ((rc = walloc(w.get(), &w->p, off)) || (rc = walloc(w.get(), &w->g, off)) || (rc = walloc(w.get(), &w->m, off)) ||
      (rc = walloc(w.get(), &w->v, off)))
    return fail(rc);
  w->act.assign(n_layers + 1, nullptr);
  size_t maxc = 0;
  for (int l = 0; l <= n_layers; ++l) maxc = std::max<size_t>(maxc, w->C[l]);
  for (int l = 1; l <= n_layers; ++l)
    if ((rc = walloc(w.get(), &w->act[l], (size_t)max_batch * w->C[l] * n))) return fail(rc);
  if ((rc = walloc(w.get(), &w->d0, (size_t)max_batch * maxc * n)) ||
      (rc = walloc(w.get(), &w->d1, (size_t)max_batch * maxc * n)))
    return fail(rc);
  // the layouts of all layers in one piece, zero where they are padded; the part sums
  size_t parts = 0, lay = 0;
  std::vector<Layer> layers(n_layers);
  for (int l = 0; l < n_layers; ++l) {
    const int cin = w->C[l], cout = w->C[l + 1];
    lay += (size_t)cin * ksize * pad4(cout) + (size_t)cout * ksize * pad4(cin);
    parts = std::max(parts, part_floats(wgrad_tiles(cin, cout, ksize), wgrad_segs(n, max_batch)));
  }
  w->part_count = parts;
  float* at = nullptr;
  if ((rc = walloc(w.get(), &at, lay)) || (rc = walloc(w.get(), &w->wparts, parts)) || (rc = prepare_of(ksize)()))
    return fail(rc);
  if (cudaMemsetAsync(at, 0, lay * sizeof(float), s) != cudaSuccess) return fail(VP_ERR_CUDA);
  for (int l = 0; l < n_layers; ++l) {
    const int cin = w->C[l], cout = w->C[l + 1];
    float* wb = at + (size_t)cin * ksize * pad4(cout);
    layers[l] = {w->woff[l], w->boff[l], cin, cout, at, wb};
    w->wf.push_back(at);
    w->wb.push_back(wb);
    at = wb + (size_t)cout * ksize * pad4(cin);
  }
  {
    void* q = nullptr;
    const size_t sums = 256 * sizeof(double), bytes = layers.size() * sizeof(Layer);
    if (cudaMalloc(&q, sums + bytes) != cudaSuccess) return fail(VP_ERR_OOM);
    w->allocs.push_back(q);
    w->part = static_cast<double*>(q);
    w->layers = reinterpret_cast<Layer*>(w->part + 256);
    if (cudaMemcpyAsync(w->layers, layers.data(), bytes, cudaMemcpyHostToDevice, s) != cudaSuccess) return fail(VP_ERR_CUDA);
  }
  // initial parameters: uniform in +-1/sqrt(fan_in) from a seeded splitmix64 stream
  std::vector<float> host(off);
  uint64_t st = seed;
  for (int l = 0; l < n_layers; ++l) {
    const float bound = 1.f / std::sqrt((float)(w->C[l] * ksize));
    for (size_t i = w->woff[l]; i < w->boff[l] + w->C[l + 1]; ++i) {
      const double u = (double)(splitmix64(st) >> 11) * (1.0 / 9007199254740992.0);
      host[i] = (float)((2.0 * u - 1.0) * bound);
    }
  }
  if (cudaMemcpyAsync(w->p, host.data(), off * sizeof(float), cudaMemcpyHostToDevice, s) != cudaSuccess ||
      layout(w.get(), s) != VP_OK || cudaMemsetAsync(w->m, 0, off * sizeof(float), s) != cudaSuccess ||
      cudaMemsetAsync(w->v, 0, off * sizeof(float), s) != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess)
    return fail(VP_ERR_CUDA);
  *out = w.release();
  return VP_OK;
}

extern "C" int ws_num_params(ws_net net, int64_t* count) {
  if (!net || !count) return VP_ERR_ARG;
  *count = (int64_t)net->nparams;
  return VP_OK;
}

extern "C" int ws_params(ws_net net, float* buf, int get, void* stream) {
  if (!net || !buf) return VP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (get) TRY(cudaMemcpyAsync(buf, net->p, net->nparams * sizeof(float), cudaMemcpyDeviceToDevice, s));
  else TRY(cudaMemcpyAsync(net->p, buf, net->nparams * sizeof(float), cudaMemcpyDeviceToDevice, s));
  return get ? VP_OK : layout(net, s);
}

extern "C" int ws_forward(ws_net net, const float* x, int batch, float* y, void* stream) {
  if (!net || !x || !y || batch < 1 || batch > net->max_batch) return VP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // a single layer reads x while it writes: it goes through the activation buffer, so y may be x as before
  if (net->L > 1) return forward(net, x, batch, y, s);
  const int rc = forward(net, x, batch, net->act[1], s);
  if (rc) return rc;
  TRY(cudaMemcpyAsync(y, net->act[1], (size_t)batch * net->out_ch * net->n * sizeof(float), cudaMemcpyDeviceToDevice, s));
  return VP_OK;
}

extern "C" int ws_grad(ws_net net, const float* x, const float* t, int batch, float* g, float* loss, void* stream) {
  if (!net || !x || !t || !g) return VP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int rc = grad(net, x, t, batch, loss, s);
  if (rc) return rc;
  TRY(cudaMemcpyAsync(g, net->g, net->nparams * sizeof(float), cudaMemcpyDeviceToDevice, s));
  return VP_OK;
}

extern "C" int ws_train_step(ws_net net, const float* x, const float* t, int batch, float lr, float* loss,
                             void* stream) {
  if (!net || !x || !t || !(lr > 0.f)) return VP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int rc = grad(net, x, t, batch, loss, s);
  if (rc) return rc;
  net->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)net->step), c2 = 1.f - std::pow(b2, (float)net->step);
  k_adam<<<(unsigned)((net->nparams + 255) / 256), 256, 0, s>>>(net->nparams, net->p, net->g, net->m, net->v, lr, b1,
                                                                 b2, 1e-8f, c1, c2, net->layers, net->L, net->K);
  TRY(cudaGetLastError());
  return VP_OK;
}
