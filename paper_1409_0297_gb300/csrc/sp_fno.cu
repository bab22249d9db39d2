// Fourier-layer network for the learned initial guess of the solve: forward pass,
// backward pass, Adam, and the packing of features, guesses and targets.
//
// The network is the Fourier neural operator of Li et al. (ICLR 2021, Section 4):
// a pointwise lift, L Fourier layers v <- gelu(W v + b + K v) with K a truncated
// spectral convolution, and a two-layer pointwise projection; Adam follows Kingma and
// Ba (ICLR 2015, Algorithm 1).  Weights are used as bfloat16 (an FP32 master copy is
// updated by Adam), activations are stored as bfloat16 (or FP32 for checks) and every
// product accumulates in FP32.
//
// Layout: tensors [b][c][j0 + n j1].  The truncated transform keeps kx = 0..M-1 along
// axis 0 and ky in {0..M-1} U {n-M..n-1} along axis 1; it runs as two dense stages
// (rows: a real-to-complex DFT of each grid row onto M modes; columns: a complex DFT
// of each mode column onto 2M modes), each a small contraction against a twiddle
// table held in shared memory.  The inverse stage along rows is fused into the
// kernel that adds the pointwise branch, the bias and the activation, so the spatial
// output of the spectral branch never goes to memory.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <exception>
#include <new>
#include <vector>

#include "sp_fno.h"

namespace {

typedef __nv_bfloat16 bf16;

constexpr int kRowsCta = 128;     // grid rows per CTA of the row transform
constexpr int kRowPitch = kRowsCta + 4;
constexpr int kRowChunk = 32;     // points of a row staged at a time
constexpr int kWgChunk = 2048;    // points per CTA of the weight-gradient reduction
constexpr int kWgSub = 64;
constexpr int kLossChunks = 64;   // CTAs per sample of the loss reduction
constexpr int kNormBlocks = 256;

__device__ __forceinline__ float ldf(const float* p) { return *p; }
__device__ __forceinline__ float ldf(const bf16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ void stf(float* p, float v) { *p = v; }
__device__ __forceinline__ void stf(bf16* p, float v) { *p = __float2bfloat16_rn(v); }

// gelu(x) = x Phi(x) and its derivative Phi(x) + x phi(x)
__device__ __forceinline__ float gelu_f(float x) {
  return 0.5f * x * (1.f + erff(x * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_d(float x) {
  return 0.5f * (1.f + erff(x * 0.70710678118654752f)) +
         x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// four consecutive values (p a multiple of 4)
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const bf16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st4(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(bf16* p, const float* v) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
  uint2 u;
  u.x = *reinterpret_cast<const unsigned*>(&a);
  u.y = *reinterpret_cast<const unsigned*>(&b);
  *reinterpret_cast<uint2*>(p) = u;
}

// The kernels below keep the order in which every output adds its products (inputs, modes
// and points ascending), so a launch shape never changes a bit of the network.

// ------------------------------------------------------------------ pointwise linear
// Y[b][o][p] = act(sum_i W[o ldw + i] X[b][i][p] + bias[o]); gelu: pre receives the value
// before the activation.  P is a multiple of 4 (n a multiple of 64); aligned: X starts on a
// 16-byte boundary (a caller's input may not).
// A CTA keeps the weights and a 128-point tile in shared memory; a thread owns 8 outputs x 4
// points, so 32 FMAs take 3 shared loads (one point per thread took 3 for 8, and the shared
// pipe bound it: width 32 -> 128 with GELU, 16 x 256^2 points: 489 us).  What bounds it now:
// the FMAs and erff.
constexpr int kTP = 128;
template <class TX, class TY>
__global__ void __launch_bounds__(kTP)
    chan_linear_kernel(const TX* __restrict__ X, int ci, const bf16* __restrict__ W, int ldw,
                       const bf16* __restrict__ bias, int co, long P, int gelu,
                       TY* __restrict__ pre, TY* __restrict__ Y, int aligned) {
  extern __shared__ float4 smf4[];
  float* sm = reinterpret_cast<float*>(smf4);
  const int co8 = (co + 7) & ~7;
  float* Ws = sm;             // [ci][co8]
  float* bs = Ws + ci * co8;  // [co8]
  float* Xs = bs + co8;       // [ci][kTP]
  for (int idx = threadIdx.x; idx < ci * co8; idx += kTP) {
    const int o = idx / ci, i = idx - o * ci;
    Ws[i * co8 + o] = o < co ? __bfloat162float(W[(long)o * ldw + i]) : 0.f;
  }
  for (int o = threadIdx.x; o < co8; o += kTP) bs[o] = o < co ? __bfloat162float(bias[o]) : 0.f;
  const int b = blockIdx.y;
  const TX* Xb = X + (long)b * ci * P;
  const int pg = threadIdx.x & 31, og = threadIdx.x >> 5;
  for (long p0 = (long)blockIdx.x * kTP; p0 < P; p0 += (long)gridDim.x * kTP) {
    __syncthreads();
    for (int idx = threadIdx.x; idx < ci * (kTP / 4); idx += kTP) {
      const int i = idx >> 5, q = (idx & 31) * 4;
      const TX* src = Xb + (long)i * P + p0 + q;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (p0 + q < P) {
        if (aligned) v = ld4(src);
        else v = make_float4(ldf(src), ldf(src + 1), ldf(src + 2), ldf(src + 3));
      }
      *reinterpret_cast<float4*>(Xs + i * kTP + q) = v;
    }
    __syncthreads();
    const long p = p0 + 4 * pg;
    for (int o0 = og * 8; o0 < co8; o0 += 32) {
      float acc[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = bs[o0 + j];
#pragma unroll 4
      for (int i = 0; i < ci; ++i) {
        const float4 x = *reinterpret_cast<const float4*>(Xs + i * kTP + 4 * pg);
        const float4 w0 = *reinterpret_cast<const float4*>(Ws + i * co8 + o0);
        const float4 w1 = *reinterpret_cast<const float4*>(Ws + i * co8 + o0 + 4);
        const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
        const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[j][q] = fmaf(wv[j], xv[q], acc[j][q]);
      }
      if (p >= P) continue;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (o0 + j >= co) break;
        const long idx = ((long)b * co + o0 + j) * P + p;
        if (gelu) {
          if (pre != nullptr) st4(pre + idx, acc[j]);
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[j][q] = gelu_f(acc[j][q]);
        }
        st4(Y + idx, acc[j]);
      }
    }
  }
}

// The same for few outputs (the projection's last layer, CO <= 8): the inputs stream through
// registers, four points per thread, and nothing but the weights is staged.  Bound by
// reading X once (128 -> 2, 16 x 256^2 points, 268 MB: 330 us through the tile above, whose
// outputs are padded to 8).
template <class TX, int CO>
__global__ void __launch_bounds__(128)
    chan_narrow_kernel(const TX* __restrict__ X, int ci, const bf16* __restrict__ W, int ldw,
                       const bf16* __restrict__ bias, int co, long P, float* __restrict__ Y) {
  __shared__ float Ws[128 * CO];
  for (int idx = threadIdx.x; idx < ci * CO; idx += 128) {
    const int i = idx / CO, o = idx % CO;
    Ws[idx] = o < co ? __bfloat162float(W[(long)o * ldw + i]) : 0.f;
  }
  __syncthreads();
  const int b = blockIdx.y;
  const long p = 4 * ((long)blockIdx.x * 128 + threadIdx.x);
  if (p >= P) return;
  float acc[CO][4];
#pragma unroll
  for (int o = 0; o < CO; ++o)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[o][q] = o < co ? __bfloat162float(bias[o]) : 0.f;
  const TX* Xb = X + (long)b * ci * P + p;
#pragma unroll 8
  for (int i = 0; i < ci; ++i) {
    const float4 x = ld4(Xb + (long)i * P);
    const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int o = 0; o < CO; ++o)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[o][q] = fmaf(Ws[i * CO + o], xv[q], acc[o][q]);
  }
#pragma unroll
  for (int o = 0; o < CO; ++o)
    if (o < co) st4(Y + ((long)b * co + o) * P + p, acc[o]);
}

// ------------------------------------------------------------------ weight gradients
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// part[(b nchunk + chunk)][o ci + i] = sum over the chunk's points of dY[b][o][p] X[b][i][p],
// part[..][co ci + o] = sum dY[b][o][p].  One CTA per chunk; thread t < own adds the points of
// a 4 x 4 set of (o, i) in order (o = ob + r co4 / 4, i = ib + c ci4 / 4, so that a warp's
// reads of a tile spread over the banks), one more warp the bias sums.  The chunk streams
// through kWgStages tiles of kWgSub points in shared memory, channel-major as it lies in
// device memory (cp.async, X still in its storage type).  With plain loads of one tile at a
// time the reduction waited for memory (235 us per 32 x 32 layer at 16 x 256^2 points, whose
// FMAs take 27).  aligned = 0 (a caller's X off the 16-byte grid) copies with plain loads.
constexpr int kWgStages = 3;
template <class TX>
__global__ void __launch_bounds__(288)
    chan_wgrad_kernel(const float* __restrict__ dY, int co, const TX* __restrict__ X, int ci, long P,
                      float* __restrict__ part, int own, int aligned) {
  extern __shared__ float4 smf4[];
  constexpr int pY = kWgSub + 4, pX = kWgSub + 16 / (int)sizeof(TX);  // row pitches (16-byte rows)
  const int co4 = (co + 3) & ~3, ci4 = (ci + 3) & ~3;
  const size_t ybytes = (size_t)co4 * pY * sizeof(float), xbytes = (size_t)ci4 * pX * sizeof(TX);
  unsigned char* sm = reinterpret_cast<unsigned char*>(smf4);
  auto tY = [&](int st) { return reinterpret_cast<float*>(sm + st * (ybytes + xbytes)); };
  auto tX = [&](int st) { return reinterpret_cast<TX*>(sm + st * (ybytes + xbytes) + ybytes); };
  const int t = threadIdx.x, nth = blockDim.x;
  const int nob = co4 / 4, nib = ci4 / 4;
  const int ob = t / nib, ib = t - ob * nib;
  const bool owner = t < nob * nib;
  const int bt = t - own;  // bias channel of the extra warp's lanes
  const int b = blockIdx.y;
  const long c0 = (long)blockIdx.x * kWgChunk;
  const long c1 = c0 + kWgChunk < P ? c0 + kWgChunk : P;  // P and kWgChunk are multiples of kWgSub
  const float* Yb = dY + (long)b * co * P;
  const TX* Xb = X + (long)b * ci * P;
  const int ntile = (int)((c1 - c0) / kWgSub);
  // rows that pad the channels to a multiple of four stay zero
  for (int st = 0; st < kWgStages; ++st) {
    for (int e = t; e < (co4 - co) * pY; e += nth) tY(st)[co * pY + e] = 0.f;
    for (int e = t; e < (ci4 - ci) * pX; e += nth) stf(tX(st) + ci * pX + e, 0.f);
  }
  auto fetch = [&](int tile) {
    if (tile < ntile) {
      const long p = c0 + (long)tile * kWgSub;
      float* y = tY(tile % kWgStages);
      TX* x = tX(tile % kWgStages);
      constexpr int vY = 4, vX = 16 / (int)sizeof(TX);
      for (int e = t; e < co * (kWgSub / vY); e += nth) {
        const int o = e / (kWgSub / vY), q = vY * (e % (kWgSub / vY));
        cp_async16(y + o * pY + q, Yb + (long)o * P + p + q);
      }
      for (int e = t; e < ci * (kWgSub / vX); e += nth) {
        const int i = e / (kWgSub / vX), q = vX * (e % (kWgSub / vX));
        const TX* src = Xb + (long)i * P + p + q;
        if (aligned) {
          cp_async16(x + i * pX + q, src);
        } else {
#pragma unroll
          for (int u = 0; u < vX; ++u) x[i * pX + q + u] = src[u];
        }
      }
    }
    cp_commit();
  };
  float acc[16];
  float accb = 0.f;
#pragma unroll
  for (int j = 0; j < 16; ++j) acc[j] = 0.f;
  for (int st = 0; st < kWgStages - 1; ++st) fetch(st);
  for (int tile = 0; tile < ntile; ++tile) {
    cp_wait<kWgStages - 2>();
    __syncthreads();  // tile arrived; everyone is done with the stage that is refilled now
    fetch(tile + kWgStages - 1);
    const float* y = tY(tile % kWgStages);
    const TX* x = tX(tile % kWgStages);
    if (owner) {
#pragma unroll 2
      for (int q = 0; q < kWgSub; q += 4) {
        float yv[4][4], xv[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float4 v = *reinterpret_cast<const float4*>(y + (ob + r * nob) * pY + q);
          yv[r][0] = v.x, yv[r][1] = v.y, yv[r][2] = v.z, yv[r][3] = v.w;
          const float4 w = ld4(x + (ib + r * nib) * pX + q);
          xv[r][0] = w.x, xv[r][1] = w.y, xv[r][2] = w.z, xv[r][3] = w.w;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r * 4 + c] = fmaf(yv[r][u], xv[c][u], acc[r * 4 + c]);
      }
    } else if (bt >= 0 && bt < co) {
#pragma unroll 4
      for (int q = 0; q < kWgSub; q += 4) {
        const float4 v = *reinterpret_cast<const float4*>(y + bt * pY + q);
        accb += v.x;
        accb += v.y;
        accb += v.z;
        accb += v.w;
      }
    }
  }
  cp_wait<0>();
  float* out = part + ((long)b * gridDim.x + blockIdx.x) * (long)(co * ci + co);
  if (owner) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int o = ob + r * nob;
      if (o >= co) continue;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int i = ib + c * nib;
        if (i < ci) out[o * ci + i] = acc[r * 4 + c];
      }
    }
  }
  if (bt >= 0 && bt < co) out[co * ci + bt] = accb;
}

// Projection backward, both products of its hidden-layer gradient
// de[h][p] = (sum_o Q2[o][h] dY[o][p]) gelu'(E[h][p]): the partial sums of dQ1 (rows h, as
// chan_wgrad_kernel with the last layer's output v) and dv_i = sum_h Q1[h][i] de_h.  A tile of
// de is formed once in shared memory and never goes to device memory (H <= 128, W <= 32,
// c2 <= 8).  What bounds it: erff and expf of gelu'; formed twice, once for each product, the
// two kernels took 1.70 ms at 16 x 256^2 points.
template <class TA>
__global__ void __launch_bounds__(256)
    proj_bwd_kernel(const float* __restrict__ dY, int c2, const TA* __restrict__ E, int H,
                    const bf16* __restrict__ Q2, const bf16* __restrict__ Q1, const TA* __restrict__ V,
                    int W, long P, float* __restrict__ dv, float* __restrict__ part) {
  extern __shared__ float4 smf4[];
  constexpr int pH = 132, pW = 36;  // row pitches: 16-byte rows, spread over the banks
  float* sD = reinterpret_cast<float*>(smf4);  // [kWgSub][pH] de
  float* sV = sD + kWgSub * pH;                // [kWgSub][pW] v
  float* Q1s = sV + kWgSub * pW;               // [128][32]
  float* Q2s = Q1s + 128 * 32;                 // [8][128]
  const int t = threadIdx.x;
  for (int idx = t; idx < 128 * 32; idx += 256) {
    const int h = idx >> 5, i = idx & 31;
    Q1s[idx] = (h < H && i < W) ? __bfloat162float(Q1[h * W + i]) : 0.f;
  }
  for (int idx = t; idx < 8 * 128; idx += 256) {
    const int o = idx >> 7, h = idx & 127;
    Q2s[idx] = (o < c2 && h < H) ? __bfloat162float(Q2[o * H + h]) : 0.f;
  }
  const int ob = t >> 3, ib = t & 7;         // dQ1: rows 4 ob, columns 4 ib
  const int q1 = t & 63, hg = t >> 6;        // de: point, rows 16 k + 4 hg + r
  const int q2 = t & 31, i4 = 4 * (t >> 5);  // dv: points q2, q2 + 32, first of four channels
  float acc[16];
  float accb = 0.f;
#pragma unroll
  for (int j = 0; j < 16; ++j) acc[j] = 0.f;
  const int b = blockIdx.y;
  const long c0 = (long)blockIdx.x * kWgChunk;
  const long c1 = c0 + kWgChunk < P ? c0 + kWgChunk : P;  // P and kWgChunk are multiples of kWgSub
  const float* Db = dY + (long)b * c2 * P;
  const TA* Eb = E + (long)b * H * P;
  const TA* Vb = V + (long)b * W * P;
  // the next tile's E, v and dY values travel while the current one is used
  TA ev[32], vv[8];
  float d[8];
  auto fetch = [&](long s0) {
    const long p = s0 + q1;
#pragma unroll
    for (int o = 0; o < 8; ++o) d[o] = o < c2 ? Db[(long)o * P + p] : 0.f;
#pragma unroll
    for (int u = 0; u < 32; ++u) {
      const int h = 16 * (u >> 2) + 4 * hg + (u & 3);
      if (h < H) ev[u] = Eb[(long)h * P + p];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = 16 * (u >> 2) + 4 * hg + (u & 3);
      if (i < W) vv[u] = Vb[(long)i * P + p];
    }
  };
  fetch(c0);
  for (long s0 = c0; s0 < c1; s0 += kWgSub) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int h = 16 * k + 4 * hg;
      float v[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        v[r] = 0.f;
        if (h + r < H) {
          float a = 0.f;
#pragma unroll
          for (int o = 0; o < 8; ++o)
            if (o < c2) a = fmaf(Q2s[o * 128 + h + r], d[o], a);
          v[r] = a * gelu_d(ldf(&ev[4 * k + r]));
        }
      }
      *reinterpret_cast<float4*>(sD + q1 * pH + h) = make_float4(v[0], v[1], v[2], v[3]);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = 16 * k + 4 * hg;
      float v[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) v[r] = i + r < W ? ldf(&vv[4 * k + r]) : 0.f;
      *reinterpret_cast<float4*>(sV + q1 * pW + i) = make_float4(v[0], v[1], v[2], v[3]);
    }
    if (s0 + kWgSub < c1) fetch(s0 + kWgSub);
    __syncthreads();
    float dvr[4][2];
#pragma unroll
    for (int j = 0; j < 4; ++j) dvr[j][0] = dvr[j][1] = 0.f;
    // four rows h at a time (the rows past H hold zeros), one 16-byte load per point
#pragma unroll 2
    for (int h = 0; h < H; h += 4) {
      const float4 a = *reinterpret_cast<const float4*>(sD + q2 * pH + h);
      const float4 c = *reinterpret_cast<const float4*>(sD + (q2 + 32) * pH + h);
      const float av[4] = {a.x, a.y, a.z, a.w}, cv[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 w = *reinterpret_cast<const float4*>(Q1s + (h + u) * 32 + i4);
        const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          dvr[j][0] = fmaf(wv[j], av[u], dvr[j][0]);
          dvr[j][1] = fmaf(wv[j], cv[u], dvr[j][1]);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (i4 + j < W) {
        float* out = dv + ((long)b * W + i4 + j) * P + s0 + q2;
        out[0] = dvr[j][0];
        out[32] = dvr[j][1];
      }
#pragma unroll 4
    for (int q = 0; q < kWgSub; ++q) {
      const float4 y = *reinterpret_cast<const float4*>(sD + q * pH + 4 * ob);
      const float4 x = *reinterpret_cast<const float4*>(sV + q * pW + 4 * ib);
      const float yv[4] = {y.x, y.y, y.z, y.w}, xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r * 4 + c] = fmaf(yv[r], xv[c], acc[r * 4 + c]);
    }
    if (t < H)
#pragma unroll 16
      for (int q = 0; q < kWgSub; ++q) accb += sD[q * pH + t];
  }
  float* out = part + ((long)b * gridDim.x + blockIdx.x) * (long)(H * W + H);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int h = 4 * ob + r;
    if (h >= H) continue;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int i = 4 * ib + c;
      if (i < W) out[h * W + i] = acc[r * 4 + c];
    }
  }
  if (t < H) out[H * W + t] = accb;
}

// grad[j] = sum over the nparts partials (fixed order) of part[k][j], j < len
__global__ void sum_parts_kernel(const float* __restrict__ part, int nparts, int len,
                                 float* __restrict__ grad) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= len) return;
  float s = 0.f;
  for (int k = 0; k < nparts; ++k) s += part[(long)k * len + j];
  grad[j] = s;
}

// ------------------------------------------------------------------ truncated DFT
// Rows: A[row][kx] = sum_j0 X[row][j0] e^{-2 pi i kx j0 / n}, row = (b C + c) n + j1.
// 128 rows per CTA, 32 points of them staged at a time (transposed, x[j0][row]); a thread
// owns two modes of eight rows: 32 FMAs for three 16-byte shared loads (one mode of four
// rows: 8 for two, 125 us at 16 x 32 x 256 rows of 256).
template <class TX>
__global__ void __launch_bounds__(128, sizeof(TX) == 4 ? 3 : 4)
    dft_rows_fwd_kernel(const TX* __restrict__ X, long rows, int n, int M,
                        const float2* __restrict__ twr, float2* __restrict__ A) {
  __shared__ __align__(16) float xs[kRowChunk * kRowPitch];
  __shared__ __align__(16) float2 tw[kRowChunk * 16];
  const long r0 = (long)blockIdx.x * kRowsCta;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int kp = t & 7, rg = t >> 3;  // modes 2 kp, 2 kp + 1 of rows 8 rg ..
  float ar[2][8], ai[2][8];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int q = 0; q < 8; ++q) ar[u][q] = ai[u][q] = 0.f;
  // the next chunk's values travel while the current one is multiplied
  TX pre[kRowsCta / 4];
  auto fetch = [&](int c0) {
#pragma unroll
    for (int u = 0; u < kRowsCta / 4; ++u) {
      const long r = r0 + 16 * (u >> 2) + 4 * warp + (u & 3);
      if (r < rows) pre[u] = X[r * n + c0 + lane];
    }
  };
  fetch(0);
  for (int c0 = 0; c0 < n; c0 += kRowChunk) {
    __syncthreads();
#pragma unroll
    for (int v = 0; v < kRowsCta / 16; ++v) {
      float4 x;
      const long r = r0 + 16 * v + 4 * warp;
      x.x = r + 0 < rows ? ldf(&pre[4 * v]) : 0.f;
      x.y = r + 1 < rows ? ldf(&pre[4 * v + 1]) : 0.f;
      x.z = r + 2 < rows ? ldf(&pre[4 * v + 2]) : 0.f;
      x.w = r + 3 < rows ? ldf(&pre[4 * v + 3]) : 0.f;
      *reinterpret_cast<float4*>(xs + lane * kRowPitch + 16 * v + 4 * warp) = x;
    }
    for (int idx = t; idx < kRowChunk * 16; idx += 128) tw[idx] = twr[c0 * 16 + idx];
    if (c0 + kRowChunk < n) fetch(c0 + kRowChunk);
    __syncthreads();
#pragma unroll 4
    for (int j = 0; j < kRowChunk; ++j) {
      const float4 x0 = *reinterpret_cast<const float4*>(xs + j * kRowPitch + 8 * rg);
      const float4 x1 = *reinterpret_cast<const float4*>(xs + j * kRowPitch + 8 * rg + 4);
      const float4 w = *reinterpret_cast<const float4*>(tw + j * 16 + 2 * kp);
      const float xv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        ar[0][q] = fmaf(xv[q], w.x, ar[0][q]);
        ai[0][q] = fmaf(xv[q], w.y, ai[0][q]);
        ar[1][q] = fmaf(xv[q], w.z, ar[1][q]);
        ai[1][q] = fmaf(xv[q], w.w, ai[1][q]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const long r = r0 + 8 * rg + q;
    if (r >= rows) continue;
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (2 * kp + u < M) A[r * M + 2 * kp + u] = make_float2(ar[u][q], ai[u][q]);
  }
}

__device__ __forceinline__ int ky_of(int kq, int n, int M) { return kq < M ? kq : n - 2 * M + kq; }

// Columns: V[bc][ky'][kx] = s_kx sum_j1 A[bc][j1][kx] e^{-2 pi i ky j1 / n}
// (s_0 = s0, s_kx = s1 for kx >= 1); one CTA per (b, c), a thread its two modes
// ky' = g, g + 16 of a kx together (one load of A for both).
__global__ void __launch_bounds__(256)
    dft_cols_fwd_kernel(const float2* __restrict__ A, int n, int M, const float2* __restrict__ twb,
                        float s0, float s1, float2* __restrict__ V) {
  extern __shared__ float4 smf4[];
  float2* As = reinterpret_cast<float2*>(smf4);  // [n][M]
  float2* tb = As + n * M;                        // [n]
  const long bc = blockIdx.x;
  const int t = threadIdx.x;
  for (int idx = t; idx < n * M; idx += 256) As[idx] = A[bc * n * M + idx];
  for (int idx = t; idx < n; idx += 256) tb[idx] = twb[idx];
  __syncthreads();
  const int kx = t & 15, g = t >> 4;
  const int K2 = 2 * M;
  if (kx >= M || g >= K2) return;
  const float s = kx == 0 ? s0 : s1;
  const int kb = g + 16;
  const int ka = ky_of(g, n, M), kc = kb < K2 ? ky_of(kb, n, M) : 0;
  float re[2] = {0.f, 0.f}, im[2] = {0.f, 0.f};
  int e0 = 0, e1 = 0;
#pragma unroll 4
  for (int j1 = 0; j1 < n; ++j1) {
    const float2 a = As[j1 * M + kx], w = tb[e0], v = tb[e1];
    re[0] = fmaf(a.x, w.x, fmaf(-a.y, w.y, re[0]));
    im[0] = fmaf(a.x, w.y, fmaf(a.y, w.x, im[0]));
    re[1] = fmaf(a.x, v.x, fmaf(-a.y, v.y, re[1]));
    im[1] = fmaf(a.x, v.y, fmaf(a.y, v.x, im[1]));
    e0 += ka;
    if (e0 >= n) e0 -= n;
    e1 += kc;
    if (e1 >= n) e1 -= n;
  }
  V[(bc * K2 + g) * M + kx] = make_float2(s * re[0], s * im[0]);
  if (kb < K2) V[(bc * K2 + kb) * M + kx] = make_float2(s * re[1], s * im[1]);
}

// Columns, inverse: Bc[bc][j1][kx] = sum_ky' Y[bc][ky'][kx] e^{+2 pi i ky j1 / n}.
// Thread (kx, g) owns the rows j1 = g, g + 16, ... of its CTA's share of the rows
// (blockIdx.y, RT rows a thread) for NC channels, which share every twiddle load; the
// twiddle index of a mode advances by 16 ky (mod n) from one of its rows to the next.
// n % 64 == 0.  NC = 2, RT = n / 16 for a training batch (74 us a call with one channel),
// NC = 1 and the rows over four CTAs for a single sample (35 us with one CTA per channel).
template <int NC, int RT>
__global__ void __launch_bounds__(256)
    dft_cols_inv_kernel(const float2* __restrict__ Y, int n, int M, int nbc,
                        const float2* __restrict__ twb, float2* __restrict__ Bc) {
  extern __shared__ float4 smf4[];
  const int K2 = 2 * M;
  float2* Ys = reinterpret_cast<float2*>(smf4);  // [NC][2M][M]
  float2* tb = Ys + NC * K2 * M;                  // [n]
  const long bc = (long)blockIdx.x * NC;
  const int t = threadIdx.x;
  const int have = min(NC, (int)(nbc - bc));
  for (int idx = t; idx < have * K2 * M; idx += 256) Ys[idx] = Y[bc * K2 * M + idx];
  for (int idx = t; idx < n; idx += 256) tb[idx] = twb[idx];
  __syncthreads();
  const int kx = t & 15, g = t >> 4;
  if (kx >= M) return;
  const int R = n >> 4;                      // rows per (kx, g) over all CTAs
  const int first = blockIdx.y * RT;         // rows g + 16 (first + r), r < RT
  const int last = min(R, first + RT) - first;
  float re[NC][RT], im[NC][RT];
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int r = 0; r < RT; ++r) re[c][r] = im[c][r] = 0.f;
  for (int kq = 0; kq < K2; ++kq) {
    const int ky = ky_of(kq, n, M);
    float2 y[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) y[c] = c < have ? Ys[(c * K2 + kq) * M + kx] : make_float2(0.f, 0.f);
    int e = (int)(((long)ky * (g + 16 * first)) % n);
    const int step = (int)(((long)ky * 16) % n);
#pragma unroll
    for (int r = 0; r < RT; ++r)
      if (r < last) {
        const float2 w = tb[e];  // e^{+i theta} = conj(w)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          re[c][r] = fmaf(y[c].x, w.x, fmaf(y[c].y, w.y, re[c][r]));
          im[c][r] = fmaf(y[c].y, w.x, fmaf(-y[c].x, w.y, im[c][r]));
        }
        e += step;
        if (e >= n) e -= n;
      }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int r = 0; r < RT; ++r)
      if (c < have && r < last)
        Bc[((bc + c) * n + g + 16 * (first + r)) * M + kx] = make_float2(re[c][r], im[c][r]);
}

// Mode mixing: Y[b][o][k] = sum_i V[b][i][k] R[k][i][o]; one CTA per mode k.
__global__ void __launch_bounds__(256)
    spec_mix_kernel(const float2* __restrict__ V, const bf16* __restrict__ R, int B, int W, int K,
                    float2* __restrict__ Y) {
  extern __shared__ float4 smf4[];
  float2* Rs = reinterpret_cast<float2*>(smf4);  // [W][W]
  float2* Vs = Rs + W * W;                        // [B][W]
  const int k = blockIdx.x, t = threadIdx.x;
  const bf16* Rk = R + (long)k * W * W * 2;
  for (int idx = t; idx < W * W; idx += 256)
    Rs[idx] = make_float2(__bfloat162float(Rk[2 * idx]), __bfloat162float(Rk[2 * idx + 1]));
  for (int idx = t; idx < B * W; idx += 256) Vs[idx] = V[(long)idx * K + k];
  __syncthreads();
  for (int idx = t; idx < B * W; idx += 256) {
    const int b = idx / W, o = idx % W;
    float re = 0.f, im = 0.f;
    for (int i = 0; i < W; ++i) {
      const float2 v = Vs[b * W + i], r = Rs[i * W + o];
      re = fmaf(v.x, r.x, fmaf(-v.y, r.y, re));
      im = fmaf(v.x, r.y, fmaf(v.y, r.x, im));
    }
    Y[(long)idx * K + k] = make_float2(re, im);
  }
}

// Mode mixing, backward: dV[b][i][k] = sum_o dY[b][o][k] conj(R[k][i][o]) and
// dR[k][i][o] = sum_b dY[b][o][k] conj(V[b][i][k]) (written as (re, im) floats).
__global__ void __launch_bounds__(256)
    spec_mix_bwd_kernel(const float2* __restrict__ dY, const float2* __restrict__ V,
                        const bf16* __restrict__ R, int B, int W, int K, float2* __restrict__ dV,
                        float* __restrict__ dR) {
  extern __shared__ float4 smf4[];
  float2* Rs = reinterpret_cast<float2*>(smf4);  // [W][W]
  float2* Ds = Rs + W * W;                        // [B][W]
  float2* Vs = Ds + B * W;                        // [B][W]
  const int k = blockIdx.x, t = threadIdx.x;
  const bf16* Rk = R + (long)k * W * W * 2;
  for (int idx = t; idx < W * W; idx += 256)
    Rs[idx] = make_float2(__bfloat162float(Rk[2 * idx]), __bfloat162float(Rk[2 * idx + 1]));
  for (int idx = t; idx < B * W; idx += 256) {
    Ds[idx] = dY[(long)idx * K + k];
    Vs[idx] = V[(long)idx * K + k];
  }
  __syncthreads();
  for (int idx = t; idx < B * W; idx += 256) {
    const int b = idx / W, i = idx % W;
    float re = 0.f, im = 0.f;
    for (int o = 0; o < W; ++o) {
      const float2 d = Ds[b * W + o], r = Rs[i * W + o];
      re = fmaf(d.x, r.x, fmaf(d.y, r.y, re));
      im = fmaf(d.y, r.x, fmaf(-d.x, r.y, im));
    }
    dV[(long)idx * K + k] = make_float2(re, im);
  }
  float* dRk = dR + (long)k * W * W * 2;
  for (int idx = t; idx < W * W; idx += 256) {
    const int i = idx / W, o = idx % W;
    float re = 0.f, im = 0.f;
    for (int b = 0; b < B; ++b) {
      const float2 d = Ds[b * W + o], v = Vs[b * W + i];
      re = fmaf(d.x, v.x, fmaf(d.y, v.y, re));
      im = fmaf(d.y, v.x, fmaf(-d.x, v.y, im));
    }
    dRk[2 * idx] = re;
    dRk[2 * idx + 1] = im;
  }
}

// Layer output: out[b][o][j1][j0] = sum_i Wt(o, i) X[b][i][j1][j0] + bias[o]
//   + sum_kx w_kx Re(Bc[b][o][j1][kx] e^{+2 pi i kx j0 / n}),  w_0 = w0, w_kx = w1;
// with gelu, pre <- the value and out <- gelu(value).  C <= 32, M <= 16.
// One product of depth C + 2 M per grid row: a CTA of n threads keeps the scaled twiddles of
// all points and one row's inputs in shared memory (2 x 32 x n floats) and walks `rows` grid
// rows; a thread owns 8 outputs x 4 points (32 FMAs for 3 shared loads; with one point per
// thread a load fed 4 and a single chain of 64 FMAs: 354 us at 16 x 256^2 with GELU).
template <class TX, class TY, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT <= 256 ? 3 : 1)
    combine_kernel(const TX* __restrict__ X, int C, const bf16* __restrict__ W, int trans,
                   const bf16* __restrict__ bias, const float2* __restrict__ Bc, int n, int M,
                   const float2* __restrict__ twr, float w0, float w1, int gelu,
                   TY* __restrict__ pre, TY* __restrict__ out, int rows) {
  extern __shared__ float4 smf4[];
  float* xs = reinterpret_cast<float*>(smf4);  // [32][n]
  float* ts = xs + 32 * n;                     // [32][n]: rows 2 kx (cos), 2 kx + 1 (-sin), scaled
  __shared__ __align__(16) float Ws[32 * 32];  // [i][o]
  __shared__ __align__(16) float Bs[32 * 32];  // [2 kx + (0: re, 1: im)][o]
  __shared__ __align__(16) float bs[32];
  const int b = blockIdx.y, t = threadIdx.x;
  for (int idx = t; idx < 32 * 32; idx += blockDim.x) {
    const int i = idx >> 5, o = idx & 31;
    float w = 0.f;
    if (o < C && i < C) w = __bfloat162float(trans ? W[i * C + o] : W[o * C + i]);
    Ws[idx] = w;
  }
  for (int o = t; o < 32; o += blockDim.x)
    bs[o] = (bias != nullptr && o < C) ? __bfloat162float(bias[o]) : 0.f;
  for (int idx = t; idx < 16 * n; idx += blockDim.x) {
    const int j0 = idx >> 4, kx = idx & 15;
    const float2 w = kx < M ? twr[idx] : make_float2(0.f, 0.f);
    const float s = kx == 0 ? w0 : w1;
    ts[(2 * kx) * n + j0] = s * w.x;
    ts[(2 * kx + 1) * n + j0] = s * w.y;
  }
  const long P = (long)n * n;
  const int ng = n >> 2;  // point groups of four
  const int og = t / ng, j0 = 4 * (t - og * ng), o0 = 8 * og;
  const int j1e = min(n, (int)(blockIdx.x + 1) * rows);
  for (int j1 = blockIdx.x * rows; j1 < j1e; ++j1) {
    __syncthreads();
    for (int idx = t; idx < C * ng; idx += blockDim.x) {
      const int i = idx / ng, q = 4 * (idx - i * ng);
      *reinterpret_cast<float4*>(xs + i * n + q) = ld4(X + ((long)b * C + i) * P + (long)j1 * n + q);
    }
    for (int idx = t; idx < 32 * 16; idx += blockDim.x) {
      const int o = idx >> 4, kx = idx & 15;
      const float2 v = (o < C && kx < M) ? Bc[(((long)b * C + o) * n + j1) * M + kx] : make_float2(0.f, 0.f);
      Bs[(2 * kx) * 32 + o] = v.x;
      Bs[(2 * kx + 1) * 32 + o] = v.y;
    }
    __syncthreads();
    float acc[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[j][q] = bs[o0 + j];
    auto step = [&](const float* a, const float* v) {
      const float4 a0 = *reinterpret_cast<const float4*>(a + o0);
      const float4 a1 = *reinterpret_cast<const float4*>(a + o0 + 4);
      const float4 x = *reinterpret_cast<const float4*>(v + j0);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = fmaf(av[j], xv[q], acc[j][q]);
    };
#pragma unroll 2
    for (int i = 0; i < C; ++i) step(Ws + i * 32, xs + i * n);
    // Re(B e^{+i theta}) with the twiddles s e^{-i theta}: the imaginary product first
#pragma unroll 1
    for (int kx = 0; kx < M; ++kx) {
      step(Bs + (2 * kx + 1) * 32, ts + (2 * kx + 1) * n);
      step(Bs + (2 * kx) * 32, ts + (2 * kx) * n);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (o0 + j >= C) break;
      const long idx = ((long)b * C + o0 + j) * P + (long)j1 * n + j0;
      if (gelu) {
        if (pre != nullptr) st4(pre + idx, acc[j]);
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = gelu_f(acc[j][q]);
      }
      st4(out + idx, acc[j]);
    }
  }
}

// dh = dv gelu'(h)
template <class TA>
__global__ void gelu_bwd_kernel(const float* __restrict__ dv, const TA* __restrict__ h, long len,
                                float* __restrict__ dh) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (long)gridDim.x * blockDim.x)
    dh[i] = dv[i] * gelu_d(ldf(h + i));
}

// ------------------------------------------------------------------ loss
__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
  return s;
}

// part[b][chunk] = (sum (y - t)^2, sum t^2) over one chunk of sample b's len values
__global__ void __launch_bounds__(256)
    loss_partial_kernel(const float* __restrict__ y, const float* __restrict__ t, long len,
                        double2* __restrict__ part) {
  __shared__ double red[8];
  const int b = blockIdx.y;
  const long per = (len + gridDim.x - 1) / gridDim.x;
  const long i0 = (long)blockIdx.x * per, i1 = i0 + per < len ? i0 + per : len;
  double s1 = 0.0, s2 = 0.0;
  for (long i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    const double tv = t[(long)b * len + i], d = (double)y[(long)b * len + i] - tv;
    s1 += d * d;
    s2 += tv * tv;
  }
  s1 = block_sum(s1, red);
  s2 = block_sum(s2, red);
  if (threadIdx.x == 0) part[(long)b * gridDim.x + blockIdx.x] = make_double2(s1, s2);
}

// loss = mean_b S1_b / S2_b; scale[b] = 2 / (B S2_b) (the gradient factor); rel[b] = sqrt(S1/S2)
__global__ void loss_finish_kernel(const double2* __restrict__ part, int B, int nchunk,
                                   double* __restrict__ loss, float* __restrict__ scale) {
  // one thread per sample adds its chunks in order, then one adds the samples
  __shared__ double rs[256];
  const int b = threadIdx.x;
  if (b < B) {
    double s1 = 0.0, s2 = 0.0;
#pragma unroll 16
    for (int c = 0; c < nchunk; ++c) {
      const double2 v = part[(long)b * nchunk + c];
      s1 += v.x;
      s2 += v.y;
    }
    rs[b] = s2 > 0.0 ? s1 / s2 : 0.0;
    scale[b] = s2 > 0.0 ? (float)(2.0 / (B * s2)) : 0.f;
  }
  __syncthreads();
  if (b == 0) {
    double L = 0.0;
    for (int i = 0; i < B; ++i) L += rs[i];
    *loss = L / B;
  }
}

__global__ void loss_grad_kernel(const float* __restrict__ y, const float* __restrict__ t, long len,
                                 int B, const float* __restrict__ scale, float* __restrict__ dy) {
  const long total = len * B;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x)
    dy[i] = (y[i] - t[i]) * scale[i / len];
}

// ------------------------------------------------------------------ Adam
__global__ void adam_kernel(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ g, bf16* __restrict__ wb, long np, float lr,
                            float b1, float b2, float eps, float bc1, float bc2) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < np; i += (long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi * bc1) / (sqrtf(vi * bc2) + eps);
    w[i] = wi;
    wb[i] = __float2bfloat16_rn(wi);
  }
}

__global__ void to_bf16_kernel(const float* __restrict__ w, long np, bf16* __restrict__ wb) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < np; i += (long)gridDim.x * blockDim.x)
    wb[i] = __float2bfloat16_rn(w[i]);
}

// ------------------------------------------------------------------ features / guess / target
// Per problem the complex scale c = sigma e^{i phi}, sigma = rms |g| and
// phi = arg(sum g^2) / 2: the solution is complex-linear in g, so dividing by c turns a
// source e^{i theta} r (r real, as every real-shaped source) into the real field +-r
// and the network meets the same problem whatever the source's phase.
__global__ void __launch_bounds__(256)
    norm_partial_kernel(const double2* __restrict__ g, long N, double* __restrict__ part) {
  __shared__ double red[8];
  double s = 0.0, sr = 0.0, si = 0.0;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
    const double2 v = g[i];
    s += v.x * v.x + v.y * v.y;
    sr += v.x * v.x - v.y * v.y;
    si += 2.0 * v.x * v.y;
  }
  s = block_sum(s, red);
  sr = block_sum(sr, red);
  si = block_sum(si, red);
  if (threadIdx.x == 0) {
    part[3 * blockIdx.x] = s;
    part[3 * blockIdx.x + 1] = sr;
    part[3 * blockIdx.x + 2] = si;
  }
}

__global__ void scale_kernel(const double* __restrict__ part, int nb, long N, double2* __restrict__ c) {
  // the partial sums staged at once, each of the three sums added in order by a thread of
  // its own (as one thread's chain of loads: 43 us)
  __shared__ double ps[3 * kNormBlocks];
  __shared__ double sum[3];
  for (int i = threadIdx.x; i < 3 * nb; i += blockDim.x) ps[i] = part[i];
  __syncthreads();
  if (threadIdx.x % 32 == 0 && threadIdx.x < 96) {
    const int j = threadIdx.x / 32;
    double a = 0.0;
    for (int i = 0; i < nb; ++i) a += ps[3 * i + j];
    sum[j] = a;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  const double s = sum[0], sr = sum[1], si = sum[2];
  const double sigma = sqrt(s / (double)N);
  const double phi = (sr == 0.0 && si == 0.0) ? 0.0 : 0.5 * atan2(si, sr);
  *c = make_double2(sigma * cos(phi), sigma * sin(phi));
}

// 1 / c (0 for c = 0)
__device__ __forceinline__ double2 inv_scale(double2 c) {
  const double m = c.x * c.x + c.y * c.y;
  return m > 0.0 ? make_double2(c.x / m, -c.y / m) : make_double2(0.0, 0.0);
}

__global__ void features_kernel(const double* __restrict__ q, double qs, const double2* __restrict__ g,
                                const double2* __restrict__ c, long N, float* __restrict__ x) {
  const double2 ic = inv_scale(*c);
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
    const double2 v = g[i];
    x[i] = (float)(qs * q[i]);
    x[N + i] = (float)(v.x * ic.x - v.y * ic.y);
    x[2 * N + i] = (float)(v.x * ic.y + v.y * ic.x);
  }
}

__global__ void guess_kernel(const float* __restrict__ y, const double2* __restrict__ c, long N,
                             double2* __restrict__ u0) {
  const double2 cc = *c;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
    const double yr = y[i], yi = y[N + i];
    u0[i] = make_double2(cc.x * yr - cc.y * yi, cc.x * yi + cc.y * yr);
  }
}

__global__ void target_kernel(const double2* __restrict__ u, const double2* __restrict__ c, long N,
                              float* __restrict__ t) {
  const double2 ic = inv_scale(*c);
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
    const double2 v = u[i];
    t[i] = (float)(v.x * ic.x - v.y * ic.y);
    t[N + i] = (float)(v.x * ic.y + v.y * ic.x);
  }
}

// the same with a prior estimate z of the solution (the preconditioner applied to g):
// x[3] + i x[4] = z / c; the guess adds the network's correction to z, the target is
// the correction (u - z) / c
__global__ void features_prior_kernel(const double2* __restrict__ z, const double2* __restrict__ c,
                                      long N, float* __restrict__ x) {
  const double2 ic = inv_scale(*c);
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
    const double2 v = z[i];
    x[3 * N + i] = (float)(v.x * ic.x - v.y * ic.y);
    x[4 * N + i] = (float)(v.x * ic.y + v.y * ic.x);
  }
}

__global__ void guess_prior_kernel(const float* __restrict__ y, const double2* __restrict__ c,
                                   const double2* __restrict__ z, long N, double2* __restrict__ u0) {
  const double2 cc = *c;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
    const double yr = y[i], yi = y[N + i];
    const double2 zi = z[i];
    u0[i] = make_double2(zi.x + (cc.x * yr - cc.y * yi), zi.y + (cc.x * yi + cc.y * yr));
  }
}

__global__ void target_prior_kernel(const double2* __restrict__ u, const double2* __restrict__ c,
                                    const double2* __restrict__ z, long N, float* __restrict__ t) {
  const double2 ic = inv_scale(*c);
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
    const double2 v = make_double2(u[i].x - z[i].x, u[i].y - z[i].y);
    t[i] = (float)(v.x * ic.x - v.y * ic.y);
    t[N + i] = (float)(v.x * ic.y + v.y * ic.x);
  }
}

unsigned grid_for(long len, int threads) {
  long g = (len + threads - 1) / threads;
  if (g > 152L * 16) g = 152L * 16;
  return (unsigned)(g < 1 ? 1 : g);
}

bool dims_ok(const sp_fno_dims* D) {
  return D && D->n >= 64 && D->n <= 512 && D->n % 64 == 0 && D->c_in >= 1 && D->c_in <= 32 &&
         D->width >= 1 && D->width <= 32 && D->modes >= 1 && D->modes <= 16 &&
         2 * D->modes <= D->n && D->layers >= 1 && D->layers <= 8 && D->hidden >= 1 &&
         D->hidden <= 128 && D->c_out >= 1 && D->c_out <= 8 && D->batch_max >= 1 &&
         D->batch_max <= 256 && (D->act_fp32 == 0 || D->act_fp32 == 1);
}

long long count_params(const sp_fno_dims* D) {
  const long long W = D->width, M = D->modes;
  long long n = W * D->c_in + W;
  n += D->layers * (2 * M * M * W * W * 2 + W * W + W);
  n += (long long)D->hidden * W + D->hidden + (long long)D->c_out * D->hidden + D->c_out;
  return n;
}

}  // namespace

struct sp_fno {
  sp_fno_dims D{};
  cudaStream_t st = nullptr;
  long long np = 0;
  long P = 0;
  int K = 0;
  long long offP = 0, offQ1 = 0, offQ2 = 0;
  std::vector<long long> offR, offW;
  float *w = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;
  bf16* wb = nullptr;
  long long step = 0;
  float2 *twr = nullptr, *twb = nullptr;
  std::vector<void*> vv, hh;
  void *e = nullptr, *ge = nullptr;
  std::vector<float2*> Vh;
  float2 *A = nullptr, *Yh = nullptr, *dVh = nullptr, *Bc = nullptr;
  float *y = nullptr, *dy = nullptr, *dv[2] = {nullptr, nullptr}, *dh = nullptr;
  float *part = nullptr, *lscale = nullptr;
  double2* lpart = nullptr;
  double *dloss = nullptr, *npart = nullptr, *hloss = nullptr;
  std::vector<void*> allocs;
  ~sp_fno() {
    for (void* p : allocs) cudaFree(p);
    if (hloss) cudaFreeHost(hloss);
  }
};

namespace {

template <class T>
cudaError_t dalloc(sp_fno* f, T** p, size_t bytes) {
  void* q = nullptr;
  cudaError_t e = cudaMalloc(&q, bytes > 0 ? bytes : 16);
  if (e != cudaSuccess) return e;
  f->allocs.push_back(q);
  *p = reinterpret_cast<T*>(q);
  return cudaSuccess;
}

sp_status cuda_st(cudaError_t e) {
  if (e == cudaSuccess) return SP_OK;
  if (e == cudaErrorMemoryAllocation) return SP_ERR_OOM;
  return SP_ERR_CUDA;
}

#define FNO_CK(x)                        \
  do {                                   \
    cudaError_t e_ = (x);                \
    if (e_ != cudaSuccess) return cuda_st(e_); \
  } while (0)

constexpr size_t kProjSmem = ((size_t)kWgSub * (132 + 36) + 128 * 32 + 8 * 128) * sizeof(float);
constexpr size_t kWgSmemMax = 200 * 1024;  // staged tiles of a weight-gradient CTA
constexpr size_t kColsSmemMax = (512 * 16 + 512) * sizeof(float2);
constexpr size_t kCombineSmemMax = 64 * 512 * sizeof(float);

// mode mixing at the widest network and the largest batch that dims_ok accepts: a network's own
// size would lower the limit under the launches of a larger one that is alive
constexpr size_t kMixSmemMax = (32 * 32 + 2 * 256 * 32) * sizeof(float2);

template <class TA>
cudaError_t set_attrs() {
  cudaError_t e;
  const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  if ((e = cudaFuncSetAttribute(chan_wgrad_kernel<TA>, at, (int)kWgSmemMax))) return e;
  if ((e = cudaFuncSetAttribute(chan_wgrad_kernel<float>, at, (int)kWgSmemMax))) return e;
  if ((e = cudaFuncSetAttribute(proj_bwd_kernel<TA>, at, (int)kProjSmem))) return e;
  if ((e = cudaFuncSetAttribute(combine_kernel<TA, TA, 256>, at, (int)kCombineSmemMax))) return e;
  if ((e = cudaFuncSetAttribute(combine_kernel<TA, TA, 512>, at, (int)kCombineSmemMax))) return e;
  if ((e = cudaFuncSetAttribute(combine_kernel<float, float, 256>, at, (int)kCombineSmemMax))) return e;
  if ((e = cudaFuncSetAttribute(combine_kernel<float, float, 512>, at, (int)kCombineSmemMax))) return e;
  if ((e = cudaFuncSetAttribute(dft_cols_fwd_kernel, at, (int)kColsSmemMax))) return e;
  if ((e = cudaFuncSetAttribute(spec_mix_kernel, at, (int)kMixSmemMax))) return e;
  return cudaFuncSetAttribute(spec_mix_bwd_kernel, at, (int)kMixSmemMax);
}

// a tiled pointwise layer (ci <= 32); ~8 CTAs per SM, each keeping its weights over its tiles
template <class TX, class TY>
void linear(sp_fno* f, int B, const TX* X, int ci, const bf16* W, const bf16* bias, int co, int gelu,
            TY* pre, TY* Y) {
  const int co8 = (co + 7) & ~7;
  const size_t smem = (size_t)(ci * co8 + co8 + ci * kTP) * sizeof(float);
  const long tiles = (f->P + kTP - 1) / kTP;
  dim3 grid((unsigned)std::min<long>(tiles, std::max<long>(1, 1216 / B)), (unsigned)B);
  chan_linear_kernel<TX, TY><<<grid, kTP, smem, f->st>>>(X, ci, W, ci, bias, co, f->P, gelu, pre, Y,
                                                         ((size_t)X & 15) == 0 ? 1 : 0);
}

// gradient of a pointwise layer's weight [co][ci] and bias [co] (adjacent in the
// parameter vector at off)
template <class TX>
void wgrad(sp_fno* f, int B, const float* dY, int co, const TX* X, int ci, long long off) {
  const int nchunk = (int)((f->P + kWgChunk - 1) / kWgChunk);
  const int co4 = (co + 3) & ~3, ci4 = (ci + 3) & ~3;
  const int own = ((co4 / 4) * (ci4 / 4) + 31) & ~31;
  const size_t smem = kWgStages * ((size_t)co4 * (kWgSub + 4) * sizeof(float) +
                                   (size_t)ci4 * (kWgSub * sizeof(TX) + 16));
  chan_wgrad_kernel<TX><<<dim3((unsigned)nchunk, (unsigned)B), own + 32, smem, f->st>>>(
      dY, co, X, ci, f->P, f->part, own, ((size_t)X & 15) == 0 ? 1 : 0);
  const int len = co * ci + co;
  sum_parts_kernel<<<(len + 255) / 256, 256, 0, f->st>>>(f->part, B * nchunk, len, f->g + off);
}

template <class TX>
void dft_forward(sp_fno* f, int B, const TX* X, float s0, float s1, float2* V) {
  const int n = f->D.n, M = f->D.modes, C = f->D.width;
  const long rows = (long)B * C * n;
  dft_rows_fwd_kernel<TX><<<(unsigned)((rows + kRowsCta - 1) / kRowsCta), 128, 0, f->st>>>(
      X, rows, n, M, f->twr, f->A);
  const size_t cs = (size_t)(n * M + n) * sizeof(float2);
  dft_cols_fwd_kernel<<<(unsigned)(B * C), 256, cs, f->st>>>(f->A, n, M, f->twb, s0, s1, V);
}

void dft_cols_inverse(sp_fno* f, int B, const float2* Y) {
  const int n = f->D.n, M = f->D.modes, C = f->D.width, R = n / 16;
  const int nbc = B * C;
  if (nbc >= 256) {  // enough channels to fill the GPU: pairs share the twiddle loads
    const size_t cs = (size_t)(2 * 2 * M * M + n) * sizeof(float2);
    dft_cols_inv_kernel<2, 16><<<dim3((unsigned)((nbc + 1) / 2), (unsigned)((R + 15) / 16)), 256, cs,
                                 f->st>>>(Y, n, M, nbc, f->twb, f->Bc);
  } else {
    const size_t cs = (size_t)(2 * M * M + n) * sizeof(float2);
    dft_cols_inv_kernel<1, 4><<<dim3((unsigned)nbc, (unsigned)((R + 3) / 4)), 256, cs, f->st>>>(
        Y, n, M, nbc, f->twb, f->Bc);
  }
}

// the layer output kernel: n threads, ~6 CTAs per SM walking the grid rows of a sample
template <class TX, class TY>
void combine(sp_fno* f, int B, const TX* X, const bf16* W, int trans, const bf16* bias, float w0,
             float w1, int gelu, TY* pre, TY* out) {
  const int n = f->D.n;
  const int rows = std::max(1, (int)((long)B * n / 912));
  auto kern = n <= 256 ? combine_kernel<TX, TY, 256> : combine_kernel<TX, TY, 512>;
  kern<<<dim3((unsigned)((n + rows - 1) / rows), (unsigned)B), n, (size_t)64 * n * sizeof(float), f->st>>>(
      X, f->D.width, W, trans, bias, f->Bc, n, f->D.modes, f->twr, w0, w1, gelu, pre, out, rows);
}

template <class TA>
cudaError_t forward_t(sp_fno* f, int B, const float* x) {
  const sp_fno_dims& D = f->D;
  const int W = D.width, L = D.layers, n = D.n;
  const bf16* wb = f->wb;
  linear<float, TA>(f, B, x, D.c_in, wb + f->offP, wb + f->offP + (long long)W * D.c_in, W, 0, nullptr,
                    (TA*)f->vv[0]);
  const float inv2 = 1.f / ((float)n * (float)n);
  for (int l = 0; l < L; ++l) {
    dft_forward<TA>(f, B, (const TA*)f->vv[l], 1.f, 1.f, f->Vh[l]);
    const size_t ms = (size_t)(W * W + B * W) * sizeof(float2);
    spec_mix_kernel<<<f->K, 256, ms, f->st>>>(f->Vh[l], wb + f->offR[l], B, W, f->K, f->Yh);
    dft_cols_inverse(f, B, f->Yh);
    const bool act = l < L - 1;
    const bf16* Wl = wb + f->offW[l];
    combine<TA, TA>(f, B, (const TA*)f->vv[l], Wl, 0, Wl + W * W, inv2, 2.f * inv2, act ? 1 : 0,
                    act ? (TA*)f->hh[l] : (TA*)nullptr, (TA*)f->vv[l + 1]);
  }
  const int H = D.hidden;
  linear<TA, TA>(f, B, (const TA*)f->vv[L], W, wb + f->offQ1, wb + f->offQ1 + (long long)H * W, H, 1,
                 (TA*)f->e, (TA*)f->ge);
  const bf16 *q2 = wb + f->offQ2, *c2 = q2 + (long long)D.c_out * H;
  const dim3 gn((unsigned)((f->P / 4 + 127) / 128), (unsigned)B);
  if (D.c_out <= 2)
    chan_narrow_kernel<TA, 2><<<gn, 128, 0, f->st>>>((const TA*)f->ge, H, q2, H, c2, D.c_out, f->P, f->y);
  else
    chan_narrow_kernel<TA, 8><<<gn, 128, 0, f->st>>>((const TA*)f->ge, H, q2, H, c2, D.c_out, f->P, f->y);
  return cudaGetLastError();
}

template <class TA>
cudaError_t backward_t(sp_fno* f, int B, const float* x, const float* t) {
  const sp_fno_dims& D = f->D;
  const int W = D.width, L = D.layers, n = D.n, H = D.hidden, co = D.c_out;
  const bf16* wb = f->wb;
  const long len = (long)co * f->P;
  loss_partial_kernel<<<dim3(kLossChunks, (unsigned)B), 256, 0, f->st>>>(f->y, t, len, f->lpart);
  loss_finish_kernel<<<1, 256, 0, f->st>>>(f->lpart, B, kLossChunks, f->dloss, f->lscale);
  loss_grad_kernel<<<grid_for(len * B, 256), 256, 0, f->st>>>(f->y, t, len, B, f->lscale, f->dy);
  // projection: dQ2 from (dy, gelu(e)); dQ1 and dv from de = (Q2^T dy) gelu'(e) in one kernel
  wgrad<TA>(f, B, f->dy, co, (const TA*)f->ge, H, f->offQ2);
  int cur = 0;
  {
    const int nchunk = (int)((f->P + kWgChunk - 1) / kWgChunk), len = H * W + H;
    proj_bwd_kernel<TA><<<dim3((unsigned)nchunk, (unsigned)B), 256, kProjSmem, f->st>>>(
        f->dy, co, (const TA*)f->e, H, wb + f->offQ2, wb + f->offQ1, (const TA*)f->vv[L], W, f->P,
        f->dv[cur], f->part);
    sum_parts_kernel<<<(len + 255) / 256, 256, 0, f->st>>>(f->part, B * nchunk, len, f->g + f->offQ1);
  }
  const float inv2 = 1.f / ((float)n * (float)n);
  const long act_len = (long)B * W * f->P;
  for (int l = L - 1; l >= 0; --l) {
    const float* dhp = f->dv[cur];
    if (l < L - 1) {
      gelu_bwd_kernel<TA><<<grid_for(act_len, 256), 256, 0, f->st>>>(f->dv[cur], (const TA*)f->hh[l],
                                                                      act_len, f->dh);
      dhp = f->dh;
    }
    wgrad<TA>(f, B, dhp, W, (const TA*)f->vv[l], W, f->offW[l]);
    // spectral branch: dY = w_kx DFT(dh), dV = dY conj(R), dR = dY conj(V), dv += Re IDFT(dV)
    dft_forward<float>(f, B, dhp, inv2, 2.f * inv2, f->Yh);
    const size_t ms = (size_t)(W * W + 2 * B * W) * sizeof(float2);
    spec_mix_bwd_kernel<<<f->K, 256, ms, f->st>>>(f->Yh, f->Vh[l], wb + f->offR[l], B, W, f->K, f->dVh,
                                                  f->g + f->offR[l]);
    dft_cols_inverse(f, B, f->dVh);
    const int nxt = cur ^ 1;
    combine<float, float>(f, B, dhp, wb + f->offW[l], 1, nullptr, 1.f, 1.f, 0, (float*)nullptr, f->dv[nxt]);
    cur = nxt;
  }
  wgrad<float>(f, B, f->dv[cur], W, x, D.c_in, f->offP);  // lift
  return cudaGetLastError();
}

sp_status run_forward(sp_fno* f, int B, const float* x) {
  return cuda_st(f->D.act_fp32 ? forward_t<float>(f, B, x) : forward_t<bf16>(f, B, x));
}

sp_status run_backward(sp_fno* f, int B, const float* x, const float* t) {
  return cuda_st(f->D.act_fp32 ? backward_t<float>(f, B, x, t) : backward_t<bf16>(f, B, x, t));
}

}  // namespace

extern "C" {

long long sp_fno_param_count(const sp_fno_dims* dims) {
  return dims_ok(dims) ? count_params(dims) : 0;
}

}  // extern "C"

namespace {

// Everything sp_fno_create does after allocating the handle: sizes, device buffers,
// twiddles and the parameters.  On failure the caller deletes f, which frees every
// device buffer recorded so far.
sp_status fno_init(sp_fno* f, const sp_fno_dims* dims, const float* params_host, void* stream) {
  f->D = *dims;
  f->st = (cudaStream_t)stream;
  const sp_fno_dims& D = f->D;
  const int W = D.width, M = D.modes, L = D.layers, n = D.n, H = D.hidden, B = D.batch_max;
  f->np = count_params(&D);
  f->P = (long)n * n;
  f->K = 2 * M * M;
  long long off = 0;
  f->offP = off;
  off += (long long)W * D.c_in + W;
  for (int l = 0; l < L; ++l) {
    f->offR.push_back(off);
    off += 2LL * f->K * W * W;
    f->offW.push_back(off);
    off += (long long)W * W + W;
  }
  f->offQ1 = off;
  off += (long long)H * W + H;
  f->offQ2 = off;
  const size_t es = D.act_fp32 ? sizeof(float) : sizeof(bf16);
  const size_t act = (size_t)B * W * f->P * es;
  cudaError_t e = cudaSuccess;
  f->allocs.reserve((size_t)3 * L + 32);  // every dalloc below records without reallocating
  auto fail = [](cudaError_t err) { return cuda_st(err); };
  if ((e = dalloc(f, &f->w, f->np * sizeof(float))) || (e = dalloc(f, &f->m, f->np * sizeof(float))) ||
      (e = dalloc(f, &f->v, f->np * sizeof(float))) || (e = dalloc(f, &f->g, f->np * sizeof(float))) ||
      (e = dalloc(f, &f->wb, f->np * sizeof(bf16))) ||
      (e = dalloc(f, &f->twr, (size_t)n * 16 * sizeof(float2))) ||
      (e = dalloc(f, &f->twb, (size_t)n * sizeof(float2))))
    return fail(e);
  f->vv.assign(L + 1, nullptr);
  f->hh.assign(L, nullptr);
  f->Vh.assign(L, nullptr);
  for (int l = 0; l <= L; ++l)
    if ((e = dalloc(f, &f->vv[l], act))) return fail(e);
  for (int l = 0; l < L; ++l)
    if ((e = dalloc(f, &f->hh[l], act)) || (e = dalloc(f, &f->Vh[l], (size_t)B * W * f->K * sizeof(float2))))
      return fail(e);
  const int nchunk = (int)((f->P + kWgChunk - 1) / kWgChunk);
  long long plen = (long long)W * D.c_in + W;
  plen = std::max(plen, (long long)W * W + W);
  plen = std::max(plen, (long long)H * W + H);
  plen = std::max(plen, (long long)D.c_out * H + D.c_out);
  if ((e = dalloc(f, &f->e, (size_t)B * H * f->P * es)) || (e = dalloc(f, &f->ge, (size_t)B * H * f->P * es)) ||
      (e = dalloc(f, &f->A, (size_t)B * W * n * M * sizeof(float2))) ||
      (e = dalloc(f, &f->Bc, (size_t)B * W * n * M * sizeof(float2))) ||
      (e = dalloc(f, &f->Yh, (size_t)B * W * f->K * sizeof(float2))) ||
      (e = dalloc(f, &f->dVh, (size_t)B * W * f->K * sizeof(float2))) ||
      (e = dalloc(f, &f->y, (size_t)B * D.c_out * f->P * sizeof(float))) ||
      (e = dalloc(f, &f->dy, (size_t)B * D.c_out * f->P * sizeof(float))) ||
      (e = dalloc(f, &f->dv[0], (size_t)B * W * f->P * sizeof(float))) ||
      (e = dalloc(f, &f->dv[1], (size_t)B * W * f->P * sizeof(float))) ||
      (e = dalloc(f, &f->dh, (size_t)B * W * f->P * sizeof(float))) ||
      (e = dalloc(f, &f->part, (size_t)B * nchunk * plen * sizeof(float))) ||
      (e = dalloc(f, &f->lpart, (size_t)B * kLossChunks * sizeof(double2))) ||
      (e = dalloc(f, &f->lscale, (size_t)B * sizeof(float))) || (e = dalloc(f, &f->dloss, sizeof(double))) ||
      (e = dalloc(f, &f->npart, (size_t)3 * kNormBlocks * sizeof(double))))
    return fail(e);
  if ((e = cudaMallocHost(&f->hloss, sizeof(double)))) return fail(e);
  if ((e = D.act_fp32 ? set_attrs<float>() : set_attrs<bf16>())) return fail(e);
  // twiddles e^{-2 pi i m / n}, with the product kx j0 reduced mod n before the angle
  std::vector<float2> twr((size_t)n * 16), twb(n);
  const double tau = 6.283185307179586476925286766559;
  for (int j0 = 0; j0 < n; ++j0)
    for (int kx = 0; kx < 16; ++kx) {
      const double a = tau * (double)((long)kx * j0 % n) / n;
      twr[(size_t)j0 * 16 + kx] = make_float2((float)std::cos(a), (float)-std::sin(a));
    }
  for (int mm = 0; mm < n; ++mm) {
    const double a = tau * mm / n;
    twb[mm] = make_float2((float)std::cos(a), (float)-std::sin(a));
  }
  if ((e = cudaMemcpyAsync(f->twr, twr.data(), twr.size() * sizeof(float2), cudaMemcpyHostToDevice, f->st)) ||
      (e = cudaMemcpyAsync(f->twb, twb.data(), twb.size() * sizeof(float2), cudaMemcpyHostToDevice, f->st)) ||
      (e = cudaStreamSynchronize(f->st)))
    return fail(e);
  return sp_fno_set_params(f, params_host);
}

}  // namespace

extern "C" {

sp_status sp_fno_create(const sp_fno_dims* dims, const float* params_host, void* stream,
                        sp_fno** out) {
  if (!out || !params_host || !dims_ok(dims)) return SP_ERR_ARG;
  *out = nullptr;
  sp_fno* f = new (std::nothrow) sp_fno;
  if (!f) return SP_ERR_OOM;
  sp_status s;
  try {
    s = fno_init(f, dims, params_host, stream);
  } catch (const std::exception&) {  // host memory: no exception crosses the ABI
    s = SP_ERR_OOM;
  }
  if (s != SP_OK) {
    delete f;
    return s;
  }
  *out = f;
  return SP_OK;
}

void sp_fno_destroy(sp_fno* f) {
  if (!f) return;
  cudaStreamSynchronize(f->st);
  delete f;
}

sp_status sp_fno_set_params(sp_fno* f, const float* params_host) {
  if (!f || !params_host) return SP_ERR_ARG;
  FNO_CK(cudaMemcpyAsync(f->w, params_host, f->np * sizeof(float), cudaMemcpyHostToDevice, f->st));
  FNO_CK(cudaMemsetAsync(f->m, 0, f->np * sizeof(float), f->st));
  FNO_CK(cudaMemsetAsync(f->v, 0, f->np * sizeof(float), f->st));
  to_bf16_kernel<<<grid_for(f->np, 256), 256, 0, f->st>>>(f->w, f->np, f->wb);
  FNO_CK(cudaGetLastError());
  f->step = 0;
  return cuda_st(cudaStreamSynchronize(f->st));
}

sp_status sp_fno_get_params(sp_fno* f, float* params_host) {
  if (!f || !params_host) return SP_ERR_ARG;
  FNO_CK(cudaMemcpyAsync(params_host, f->w, f->np * sizeof(float), cudaMemcpyDeviceToHost, f->st));
  return cuda_st(cudaStreamSynchronize(f->st));
}

sp_status sp_fno_forward(sp_fno* f, int batch, const float* x_dev, float* y_dev) {
  if (!f || !x_dev || !y_dev || batch < 1 || batch > f->D.batch_max) return SP_ERR_ARG;
  sp_status s = run_forward(f, batch, x_dev);
  if (s != SP_OK) return s;
  return cuda_st(cudaMemcpyAsync(y_dev, f->y, (size_t)batch * f->D.c_out * f->P * sizeof(float),
                                 cudaMemcpyDeviceToDevice, f->st));
}

sp_status sp_fno_gradient(sp_fno* f, int batch, const float* x_dev, const float* t_dev, float* y_dev,
                          double* loss_host, float* grad_host) {
  if (!f || !x_dev || !t_dev || batch < 1 || batch > f->D.batch_max) return SP_ERR_ARG;
  sp_status s = run_forward(f, batch, x_dev);
  if (s == SP_OK) s = run_backward(f, batch, x_dev, t_dev);
  if (s != SP_OK) return s;
  if (y_dev)
    FNO_CK(cudaMemcpyAsync(y_dev, f->y, (size_t)batch * f->D.c_out * f->P * sizeof(float),
                           cudaMemcpyDeviceToDevice, f->st));
  if (grad_host)
    FNO_CK(cudaMemcpyAsync(grad_host, f->g, f->np * sizeof(float), cudaMemcpyDeviceToHost, f->st));
  FNO_CK(cudaMemcpyAsync(f->hloss, f->dloss, sizeof(double), cudaMemcpyDeviceToHost, f->st));
  FNO_CK(cudaStreamSynchronize(f->st));
  if (loss_host) *loss_host = *f->hloss;
  return SP_OK;
}

sp_status sp_fno_train_step(sp_fno* f, int batch, const float* x_dev, const float* t_dev,
                            const sp_adam* opt, double* loss_host) {
  if (!f || !x_dev || !t_dev || !opt || batch < 1 || batch > f->D.batch_max || !(opt->lr > 0.0) ||
      !(opt->beta1 >= 0.0 && opt->beta1 < 1.0) || !(opt->beta2 >= 0.0 && opt->beta2 < 1.0) ||
      !(opt->eps > 0.0))
    return SP_ERR_ARG;
  sp_status s = run_forward(f, batch, x_dev);
  if (s == SP_OK) s = run_backward(f, batch, x_dev, t_dev);
  if (s != SP_OK) return s;
  f->step += 1;
  const double bc1 = 1.0 / (1.0 - std::pow(opt->beta1, (double)f->step));
  const double bc2 = 1.0 / (1.0 - std::pow(opt->beta2, (double)f->step));
  adam_kernel<<<grid_for(f->np, 256), 256, 0, f->st>>>(f->w, f->m, f->v, f->g, f->wb, f->np,
                                                       (float)opt->lr, (float)opt->beta1,
                                                       (float)opt->beta2, (float)opt->eps, (float)bc1,
                                                       (float)bc2);
  FNO_CK(cudaGetLastError());
  if (loss_host) {
    FNO_CK(cudaMemcpyAsync(f->hloss, f->dloss, sizeof(double), cudaMemcpyDeviceToHost, f->st));
    FNO_CK(cudaStreamSynchronize(f->st));
    *loss_host = *f->hloss;
  }
  return SP_OK;
}

sp_status sp_fno_features(sp_fno* f, const double* q_dev, double q_scale, const void* g_dev,
                          float* x_dev, void* scale_dev) {
  if (!f || !q_dev || !g_dev || !x_dev || !scale_dev || f->D.c_in != 3) return SP_ERR_ARG;
  const long N = f->P;
  norm_partial_kernel<<<kNormBlocks, 256, 0, f->st>>>((const double2*)g_dev, N, f->npart);
  scale_kernel<<<1, 256, 0, f->st>>>(f->npart, kNormBlocks, N, (double2*)scale_dev);
  features_kernel<<<grid_for(N, 256), 256, 0, f->st>>>(q_dev, q_scale, (const double2*)g_dev,
                                                       (const double2*)scale_dev, N, x_dev);
  return cuda_st(cudaGetLastError());
}

sp_status sp_fno_features_prior(sp_fno* f, const double* q_dev, double q_scale, const void* g_dev,
                                const void* z_dev, float* x_dev, void* scale_dev) {
  if (!f || !q_dev || !g_dev || !z_dev || !x_dev || !scale_dev || f->D.c_in != 5) return SP_ERR_ARG;
  const long N = f->P;
  norm_partial_kernel<<<kNormBlocks, 256, 0, f->st>>>((const double2*)g_dev, N, f->npart);
  scale_kernel<<<1, 256, 0, f->st>>>(f->npart, kNormBlocks, N, (double2*)scale_dev);
  features_kernel<<<grid_for(N, 256), 256, 0, f->st>>>(q_dev, q_scale, (const double2*)g_dev,
                                                       (const double2*)scale_dev, N, x_dev);
  features_prior_kernel<<<grid_for(N, 256), 256, 0, f->st>>>((const double2*)z_dev,
                                                             (const double2*)scale_dev, N, x_dev);
  return cuda_st(cudaGetLastError());
}

sp_status sp_fno_guess_prior(sp_fno* f, const float* y_dev, const void* scale_dev, const void* z_dev,
                             void* u0_dev) {
  if (!f || !y_dev || !scale_dev || !z_dev || !u0_dev || f->D.c_out != 2) return SP_ERR_ARG;
  guess_prior_kernel<<<grid_for(f->P, 256), 256, 0, f->st>>>(
      y_dev, (const double2*)scale_dev, (const double2*)z_dev, f->P, (double2*)u0_dev);
  return cuda_st(cudaGetLastError());
}

sp_status sp_fno_target_prior(sp_fno* f, const void* u_dev, const void* scale_dev, const void* z_dev,
                              float* t_dev) {
  if (!f || !u_dev || !scale_dev || !z_dev || !t_dev || f->D.c_out != 2) return SP_ERR_ARG;
  target_prior_kernel<<<grid_for(f->P, 256), 256, 0, f->st>>>(
      (const double2*)u_dev, (const double2*)scale_dev, (const double2*)z_dev, f->P, t_dev);
  return cuda_st(cudaGetLastError());
}

sp_status sp_fno_guess(sp_fno* f, const float* y_dev, const void* scale_dev, void* u0_dev) {
  if (!f || !y_dev || !scale_dev || !u0_dev || f->D.c_out != 2) return SP_ERR_ARG;
  guess_kernel<<<grid_for(f->P, 256), 256, 0, f->st>>>(y_dev, (const double2*)scale_dev, f->P,
                                                       (double2*)u0_dev);
  return cuda_st(cudaGetLastError());
}

sp_status sp_fno_target(sp_fno* f, const void* u_dev, const void* scale_dev, float* t_dev) {
  if (!f || !u_dev || !scale_dev || !t_dev || f->D.c_out != 2) return SP_ERR_ARG;
  target_kernel<<<grid_for(f->P, 256), 256, 0, f->st>>>((const double2*)u_dev, (const double2*)scale_dev,
                                                        f->P, t_dev);
  return cuda_st(cudaGetLastError());
}

}  // extern "C"
