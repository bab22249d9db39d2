// Complex FFT passes for the pseudospectral operator (Section 2.1, Eq. G), in
// FP64 (double2) and, for the inner solve of the mixed-precision form, FP32 (float2).
//
//   G x = F^{-1} diag(1/(4 pi^2 |k|^2 - s)) F x       (Eq. G)
//   A x = x + G (q x)                                   (Section 2.2)
//
// The n^d transform is done axis by axis; a CTA owns W neighbouring lines of one axis, n = 2^p or
// 3 2^p.  Fused pointwise work:
//   first pass   x -> q x              (PRE_Q)
//   last axis    forward, * D/N, inverse in one pass (MID)
//   final pass   out = x + result      (POST_ADD)
// Two forms, chosen by the length (run_pass), lines in registers and lines in shared memory, with
// the same operations: a step of radix 2 when p is odd, steps of radix 4, then the radix 3;
// twiddles before the forward butterflies and behind the inverse ones, which run in reverse; q
// and D / N rounded before they enter a butterfly.  So the bits do not depend on the form.  (FP32
// preconditioners turn a last bit of the operator into another residual at 1e-12.)
//
// Registers: self-sorting (Stockham) steps.  With l the product of the radices before a step of
// radix r, butterfly b takes x[b + k n / r] (k < r), multiplies by w_{l r}^{(b mod l) k},
// transforms and writes y[(b - b mod l) r + b mod l + k l].  The inverse is its mirror image:
// the steps in reverse, each reading where the forward step wrote, transforming, multiplying by
// the conjugate twiddles and writing where the forward step read.  A thread keeps its butterflies
// in registers; the first step reads device memory, the last writes it, in between the line
// passes through shared memory once a step, and the inverse of a middle pass starts from the
// values that the forward transform left in the registers.  A line of 64 points costs two
// exchanges and no bit reversal.
// What bounds it: the FP64 pipe (28 instructions per radix-4 butterfly, two lanes per SM cycle)
// on large grids, the chain of three launches on small ones.
#include <algorithm>
#include <type_traits>

#include "sp_internal.h"

namespace sp {

namespace {

template <class VT> struct Real;
template <> struct Real<double2> { using T = double; };
template <> struct Real<float2> { using T = float; };

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

// a product that is rounded before it is added to anything
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }

constexpr int kMaxSteps = 16;
constexpr int kThreads = 256;  // of a CTA with its lines in shared memory

template <class VT>
struct PassArgs {
  using T = typename Real<VT>::T;
  const VT* in;
  VT* out;
  const T* q;      // PRE_Q
  const T* Dn;     // MID
  const VT* addx;  // POST_ADD
  const VT* tw;         // w_n^t = exp(-2 pi i t / n), t < n / 2
  unsigned S;           // stride between consecutive elements of a line
  unsigned nlines;      // number of lines of this axis, all vectors
  unsigned vlines;      // lines per vector
  long vstride;         // entries per vector (vectors stacked)
  int n, W;             // W lines per CTA
  int ld;               // entries between two lines in shared memory
  int U;                // register form: threads per line
  int steps;
  int rad[kMaxSteps];   // radices of the forward transform; the inverse runs them in reverse
  int sh_last;          // log2 of the product of the radices before the last
  int M, logM;          // shared-memory form: n = M or 3 M, M = 2^logM
  int mode;             // 0 forward, 1 inverse, 2 middle (forward, scale, inverse)
  int qper;             // q and Dn per vector: vector v reads those of v % qper (vstride apart)
};

// shared-memory position of element i of a line: one entry of padding per eight keeps the
// strided writes of a step (stride r) off each other's banks
__device__ __forceinline__ int spos(int i) { return i + (i >> 3); }

template <class VT>
__device__ __forceinline__ VT mul_i(VT v) {  // i v
  VT r;
  r.x = -v.y;
  r.y = v.x;
  return r;
}
template <class VT>
__device__ __forceinline__ VT mul_mi(VT v) {  // -i v
  VT r;
  r.x = v.y;
  r.y = -v.x;
  return r;
}

// in-register transform of r values, sign -1 (forward) or +1 (INV) in the exponent
template <int r, bool INV, class VT>
__device__ __forceinline__ void dft_reg(VT* v) {
  using T = typename Real<VT>::T;
  if constexpr (r == 3) {
    const T h3 = (T)0.86602540378443864676372317075294;  // sin(2 pi / 3)
    const VT t1 = cadd(v[1], v[2]), t2 = csub(v[1], v[2]);
    VT m = v[0];
    m.x -= (T)0.5 * t1.x;
    m.y -= (T)0.5 * t1.y;
    VT rot = INV ? mul_i(t2) : mul_mi(t2);
    rot.x *= h3;
    rot.y *= h3;
    v[0] = cadd(v[0], t1);
    v[1] = cadd(m, rot);
    v[2] = csub(m, rot);
  } else {
    const VT s0 = cadd(v[0], v[2]), s1 = csub(v[0], v[2]), s2 = cadd(v[1], v[3]);
    const VT d = csub(v[1], v[3]);
    const VT s3 = INV ? mul_i(d) : mul_mi(d);
    v[0] = cadd(s0, s2);
    v[1] = cadd(s1, s3);
    v[2] = csub(s0, s2);
    v[3] = csub(s1, s3);
  }
}

// w_n^t (INV: its conjugate) for 0 <= t < n (w_n^(t + n/2) = -w_n^t)
template <bool INV, class VT>
__device__ __forceinline__ VT tw_at(const PassArgs<VT>& a, int t) {
  const int h = a.n >> 1;
  const bool up = t >= h;
  VT v = a.tw[up ? t - h : t];
  if (up) {
    v.x = -v.x;
    v.y = -v.y;
  }
  if (INV) v.y = -v.y;
  return v;
}

// butterflies of a thread: one of radix 4 or two of radix 3, so six values
constexpr int kVal = 6;
template <int r>
constexpr int kPer = r == 4 ? 1 : 2;

// The twiddles of a step of radix r at l = 2^sh, w_{l r}^{(b mod l) k} for k = 1 .. r - 1 of
// each butterfly, loaded ahead of the exchange that the step waits for.
template <int r, bool INV, class VT>
__device__ __forceinline__ void load_tw(const PassArgs<VT>& a, int bb, int sh, VT* tw) {
  const int nb = a.n / r;
#pragma unroll
  for (int j = 0; j < kPer<r>; ++j) {
    const int b = bb + j * a.U;
    const int t = b < nb ? (b & ((1 << sh) - 1)) * (nb >> sh) : 0;  // w_{l r}^1 = w_n^(n / (l r))
#pragma unroll
    for (int k = 1; k < r; ++k) tw[j * (r - 1) + k - 1] = tw_at<INV>(a, t * k);
  }
}

// One step of radix r at l = 2^sh for the butterflies b = bb + j U of a line: from the values
// in v (reg: already there) or from the line in shared memory, to registers.
template <int r, bool INV, class VT>
__device__ __forceinline__ void step_reg(const PassArgs<VT>& a, const VT* line, int bb, bool reg,
                                         int sh, const VT* tw, VT* v) {
  const int nb = a.n / r, lm = (1 << sh) - 1;
#pragma unroll
  for (int j = 0; j < kPer<r>; ++j) {
    const int b = bb + j * a.U;
    if (b >= nb) continue;
    VT* x = v + j * r;
    const int m = b & lm;
    if (!reg) {
      const int o = (b - m) * r + m;
#pragma unroll
      for (int k = 0; k < r; ++k) x[k] = line[spos(INV ? o + (k << sh) : b + k * nb)];
    }
    if (INV) dft_reg<r, INV>(x);
    if (sh > 0) {
#pragma unroll
      for (int k = 1; k < r; ++k)
        x[k] = cmul(x[k], tw[j * (r - 1) + k - 1]);
    }
    if (!INV) dft_reg<r, INV>(x);
  }
}
template <int r, bool INV, class VT>
__device__ __forceinline__ void put_line(const PassArgs<VT>& a, VT* line, int bb, int sh, const VT* v) {
  const int nb = a.n / r, lm = (1 << sh) - 1;
#pragma unroll
  for (int j = 0; j < kPer<r>; ++j) {
    const int b = bb + j * a.U;
    if (b >= nb) continue;
    const int m = b & lm, o = (b - m) * r + m;
#pragma unroll
    for (int k = 0; k < r; ++k) line[spos(INV ? b + k * nb : o + (k << sh))] = v[j * r + k];
  }
}

// The transform of one line: forward, on entry the first step's inputs are in v, on return the
// last step's outputs (element b + k n / r of butterfly b); INV the other way round.
template <bool INV, class VT>
__device__ __forceinline__ void transform(const PassArgs<VT>& a, VT* line, int bb, bool live, VT* v) {
  VT tw[4];  // kPer (r - 1) twiddles of the next step
  auto fetch = [&](int r, int sh) {
    if (!live || sh == 0) return;
    if (r == 4) load_tw<4, INV>(a, bb, sh, tw);
    else load_tw<3, INV>(a, bb, sh, tw);
  };
  int sh = INV ? a.sh_last : 0;
  if (INV) fetch(a.rad[a.steps - 1], sh);
  for (int s = 0; s < a.steps; ++s) {
    const int r = a.rad[INV ? a.steps - 1 - s : s];
    if (live) {
      if (r == 4) step_reg<4, INV>(a, line, bb, s == 0, sh, tw, v);
      else step_reg<3, INV>(a, line, bb, s == 0, sh, tw, v);
    }
    if (s == a.steps - 1) break;
    const int rn = a.rad[INV ? a.steps - 2 - s : s + 1];
    const int shn = INV ? sh - 2 : sh + 2;  // a radix 3 is the last step
    fetch(rn, shn);
    __syncthreads();  // the line has been read
    if (live) {
      if (r == 4) put_line<4, INV>(a, line, bb, sh, v);
      else put_line<3, INV>(a, line, bb, sh, v);
    }
    __syncthreads();
    sh = shn;
  }
}

// fn(value, element index) for the values of a step of radix r read or written at
// b + k n / r
template <class VT, class Fn>
__device__ __forceinline__ void each_value(const PassArgs<VT>& a, int r, int bb, VT* v, Fn fn) {
  const int nb = a.n / r;
  auto go = [&](auto rr) {
    constexpr int R = decltype(rr)::value;
#pragma unroll
    for (int j = 0; j < kPer<R>; ++j) {
      const int b = bb + j * a.U;
      if (b >= nb) continue;
#pragma unroll
      for (int k = 0; k < R; ++k) fn(v[j * R + k], b + k * nb);
    }
  };
  if (r == 4) go(std::integral_constant<int, 4>{});
  else go(std::integral_constant<int, 3>{});
}

template <class VT>
__global__ void __launch_bounds__(1024) fft_reg_kernel(PassArgs<VT> a) {
  using T = typename Real<VT>::T;
  extern __shared__ __align__(16) unsigned char smraw[];
  const bool axis0 = a.S == 1;
  // lines side by side along axis 0, element-interleaved along the others (coalesced)
  const int tid = threadIdx.x;
  const int w = axis0 ? tid / a.U : tid % a.W, bb = axis0 ? tid - w * a.U : tid / a.W;
  const unsigned t = blockIdx.x * (unsigned)a.W + (unsigned)w;
  const bool live = w < a.W && bb < a.U && t < a.nlines;
  VT* line = reinterpret_cast<VT*>(smraw) + (long)w * a.ld;
  const unsigned vec = a.nlines == a.vlines ? 0u : t / a.vlines, tl = t - vec * a.vlines;
  const unsigned hi = axis0 ? tl : tl / a.S;
  const long base = (long)(tl - hi * a.S) + (long)hi * a.S * a.n;  // within the vector
  const long voff = vec * a.vstride;
  const long qoff = (a.qper > 1 ? vec % (unsigned)a.qper * a.vstride : 0) + base;
  const VT* in = a.in + voff + base;
  VT v[kVal];
  const int rf = a.mode == 1 ? a.rad[a.steps - 1] : a.rad[0];                 // radix read first
  const int rl = a.mode == 0 ? a.rad[a.steps - 1] : a.rad[0];                 // radix written last
  if (live) {
    each_value(a, rf, bb, v, [&](VT& x, int i) { x = in[(long)i * a.S]; });
    if (a.q)
      each_value(a, rf, bb, v, [&](VT& x, int i) {
        const T qq = a.q[qoff + (long)i * a.S];
        x.x = mul_rn(x.x, qq);
        x.y = mul_rn(x.y, qq);
      });
  }
  if (a.mode != 1) transform<false>(a, line, bb, live, v);
  if (a.mode == 2) {
    if (live)
      each_value(a, a.rad[a.steps - 1], bb, v, [&](VT& x, int i) {
        const T dn = a.Dn[qoff + (long)i * a.S];
        x.x = mul_rn(x.x, dn);
        x.y = mul_rn(x.y, dn);
      });
  }
  if (a.mode != 0) transform<true>(a, line, bb, live, v);
  if (live) {
    VT* out = a.out + voff + base;
    if (a.addx) {
      const VT* add = a.addx + voff + base;
      each_value(a, rl, bb, v, [&](VT& x, int i) { x = cadd(x, add[(long)i * a.S]); });
    }
    each_value(a, rl, bb, v, [&](VT& x, int i) { out[(long)i * a.S] = x; });
  }
}

// ---- lines in shared memory ---------------------------------------------------------
// The same transforms on lines that stay in shared memory, 256 threads a CTA whatever the
// line: in place, the forward order bit-reversed on load, the inverse's on store, each stage a
// strided loop over the butterflies.  A CTA needs few registers, so more of them share an SM,
// and every butterfly has a thread of its own where a line is short: better on few or long
// lines (run_pass).  Every operation is that of the register form (its radix-2 step first, twiddles
// before the forward and behind the inverse butterflies), so both give the same bits.
//   DIT stages s, s+1 (h = 2^(s-1)): with t1 = w_{2h}^j, t2 = w_{4h}^j,
//     u0 = x0, u1 = t1 x1, u2 = t2 x2, u3 = t1 t2 x3 (x_q at base + j + q h),
//     y0 = (u0 + u1) + (u2 + u3), y2 = (u0 + u1) - (u2 + u3),
//     y1 = (u0 - u1) - i (u2 - u3), y3 = (u0 - u1) + i (u2 - u3);
//   DIF stages s, s-1 (q = 2^(s-2)) of the conjugate (inverse) transform: with
//     t1 = conj w_{4q}^j, t2 = conj w_{2q}^j, s0 = x0 + x2, s1 = x0 - x2, s2 = x1 + x3,
//     s3 = x1 - x3 (x_r at base + j + r q): y0 = s0 + s2, y1 = (s0 - s2) t2,
//     y2 = (s1 + i s3) t1, y3 = (s1 - i s3) t1 t2.
// An odd stage count leaves one radix-2 stage (first for DIT, last for DIF).
// position in the staged row of element i of a line in permuted (DIT input /
// DIF output) order
template <int R, class VT>
__device__ __forceinline__ int perm_pos(const PassArgs<VT>& a, int i) {
  const int r = i % R, j = i / R;
  return r * a.M + (a.logM ? (int)(__brev((unsigned)j) >> (32 - a.logM)) : 0);
}
template <int R, class VT>
__device__ __forceinline__ void dit_stages4(VT* sm, const PassArgs<VT>& a) {
  const int M = a.M, ld = a.ld;
  int s = 1;
  if (a.logM & 1) {  // one radix-2 stage first (twiddle 1)
    const int work = a.W * R * (M >> 1);
    for (int it = threadIdx.x; it < work; it += blockDim.x) {
      const int u = it / (M >> 1), p = it - u * (M >> 1);
      const int w = u / R, r = u - w * R;
      VT* row = sm + w * ld + r * M;
      const int i0 = 2 * p;
      const VT x0 = row[i0], x1 = row[i0 + 1];
      row[i0] = cadd(x0, x1);
      row[i0 + 1] = csub(x0, x1);
    }
    __syncthreads();
    s = 2;
  }
  const int quarter = M >> 2;
  const int work = a.W * R * quarter;
  for (; s + 1 <= a.logM; s += 2) {
    const int h = 1 << (s - 1);
    for (int it = threadIdx.x; it < work; it += blockDim.x) {
      const int u = it / quarter, p = it - u * quarter;
      const int w = u / R, r = u - w * R;
      const int j = p & (h - 1);
      const int base = ((p >> (s - 1)) << (s + 1)) + j;
      VT* row = sm + w * ld + r * M;
      const VT t1 = a.tw[(j << (a.logM - s)) * R];
      const VT t2 = a.tw[(j << (a.logM - s - 1)) * R];
      const VT t3 = tw_at<false>(a, (3 * j << (a.logM - s - 1)) * R);
      const VT u0 = row[base], u1 = cmul(row[base + h], t1);
      const VT u2 = cmul(row[base + 2 * h], t2), u3 = cmul(row[base + 3 * h], t3);
      const VT s0 = cadd(u0, u1), s1 = csub(u0, u1), s2 = cadd(u2, u3), s3 = mul_i(csub(u2, u3));
      row[base] = cadd(s0, s2);
      row[base + 2 * h] = csub(s0, s2);
      row[base + h] = csub(s1, s3);
      row[base + 3 * h] = cadd(s1, s3);
    }
    __syncthreads();
  }
}
template <int R, class VT>
__device__ __forceinline__ void dif_stages4_conj(VT* sm, const PassArgs<VT>& a) {
  const int M = a.M, ld = a.ld;
  const int quarter = M >> 2;
  const int work4 = a.W * R * quarter;
  int s = a.logM;
  for (; s >= 2; s -= 2) {
    const int q = 1 << (s - 2);
    for (int it = threadIdx.x; it < work4; it += blockDim.x) {
      const int u = it / quarter, p = it - u * quarter;
      const int w = u / R, r = u - w * R;
      const int j = p & (q - 1);
      const int base = ((p >> (s - 2)) << s) + j;
      VT* row = sm + w * ld + r * M;
      VT t1 = a.tw[(j << (a.logM - s)) * R];
      VT t2 = a.tw[(j << (a.logM - s + 1)) * R];
      VT t3 = tw_at<false>(a, (3 * j << (a.logM - s)) * R);
      t1.y = -t1.y;
      t2.y = -t2.y;
      t3.y = -t3.y;
      const VT x0 = row[base], x1 = row[base + q], x2 = row[base + 2 * q], x3 = row[base + 3 * q];
      const VT s0 = cadd(x0, x2), s1 = csub(x0, x2), s2 = cadd(x1, x3), s3 = mul_i(csub(x1, x3));
      row[base] = cadd(s0, s2);
      row[base + q] = cmul(csub(s0, s2), t2);
      row[base + 2 * q] = cmul(cadd(s1, s3), t1);
      row[base + 3 * q] = cmul(csub(s1, s3), t3);
    }
    __syncthreads();
  }
  if (s == 1) {  // one radix-2 stage last (twiddle 1)
    const int work = a.W * R * (M >> 1);
    for (int it = threadIdx.x; it < work; it += blockDim.x) {
      const int u = it / (M >> 1), p = it - u * (M >> 1);
      const int w = u / R, r = u - w * R;
      VT* row = sm + w * ld + r * M;
      const int i0 = 2 * p;
      const VT x0 = row[i0], x1 = row[i0 + 1];
      row[i0] = cadd(x0, x1);
      row[i0 + 1] = csub(x0, x1);
    }
    __syncthreads();
  }
}

// radix-3 step over the three sub-lines of every row (R = 3 only).  Forward:
// X[k1 + M k2] = sum_r w_3^(r k2) (w_n^(r k1) Y_r[k1]); inverse (conjugate):
// Z_r[k1] = w_n^(-r k1) sum_k2 w_3^(-r k2) X[k1 + M k2].
template <class VT>
__device__ __forceinline__ void radix3_step(VT* sm, const PassArgs<VT>& a, bool inverse) {
  using T = typename Real<VT>::T;
  const int M = a.M, ld = a.ld;
  const T h3 = (T)0.86602540378443864676372317075294;  // sin(2 pi / 3)
  for (int it = threadIdx.x; it < a.W * M; it += blockDim.x) {
    const int w = it / M, k1 = it - w * M;
    VT* row = sm + w * ld;
    VT w1 = tw_at<false>(a, k1), w2 = tw_at<false>(a, 2 * k1);
    if (!inverse) {
      const VT a0 = row[k1], b1 = cmul(row[M + k1], w1), b2 = cmul(row[2 * M + k1], w2);
      const VT t1 = cadd(b1, b2), t2 = csub(b1, b2);
      VT mm = a0;
      mm.x -= (T)0.5 * t1.x;
      mm.y -= (T)0.5 * t1.y;
      VT rot;  // -i sin(2 pi / 3) t2
      rot.x = h3 * t2.y;
      rot.y = -h3 * t2.x;
      row[k1] = cadd(a0, t1);
      row[M + k1] = cadd(mm, rot);
      row[2 * M + k1] = csub(mm, rot);
    } else {
      const VT x0 = row[k1], x1 = row[M + k1], x2 = row[2 * M + k1];
      const VT u1 = cadd(x1, x2), u2 = csub(x1, x2);
      VT mm = x0;
      mm.x -= (T)0.5 * u1.x;
      mm.y -= (T)0.5 * u1.y;
      VT rot;  // +i sin(2 pi / 3) u2
      rot.x = -h3 * u2.y;
      rot.y = h3 * u2.x;
      w1.y = -w1.y;
      w2.y = -w2.y;
      row[k1] = cadd(x0, u1);
      row[M + k1] = cmul(cadd(mm, rot), w1);
      row[2 * M + k1] = cmul(csub(mm, rot), w2);
    }
  }
  __syncthreads();
}

template <class VT, int R>
__global__ void __launch_bounds__(kThreads) fft_smem_kernel(PassArgs<VT> a) {
  using T = typename Real<VT>::T;
  extern __shared__ __align__(16) unsigned char smraw[];
  VT* sm = reinterpret_cast<VT*>(smraw);
  const int n = a.n, ld = a.ld, W = a.W;
  const unsigned t0 = blockIdx.x * (unsigned)W;
  const int total = W * n;
  // element i of line t: its offset within the vector, the vector
  auto addr = [&](unsigned t, int i) {
    const unsigned tl = t % a.vlines, hi = tl / a.S;
    return (long)(tl - hi * a.S) + (long)hi * a.S * n + (long)i * a.S;
  };
  auto vec_at = [&](unsigned t) { return (long)(t / a.vlines) * a.vstride; };
  auto q_at = [&](unsigned t) { return a.qper > 1 ? t / a.vlines % (unsigned)a.qper * a.vstride : 0; };
  const bool axis0 = (a.S == 1);
  const bool bitrev_load = (a.mode != 1);  // forward transforms are DIT
  // ---- load (coalesced), optional q multiply, bit-reversed placement for DIT
  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    int w, i;
    if (axis0) {
      w = e / n;
      i = e - w * n;
    } else {
      i = e / W;
      w = e - i * W;
    }
    const unsigned t = t0 + w;
    if (t >= a.nlines) continue;
    const long g = addr(t, i);
    VT v = a.in[vec_at(t) + g];
    if (a.q) {
      T qq = a.q[q_at(t) + g];
      v.x *= qq;
      v.y *= qq;
    }
    int pos = bitrev_load ? perm_pos<R>(a, i) : i;
    sm[w * ld + pos] = v;
  }
  __syncthreads();
  if (a.mode == 0) {
    dit_stages4<R>(sm, a);
    if (R == 3) radix3_step(sm, a, false);
  } else if (a.mode == 1) {
    if (R == 3) radix3_step(sm, a, true);
    dif_stages4_conj<R>(sm, a);
  } else {
    dit_stages4<R>(sm, a);
    if (R == 3) radix3_step(sm, a, false);
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
      int w, i;
      if (axis0) {
        w = e / n;
        i = e - w * n;
      } else {
        i = e / W;
        w = e - i * W;
      }
      const unsigned t = t0 + w;
      if (t >= a.nlines) continue;
      T dn = a.Dn[q_at(t) + addr(t, i)];
      VT* p = &sm[w * ld + i];
      p->x *= dn;
      p->y *= dn;
    }
    __syncthreads();
    if (R == 3) radix3_step(sm, a, true);
    dif_stages4_conj<R>(sm, a);
  }
  const bool bitrev_store = (a.mode != 0);  // inverse transforms are DIF
  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    int w, i;
    if (axis0) {
      w = e / n;
      i = e - w * n;
    } else {
      i = e / W;
      w = e - i * W;
    }
    const unsigned t = t0 + w;
    if (t >= a.nlines) continue;
    const long g = vec_at(t) + addr(t, i);
    int pos = bitrev_store ? perm_pos<R>(a, i) : i;
    VT v = sm[w * ld + pos];
    if (a.addx) v = cadd(v, a.addx[g]);
    a.out[g] = v;
  }
}

template <class VT>
cudaError_t run_pass(int d, int n, const VT* tw, const typename Real<VT>::T* Dn, int axis,
                     int mode, const VT* in, VT* out, const typename Real<VT>::T* q,
                     const VT* addx, int nvec, int qper, cudaStream_t st) {
  PassArgs<VT> a{};
  a.mode = mode;
  a.qper = qper;
  a.in = in;
  a.out = out;
  a.q = q;
  a.Dn = (mode == 2) ? Dn : nullptr;
  a.addx = addx;
  a.tw = tw;
  a.n = n;
  const bool three = n % 3 == 0;
  a.M = three ? n / 3 : n;
  while ((1 << a.logM) < a.M) ++a.logM;
  long S = 1;
  for (int i = 0; i < axis; ++i) S *= n;
  a.S = (unsigned)S;
  long N = 1;
  for (int i = 0; i < d; ++i) N *= n;
  if (N / n * nvec > 0x7fffffffL) return cudaErrorInvalidValue;  // beyond every context's size
  a.vlines = (unsigned)(N / n);
  a.vstride = N;
  a.nlines = a.vlines * (unsigned)nvec;
  // Lines in registers where every step is of radix 4, or all but the last of a long line: two
  // butterflies of radix 2 (or 3, on short lines) in one thread are a chain of FP64 instructions
  // twice as long, and a warp issues one in 64 cycles.  G f, register / shared-memory form: 3D 16^3
  // 33.1 / 35.2, 64^3 94.1 / 117.2, 2D 64^2 and 256^2 the same, four 256^2 82.3 / 92.5, 768^2 221.6 /
  // 233.9, 1024^2 334 / 349 us; but 2D 96^2 37.2 / 29.0, four 192^2 63.9 / 61.8, 384^2 78.1 / 63.9,
  // 512^2 104.8 / 96.8, 3D 24^3 47.2 / 38.3, and beyond 1024 points, where one line fills a CTA's
  // registers, 1536^2 883 / 842, 2048^2 1502 / 1391.
  const bool reg = a.logM % 2 == 0 && n <= 1024 && (!three || n >= 512);
  const long esz = sizeof(VT);
  if (reg) {
    for (int i = 0; i < a.logM / 2; ++i) a.rad[a.steps++] = 4;
    if (three) a.rad[a.steps++] = 3;
    a.sh_last = three ? a.logM : a.logM - 2;
    a.U = n / 4;
    // lines per CTA: eight (whole 128-byte lines across an axis > 0) while there are six CTAs
    // per SM, down to two (whole sectors) and to a full warp; one from 1024 points on, where
    // pairs leave too few CTAs to even out (an application at 1024^2: 364 us in pairs, 341 alone)
    int least = axis > 0 && n < 1024 ? 2 : 1;
    while (least * a.U < 32) least *= 2;
    a.W = n < 1024 ? std::max(8, least) : 1;
    while (a.W > least && (int)a.nlines / a.W < 912) a.W /= 2;
    a.ld = (n + n / 8 + 1) | 1;
    while (a.W > 1 && (a.W * a.U > 1024 || a.W * a.ld * esz > 128 * 1024)) a.W /= 2;
  } else {
    // enough lines for 256 butterflies per stage, at most 64 KB of lines, and ~2 CTAs per SM
    // when the grid allows it
    a.W = 1;
    while (a.W * n < 2 * kThreads && a.W < 64) a.W *= 2;
    while (a.W > 1 && (a.W * n * esz > 64 * 1024 || (int)a.nlines / a.W < 304)) a.W /= 2;
    a.ld = n + 1;
  }
  while (axis > 0 && a.W > 1 && S % a.W) a.W /= 2;  // a CTA's lines lie inside one S-block
  const size_t smem = (size_t)a.W * a.ld * sizeof(VT);
  const unsigned grid = (unsigned)((a.nlines + a.W - 1) / a.W);
  const auto kern = reg ? fft_reg_kernel<VT> : three ? fft_smem_kernel<VT, 3> : fft_smem_kernel<VT, 1>;
  const unsigned threads = reg ? (unsigned)((a.W * a.U + 31) / 32 * 32) : (unsigned)kThreads;
  static PerDevice attr;
  const cudaError_t ea = attr.run([] {
    const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(fft_reg_kernel<VT>, at, 200 * 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fft_smem_kernel<VT, 1>, at, 200 * 1024);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(fft_smem_kernel<VT, 3>, at, 200 * 1024);
  });
  if (ea != cudaSuccess) return ea;
  const double es = sizeof(VT);
  ProfScope ps(PROF_FFT, st);
  kern<<<grid, threads, smem, st>>>(a);
  ps.done((double)N * nvec * (2 * es + (q ? es / 2 : 0.0) + (mode == 2 ? es / 2 : 0.0) +
                             (addx ? es : 0.0)),
          1, st);
  return cudaGetLastError();
}

template <class VT>
cudaError_t green_apply_t(int d, int n, const VT* tw, const typename Real<VT>::T* Dn,
                          VT* tmp, const VT* x, const typename Real<VT>::T* q, bool add_x, VT* out,
                          int nvec, int qper, cudaStream_t st) {
  cudaError_t e;
  // forward along axes 0..d-2, middle pass on axis d-1, inverse along d-2..0
  const VT* src = x;
  for (int ax = 0; ax < d - 1; ++ax) {
    e = run_pass<VT>(d, n, tw, Dn, ax, 0, src, tmp, ax == 0 ? q : nullptr, nullptr, nvec, qper, st);
    if (e != cudaSuccess) return e;
    src = tmp;
  }
  e = run_pass<VT>(d, n, tw, Dn, d - 1, 2, src, tmp, nullptr, nullptr, nvec, qper, st);
  if (e != cudaSuccess) return e;
  for (int ax = d - 2; ax >= 0; --ax) {
    bool last = (ax == 0);
    e = run_pass<VT>(d, n, tw, Dn, ax, 1, tmp, last ? out : tmp, nullptr,
                     (last && add_x) ? x : nullptr, nvec, qper, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

__global__ void to_float_kernel(const double* a, float* b, long N) {
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) b[i] = (float)a[i];
}

}  // namespace

cudaError_t fft_green_apply(const FftPlan& P, const double2* x, const double* q, bool add_x,
                            double2* out, cudaStream_t st, int nvec, int qper) {
  if (qper < 1 || nvec % qper) return cudaErrorInvalidValue;
  return green_apply_t<double2>(P.d, P.n, P.tw, P.Dn, P.tmp, x, q, add_x, out, nvec, qper, st);
}

cudaError_t fft_green_apply32(const FftPlan& P, const float2* x, const float* q, bool add_x,
                              float2* out, cudaStream_t st) {
  return green_apply_t<float2>(P.d, P.n, P.tw32, P.Dn32, P.tmp32, x, q, add_x, out, 1, 1, st);
}

cudaError_t to_float(const double* a, float* b, long N, cudaStream_t st) {
  to_float_kernel<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(a, b, N);
  return cudaGetLastError();
}

}  // namespace sp
