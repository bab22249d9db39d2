// Complex FFT passes for the pseudospectral operator (Section 2.1, Eq. G), in
// FP64 (double2) and, for the inner solve of the mixed-precision form, FP32 (float2).
//
//   G x = F^{-1} diag(1/(4 pi^2 |k|^2 - s)) F x       (Eq. G)
//   A x = x + G (q x)                                   (Section 2.2)
//
// The n^d transform is done axis by axis; a CTA owns W neighbouring lines of one axis.  A
// line is transformed by self-sorting (Stockham) steps: with l the product of the radices
// before a step of radix r, butterfly b takes x[b + k n / r] (k < r), multiplies by
// w_{l r}^{(b mod l) k}, transforms and writes y[(b - b mod l) r + b mod l + k l].  The
// inverse is its mirror image: the steps in reverse, each reading where the forward step
// wrote, transforming, multiplying by the conjugate twiddles and writing where the forward
// step read.  A thread
// keeps its butterflies in registers; the first step reads device memory, the last writes
// it, and between steps the line passes through shared memory once, so a line of 64 points
// (three steps of radix 4) costs two exchanges and no bit reversal, and the steps at l = 1 no
// twiddles.  Fused pointwise work:
//   first pass   x -> q x              (PRE_Q)
//   last axis    forward, * D/N, inverse in one pass (MID): the inverse's first step wants
//                exactly the elements that the last forward step left in the thread's registers
//   final pass   out = x + result      (POST_ADD)
// n = 2^p or 3 2^p: a step of radix 2 when p is odd, steps of radix 4, then the radix 3, so l
// is always a power of two.  The bits do not depend on the launch shape: twiddles before the
// forward and behind the inverse butterflies, q and D / N rounded before they enter one.
// (FP32 preconditioners turn a last bit of the operator into another residual at 1e-12.)
// What bounds it: the FP64 pipe (28 instructions per radix-4 butterfly, two lanes per SM
// cycle) on large grids, the chain of three launches on small ones.
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
  int n, W, U;          // U threads per line
  int ld;               // entries between two lines in shared memory
  int steps;
  int rad[kMaxSteps];   // radices of the forward transform; the inverse runs them in reverse
  int sh_last;          // log2 of the product of the radices before the last
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
  if constexpr (r == 2) {
    const VT t = v[0];
    v[0] = cadd(t, v[1]);
    v[1] = csub(t, v[1]);
  } else if constexpr (r == 3) {
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

// values a thread holds: G butterflies of radix 4, 2 G of radix 2 or 3 (G = 2 for n >= 1536,
// so that a line of 8192 points is one CTA and more than two CTAs of a shorter one share an
// SM: an application at 1536^2 takes 880 us, with G = 1 904)
template <int G>
constexpr int kVal = 6 * G;
template <int r, int G>
constexpr int kPer = (r == 4 ? 1 : 2) * G;

// The twiddles of a step of radix r at l = 2^sh, w_{l r}^{(b mod l) k} for k = 1 .. r - 1 of
// each butterfly, loaded ahead of the exchange that the step waits for (G = 1; the threads of
// longer lines have no registers left for them and load them in the step).
template <int r, bool INV, class VT>
__device__ __forceinline__ void load_tw(const PassArgs<VT>& a, int bb, int sh, VT* tw) {
  const int nb = a.n / r;
#pragma unroll
  for (int j = 0; j < kPer<r, 1>; ++j) {
    const int b = bb + j * a.U;
    const int t = b < nb ? (b & ((1 << sh) - 1)) * (nb >> sh) : 0;  // w_{l r}^1 = w_n^(n / (l r))
#pragma unroll
    for (int k = 1; k < r; ++k) tw[j * (r - 1) + k - 1] = tw_at<INV>(a, t * k);
  }
}

// One step of radix r at l = 2^sh for the butterflies b = bb + j U of a line: from the values
// in v (reg: already there) or from the line in shared memory, to registers.
template <int r, bool INV, int G, class VT>
__device__ __forceinline__ void step_reg(const PassArgs<VT>& a, const VT* line, int bb, bool reg,
                                         int sh, const VT* tw, VT* v) {
  const int nb = a.n / r, lm = (1 << sh) - 1;
#pragma unroll
  for (int j = 0; j < kPer<r, G>; ++j) {
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
      const int t = m * (nb >> sh);
#pragma unroll
      for (int k = 1; k < r; ++k)
        x[k] = cmul(x[k], G > 1 ? tw_at<INV>(a, t * k) : tw[j * (r - 1) + k - 1]);
    }
    if (!INV) dft_reg<r, INV>(x);
  }
}
template <int r, bool INV, int G, class VT>
__device__ __forceinline__ void put_line(const PassArgs<VT>& a, VT* line, int bb, int sh, const VT* v) {
  const int nb = a.n / r, lm = (1 << sh) - 1;
#pragma unroll
  for (int j = 0; j < kPer<r, G>; ++j) {
    const int b = bb + j * a.U;
    if (b >= nb) continue;
    const int m = b & lm, o = (b - m) * r + m;
#pragma unroll
    for (int k = 0; k < r; ++k) line[spos(INV ? b + k * nb : o + (k << sh))] = v[j * r + k];
  }
}

// The transform of one line: forward, on entry the first step's inputs are in v, on return the
// last step's outputs (element b + k n / r of butterfly b); INV the other way round.
template <bool INV, int G, class VT>
__device__ __forceinline__ void transform(const PassArgs<VT>& a, VT* line, int bb, bool live, VT* v) {
  VT tw[4];  // G = 1: kPer (r - 1) twiddles of the next step
  auto fetch = [&](int r, int sh) {
    if (G != 1 || !live || sh == 0) return;
    if (r == 4) load_tw<4, INV>(a, bb, sh, tw);
    else if (r == 2) load_tw<2, INV>(a, bb, sh, tw);
    else load_tw<3, INV>(a, bb, sh, tw);
  };
  int sh = INV ? a.sh_last : 0;
  if (INV) fetch(a.rad[a.steps - 1], sh);
  for (int s = 0; s < a.steps; ++s) {
    const int r = a.rad[INV ? a.steps - 1 - s : s];
    if (live) {
      if (r == 4) step_reg<4, INV, G>(a, line, bb, s == 0, sh, tw, v);
      else if (r == 2) step_reg<2, INV, G>(a, line, bb, s == 0, sh, tw, v);
      else step_reg<3, INV, G>(a, line, bb, s == 0, sh, tw, v);
    }
    if (s == a.steps - 1) break;
    const int rn = a.rad[INV ? a.steps - 2 - s : s + 1];
    const int shn = INV ? sh - (rn >> 1) : sh + (r >> 1);  // log2 of 2 and 4; 3 is the last step
    fetch(rn, shn);
    __syncthreads();  // the line has been read
    if (live) {
      if (r == 4) put_line<4, INV, G>(a, line, bb, sh, v);
      else if (r == 2) put_line<2, INV, G>(a, line, bb, sh, v);
      else put_line<3, INV, G>(a, line, bb, sh, v);
    }
    __syncthreads();
    sh = shn;
  }
}

// fn(value, element index) for the values of a step of radix r read or written at
// b + k n / r
template <int G, class VT, class Fn>
__device__ __forceinline__ void each_value(const PassArgs<VT>& a, int r, int bb, VT* v, Fn fn) {
  const int nb = a.n / r;
  auto go = [&](auto rr) {
    constexpr int R = decltype(rr)::value;
#pragma unroll
    for (int j = 0; j < kPer<R, G>; ++j) {
      const int b = bb + j * a.U;
      if (b >= nb) continue;
#pragma unroll
      for (int k = 0; k < R; ++k) fn(v[j * R + k], b + k * nb);
    }
  };
  if (r == 4) go(std::integral_constant<int, 4>{});
  else if (r == 2) go(std::integral_constant<int, 2>{});
  else go(std::integral_constant<int, 3>{});
}

template <class VT, int G>
__global__ void __launch_bounds__(1024) fft_pass_kernel(PassArgs<VT> a) {
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
  VT v[kVal<G>];
  const int rf = a.mode == 1 ? a.rad[a.steps - 1] : a.rad[0];                 // radix read first
  const int rl = a.mode == 0 ? a.rad[a.steps - 1] : a.rad[0];                 // radix written last
  if (live) {
    each_value<G>(a, rf, bb, v, [&](VT& x, int i) { x = in[(long)i * a.S]; });
    if (a.q)
      each_value<G>(a, rf, bb, v, [&](VT& x, int i) {
        const T qq = a.q[qoff + (long)i * a.S];
        x.x = mul_rn(x.x, qq);
        x.y = mul_rn(x.y, qq);
      });
  }
  if (a.mode != 1) transform<false, G>(a, line, bb, live, v);
  if (a.mode == 2) {
    if (live)
      each_value<G>(a, a.rad[a.steps - 1], bb, v, [&](VT& x, int i) {
        const T dn = a.Dn[qoff + (long)i * a.S];
        x.x = mul_rn(x.x, dn);
        x.y = mul_rn(x.y, dn);
      });
  }
  if (a.mode != 0) transform<true, G>(a, line, bb, live, v);
  if (live) {
    VT* out = a.out + voff + base;
    if (a.addx) {
      const VT* add = a.addx + voff + base;
      each_value<G>(a, rl, bb, v, [&](VT& x, int i) { x = cadd(x, add[(long)i * a.S]); });
    }
    each_value<G>(a, rl, bb, v, [&](VT& x, int i) { out[(long)i * a.S] = x; });
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
  {  // radices: a 2 for an odd power, fours, a 3
    int p = 0;
    while ((n % 3 == 0 ? n / 3 : n) >> (p + 1)) ++p;
    if (p & 1) a.rad[a.steps++] = 2;
    for (int i = 0; i < p / 2; ++i) a.rad[a.steps++] = 4;
    if (n % 3 == 0) a.rad[a.steps++] = 3;
    a.sh_last = n % 3 == 0 ? p : p - a.rad[a.steps - 1] / 2;
  }
  long S = 1;
  for (int i = 0; i < axis; ++i) S *= n;
  a.S = (unsigned)S;
  long N = 1;
  for (int i = 0; i < d; ++i) N *= n;
  if (N / n * nvec > 0x7fffffffL) return cudaErrorInvalidValue;  // beyond every context's size
  a.vlines = (unsigned)(N / n);
  a.vstride = N;
  a.nlines = a.vlines * (unsigned)nvec;
  const int G = n >= 1536 ? 2 : 1;
  a.U = (n + 4 * G - 1) / (4 * G);
  if (a.U > 1024) return cudaErrorInvalidValue;
  // lines per CTA: eight (whole 128-byte lines across an axis > 0) while there are six CTAs
  // per SM, down to two (whole sectors) and to a full warp; one from 1024 points on, where
  // pairs leave too few CTAs to even out (an application at 1024^2: 364 us in pairs, 341
  // alone; at 2048^2: 1526 and 1513)
  int least = axis > 0 && n < 1024 ? 2 : 1;
  while (least * a.U < 32) least *= 2;
  a.W = n < 1024 ? std::max(8, least) : 1;
  while (a.W > least && (int)a.nlines / a.W < 912) a.W /= 2;
  a.ld = (n + n / 8 + 1) | 1;
  while (a.W > 1 && (a.W * a.U > 1024 || (long)a.W * a.ld * sizeof(VT) > 128 * 1024 ||
                     (axis > 0 && S % a.W)))
    a.W /= 2;
  const size_t smem = (size_t)a.W * a.ld * sizeof(VT);
  const unsigned grid = (unsigned)((a.nlines + a.W - 1) / a.W);
  static PerDevice attr;
  const cudaError_t ea = attr.run([] {
    const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(fft_pass_kernel<VT, 1>, at, 200 * 1024);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(fft_pass_kernel<VT, 2>, at, 200 * 1024);
  });
  if (ea != cudaSuccess) return ea;
  const double es = sizeof(VT);
  ProfScope ps(PROF_FFT, st);
  auto kern = G == 2 ? fft_pass_kernel<VT, 2> : fft_pass_kernel<VT, 1>;
  kern<<<grid, (unsigned)((a.W * a.U + 31) / 32 * 32), smem, st>>>(a);
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
