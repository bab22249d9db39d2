// Numeric multifrontal factorisation of P = Q + C q on the periodic nested-dissection
// tree (Section 2.2-2.3, Fig. nd): per level, leaves to root,
//   1. assemble the original entries P(j, i) = Q(j, i) + C(j, i) q_i whose
//      earlier-eliminated endpoint belongs to the front (Section 2.2: P = Q + C q);
//   2. extend-add the children's Schur complements (one launch per child position,
//      so no two threads of a launch add into the same entry);
//   3. blocked right-looking LU of the front with partial pivoting restricted to
//      the k eliminated rows (the paper does not say how fronts are pivoted; this
//      is the reading used throughout): panel factorisation, row-block triangular
//      solve and a tiled Schur-complement update that also forms
//      S = F22 - L21 U12, the block handed to the parent.
// Every front of a level has the same size, so each step is one batched launch
// over all fronts of the level.  Fronts are column-major m x m.  T = double for
// the FP64 form, float for the FP32 preconditioner form.
#include <cooperative_groups.h>

#include <functional>
#include <type_traits>
#include <vector>

#include <algorithm>
#include <cfloat>

#include <cuda_fp16.h>

#include "sp_internal.h"

namespace sp {

namespace {

constexpr int kNB = 32;       // panel width
constexpr int kTile = 64;     // Schur update tile (kTile x kTile per CTA)
constexpr int kTcMinFront = 1024;         // smallest front blocked for the tensor cores
constexpr int kGridPanelCTAs = 152;       // CTAs of a grid-panel launch (one per SM)
constexpr size_t kGridPanelSmem = 200 * 1024;  // staged rows of one grid-panel CTA

template <class T>
__global__ void assemble_kernel(T* fronts, int m, int nasm, const int* __restrict__ row,
                                const int* __restrict__ tidx, const int* __restrict__ cvar,
                                const int* __restrict__ gidx, const double* __restrict__ Qcat,
                                const double* __restrict__ Ccat, const double* __restrict__ q,
                                int nfp, long tstride) {
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nasm) return;
  long f = blockIdx.y;
  // fronts of a problem group: problem f / nfp reads its own tables (tstride apart)
  const long ti = tidx[e] + (f / nfp) * tstride;
  const int c = cvar[e];
  double qi = q[gidx[f * m + c]];
  fronts[f * (long)m * m + row[e] + (long)c * m] = (T)fma(Ccat[ti], qi, Qcat[ti]);
}

// One launch per child position: the child's Schur block (rows and columns kc..mc-1 of
// its front) is added into the parent front through the map.  Each thread adds kEaU
// entries a block width apart in column-major order: it reads every child value, map
// entry and parent value first and writes afterwards, so kEaU independent read chains
// are in flight (the map is injective within one child position, so no two entries of a
// launch meet in the parent).
constexpr int kEaU = 4;

template <class T>
__global__ void extend_add_kernel(T* parent, int m, int nb1, const T* __restrict__ child, int mc,
                                  int kc, const int* __restrict__ map, int delta, int d) {
  const int nbd = mc - kc;
  const long nn = (long)nbd * nbd;
  const long e0 = (long)blockIdx.x * (kEaU * blockDim.x) + threadIdx.x;
  if (e0 >= nn) return;
  int f = blockIdx.y;
  // parent box coordinates -> child box id (child grid has 2*nb1 boxes per axis)
  int ff = f, cid = 0, stride = 1;
  for (int a = 0; a < d; ++a) {
    int bc = ff % nb1;
    ff /= nb1;
    cid += (2 * bc + ((delta >> a) & 1)) * stride;
    stride *= 2 * nb1;
  }
  cid += ff * stride;  // problem ff of a group: its children follow the earlier problems'
  const T* cf = child + (long)cid * mc * mc + kc + (long)kc * mc;
  T* pf = parent + (long)f * m * m;
  int i = (int)(e0 % nbd), j = (int)(e0 / nbd);
  T v[kEaU];
  long at[kEaU];
#pragma unroll
  for (int u = 0; u < kEaU; ++u) {
    at[u] = -1;
    if (e0 + (long)u * blockDim.x < nn) {
      v[u] = cf[i + (long)j * mc];
      at[u] = map[i] + (long)map[j] * m;
    }
    i += blockDim.x;  // next entry: blockDim.x further in column-major order
    j += i / nbd;
    i %= nbd;
  }
  T p[kEaU];
#pragma unroll
  for (int u = 0; u < kEaU; ++u)
    if (at[u] >= 0) p[u] = pf[at[u]];
#pragma unroll
  for (int u = 0; u < kEaU; ++u)
    if (at[u] >= 0) pf[at[u]] = p[u] + v[u];
}

// FP16 copy of the factor for the chained sweeps (sp_opts.factor_storage = 1), with a
// power-of-two scale per front column: column c of front f is stored as entry /
// 2^(e - 15), with max |entry| = mant 2^e (mant in [0.5, 1)) over the rows the sweeps
// read (all rows for c < k; rows < k, the U12 block, for c >= k), so every stored
// magnitude is below 2^15 (FP16's largest finite value is 65504), the scaling is
// exact, and a column's entries keep FP16's 11 significant bits down to 2^-29 of its
// largest.  One warp per column; columns ld16 = m rounded up to even apart (the pad
// row zero).
__global__ void f16_copy_kernel(const float* fronts, int m, int k, __half* out, float* fsc) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = blockIdx.x * (blockDim.x >> 5) + warp;
  if (c >= m) return;
  const long f = blockIdx.y, mm = (long)m * m;
  const int ld16 = (m + 1) & ~1;  // even column stride: row pairs load as half2
  const float* col = fronts + f * mm + (long)c * m;
  __half* hc = out + f * (long)m * ld16 + (long)c * ld16;
  const int rows = c < k ? m : k;
  if (lane == 0 && ld16 > m) hc[m] = __float2half_rn(0.f);
  // both passes over the column keep eight loads per lane in flight
  constexpr int kU = 8;
  float mxu[kU];
#pragma unroll
  for (int u = 0; u < kU; ++u) mxu[u] = 0.f;
  int r = lane;
  for (; r + 32 * (kU - 1) < rows; r += 32 * kU) {
    float v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) v[u] = col[r + 32 * u];
#pragma unroll
    for (int u = 0; u < kU; ++u) mxu[u] = fmaxf(mxu[u], fabsf(v[u]));
  }
  for (; r < rows; r += 32) mxu[0] = fmaxf(mxu[0], fabsf(col[r]));
  float mx = mxu[0];
#pragma unroll
  for (int u = 1; u < kU; ++u) mx = fmaxf(mx, mxu[u]);
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  int e = 0;
  if (mx > 0.f) frexpf(mx, &e);
  const float inv = ldexpf(1.0f, 15 - e);
  if (lane == 0) fsc[f * m + c] = ldexpf(1.0f, e - 15);
  r = lane;
  for (; r + 32 * (kU - 1) < rows; r += 32 * kU) {
    float v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) v[u] = col[r + 32 * u];
#pragma unroll
    for (int u = 0; u < kU; ++u) hc[r + 32 * u] = __float2half_rn(v[u] * inv);
  }
  for (; r < rows; r += 32) hc[r] = __float2half_rn(col[r] * inv);
}

// max |entry| of every front: CTAs over (chunk, front).  Magnitudes order like their bit
// patterns, so the maximum is an integer one (NaNs count as 0): as FP64 fmax it held the
// pass at 1 TB/s in FP32 (3D 64^3 leaves, 1.1 GB: 1.05 ms).  scale must be zeroed first.
__device__ __forceinline__ unsigned mag_word(float v) {
  const unsigned u = __float_as_uint(v) & 0x7fffffffu;
  return u > 0x7f800000u ? 0u : u;
}
__device__ __forceinline__ unsigned long long mag_word(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  return u > 0x7ff0000000000000ull ? 0ull : u;
}
__device__ __forceinline__ double mag_value(unsigned u) { return (double)__uint_as_float(u); }
__device__ __forceinline__ double mag_value(unsigned long long u) { return __longlong_as_double((long long)u); }
template <class T>
__global__ void __launch_bounds__(256) front_scale_kernel(const T* fronts, long mm, double* scale) {
  const T* A = fronts + blockIdx.y * mm;
  // eight independent loads in flight per thread (a loop-carried max with one load per
  // trip is bound by memory latency, not bandwidth)
  constexpr int kU = 8;
  using W = decltype(mag_word(T()));
  const long stride = (long)gridDim.x * blockDim.x;
  W mx = 0;
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + (kU - 1) * stride < mm; i += kU * stride) {
    T v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) v[u] = A[i + u * stride];
#pragma unroll
    for (int u = 0; u < kU; ++u) mx = max(mx, mag_word(v[u]));
  }
  for (; i < mm; i += stride) mx = max(mx, mag_word(A[i]));
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_down_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0 && mx > 0)
    atomicMax(reinterpret_cast<unsigned long long*>(scale + blockIdx.y),
              (unsigned long long)__double_as_longlong(mag_value(mx)));
}

// Panel LU of a front too tall for the register panel below: G CTAs per front in one
// cooperative launch (every CTA resident), the fronts of a level in groups of
// nfl per launch.  CTA g stages the panel rows ("slots") [g c, (g+1) c) of rows
// [j0, m) in shared memory; rows never move during the panel.  A slot is a pivot
// candidate while its starting position is below k (interchanges only exchange
// positions below k) and it has not been a pivot yet.  Per pivot column every
// CTA publishes the row of its best candidate, then (release) one 64-bit word:
// FP32 magnitude in bits 32-63, 2^20 - 1 - slot in bits 8-27, the column tag in
// bits 0-7 (words of one column compare like their keys); each CTA polls the
// words of its front's G CTAs (acquire, all in flight at once), takes the
// largest and copies the winner's row: no other barrier.  The publication slots alternate between two
// buffers by column parity (a CTA cannot publish column j+2 before every CTA has
// published j+1, i.e. finished reading column j).  The pivot positions are
// reconstructed after the panel from the sequence of pivot slots; each CTA then
// writes its rows back in position order.  A poll that does not complete within
// wait_ns (2 s by default) sets bit 2 of *status and the CTA returns without
// writing back (CTA 0 of the front leaves identity interchanges for the panel).
constexpr int kPubWords = 1 + kNB;  // word, row (in units of 8 bytes; T <= 8 bytes)
__device__ __forceinline__ unsigned long long gtimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

template <class T>
__global__ void __launch_bounds__(256) lu_panel_grid_kernel(T* fronts, int m, int k, int j0, int jb,
                                                            int f0, int G, int* piv,
                                                            const double* scale, double ptol,
                                                            int* status,
                                                            unsigned long long* pub,
                                                            unsigned long long wait_ns) {
  const int f = f0 + blockIdx.x / G, g = blockIdx.x % G;
  T* A = fronts + (long)f * m * m;
  const int rows = m - j0, kl = k - j0;
  const int chunk = (rows + G - 1) / G;
  const int s0 = min(rows, g * chunk), s1 = min(rows, s0 + chunk), nmy = s1 - s0;
  // publication slots of this front: [parity][g][kPubWords]
  unsigned long long* pf = pub + (long)f * 2 * kGridPanelMaxG * kPubWords;
  extern __shared__ unsigned long long smraw_u64[];
  T* P = reinterpret_cast<T*>(smraw_u64);                      // chunk x jb, column-major
  unsigned char* elim = reinterpret_cast<unsigned char*>(P + (long)chunk * jb);
  __shared__ T prow[kNB];
  __shared__ unsigned long long wkey[8];
  __shared__ int pslot[kNB];
  __shared__ int ds[2 * kNB], dp[2 * kNB];
  __shared__ int s_nd, s_abort;
  const double thresh = ptol * scale[f];
  for (long e = threadIdx.x; e < (long)nmy * jb; e += blockDim.x) {
    const int r = (int)(e % nmy), c = (int)(e / nmy);
    P[r + (long)c * chunk] = A[(j0 + s0 + r) + (long)(j0 + c) * m];
  }
  for (int r = threadIdx.x; r < nmy; r += blockDim.x) elim[r] = 0;
  if (threadIdx.x == 0) s_abort = 0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  for (int jj = 0; jj < jb; ++jj) {
    const unsigned long long tag = (unsigned long long)(jj + 1);
    unsigned long long key = 0ull;
    for (int r = threadIdx.x; r < nmy; r += blockDim.x) {
      const int sl = s0 + r;
      if (sl >= kl || elim[r]) continue;
      const float v = (float)fabs((double)P[r + (long)jj * chunk]);
      const unsigned long long kk = ((unsigned long long)__float_as_uint(v) << 32) |
                                    ((unsigned long long)(0xFFFFFu - (unsigned)sl) << 8);
      key = kk > key ? kk : key;
    }
    for (int o = 16; o > 0; o >>= 1) {
      unsigned long long ok = __shfl_down_sync(0xffffffffu, key, o);
      key = ok > key ? ok : key;
    }
    if (lane == 0) wkey[warp] = key;
    __syncthreads();
    unsigned long long* base = pf + (long)(jj & 1) * kGridPanelMaxG * kPubWords;
    if (warp == 0) {
      unsigned long long kb = wkey[lane & 7];
      for (int o = 4; o > 0; o >>= 1) {
        unsigned long long ok = __shfl_down_sync(0xffffffffu, kb, o);
        kb = ok > kb ? ok : kb;
      }
      if (lane == 0) {
        unsigned long long* mine = base + (long)g * kPubWords;
        if (kb) {
          const int r = (int)(0xFFFFFu - (unsigned)((kb >> 8) & 0xFFFFFu)) - s0;
          T* row = reinterpret_cast<T*>(mine + 1);
          for (int c = 0; c < jb; ++c) row[c] = P[r + (long)c * chunk];
        }
        st_release64(mine, kb | tag);  // orders the row stores before the word
      }
      // the G words of this column, all loads in flight at once
      constexpr int kPer = (kGridPanelMaxG + 31) / 32;
      unsigned long long w[kPer];
      bool rdy[kPer];
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        w[i] = 0ull;
        rdy[i] = lane + 32 * i >= G;
      }
      const unsigned long long t0 = gtimer_ns();
      bool ok = true;
      while (true) {
#pragma unroll
        for (int i = 0; i < kPer; ++i)
          if (!rdy[i]) w[i] = ld_acquire64(base + (long)(lane + 32 * i) * kPubWords);
        bool mine_ok = true;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          if (!rdy[i]) rdy[i] = (w[i] & 0xFFull) == tag;
          mine_ok = mine_ok && rdy[i];
        }
        if (__all_sync(0xffffffffu, mine_ok)) break;
        if (gtimer_ns() - t0 > wait_ns) {
          ok = false;
          break;
        }
      }
      __syncwarp();  // the lanes' acquires order the row reads of every lane below
      unsigned long long best = 0ull;
#pragma unroll
      for (int i = 0; i < kPer; ++i)
        if (lane + 32 * i < G) best = w[i] > best ? w[i] : best;
      for (int o = 16; o > 0; o >>= 1) {
        unsigned long long ob = __shfl_down_sync(0xffffffffu, best, o);
        best = ob > best ? ob : best;
      }
      best = __shfl_sync(0xffffffffu, best, 0);
      int sb = (int)(0xFFFFFu - (unsigned)((best >> 8) & 0xFFFFFu));
      const bool valid = ok && (best >> 8) != 0ull && sb >= 0 && sb < rows;
      if (!valid) {
        if (lane == 0) {
          s_abort = 1;
          atomicOr(status, ok ? 1 : 2);
        }
        sb = 0;
      } else {
        const T* orow = reinterpret_cast<const T*>(base + (long)(sb / chunk) * kPubWords + 1);
        if (lane < jb) prow[lane] = __ldcg(orow + lane);
      }
      if (lane == 0) {
        pslot[jj] = sb;
        if (sb >= s0 && sb < s1) elim[sb - s0] = 1;
      }
    }
    __syncthreads();
    if (s_abort) {
      // the panel stops here; later kernels of the factorisation still read this
      // panel's interchanges, so leave in-range (identity) ones
      if (g == 0)
        for (int c = threadIdx.x; c < jb; c += blockDim.x) piv[(long)f * k + j0 + c] = j0 + c;
      return;
    }
    T pv = prow[jj];
    if (g == 0 && threadIdx.x == 0 && !(fabs((double)pv) > thresh)) atomicOr(status, 1);
    if (!(fabs((double)pv) > 0.0)) pv = (T)(thresh > 0 ? thresh : 1e-30);
    const T inv = (T)1 / pv;
    for (int r = threadIdx.x; r < nmy; r += blockDim.x) {
      if (elim[r]) continue;
      T* pr = P + r;
      const T l = pr[(long)jj * chunk] * inv;
      pr[(long)jj * chunk] = l;
      for (int c = jj + 1; c < jb; ++c) pr[(long)c * chunk] -= l * prow[c];
    }
  }
  // positions: replay the interchanges (pivot slot pslot[jj] moves to position jj,
  // the slot at jj moves to the pivot's position); displaced slots in ds/dp
  if (threadIdx.x == 0) {
    int nd = 0;
    for (int jj = 0; jj < jb; ++jj) {
      const int sb = pslot[jj];
      int p = sb, ib = -1, sa = jj, ia = -1;
      for (int i = 0; i < nd; ++i) {
        if (ds[i] == sb) {
          p = dp[i];
          ib = i;
        }
      }
      for (int i = 0; i < nd; ++i)
        if (dp[i] == jj) {
          sa = ds[i];
          ia = i;
        }
      if (ia < 0)
        for (int i = 0; i < nd; ++i)
          if (ds[i] == sa) ia = i;
      if (ib < 0) {
        ib = nd++;
        ds[ib] = sb;
      }
      dp[ib] = jj;
      if (sa != sb) {
        if (ia < 0) {
          ia = nd++;
          ds[ia] = sa;
        }
        dp[ia] = p;
      }
      if (g == 0) piv[(long)f * k + j0 + jj] = j0 + p;
    }
    s_nd = nd;
  }
  __syncthreads();
  const int nd = s_nd;
  for (long e = threadIdx.x; e < (long)nmy * jb; e += blockDim.x) {
    const int r = (int)(e % nmy), c = (int)(e / nmy);
    const int sl = s0 + r;
    int pos = sl;
    for (int i = 0; i < nd; ++i)
      if (ds[i] == sl) pos = dp[i];
    A[(j0 + pos) + (long)(j0 + c) * m] = P[r + (long)c * chunk];
  }
}

// ---- panel LU with the panel in registers ------------------------------------------
// LU of the panel columns [j0, j0 + jb) of every front, rows [j0, m) ("slots", local
// index 0 .. rows - 1), by a cluster of C CTAs of NT threads per front (C = 1: an
// ordinary launch).  Thread t of CTA q keeps R whole panel rows in registers, slot
// q NT R + r NT + t (r < R), so a pivot step touches shared memory only to publish one
// candidate row.  Rows never move: a slot is a pivot candidate while its position is
// below k (interchanges only exchange positions below k, so: slot < k - j0) and it has
// not been a pivot; the positions are replayed once at the end.
//
// The pivot is the largest magnitude of the column (FP64: all bits of it), ties to the
// smallest position, as in the textbook loop over the rows in place.  A row is at its own
// slot until an interchange moves it, and the only rows that an interchange moves without
// making them pivots are those of the slots 0 .. 31, so the position is one register (of
// row r = 0) that follows the interchanges.
//
// Pivot step.  Each warp reduces its candidates' magnitude bits and the owner of the
// largest posts its row; one CTA barrier; every
// warp picks the CTA's best.  With C > 1 each CTA then pushes its best row and key into
// all C CTAs with st.async on the receiver's mbarrier (double-buffered by the step's
// parity: a CTA pushes step j + 2 only after it holds every push of step j + 1, which
// its peers sent after they had read step j), so a step costs one CTA barrier and one
// one-way trip through distributed shared memory.  A wait that lasts longer than wait_ns
// makes the panel report a timeout (status bit 2, identity interchanges, no write-back), but
// the CTA goes on with the steps: its peers' pushes are in flight then, and a CTA that left
// would be written to after its shared memory was handed on.  Only a wait of kPushDrainNs
// more, which the resident CTAs of a cluster cannot cause, ends the panel at once.
//
// The 32 columns are taken in four blocks of eight: the eight steps are unrolled with
// the current block in registers 0-7, the columns right of it updated in groups of
// eight (finished groups skipped), then the registers rotate by eight; the code stays
// at eight unrolled steps.
//
// What bounds it: the chain of pivot steps (FP32) and the SM's two FP64 FMAs per cycle
// (FP64), so FP32 panels take the fewest CTAs whose registers hold them and FP64 panels
// as many as the level leaves free (panel_shape).
constexpr int kPanelMaxC = 16;
constexpr unsigned long long kPushDrainNs = 2000000000ull;

// magnitudes as integers of the same order; a NaN is never the largest
__device__ __forceinline__ unsigned mag_bits(float v) {
  const unsigned u = __float_as_uint(v) & 0x7fffffffu;
  return u > 0x7f800000u ? 0u : u;
}
__device__ __forceinline__ unsigned long long mag_bits(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  return u > 0x7ff0000000000000ull ? 0ull : u;
}
// the largest key of the warp and, of the lanes that hold it, the smallest position
__device__ __forceinline__ void pick(unsigned* key, unsigned* pos) {
  const unsigned best = __reduce_max_sync(0xffffffffu, *key);
  *pos = __reduce_min_sync(0xffffffffu, *key == best ? *pos : 0xffffffffu);
  *key = best;
}
__device__ __forceinline__ void pick(unsigned long long* key, unsigned* pos) {
  const unsigned hi = (unsigned)(*key >> 32), bh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned bl = __reduce_max_sync(0xffffffffu, hi == bh ? (unsigned)*key : 0u);
  const unsigned long long best = (unsigned long long)bh << 32 | bl;
  *pos = __reduce_min_sync(0xffffffffu, *key == best ? *pos : 0xffffffffu);
  *key = best;
}
// the panel row's columns [8 g, 8 g + 8) of `src` in shared memory (16-byte aligned)
__device__ __forceinline__ void load8(const float* src, float* v) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float4 t = reinterpret_cast<const float4*>(src)[i];
    v[4 * i] = t.x;
    v[4 * i + 1] = t.y;
    v[4 * i + 2] = t.z;
    v[4 * i + 3] = t.w;
  }
}
__device__ __forceinline__ void load8(const double* src, double* v) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double2 t = reinterpret_cast<const double2*>(src)[i];
    v[2 * i] = t.x;
    v[2 * i + 1] = t.y;
  }
}
__device__ __forceinline__ void store8(float* dst, const float* v) {
#pragma unroll
  for (int i = 0; i < 2; ++i)
    reinterpret_cast<float4*>(dst)[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
}
__device__ __forceinline__ void store8(double* dst, const double* v) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    reinterpret_cast<double2*>(dst)[i] = make_double2(v[2 * i], v[2 * i + 1]);
}
__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
// address in CTA `rank` of the cluster of the same shared-memory location
__device__ __forceinline__ unsigned peer_addr(unsigned a, int rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void push(unsigned dst, unsigned bar, unsigned v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst),
               "r"(v), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void push(unsigned dst, unsigned bar, unsigned long long v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst),
               "l"(v), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void push(unsigned dst, unsigned bar, float v) {
  push(dst, bar, __float_as_uint(v));
}
__device__ __forceinline__ void push(unsigned dst, unsigned bar, double v) {
  push(dst, bar, (unsigned long long)__double_as_longlong(v));
}
// bounded wait for the phase of the given parity (acquire at cluster scope: the peers' pushes):
// *late after wait_ns, given up kPushDrainNs later
__device__ __forceinline__ bool bar_wait(unsigned bar, unsigned parity, unsigned long long wait_ns,
                                         bool* late) {
  const unsigned long long t0 = gtimer_ns();
  while (true) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    const unsigned long long t = gtimer_ns() - t0;
    if (t > wait_ns) *late = true;
    if (t > wait_ns + kPushDrainNs) return false;
  }
}

template <class T, int NT, int R>
__global__ void __launch_bounds__(NT)
    lu_panel_reg_kernel(T* fronts, int m, int k, int j0, int jb, int C, int* piv, int* pmap, int* perm,
                        const double* scale, double ptol, int* status, unsigned long long wait_ns) {
  constexpr int W = NT / 32;
  using Mag = decltype(mag_bits(T()));
  const int q = C > 1 ? (int)(blockIdx.x % C) : 0;
  const long f = blockIdx.x / C;
  T* A = fronts + f * (long)m * m + j0 + (long)j0 * m;
  const int rows = m - j0, kl = k - j0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int s0 = q * NT * R + tid;  // slot of row r: s0 + r NT
  __shared__ __align__(16) T wrow[2][W][kNB];   // posted candidate row of each warp
  __shared__ Mag wmag[2][W];
  __shared__ unsigned wpos[2][W];
  __shared__ __align__(16) T crow[2][kPanelMaxC][kNB];  // pushed rows of the cluster's CTAs
  constexpr bool kWide = sizeof(Mag) == 8;  // FP64: the position does not fit beside the magnitude
  __shared__ __align__(8) unsigned long long ckey[2][kPanelMaxC];
  __shared__ unsigned cpos[2][kWide ? kPanelMaxC : 1];
  __shared__ __align__(8) unsigned long long cbar[2];
  __shared__ int spiv[kNB];   // pivot positions in order
  __shared__ T spv[kNB];      // pivots
  const double thresh = ptol * scale[f];
  if (C > 1) {
    if (tid == 0) {
      for (int i = 0; i < 2; ++i)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&cbar[i])) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
  }
  T a[R][kNB];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < kNB; ++c) {
      const int sl = s0 + r * NT;
      a[r][c] = (sl < rows && c < jb) ? A[sl + (long)c * m] : (T)0;
    }
  int pj[R];  // pivot step of the row, -1: not a pivot
#pragma unroll
  for (int r = 0; r < R; ++r) pj[r] = -1;
  int pos0 = s0;  // position of row r = 0; the other rows stay at their slots
  bool ok = true, stop = false;  // this warp's last wait; the CTA gave up
  bool late = false;             // a wait of this warp ran over its limit
#pragma unroll 1
  for (int o = 0; o < kNB / 8; ++o) {
    const int live = kNB / 8 - o;  // column groups of eight not finished (the current one included)
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int jj = 8 * o + u;
      if (jj < jb && !stop) {
        const int buf = u & 1;
        // this thread's candidate: magnitude + 1 (0: none) and position (rows r > 0 in the
        // order of their positions)
        Mag mg = 0;
        unsigned mpos = 0xffffffffu;
#pragma unroll
        for (int r = 1; r < R; ++r) {
          const Mag v = pj[r] < 0 && s0 + r * NT < kl ? mag_bits(a[r][u]) + 1 : 0;
          if (v > mg) {
            mg = v;
            mpos = (unsigned)(s0 + r * NT);
          }
        }
        {
          const Mag v = pj[0] < 0 && s0 < kl ? mag_bits(a[0][u]) + 1 : 0;
          if (v && (v > mg || (v == mg && (unsigned)pos0 < mpos))) {
            mg = v;
            mpos = (unsigned)pos0;
          }
        }
        Mag wm = mg;
        unsigned wp = mpos;
        pick(&wm, &wp);
        if (mg == wm && mpos == wp && wm) {
#pragma unroll
          for (int r = 0; r < R; ++r)
            if (pj[r] < 0 && (unsigned)(r == 0 ? pos0 : s0 + r * NT) == mpos) {
#pragma unroll
              for (int g = 0; g < kNB / 8; ++g)
                if (g < live) store8(&wrow[buf][warp][8 * g], &a[r][8 * g]);
            }
        }
        if (lane == 0) {
          wmag[buf][warp] = wm;
          wpos[buf][warp] = wp;
        }
        if (C > 1) {
          // a warp whose last wait gave up stops its whole CTA here
          stop = __syncthreads_or(!ok) != 0;
          if (stop) continue;
        } else if (W > 1) {
          __syncthreads();
        } else {
          __syncwarp();
        }
        // the CTA's best
        Mag best = wm;
        unsigned bpos = wp;
        int wb = 0;
        if (W > 1) {
          const Mag bm = lane < W ? wmag[buf][lane] : 0;
          const unsigned bp = lane < W ? wpos[buf][lane] : 0xffffffffu;
          best = bm;
          bpos = bp;
          pick(&best, &bpos);
          wb = __ffs(__ballot_sync(0xffffffffu, bm == best && bp == bpos)) - 1;
        }
        const T* prow = wrow[buf][wb];
        if (C > 1) {
          // push the row and its key to every CTA of the cluster (destinations spread
          // over the warps), then wait for the C pushes of this step
          const unsigned rdst = smem_addr(&crow[buf][q][lane]);
          const unsigned kdst = smem_addr(&ckey[buf][q]), pdst = smem_addr(&cpos[buf][kWide ? q : 0]);
          const unsigned bar = smem_addr(&cbar[buf]);
          const T rv = wrow[buf][wb][lane];
          const unsigned long long key = kWide ? (unsigned long long)best : (unsigned long long)best << 32 | bpos;
          if (tid == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                         "r"((unsigned)(C * (kNB * sizeof(T) + 8 + (kWide ? 4 : 0))))
                         : "memory");
          for (int dst = warp; dst < C; dst += W) {
            const unsigned rb = peer_addr(bar, dst);
            push(peer_addr(rdst, dst), rb, rv);
            if (lane == 0) push(peer_addr(kdst, dst), rb, key);
            if (kWide && lane == 1) push(peer_addr(pdst, dst), rb, bpos);
          }
          ok = __all_sync(0xffffffffu, bar_wait(bar, (jj >> 1) & 1, wait_ns, &late));
          const unsigned long long kk = lane < C ? ckey[buf][lane] : 0xffffffffull;
          const Mag km = kWide ? (lane < C ? (Mag)kk : 0) : (Mag)(kk >> 32);
          const unsigned kp = kWide && lane < C ? cpos[buf][lane] : (unsigned)kk;
          best = km;
          bpos = kp;
          pick(&best, &bpos);
          const int cb = __ffs(__ballot_sync(0xffffffffu, km == best && kp == bpos)) - 1;
          prow = crow[buf][cb];
        }
        if (ok) {
          T pv = prow[u];
          if (tid == 0) {
            spiv[jj] = best ? (int)bpos : jj;  // there is a candidate inside k columns, always
            spv[jj] = best ? pv : (T)0;
          }
          if (mag_bits(pv) == 0) pv = (T)(thresh > 0 ? thresh : 1e-30);
          const T inv = (T)1 / pv;
          T l[R];
#pragma unroll
          for (int r = 0; r < R; ++r) {
            if (pj[r] < 0 && (unsigned)(r == 0 ? pos0 : s0 + r * NT) == bpos) pj[r] = jj;
            l[r] = pj[r] < 0 ? a[r][u] * inv : (T)0;
            if (pj[r] < 0) a[r][u] = l[r];
          }
          if (pj[0] < 0 && pos0 == jj) pos0 = (int)bpos;  // the interchange moves the row at jj
#pragma unroll
          for (int g = 0; g < kNB / 8; ++g)
            if (g < live) {
              T p[8];
              load8(prow + 8 * g, p);
#pragma unroll
              for (int c = 0; c < 8; ++c) {
                if (8 * g + c <= u) continue;
#pragma unroll
                for (int r = 0; r < R; ++r)
                  if (pj[r] < 0) a[r][8 * g + c] = fma(-l[r], p[c], a[r][8 * g + c]);
              }
            }
        }
      }
    }
    // the finished block of eight columns goes to the back
#pragma unroll
    for (int r = 0; r < R; ++r) {
      T t[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) t[c] = a[r][c];
#pragma unroll
      for (int c = 0; c < kNB - 8; ++c) a[r][c] = a[r][c + 8];
#pragma unroll
      for (int c = 0; c < 8; ++c) a[r][kNB - 8 + c] = t[c];
    }
  }
  int* pvf = piv + f * k + j0;
  int* mpf = pmap + (f * ((k + kNB - 1) / kNB) + j0 / kNB) * (2 * kNB);
  if (C > 1 && __syncthreads_or(!ok || stop || late)) {
    // later kernels of the factorisation still read this panel's interchanges
    if (tid == 0) atomicOr(status, 2);
    if (q == 0)
      for (int c = tid; c < jb; c += NT) {
        pvf[c] = j0 + c;
        mpf[c] = c;
        mpf[kNB + c] = -1;
      }
  } else {
    // Replay of the interchanges from the pivots' positions, as in panel_map_kernel: step j
    // moves the pivot's slot to position j and the slot there to the pivot's old position.
    // Only the slots 0 .. 31 (whose position lane i tracks) and the pivots ever leave their
    // own position.
    if (W > 1) __syncthreads();
    else __syncwarp();
    if (warp == 0 && q == 0) {
      if (lane < jb && !(fabs((double)spv[lane]) > thresh)) atomicOr(status, 1);
      int pos = lane, fin = 0, pslot = lane;
      const int pdst = lane < jb ? spiv[lane] : lane;
      for (int j = 0; j < jb; ++j) {
        const int p = __shfl_sync(0xffffffffu, pdst, j);
        const unsigned at = __ballot_sync(0xffffffffu, pos == p && !fin);
        const int sb = at ? __ffs(at) - 1 : p;  // slot at position p
        const unsigned here = __ballot_sync(0xffffffffu, pos == j && !fin);
        const int ia = __ffs(here) - 1;  // slot at position j
        if (lane == ia) pos = p;
        if (lane == sb) {
          pos = j;
          fin = 1;
        }
        if (lane == j) pslot = sb;
      }
      if (lane < jb) {
        pvf[lane] = j0 + pdst;
        mpf[lane] = pslot;
        mpf[kNB + lane] = fin ? -1 : pos;
      }
      // the row permutation of the eliminated block, kept up to date
      int* pm = perm + f * k + j0;
      const int vs = lane < kl ? pm[lane] : 0;                 // at slot `lane`
      const int vp = lane < jb ? pm[pslot] : 0;                // at this step's pivot slot
      __syncwarp();
      if (lane < kl && !fin) pm[pos] = vs;
      if (lane < jb) pm[lane] = vp;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int sl = s0 + r * NT;
      if (sl < rows) {
        const int pos = pj[r] >= 0 ? pj[r] : (r == 0 ? pos0 : sl);
#pragma unroll
        for (int c = 0; c < kNB; ++c)
          if (c < jb) A[pos + (long)c * m] = a[r][c];
      }
    }
  }
  // no CTA leaves while a peer may still push into its shared memory
  if (C > 1)
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

// ---- tournament pivoting of the grid panel (FP32 forms) -------------------------
// Communication-avoiding LU of the panel (Grigori, Demmel and Xiang, "CALU", 2011):
// instead of one publication round per pivot column, the jb pivot rows are chosen
// by a tournament, then every row is eliminated against them at once.
//   1. each CTA runs partial-pivoting elimination on its candidate rows (slot below
//      k - j0) and publishes the ORIGINAL values of its jb winners (read again
//      from the front, which the panel does not change until its write-back);
//   2. the first CTA of every group of kCaluGroup CTAs gathers the group's winners,
//      runs the same elimination on them and publishes its jb winners' originals;
//   3. every CTA gathers the groups' winners and runs the same elimination, which
//      fixes the panel's pivot rows in order and their factored values [L11 | U11]
//      (every CTA computes identical values from identical inputs);
//   4. every other row gets its multipliers l = a U11^{-1} from its original values;
//   5. the interchanges and the write-back are those of lu_panel_grid_kernel.
// Pivots are chosen by FP32 magnitude with ties to the smaller slot.  Each wait on a
// publication gives up after wait_ns (status bit 2, identity interchanges, return).
constexpr int kCaluGroup = 16;
constexpr int kCaluMaxGroups = (kGridPanelMaxG + kCaluGroup - 1) / kCaluGroup;
constexpr int kCaluRow = kNB + 1;  // words of a published row: jb values, then the slot
constexpr long kCaluTagWords = 256;  // u64 words: tags of level 1 (G) and level 2 (groups)
constexpr long kCaluFrontWords =
    kCaluTagWords + ((long)(kGridPanelMaxG + kCaluMaxGroups) * kNB * kCaluRow + 1) / 2;
constexpr size_t kCaluBuf = sizeof(float) * (size_t)kCaluGroup * kNB * kCaluRow;  // gather buffer

// Partial-pivoting elimination of the rows [0, R) of the shared-memory matrix
// M(r, c) = M[r rs + c cs] (jb columns), candidates cand(r); up to jb pivots in order
// into sel[] (row indices), *nsel their count.  Rows are owned round-robin by the
// threads; two barriers per pivot.  used: R bytes of shared memory.
template <class Cand, class Slot>
__device__ void calu_gepp(float* M, int rs, int cs, int R, int jb, Cand cand, Slot slot,
                          unsigned char* used, int* sel, int* nsel, unsigned long long* wkey) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  auto keyof = [&](int r, int c) -> unsigned long long {
    const float v = fabsf(M[r * rs + c * cs]);
    return ((unsigned long long)__float_as_uint(v) << 32) |
           ((unsigned long long)(0xFFFFFu - (unsigned)slot(r)) << 12) | (unsigned long long)r;
  };
  for (int r = threadIdx.x; r < R; r += blockDim.x) used[r] = cand(r) ? 0 : 1;
  __syncthreads();
  unsigned long long key = 0ull;
  for (int r = threadIdx.x; r < R; r += blockDim.x)
    if (!used[r]) {
      const unsigned long long kk = keyof(r, 0);  // nonzero even for a zero entry (slot field)
      key = (kk > key) ? kk : key;
    }
  int n = 0;
  for (int jj = 0; jj < jb; ++jj) {
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long ok = __shfl_down_sync(0xffffffffu, key, o);
      key = ok > key ? ok : key;
    }
    if (lane == 0) wkey[warp] = key;
    __syncthreads();
    unsigned long long kb = 0ull;
    for (int w = 0; w < nw; ++w) kb = wkey[w] > kb ? wkey[w] : kb;
    // a candidate row always carries a key > 0 (its slot field is nonzero)
    if (kb == 0ull) break;
    const int p = (int)(kb & 0xFFFull);
    if (threadIdx.x == 0) sel[jj] = p;
    n = jj + 1;
    float pv = M[p * rs + jj * cs];
    if (!(fabsf(pv) > 0.f)) pv = 1e-30f;
    const float inv = 1.f / pv;
    key = 0ull;
    for (int r = threadIdx.x; r < R; r += blockDim.x) {
      if (used[r]) continue;
      if (r == p) {
        used[r] = 1;
        continue;
      }
      const float l = M[r * rs + jj * cs] * inv;
      M[r * rs + jj * cs] = l;
      for (int c = jj + 1; c < jb; ++c) M[r * rs + c * cs] -= l * M[p * rs + c * cs];
      if (jj + 1 < jb) {
        const unsigned long long kk = keyof(r, jj + 1);
        key = kk > key ? kk : key;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *nsel = n;
  __syncthreads();
}

__global__ void __launch_bounds__(256) lu_panel_calu_kernel(float* fronts, int m, int k, int j0,
                                                             int jb, int f0, int G, int* piv,
                                                             const double* scale, double ptol,
                                                             int* status, unsigned long long* pub,
                                                             unsigned long long wait_ns) {
  const int fl = blockIdx.x / G, g = blockIdx.x % G;
  const int f = f0 + fl;
  float* A = fronts + (long)f * m * m;
  const int rows = m - j0, kl = k - j0;
  const int chunk = (rows + G - 1) / G;
  const int s0 = min(rows, g * chunk), s1 = min(rows, s0 + chunk), nmy = s1 - s0;
  const int ngroups = (G + kCaluGroup - 1) / kCaluGroup;
  unsigned long long* tags = pub + (long)f * kCaluFrontWords;  // [G] then [ngroups]
  float* cand1 = reinterpret_cast<float*>(tags + kCaluTagWords);  // [G][jb][kCaluRow]
  float* cand2 = cand1 + (long)kGridPanelMaxG * kNB * kCaluRow;   // [groups][jb][kCaluRow]
  extern __shared__ unsigned long long smraw_u64[];
  float* P = reinterpret_cast<float*>(smraw_u64);              // chunk x jb, column-major
  float* Bf = P + (long)chunk * jb;                              // gather buffer, row-major
  unsigned char* used = reinterpret_cast<unsigned char*>(Bf + (long)kCaluGroup * kNB * kCaluRow);
  // used: max(chunk, kCaluGroup jb) bytes; pivj: chunk ints after it
  int* pivj = reinterpret_cast<int*>(used + ((max(chunk, kCaluGroup * kNB) + 15) & ~15));
  __shared__ float UF[kNB][kNB + 1];
  __shared__ int sel[kNB], pslot[kNB], bslot[kCaluGroup * kNB];
  __shared__ unsigned long long wkey[8];
  __shared__ int s_n, s_abort;
  __shared__ int ds[2 * kNB], dp[2 * kNB];
  __shared__ int s_nd, s_ok;
  __shared__ int cnt[kGridPanelMaxG], offs[kGridPanelMaxG + 1];
  const double thresh = ptol * scale[f];
  if (threadIdx.x == 0) s_abort = 0;
  // ---- 1. local tournament on the chunk
  for (long e = threadIdx.x; e < (long)nmy * jb; e += blockDim.x) {
    const int r = (int)(e % nmy), c = (int)(e / nmy);
    P[r + (long)c * chunk] = A[(j0 + s0 + r) + (long)(j0 + c) * m];
  }
  __syncthreads();
  calu_gepp(P, 1, chunk, nmy, jb, [&](int r) { return s0 + r < kl; }, [&](int r) { return s0 + r; },
            used, sel, &s_n, wkey);
  const int n1 = s_n;
  {
    float* out = cand1 + (long)g * kNB * kCaluRow;  // this CTA's level-1 block of its front
    for (int e = threadIdx.x; e < n1 * jb; e += blockDim.x) {
      const int i = e / jb, c = e % jb;
      const int r = sel[i];
      out[(long)i * kCaluRow + c] = A[(j0 + s0 + r) + (long)(j0 + c) * m];
      if (c == 0) out[(long)i * kCaluRow + jb] = __int_as_float(s0 + r);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) st_release64(tags + g, ((unsigned long long)n1 << 8) | 1ull);
  }
  // bounded wait for the tags [t0, t1) of `tags`; returns the candidate counts in cnt
  auto wait_tags = [&](const unsigned long long* tg, int t0, int t1) -> bool {
    if (threadIdx.x < 32) {
      const unsigned long long tstart = gtimer_ns();
      bool ok = true;
      for (int i = t0 + (int)threadIdx.x; i < t1; i += 32) {
        unsigned long long v = ld_acquire64(tg + i);
        while ((v & 0xFFull) != 1ull) {
          if (gtimer_ns() - tstart > wait_ns) {
            ok = false;
            break;
          }
          v = ld_acquire64(tg + i);
        }
        if (!ok) break;
        cnt[i - t0] = (int)(v >> 8);
      }
      ok = __all_sync(0xffffffffu, ok);
      if (threadIdx.x == 0) s_ok = ok ? 1 : 0;
    }
    __syncthreads();
    return s_ok != 0;
  };
  // gathers the candidate blocks [b0, b1) of `src` (counts in cnt) into Bf (row-major,
  // kCaluRow words per row; block b's rows start at offs[b - b0])
  auto gather = [&](const float* src, int b0, int b1) -> int {
    if (threadIdx.x == 0) {
      offs[0] = 0;
      for (int b = b0; b < b1; ++b) offs[b - b0 + 1] = offs[b - b0] + cnt[b - b0];
    }
    __syncthreads();
    const int tot = offs[b1 - b0];
    for (int b = b0; b < b1; ++b) {
      const float* blk = src + (long)b * kNB * kCaluRow;
      const int nb = cnt[b - b0], o = offs[b - b0];
      for (int e = threadIdx.x; e < nb * kCaluRow; e += blockDim.x)
        Bf[(long)o * kCaluRow + e] = __ldcg(blk + e);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < tot; i += blockDim.x) bslot[i] = __float_as_int(Bf[(long)i * kCaluRow + jb]);
    __syncthreads();
    return tot;
  };
  // ---- 2. group tournament (first CTA of each group)
  const int grp = g / kCaluGroup;
  if (g % kCaluGroup == 0) {
    const int b0 = grp * kCaluGroup, b1 = min(G, b0 + kCaluGroup);
    if (!wait_tags(tags, b0, b1)) {
      if (threadIdx.x == 0) {
        s_abort = 1;
        atomicOr(status, 2);
      }
    } else {
      const int tot = gather(cand1, b0, b1);
      calu_gepp(Bf, kCaluRow, 1, tot, jb, [&](int) { return true; }, [&](int r) { return bslot[r]; },
                used, sel, &s_n, wkey);
      const int n2 = s_n;
      float* out = cand2 + (long)grp * kNB * kCaluRow;
      // the winners' original rows: re-read from the level-1 area (Bf was eliminated)
      for (int e = threadIdx.x; e < n2 * kCaluRow; e += blockDim.x) {
        const int i = e / kCaluRow, c = e % kCaluRow;
        const int r = sel[i];
        // row r of Bf came from level-1 block b at row r - offs[b - b0]
        int b = b0;
        while (b + 1 < b1 && r >= offs[b + 1 - b0]) ++b;
        out[(long)i * kCaluRow + c] =
            __ldcg(cand1 + (long)b * kNB * kCaluRow + (long)(r - offs[b - b0]) * kCaluRow + c);
      }
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) st_release64(tags + G + grp, ((unsigned long long)n2 << 8) | 1ull);
    }
  }
  __syncthreads();
  // ---- 3. final tournament (every CTA)
  if (!s_abort) {
    if (!wait_tags(tags + G, 0, ngroups)) {
      if (threadIdx.x == 0) {
        s_abort = 1;
        atomicOr(status, 2);
      }
    }
  }
  __syncthreads();
  if (s_abort) {
    if (g == 0)
      for (int c = threadIdx.x; c < jb; c += blockDim.x) piv[(long)f * k + j0 + c] = j0 + c;
    return;
  }
  {
    const int tot = gather(cand2, 0, ngroups);
    calu_gepp(Bf, kCaluRow, 1, tot, jb, [&](int) { return true; }, [&](int r) { return bslot[r]; },
              used, sel, &s_n, wkey);
    if (s_n < jb) {  // fewer candidates than columns: cannot happen inside k
      if (threadIdx.x == 0) atomicOr(status, 1);
    }
    for (int e = threadIdx.x; e < jb * jb; e += blockDim.x) {
      const int j = e / jb, c = e % jb;
      UF[j][c] = j < s_n ? Bf[(long)sel[j] * kCaluRow + c] : (c == j ? 1.f : 0.f);
    }
    for (int j = threadIdx.x; j < jb; j += blockDim.x) pslot[j] = j < s_n ? bslot[sel[j]] : -1;
    __syncthreads();
    for (int j = threadIdx.x; j < jb; j += blockDim.x) {
      float d = UF[j][j];
      if (g == 0 && !(fabs((double)d) > thresh)) atomicOr(status, 1);
      if (!(fabsf(d) > 0.f)) UF[j][j] = (float)(thresh > 0 ? thresh : 1e-30);
    }
  }
  // ---- 4. rows of the chunk: pivot rows take their factored values, the others
  // their multipliers from the original values
  for (int r = threadIdx.x; r < nmy; r += blockDim.x) pivj[r] = -1;
  __syncthreads();
  for (int j = threadIdx.x; j < jb; j += blockDim.x)
    if (pslot[j] >= s0 && pslot[j] < s1) pivj[pslot[j] - s0] = j;
  for (long e = threadIdx.x; e < (long)nmy * jb; e += blockDim.x) {
    const int r = (int)(e % nmy), c = (int)(e / nmy);
    P[r + (long)c * chunk] = A[(j0 + s0 + r) + (long)(j0 + c) * m];
  }
  __syncthreads();
  for (int r = threadIdx.x; r < nmy; r += blockDim.x) {
    float* pr = P + r;
    const int j = pivj[r];
    if (j >= 0) {
      for (int c = 0; c < jb; ++c) pr[(long)c * chunk] = UF[j][c];
      continue;
    }
    for (int c = 0; c < jb; ++c) {
      float a = pr[(long)c * chunk];
      for (int i = 0; i < c; ++i) a -= pr[(long)i * chunk] * UF[i][c];
      pr[(long)c * chunk] = a / UF[c][c];
    }
  }
  // ---- 5. positions of the interchanges (pivot slot pslot[jj] to position jj) and
  // the write-back, as in lu_panel_grid_kernel
  if (threadIdx.x == 0) {
    int nd = 0;
    for (int jj = 0; jj < jb; ++jj) {
      const int sb = pslot[jj];
      int p = sb, ib = -1, sa = jj, ia = -1;
      for (int i = 0; i < nd; ++i) {
        if (ds[i] == sb) {
          p = dp[i];
          ib = i;
        }
      }
      for (int i = 0; i < nd; ++i)
        if (dp[i] == jj) {
          sa = ds[i];
          ia = i;
        }
      if (ia < 0)
        for (int i = 0; i < nd; ++i)
          if (ds[i] == sa) ia = i;
      if (ib < 0) {
        ib = nd++;
        ds[ib] = sb;
      }
      dp[ib] = jj;
      if (sa != sb) {
        if (ia < 0) {
          ia = nd++;
          ds[ia] = sa;
        }
        dp[ia] = p;
      }
      if (g == 0) piv[(long)f * k + j0 + jj] = j0 + p;
    }
    s_nd = nd;
  }
  __syncthreads();
  const int nd = s_nd;
  for (long e = threadIdx.x; e < (long)nmy * jb; e += blockDim.x) {
    const int r = (int)(e % nmy), c = (int)(e / nmy);
    const int sl = s0 + r;
    int pos = sl;
    for (int i = 0; i < nd; ++i)
      if (ds[i] == sl) pos = dp[i];
    A[(j0 + pos) + (long)(j0 + c) * m] = P[r + (long)c * chunk];
  }
}

// The interchanges of a panel as a map (per front and panel 2 x 32 ints, local rows):
// map[i] = the row whose content goes to row i (the i-th pivot), map[32 + i] = the row that
// takes row i's content, -1 when row i is a pivot itself.  Rows outside the map stay.  All
// reads come before all writes, so a column takes one memory latency where the 32
// exchanges in order took 32.  The register panel writes its map; this kernel makes it
// from the pivot rows of the other panels (one warp per front).
__global__ void panel_map_kernel(const int* piv, int* pmap, int k, int j0, int jb) {
  const long f = blockIdx.x;
  const int lane = threadIdx.x;
  const int pv = lane < jb ? piv[f * k + j0 + lane] - j0 : lane;
  int pos = lane, fin = 0, pslot = lane;
  for (int j = 0; j < jb; ++j) {
    const int p = __shfl_sync(0xffffffffu, pv, j);
    const unsigned at = __ballot_sync(0xffffffffu, pos == p && !fin);
    const int sb = at ? __ffs(at) - 1 : p;  // row at position p
    const unsigned here = __ballot_sync(0xffffffffu, pos == j && !fin);
    const int ia = __ffs(here) - 1;  // row at position j
    if (lane == ia) pos = p;
    if (lane == sb) {
      pos = j;
      fin = 1;
    }
    if (lane == j) pslot = sb;
  }
  int* mp = pmap + (f * ((k + kNB - 1) / kNB) + j0 / kNB) * (2 * kNB);
  if (lane < jb) {
    mp[lane] = pslot;
    mp[kNB + lane] = fin ? -1 : pos;
  }
}

// Interchanges of the panel's pivots and the row-block solve
// A[j0:j0+jb, c] = L_pp^{-1} A[j0:j0+jb, c] on the columns c in [c_lo, c_hi)
// outside the panel [j0, j0+jb): columns left of the panel get the interchanges
// only, columns right of it the interchanges (when do_swap) and the solve.
// The full-front form is c_lo = 0, c_hi = m, do_swap = 1.
// Four lanes per column (rows i = 4 r + lane % 4 in registers), eight columns per warp:
// a solve is 144 FMA instructions and 32 shuffles deep where one thread per column took
// 496 (in FP64, 64 cycles each), four times as many warps cover the SMs, and a column's
// rows load as whole sectors.  3D 32^3 FP64: 29 us a launch with one thread per column.
constexpr int kTrsmCols = 32;  // columns per CTA
template <class T>
__global__ void __launch_bounds__(4 * kTrsmCols) lu_trsm_kernel(T* fronts, int m, int k, int j0,
                                                                int jb, const int* pmap, int c_lo,
                                                                int c_hi, int do_swap) {
  T* A = fronts + (long)blockIdx.y * m * m;
  __shared__ T Lp[kNB][kNB + 1];
  __shared__ int mp[2 * kNB];
  for (int e = threadIdx.x; e < kNB * kNB; e += blockDim.x) {
    const int i = e % kNB, l = e / kNB;
    Lp[i][l] = (i < jb && l < i) ? A[(j0 + i) + (long)(j0 + l) * m] : (T)0;
  }
  if (do_swap && threadIdx.x < 2 * kNB)
    mp[threadIdx.x] =
        pmap[((long)blockIdx.y * ((k + kNB - 1) / kNB) + j0 / kNB) * (2 * kNB) + threadIdx.x];
  __syncthreads();
  const int nleft = max(0, min(j0, c_hi) - c_lo);
  const int rbeg = max(j0 + jb, c_lo);
  const int sub = threadIdx.x & 3;
  const int cc = blockIdx.x * kTrsmCols + (threadIdx.x >> 2);
  const int c = cc < nleft ? c_lo + cc : rbeg + (cc - nleft);
  const bool live = c < c_hi;
  T* col = A + (long)c * m + j0;
  constexpr int R = kNB / 4;
  T x[R], y[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = 4 * r + sub;
    const bool in = live && i < jb;
    y[r] = in ? col[i] : (T)0;
    x[r] = do_swap && in ? col[mp[i]] : y[r];
  }
  if (do_swap) {
    __syncwarp();  // the four lanes of a column have read it
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = 4 * r + sub;
      if (live && i < jb && mp[kNB + i] >= 0) col[mp[kNB + i]] = y[r];
    }
    __syncwarp();
  }
#pragma unroll
  for (int l = 0; l < kNB - 1; ++l) {
    const T xl = __shfl_sync(0xffffffffu, x[l >> 2], (threadIdx.x & 28) | (l & 3));
    if (cc >= nleft) {
#pragma unroll
      for (int r = l >> 2; r < R; ++r)
        if (r > (l >> 2) || sub > (l & 3)) x[r] = fma(-Lp[4 * r + sub][l], xl, x[r]);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = 4 * r + sub;
    if (live && i < jb) col[i] = x[r];
  }
}

// Row interchanges of the panels covering [p0, p0 + cnt) (in order, p0 a multiple of 32)
// on the columns [a0, a1) and [b0, b1) of every front: one warp per column, one panel's map
// at a time (two loads and two stores per lane).  One thread per column and one exchange
// after the other took up to 430 us a launch at 3D 64^3.
template <class T>
__global__ void __launch_bounds__(256) lu_laswp_kernel(T* fronts, int m, int k, int p0, int cnt,
                                                       const int* pmap, int a0, int a1, int b0,
                                                       int b1) {
  T* A = fronts + (long)blockIdx.y * m * m;
  const int lane = threadIdx.x & 31;
  const int cc = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int na = a1 - a0;
  const int c = cc < na ? a0 + cc : b0 + (cc - na);
  if (c >= (cc < na ? a1 : b1)) return;
  T* col = A + (long)c * m;
  const int* mp = pmap + ((long)blockIdx.y * ((k + kNB - 1) / kNB) + p0 / kNB) * (2 * kNB);
  int src = mp[lane], dst = mp[kNB + lane];
  for (int j0 = p0; j0 < p0 + cnt; j0 += kNB) {
    const int jb = min(kNB, p0 + cnt - j0);
    T* cj = col + j0;
    T x = 0, y = 0;
    if (lane < jb) {
      x = cj[src];
      y = cj[lane];
    }
    const int d = dst;
    mp += 2 * kNB;
    if (j0 + kNB < p0 + cnt) {
      src = mp[lane];
      dst = mp[kNB + lane];
    }
    __syncwarp();
    if (lane < jb) {
      cj[lane] = x;
      if (d >= 0) cj[d] = y;
    }
    __syncwarp();
  }
}

// Batched C[M x N] -= A[M x K] B[K x N], K <= kNB, column-major with leading
// dimensions lda/ldb/ldc and per-batch strides (blockIdx.y = batch); FP32.  TILE x TILE
// per CTA (TILE = 64: 4 x 4 per thread, TILE = 32: 2 x 2 per thread; the launcher
// picks the one that wastes less work on the padding of the last tile row and
// column): rows tx + 16 a, columns ty + 16 b, so a warp's C accesses stay contiguous.  The
// staged rows of A hold a thread's values side by side and those of B four steps of depth,
// so vector loads feed it (two per sixteen FMAs; as scalars, eight).  Bound by C traffic and
// the latency of one depth-32 pass per launch.  3D 64^3, root launches of the 32-wide tile:
// 10.2 -> 6.3 us, of the 64-wide 11.2 -> 8.2 us; 8 x 4 per thread (128 x 64) was slower on the
// leaves (two CTAs per SM).  Every entry adds its products in the order of l.
template <class T, int TILE>
__global__ void __launch_bounds__(256) gemm_sub_kernel(int M, int N, int K, const T* A, int lda,
                                                       long sA, const T* B, int ldb, long sB,
                                                       T* C, int ldc, long sC, int tilesM) {
  constexpr int R = TILE / 16;
  constexpr int pB = kNB + 4;  // B rows: 16-byte steps, spread over the banks
  A += blockIdx.y * sA;
  B += blockIdx.y * sB;
  C += blockIdx.y * sC;
  const int tr = blockIdx.x % tilesM, tc = blockIdx.x / tilesM;
  const int r0 = tr * TILE, c0 = tc * TILE;
  __shared__ __align__(16) T As[kNB][TILE];   // [l][(i % 16) R + i / 16]
  __shared__ __align__(16) T Bs[TILE][pB];    // [c][l]
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  // this thread's C entries are loaded first, so their latency overlaps the staging of
  // A and B and the products (the update is bound by C traffic)
  T cpre[R][R];
#pragma unroll
  for (int b = 0; b < R; ++b) {
    const int c = c0 + ty + 16 * b;
#pragma unroll
    for (int a = 0; a < R; ++a) {
      const int r = r0 + tx + 16 * a;
      cpre[a][b] = (r < M && c < N) ? C[r + (long)c * ldc] : (T)0;
    }
  }
  // the depth is padded to a multiple of four with zeros
  const int K4 = (K + 3) & ~3;
  for (int e = threadIdx.x; e < K4 * TILE; e += 256) {
    const int sl = e % TILE, l = e / TILE;
    const int r = r0 + (sl % R) * 16 + sl / R;
    As[l][sl] = (r < M && l < K) ? A[r + (long)l * lda] : (T)0;
  }
  for (int e = threadIdx.x; e < kNB * TILE; e += 256) {
    const int l = e % kNB, jc = e / kNB;
    const int c = c0 + jc;
    Bs[jc][l] = (c < N && l < K) ? B[l + (long)c * ldb] : (T)0;
  }
  __syncthreads();
  struct alignas(R * sizeof(T)) VecA {
    T v[R];
  };
  struct alignas(4 * sizeof(T)) VecB {
    T v[4];
  };
  T acc[R][R];
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) acc[a][b] = 0;
#pragma unroll 2
  for (int l = 0; l < K4; l += 4) {
    VecB bv[R];
#pragma unroll
    for (int b = 0; b < R; ++b) bv[b] = *reinterpret_cast<const VecB*>(&Bs[ty + 16 * b][l]);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const VecA av = *reinterpret_cast<const VecA*>(&As[l + u][tx * R]);
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) acc[a][b] += av.v[a] * bv[b].v[u];
    }
  }
#pragma unroll
  for (int b = 0; b < R; ++b) {
    int c = c0 + ty + 16 * b;
    if (c >= N) continue;
#pragma unroll
    for (int a = 0; a < R; ++a) {
      int r = r0 + tx + 16 * a;
      if (r < M) C[r + (long)c * ldc] = cpre[a][b] - acc[a][b];
    }
  }
}

// One batched product C = beta C + alpha A B (column-major, any K) with triangle-aware K
// ranges: tri_a = 1 when A is lower triangular (A[r, l] = 0 for l > r), 2 when
// upper (A[r, l] = 0 for l < r); tri_b = 1 when B is lower (B[l, c] = 0 for
// l < c), 2 when upper (B[l, c] = 0 for l > c).  Zero tiles are skipped, entries
// inside a computed tile must hold their zeros.  beta is 0 or 1.
// batch index = outer * nb2 + inner with strides (sA, sB, sC) and (sA2, sB2, sC2)
template <class T>
struct GemmSide {
  int M = 0, N = 0, K = 0;
  const T* A = nullptr;
  int lda = 0;
  long sA = 0, sA2 = 0;
  const T* B = nullptr;
  int ldb = 0;
  long sB = 0, sB2 = 0;
  T* C = nullptr;
  int ldc = 0;
  long sC = 0, sC2 = 0;
  int tri_a = 0, tri_b = 0;
};

// A launch takes one product or two independent ones of a batch (blockIdx.z: the inverses
// of L and U, whose chains of small products then cost one launch each instead of two).
template <class T, int TILE>
__global__ void __launch_bounds__(256) gemm_gen_kernel(GemmSide<T> g0, GemmSide<T> g1, T alpha,
                                                       int beta_one, int nb2) {
  constexpr int R = TILE / 16;  // outputs per thread along each dimension
  const GemmSide<T> g = blockIdx.z ? g1 : g0;
  const int M = g.M, N = g.N, lda = g.lda, ldb = g.ldb, ldc = g.ldc;
  const int tilesM = (M + TILE - 1) / TILE, tilesN = (N + TILE - 1) / TILE;
  if ((int)blockIdx.x >= tilesM * tilesN) return;
  const long bo = blockIdx.y / nb2, bi = blockIdx.y % nb2;
  const T* A = g.A + bo * g.sA + bi * g.sA2;
  const T* B = g.B + bo * g.sB + bi * g.sB2;
  T* C = g.C + bo * g.sC + bi * g.sC2;
  const int tr = blockIdx.x % tilesM, tc = blockIdx.x / tilesM;
  const int r0 = tr * TILE, c0 = tc * TILE;
  int klo = 0, khi = g.K;
  if (g.tri_a == 1) khi = min(khi, r0 + TILE);
  if (g.tri_a == 2) klo = max(klo, r0);
  if (g.tri_b == 1) klo = max(klo, c0);
  if (g.tri_b == 2) khi = min(khi, c0 + TILE);
  __shared__ T As[kNB][TILE];
  __shared__ T Bs[kNB][TILE + 1];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  T acc[R][R];
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) acc[a][b] = 0;
  for (int k0 = klo; k0 < khi; k0 += kNB) {
    const int kc = min(kNB, khi - k0);
    for (int e = threadIdx.x; e < kNB * TILE; e += blockDim.x) {
      int i = e % TILE, l = e / TILE;
      int r = r0 + i;
      As[l][i] = (r < M && l < kc) ? A[r + (long)(k0 + l) * lda] : (T)0;
    }
    for (int e = threadIdx.x; e < kNB * TILE; e += blockDim.x) {
      int l = e % kNB, jc = e / kNB;
      int c = c0 + jc;
      Bs[l][jc] = (c < N && l < kc) ? B[(k0 + l) + (long)c * ldb] : (T)0;
    }
    __syncthreads();
#pragma unroll 4
    for (int l = 0; l < kNB; ++l) {
      T av[R], bv[R];
#pragma unroll
      for (int a = 0; a < R; ++a) av[a] = As[l][tx + 16 * a];
#pragma unroll
      for (int b = 0; b < R; ++b) bv[b] = Bs[l][ty + 16 * b];
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) acc[a][b] += av[a] * bv[b];
    }
    __syncthreads();
  }
#pragma unroll
  for (int b = 0; b < R; ++b) {
    int c = c0 + ty + 16 * b;
    if (c >= N) continue;
#pragma unroll
    for (int a = 0; a < R; ++a) {
      int r = r0 + tx + 16 * a;
      if (r < M) {
        T v = alpha * acc[a][b];
        if (beta_one) v += C[r + (long)c * ldc];
        C[r + (long)c * ldc] = v;
      }
    }
  }
}

__global__ void perm_identity_kernel(int* perm, int k, long np) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < np) perm[i] = (int)(i % k);
}

__global__ void lu_perm_kernel(const int* piv, int* perm, int k, int nf) {
  int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= nf) return;
  int* p = perm + (long)f * k;
  const int* pv = piv + (long)f * k;
  for (int j = 0; j < k; ++j) p[j] = j;
  for (int j = 0; j < k; ++j) {
    int t = p[j];
    p[j] = p[pv[j]];
    p[pv[j]] = t;
  }
}

// ---- explicit triangular inverses -------------------------------------------------
// Inverses of every 32 x 32 diagonal block of L11 (unit lower) and U11 of every front, one
// CTA per (block, front): threads 0-127 invert the L block, 128-255 the U block, four lanes
// per column (rows 4 r + lane % 4 in registers) as in lu_trsm_kernel.  Xl != null: written to the matching diagonal
// blocks of Xl and Xu (entry (i, j) at i + j ldx, front stride sX).  Xl == null: in place,
// the strict lower part from L^{-1}, the upper part with the diagonal from U^{-1}; the
// sweeps then resolve a diagonal block with a matrix-vector product instead of 32
// dependent steps.  With one thread per column (496 FMAs and 32 divisions in a row) an FP64
// launch took 64 us however few its blocks were.  The FP32 U block keeps one thread per
// column: row i subtracts its products in the order of l = i + 1 ..., which starts with the
// entry computed last, so four lanes could only take another order, and the FP32
// preconditioner's bits would change with it (2D 512^2, all inverses: 2.41 -> 2.49 ms).
template <class T>
__global__ void __launch_bounds__(256) diag32_kernel(T* fronts, int m, int k, T* Xl, T* Xu, int ldx,
                                                     long sX) {
  const int j0 = blockIdx.x * kNB;
  const int jb = min(kNB, k - j0);
  T* A = fronts + (long)blockIdx.y * m * m;
  __shared__ T Bk[kNB][kNB + 1];
  for (int e = threadIdx.x; e < kNB * kNB; e += 256) {
    const int i = e % kNB, l = e / kNB;
    Bk[i][l] = (i < jb && l < jb) ? A[(j0 + i) + (long)(j0 + l) * m] : (i == l ? (T)1 : (T)0);
  }
  __syncthreads();
  const bool upper = threadIdx.x >= 128;
  if (sizeof(T) == sizeof(float) && upper) {
    const int c = threadIdx.x - 128;
    if (c >= jb) return;
    T x[kNB];
#pragma unroll
    for (int i = 0; i < kNB; ++i) x[i] = i == c ? (T)1 : (T)0;
#pragma unroll
    for (int i = kNB - 1; i >= 0; --i) {
      T acc = x[i];
#pragma unroll
      for (int l = i + 1; l < kNB; ++l) acc = fma(-Bk[i][l], x[l], acc);
      x[i] = acc / Bk[i][i];
    }
    T* out = Xl == nullptr ? A + j0 + (long)(j0 + c) * m
                           : Xu + (long)blockIdx.y * sX + j0 + (long)(j0 + c) * ldx;
#pragma unroll
    for (int i = 0; i < kNB; ++i)
      if (i < jb && (Xl != nullptr || i <= c)) out[i] = x[i];
    return;
  }
  const int sub = threadIdx.x & 3, c = (threadIdx.x & 127) >> 2, base = threadIdx.x & 28;
  constexpr int R = kNB / 4;
  T x[R];
#pragma unroll
  for (int r = 0; r < R; ++r) x[r] = 4 * r + sub == c ? (T)1 : (T)0;
  if (!upper) {
#pragma unroll
    for (int l = 0; l < kNB - 1; ++l) {
      if (l < (c & ~7)) continue;  // still zero in the warp's eight columns
      const T xl = __shfl_sync(0xffffffffu, x[l >> 2], base | (l & 3));
#pragma unroll
      for (int r = l >> 2; r < R; ++r)
        if (r > (l >> 2) || sub > (l & 3)) x[r] = fma(-Bk[4 * r + sub][l], xl, x[r]);
    }
  } else {
#pragma unroll
    for (int l = kNB - 1; l >= 0; --l) {
      if (l > (c | 7)) continue;
      if (sub == (l & 3)) x[l >> 2] /= Bk[l][l];
      const T xl = __shfl_sync(0xffffffffu, x[l >> 2], base | (l & 3));
#pragma unroll
      for (int r = 0; r <= (l >> 2); ++r)
        if (r < (l >> 2) || sub < (l & 3)) x[r] = fma(-Bk[4 * r + sub][l], xl, x[r]);
    }
  }
  if (c >= jb) return;
  T* out = Xl == nullptr ? A + j0 + (long)(j0 + c) * m
                         : (upper ? Xu : Xl) + (long)blockIdx.y * sX + j0 + (long)(j0 + c) * ldx;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = 4 * r + sub;
    if (i < jb && (Xl != nullptr || (i > c) != upper)) out[i] = x[r];
  }
}

// F11 <- strict lower part of Linv, upper part (with the diagonal) of Uinv, on
// the diagonal blocks of size Bsz only (the off-diagonal blocks keep L11, U11).
// X entry (r, c) at r + c Bsz (front stride sX); one thread per entry of the blocks, whose
// existing part is side x side.
template <class T>
__global__ void trinv_store_kernel(T* fronts, int m, const T* Xl, const T* Xu, long sX, int k,
                                   int Bsz, int side) {
  const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long bb = (long)side * side;
  const long blk = e / bb, rem = e % bb;
  const long r = blk * Bsz + rem % side, c = blk * Bsz + rem / side;
  if (r >= k || c >= k) return;
  const long f = blockIdx.y;
  const long x = f * sX + r + c * Bsz;
  fronts[f * (long)m * m + r + c * m] = (r > c) ? Xl[x] : Xu[x];
}

// ---- FP64 products on the tensor cores -----------------------------------------------
// C = beta C +- A B in FP64 from exact integer products (the error-free splitting of
// Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by
// using fast routines of matrix multiplication", Numer. Algorithms 59, 2012).  FP64 FMAs
// run at two per SM cycle here, FP16 tensor-core products at a thousand.
//
// Per 32-deep chunk, a row of A (a column of B) is written on a common exponent E, the
// largest of its 32 entries: x = X 2^(E - 1084) with |X| < 2^62 an integer that keeps all
// 53 bits of every entry down to 2^-9 of the largest and 62 bits below that on.  X is cut
// into seven balanced digits of nine bits, X = sum_i f_i 2^(9 i), |f_i| <= 256, each an
// exact FP16 number.  The sums S_h = sum_{i + j = h + 6} sum_k f_i(A) f_j(B), h = 0 .. 6, are
// then exact in the FP32 accumulators of mma.sync (at most 7 x 32 x 2^16 < 2^24), and
// sum_k A B = 2^(Ea + Eb - 2114) sum_h S_h 2^(9 h) up to the digit pairs with i + j < 6.  The
// sum of the S_h is formed as a 64-bit integer and enters C with two FP64 FMAs.
//
// Error, in X X and whatever the entries are: digit pairs left out 2^68.6, bits cut from
// entries more than nine binades below their row's largest 2^67.  Against sum |a b| that is
// nothing where the large entries of the row meet those of the column, and everything where
// they only meet zeros or far smaller ones.  So the leading digits give a lower bound of
// sum |a b|, one more product: P = sum_k |f_6(a)| |f_6(b)|, and |X| >= (|f_6| - 0.501) 2^54.
//   P >= 2^14 (a leading digit at its smallest times another, so a row's largest entry that
//     meets a column's largest is enough): sum |X X| > 2^121, the 64-bit sum in units of 2^68
//     adds 2^68 with the first FMA; the error is below 2^-51 sum |a b|.
//   1088 <= P < 2^14: sum |X X| > 2^117.04; units of 2^63 add 2^63; below 2^-48 sum |a b|, the
//     bound of an FMA loop of 32 steps.
//   P < 1088: the FMA loop over the entries where row and column are both nonzero (a mask of 32
//     bits each); no such entry: the product is zero and C stays.
//
// One CTA: a 64 x 64 tile, eight warps of 16 x 32 (two halves of 16 x 16, so the 56
// accumulators of a half fit beside the fragments and two CTAs share an SM).  The tile's
// digits are cut once into shared memory (rows of 32 halves, 80 bytes apart: conflict-free
// for ldmatrix), 29 products of 16 x 16 x 16 per 16 x 16 block and 16 of depth.  What
// bounds it: latency between the phases of a tile (load, cut, multiply, combine) and the FMA
// loops of the outputs of low weight; no pipe is above 40 % (leaf level of 2D 512^2: FP64 38, ALU 34,
// tensor 18).  Three FP64 instructions, ~30 integer ones and 29 / 16 x 2 tensor instructions per
// output and chunk, where the FMA loop took 32 FP64 instructions.  All 101 updates of a 2D 512^2
// factor 10.2 ms (FMA loop 33), 205 of 3D 32^3 39.9 (144).
// Rows whose entries leave [2^-477, 2^477] (subnormals too), and infinities and NaNs, take the
// FMA loop for the whole tile.
constexpr int kDig = 7;          // digits of a number
constexpr int kDigT = 64;        // tile
constexpr int kDigPitch = 40;    // halves between the 32-deep rows of a digit plane
constexpr int kDigPlane = kDigT * kDigPitch;
constexpr float kDigWeight = 1088.f;  // smallest leading-digit product sum that the digits carry
constexpr float kDigFine = 16384.f;   // below: the 64-bit sum in finer units
constexpr int kDigElo = 546, kDigEhi = 1500;  // biased exponents of a row's largest entry
constexpr size_t kDigSmem = 2 * kDig * kDigPlane * sizeof(__half);

// biased exponent (1 for subnormals, 0 for zero)
__device__ __forceinline__ int f64_exp(double x) {
  const int hi = __double2hiint(x) & 0x7fffffff;
  return hi >= 0x100000 ? hi >> 20 : ((hi | __double2loint(x)) != 0 ? 1 : 0);
}

// the seven digits of eight numbers on the exponent E, written as eight consecutive halves
// of seven planes (dst: the first plane's 16 bytes)
__device__ __forceinline__ void cut_digits(const double* x, int E, __half* dst) {
  unsigned w[kDig][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    unsigned f[2][kDig];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const double v = x[2 * p + h];
      const int hi = __double2hiint(v);
      const int ex = (hi >> 20) & 0x7ff, d = E - ex;
      unsigned long long m =
          ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
      m = (ex == 0 || d > 62) ? 0ull : (m << 9) >> d;
      // every digit shifted by +256, so the fields below are unsigned
      constexpr unsigned long long kBias =
          256ull * (1ull | 1ull << 9 | 1ull << 18 | 1ull << 27 | 1ull << 36 | 1ull << 45 | 1ull << 54);
      const unsigned long long u = hi < 0 ? kBias - m : kBias + m;
      const unsigned lo = (unsigned)u, up = (unsigned)(u >> 32);
      f[h][0] = lo & 511u;
      f[h][1] = (lo >> 9) & 511u;
      f[h][2] = (lo >> 18) & 511u;
      f[h][3] = __funnelshift_r(lo, up, 27) & 511u;
      f[h][4] = (up >> 4) & 511u;
      f[h][5] = (up >> 13) & 511u;
      f[h][6] = up >> 22;
    }
#pragma unroll
    for (int i = 0; i < kDig; ++i) {
      // 0x6400 | f is the FP16 number 1024 + f; minus 1280 leaves the digit f - 256
      const unsigned t = (f[0][i] | (f[1][i] << 16)) | 0x64006400u;
      const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&t), __half2half2(__ushort_as_half(0x6500)));
      w[i][p] = *reinterpret_cast<const unsigned*>(&v);
    }
  }
#pragma unroll
  for (int i = 0; i < kDig; ++i)
    *reinterpret_cast<uint4*>(dst + i * kDigPlane) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}

__device__ __forceinline__ void ldmatrix4(unsigned* r, unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void mma_f16(float* c, const unsigned* a, unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// acc +- sum_h S_h 2^(9 h), from the 64-bit sum T of the S_h in units of 2^68 (in X X), or of
// 2^63 (fine) where the weight keeps |T| below 2^61; es the biased exponent of the unit 2^68
__device__ __forceinline__ double add_digits(double acc, const float* S, int es, bool fine, unsigned neg) {
  const int s0 = __float2int_rn(S[0]), s1 = __float2int_rn(S[1]), s2 = __float2int_rn(S[2]);
  const int s3 = __float2int_rn(S[3]), s4 = __float2int_rn(S[4]), s5 = __float2int_rn(S[5]);
  const int s6 = __float2int_rn(S[6]);
  const long long low = (long long)s3 * 262144 + ((long long)s2 * 512 + (s1 + ((s0 + 256) >> 9)));
  const long long top = (long long)s6 * 262144 + ((long long)s5 * 512 + s4);
  const long long T = fine ? (long long)((unsigned long long)top << 27) + low : (top << 22) + ((low + 16) >> 5);
  if (fine) es -= 5;
  // T = hi 2^32 + lo as two exact doubles: 2^52 + lo, and hi - 2^20 (its 2^52 cancels)
  const double dl = __hiloint2double(0x43300000, (int)(unsigned)T);
  const double dh = __hiloint2double(0x43300000, (int)(T >> 32) ^ (int)0x80000000) -
                    (4503599627370496.0 + 2147483648.0 + 1048576.0);
  const double sl = __hiloint2double((int)(((unsigned)es << 20) | neg), 0);
  const double sh = __hiloint2double((int)(((unsigned)(es + 32) << 20) | neg), 0);
  return fma(sl, dl, fma(sh, dh, acc));
}

// ONE: K <= 32 (one chunk; C read while the products run).  Arguments as gemm_gen_kernel,
// alpha = -1 (neg = the sign bit) or 1.
template <bool ONE>
__global__ void __launch_bounds__(256, ONE ? 2 : 1) gemm_f64_kernel(GemmSide<double> g0,
                                                                  GemmSide<double> g1, unsigned neg,
                                                                  int beta_one, int nb2) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __half* Ad = reinterpret_cast<__half*>(smraw);
  __half* Bd = Ad + kDig * kDigPlane;
  __shared__ int eA[4][kDigT], eB[kDigT];
  __shared__ __align__(4) unsigned char nzA[kDigT][4], nzB[kDigT][4];  // nonzero entries, eight to a byte
  __shared__ int s_plain;
  const GemmSide<double> g = blockIdx.z ? g1 : g0;
  const int M = g.M, N = g.N, lda = g.lda, ldb = g.ldb, ldc = g.ldc;
  const int tilesM = (M + kDigT - 1) / kDigT, tilesN = (N + kDigT - 1) / kDigT;
  if ((int)blockIdx.x >= tilesM * tilesN) return;
  const long bo = blockIdx.y / nb2, bi = blockIdx.y % nb2;
  const double* A = g.A + bo * g.sA + bi * g.sA2;
  const double* B = g.B + bo * g.sB + bi * g.sB2;
  double* C = g.C + bo * g.sC + bi * g.sC2;
  const int r0 = (blockIdx.x % tilesM) * kDigT, c0 = (blockIdx.x / tilesM) * kDigT;
  int klo = 0, khi = g.K;
  if (g.tri_a == 1) khi = min(khi, r0 + kDigT);
  if (g.tri_a == 2) klo = max(klo, r0);
  if (g.tri_b == 1) klo = max(klo, c0);
  if (g.tri_b == 2) khi = min(khi, c0 + kDigT);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // this thread's outputs: half s, n-tile t, register i: row rw + 8 (i / 2), column
  // cw + 16 s + 8 t + (i & 1)
  const int rw = (warp & 3) * 16 + (lane >> 2), cw = (warp >> 2) * 32 + 2 * (lane & 3);
  auto out_at = [&](int s, int i) -> long {
    const int r = r0 + rw + 8 * ((i >> 1) & 1), c = c0 + cw + 16 * s + 8 * (i >> 2) + (i & 1);
    return r < M && c < N ? r + (long)c * ldc : -1;
  };
  double acc[ONE ? 1 : 2][8];
  if (!ONE) {
#pragma unroll
    for (int s = 0; s < (ONE ? 1 : 2); ++s)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const long at = out_at(s, i);
        acc[s][i] = beta_one && at >= 0 ? C[at] : 0.0;
      }
  }
  const int ai = tid & 63, ak = (tid >> 6) * 8;       // A: row, first of eight columns
  const int bc = tid >> 2, bk = (tid & 3) * 8;        // B: column, first of eight rows
  const unsigned a_frag = smem_addr(Ad + ((warp & 3) * 16 + (lane & 15)) * kDigPitch + (lane >> 4) * 8);
  const unsigned b_frag = smem_addr(
      Bd + ((warp >> 2) * 32 + (lane >> 4) * 8 + (lane & 7)) * kDigPitch + ((lane >> 3) & 1) * 8);
  for (int k0 = klo; k0 < khi; k0 += 32) {
    const int kc = min(32, khi - k0);
    double xa[8], xb[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      xa[j] = (r0 + ai < M && ak + j < kc) ? A[r0 + ai + (long)(k0 + ak + j) * lda] : 0.0;
      xb[j] = (c0 + bc < N && bk + j < kc) ? B[k0 + bk + j + (long)(c0 + bc) * ldb] : 0.0;
    }
    if (tid == 0) s_plain = 0;
    int ea = 0, eb = 0;
    unsigned za = 0, zb = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int fa = f64_exp(xa[j]), fb = f64_exp(xb[j]);
      ea = max(ea, fa);
      eb = max(eb, fb);
      za |= (fa != 0 ? 1u : 0u) << j;
      zb |= (fb != 0 ? 1u : 0u) << j;
    }
    nzA[ai][tid >> 6] = (unsigned char)za;
    nzB[bc][tid & 3] = (unsigned char)zb;
    eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, 1));
    eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, 2));
    eA[tid >> 6][ai] = ea;
    if ((tid & 3) == 0) eB[bc] = eb;
    __syncthreads();  // exponents written; the previous chunk's digits are read
    ea = max(max(eA[0][ai], eA[1][ai]), max(eA[2][ai], eA[3][ai]));
    if ((ea != 0 && (ea < kDigElo || ea > kDigEhi)) || (eb != 0 && (eb < kDigElo || eb > kDigEhi)))
      s_plain = 1;
    cut_digits(xa, ea, Ad + ai * kDigPitch + ak);
    cut_digits(xb, eb, Bd + bc * kDigPitch + bk);
    __syncthreads();
    if (s_plain) {  // an exponent outside the range of the scales (uniform)
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const long at = out_at(s, i);
          if (at < 0) continue;
          const long r = at % ldc, c = at / ldc;
          double v = 0.0;
          for (int k = k0; k < k0 + kc; ++k) v = fma(A[r + (long)k * lda], B[k + c * ldb], v);
          if (neg) v = -v;
          if (ONE) C[at] = beta_one ? C[at] + v : v;
          else acc[ONE ? 0 : s][i] += v;
        }
      __syncthreads();
      continue;
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if (ONE) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const long at = out_at(s, i);
          acc[0][i] = beta_one && at >= 0 ? C[at] : 0.0;
        }
      }
      float P[kDig][2][4];
#pragma unroll
      for (int h = 0; h < kDig; ++h)
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
          for (int i = 0; i < 4; ++i) P[h][t][i] = 0.f;
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) {
        if (ks * 16 < kc) {
          unsigned fa[kDig][4];
#pragma unroll
          for (int i = 0; i < kDig; ++i) ldmatrix4(fa[i], a_frag + 2 * (i * kDigPlane + ks * 16));
#pragma unroll
          for (int j = 0; j < kDig; ++j) {
            unsigned fb[4];
            ldmatrix4(fb, b_frag + 2 * (j * kDigPlane + s * 16 * kDigPitch + ks * 16));
#pragma unroll
            for (int i = 0; i < kDig; ++i)
              if (i + j >= kDig - 1) {
                mma_f16(P[i + j - (kDig - 1)][0], fa[i], fb[0], fb[1]);
                mma_f16(P[i + j - (kDig - 1)][1], fa[i], fb[2], fb[3]);
              }
          }
        }
      }
      // the weight of each output's products
      float Q[2][4];
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int i = 0; i < 4; ++i) Q[t][i] = 0.f;
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) {
        if (ks * 16 < kc) {
          unsigned fa[4], fb[4];
          ldmatrix4(fa, a_frag + 2 * ((kDig - 1) * kDigPlane + ks * 16));
          ldmatrix4(fb, b_frag + 2 * ((kDig - 1) * kDigPlane + s * 16 * kDigPitch + ks * 16));
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            fa[i] &= 0x7fff7fffu;
            fb[i] &= 0x7fff7fffu;
          }
          mma_f16(Q[0], fa, fb[0], fb[1]);
          mma_f16(Q[1], fa, fb[2], fb[3]);
        }
      }
      // the digit sums of all eight outputs without a branch between them (their FP64 chains
      // overlap), then the few of low weight
      unsigned low = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int row = rw + 8 * ((i >> 1) & 1), col = cw + 16 * s + 8 * (i >> 2) + (i & 1);
        const int er = max(max(eA[0][row], eA[1][row]), max(eA[2][row], eA[3][row]));
        float v[kDig];
#pragma unroll
        for (int h = 0; h < kDig; ++h) v[h] = P[h][i >> 2][i & 3];
        double& o = acc[ONE ? 0 : s][i];
        const float q = Q[i >> 2][i & 3];
        const double t = add_digits(o, v, max(er + eB[col] - 1077, 6), q < kDigFine, neg);
        if (q >= kDigWeight) o = t;
        else low |= 1u << i;
      }
      if (low) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int row = rw + 8 * ((i >> 1) & 1), col = cw + 16 * s + 8 * (i >> 2) + (i & 1);
          unsigned both = *reinterpret_cast<const unsigned*>(nzA[row]) & *reinterpret_cast<const unsigned*>(nzB[col]);
          if (!(low >> i & 1)) both = 0;
          if (both) {
            const double* ar = A + r0 + row + (long)k0 * lda;
            const double* bc_ = B + k0 + (long)(c0 + col) * ldb;
            double sum[4] = {0.0, 0.0, 0.0, 0.0};  // an FP64 chain a quarter as long
            while (both) {
              double x[4], y[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const int k = __ffs(both) - 1;
                x[u] = both ? ar[(long)k * lda] : 0.0;
                y[u] = both ? bc_[k] : 0.0;
                both &= both - 1;
              }
#pragma unroll
              for (int u = 0; u < 4; ++u) sum[u] = fma(x[u], y[u], sum[u]);
            }
            const double v = (sum[0] + sum[1]) + (sum[2] + sum[3]);
            double& o = acc[ONE ? 0 : s][i];
            o = neg ? o - v : o + v;
          }
        }
      }
      if (ONE) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const long at = out_at(s, i);
          if (at >= 0) C[at] = acc[0][i];
        }
      }
    }
    if (!ONE) __syncthreads();  // digits and exponents read before the next chunk's
  }
  if (!ONE) {
#pragma unroll
    for (int s = 0; s < (ONE ? 1 : 2); ++s)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const long at = out_at(s, i);
        if (at >= 0) C[at] = acc[s][i];
      }
  }
}

void gemm_f64(const GemmSide<double>& g0, const GemmSide<double>* g1, bool minus, bool beta_one,
              int batch, int nb2, cudaStream_t st) {
  static PerDevice attr;
  attr.run([] {
    const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(gemm_f64_kernel<true>, at, (int)kDigSmem);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(gemm_f64_kernel<false>, at, (int)kDigSmem);
  });  // a refusal shows as the launch's error
  auto tiles = [](const GemmSide<double>& g) {
    return ((g.M + kDigT - 1) / kDigT) * ((g.N + kDigT - 1) / kDigT);
  };
  dim3 gr((unsigned)(g1 ? std::max(tiles(g0), tiles(*g1)) : tiles(g0)), (unsigned)(batch * nb2), g1 ? 2 : 1);
  const bool one = g0.K <= 32 && (!g1 || g1->K <= 32) && beta_one;
  auto kern = one ? gemm_f64_kernel<true> : gemm_f64_kernel<false>;
  kern<<<gr, 256, kDigSmem, st>>>(g0, g1 ? *g1 : g0, minus ? 0x80000000u : 0u, beta_one ? 1 : 0, nb2);
}

template <class T>
void gemm_sub(int M, int N, int K, const T* A, int lda, long sA, const T* B, int ldb, long sB,
              T* C, int ldc, long sC, int batch, cudaStream_t st, int tile = 0) {
  if (M <= 0 || N <= 0 || K <= 0) return;
  if constexpr (sizeof(T) == sizeof(double)) {
    GemmSide<T> g{M, N, K, A, lda, sA, 0, B, ldb, sB, 0, C, ldc, sC, 0, 0, 0};
    gemm_f64(g, nullptr, true, true, batch, 1, st);
  } else {
    // padded work of 64- and 32-wide tiles relative to M N
    const double w64 = (double)((M + 63) / 64 * 64) * ((N + 63) / 64 * 64);
    const double w32 = (double)((M + 31) / 32 * 32) * ((N + 31) / 32 * 32);
    const int t = tile == 32 || (tile == 0 && w64 > 1.1 * w32) ? 32 : 64;
    const int tilesM = (M + t - 1) / t, tilesN = (N + t - 1) / t;
    dim3 g(tilesM * tilesN, batch);
    auto kern = t == 32 ? gemm_sub_kernel<T, 32> : gemm_sub_kernel<T, 64>;
    kern<<<g, 256, 0, st>>>(M, N, K, A, lda, sA, B, ldb, sB, C, ldc, sC, tilesM);
  }
}

// one product (g1 null) or two, alpha = -1 (minus) or 1
template <class T>
void gemm_gen(const GemmSide<T>& g0, const GemmSide<T>* g1, bool minus, bool beta_one, int batch,
              int nb2, int tile, cudaStream_t st) {
  if (g0.M <= 0 || g0.N <= 0 || g0.K <= 0 || batch <= 0 || nb2 <= 0) return;
  if constexpr (sizeof(T) == sizeof(double)) {
    gemm_f64(g0, g1, minus, beta_one, batch, nb2, st);
  } else {
    auto tiles = [&](const GemmSide<T>& g, int t) { return (long)((g.M + t - 1) / t) * ((g.N + t - 1) / t); };
    // a small problem takes 32 x 32 tiles: four times the CTAs
    const int t = tile == 32 || (tile == 0 && tiles(g0, kTile) * batch * nb2 < 304) ? 32 : kTile;
    dim3 gr((unsigned)(g1 ? std::max(tiles(g0, t), tiles(*g1, t)) : tiles(g0, t)), (unsigned)(batch * nb2),
            g1 ? 2 : 1);
    auto kern = t == 32 ? gemm_gen_kernel<T, 32> : gemm_gen_kernel<T, kTile>;
    kern<<<gr, 256, 0, st>>>(g0, g1 ? *g1 : g0, minus ? (T)-1 : (T)1, beta_one ? 1 : 0, nb2);
  }
}

// Replace the diagonal blocks (size Bsz, a power of two >= 32) of L11 and U11 of
// every front of the level by the blocks of L11^{-1} (strict lower part; the unit
// diagonal is implied) and U11^{-1} (upper part).  The sweeps of such a level are
// then short chains of matrix-vector products spread over many CTAs.
// Recursive doubling on the diagonal blocks (32, 64, 128, ... up to Bsz):
//   [A 0; B C]^{-1} = [A^{-1} 0; -C^{-1} (B A^{-1}), C^{-1}]
//   [A B; 0 C]^{-1} = [A^{-1}, -(A^{-1} B) C^{-1}; 0 C^{-1}]
// with the two products of each merge as batched GEMMs over fronts, pairs and the two
// triangles.
// Storage: the inverses Xl, Xu keep entry (i, j) of a diagonal block at
// i + j Bsz (a column-major array with leading dimension Bsz whose columns
// overlap: the diagonal blocks never collide, and a pair's diagonal step is
// 2 s (1 + Bsz) everywhere), k (Bsz + 1) entries per front; the work arrays Wl, Wu
// hold pair p's product at rows [2ps, 2ps+s) of a k x Bsz/2 block per front.
template <class T>
void invert_triangles(DevLevel& L, T* scratch, int Bsz, cudaStream_t st) {
  const int k = L.k, m = L.m, nf = L.nf;
  const long mm = (long)m * m;
  const int ldx = Bsz;
  const long sX = (long)k * (Bsz + 1), sW = (long)k * (Bsz / 2);
  T* F = (T*)L.front;
  T* Xl = scratch;
  T* Xu = scratch + sX * nf;
  T* Wl = scratch + 2 * sX * nf;
  T* Wu = Wl + sW * nf;
  cudaMemsetAsync(Xl, 0, sizeof(T) * sX * nf, st);
  cudaMemsetAsync(Xu, 0, sizeof(T) * sX * nf, st);
  const int nb = (k + kNB - 1) / kNB;
  dim3 gd(nb, nf);
  diag32_kernel<T><<<gd, 256, 0, st>>>(F, m, k, Xl, Xu, ldx, sX);
  for (int s = kNB; s < k && s < Bsz; s *= 2) {
    // pairs p: A at [2ps, 2ps+s), C at [2ps+s, min(2ps+2s, k)); the pairs with a
    // full-size C go in one batched launch (fronts x pairs), a ragged last pair in
    // a second one.
    const int npairs = (k + 2 * s - 1) / (2 * s);
    const int last_c = k - ((npairs - 1) * 2 * s + s);
    const int nfull = (last_c >= s) ? npairs : npairs - 1;
    const long ps_x = 2L * s * (1 + ldx), ps_m = 2L * s * (1 + m), ps_w = 2L * s;
    for (int pass = 0; pass < 2; ++pass) {
      int cnt, p0, sc;
      if (pass == 0) {
        cnt = nfull;
        p0 = 0;
        sc = s;
      } else {
        if (nfull == npairs || last_c <= 0) continue;
        cnt = 1;
        p0 = npairs - 1;
        sc = last_c;
      }
      if (cnt <= 0) continue;
      const int a0 = p0 * 2 * s, c0 = a0 + s;
      // lower: Wl = B Ainv (B = L[c0.., a0..], Ainv lower), Xl[c0.., a0..] = -Cinv Wl;
      // upper: Wu = Ainv B (B = U[a0.., c0..], Ainv upper), Xu[a0.., c0..] = -Wu Cinv
      const GemmSide<T> l1{sc, s, s, F + c0 + (long)a0 * m, m, mm, ps_m, Xl + a0 + (long)a0 * ldx, ldx, sX,
                           ps_x, Wl + a0, k, sW, ps_w, 0, 1};
      const GemmSide<T> u1{s, sc, s, Xu + a0 + (long)a0 * ldx, ldx, sX, ps_x, F + a0 + (long)c0 * m, m, mm,
                           ps_m, Wu + a0, k, sW, ps_w, 2, 0};
      gemm_gen<T>(l1, &u1, false, false, nf, cnt, L.gen_tile, st);
      const GemmSide<T> l2{sc, s, sc, Xl + c0 + (long)c0 * ldx, ldx, sX, ps_x, Wl + a0, k, sW, ps_w,
                           Xl + c0 + (long)a0 * ldx, ldx, sX, ps_x, 1, 0};
      const GemmSide<T> u2{s, sc, sc, Wu + a0, k, sW, ps_w, Xu + c0 + (long)c0 * ldx, ldx, sX, ps_x,
                           Xu + a0 + (long)c0 * ldx, ldx, sX, ps_x, 0, 2};
      gemm_gen<T>(l2, &u2, true, false, nf, cnt, L.gen_tile, st);
    }
  }
  // fronts with fewer than Bsz eliminated rows have one k x k block (threads over the
  // whole Bsz x Bsz block of 4096 fronts with k = 25 took 3.2 ms)
  const int side = std::min(k, Bsz);
  const long nbk = (k + Bsz - 1) / Bsz;
  dim3 g((unsigned)((nbk * side * side + 255) / 256), nf);
  trinv_store_kernel<T><<<g, 256, 0, st>>>(F, m, Xl, Xu, sX, k, Bsz, side);
}

template <class T>
int panel_width(int m) {
  return m > 0 ? kNB : 0;
}
// Fronts per launch (nfl) and CTAs per front (G) of the grid panel for `rows`
// panel rows: every CTA's rows fit in kGridPanelSmem, nfl G <= kGridPanelCTAs.
template <class T>
void grid_panel_shape(int nf, int rows, int* nfl, int* G) {
  const long cmax = (long)(kGridPanelSmem / (sizeof(T) * kNB + 1));
  const int gmin = (int)std::max<long>(1, (rows + cmax - 1) / cmax);
  *nfl = std::max(1, std::min(nf, kGridPanelCTAs / gmin));
  *G = std::max(1, std::min(kGridPanelMaxG, std::min(kGridPanelCTAs / *nfl, (rows + 31) / 32)));
}

// the tournament panel's shared memory: the chunk (jb floats per row), the gather
// buffer, the row flags and the pivot map
size_t calu_smem(int chunk) {
  return sizeof(float) * (size_t)chunk * kNB + kCaluBuf +
         (size_t)((std::max(chunk, kCaluGroup * kNB) + 15) & ~15) + sizeof(int) * (size_t)chunk;
}
void calu_shape(int nf, int rows, int* nfl, int* G) {
  const long per_row = sizeof(float) * kNB + 1 + sizeof(int);
  const long cmax = (long)(kGridPanelSmem - kCaluBuf - kCaluGroup * kNB - 16) / per_row;
  const int gmin = (int)std::max<long>(1, (rows + cmax - 1) / cmax);
  *nfl = std::max(1, std::min(nf, kGridPanelCTAs / gmin));
  *G = std::max(1, std::min(kGridPanelMaxG, std::min(kGridPanelCTAs / *nfl, (rows + 31) / 32)));
}

// Fronts that may need the grid panel (their publication slots are allocated): those
// too tall for the registers of eight CTAs at the smaller row count of FP64 or FP32.
// panel_pivoting = 1 takes the tournament on all of them.
template <class T>
bool grid_panel_front(int m) {
  return (size_t)((m + 7) / 8) * kNB * sizeof(T) + 2 * sizeof(int) * (size_t)m > 160 * 1024;
}

// Largest cluster of the register panel on the current device: 16 CTAs (not a portable
// size) when one of its largest form can be resident, else 8.
int panel_max_cluster() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 8;
  static std::atomic<int> cache[64];  // 0: not asked yet
  if (cache[dev]) return cache[dev];
  int best = 8;
  auto kern = lu_panel_reg_kernel<double, 256, 3>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kPanelMaxC);
    cfg.blockDim = dim3(256);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kPanelMaxC;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n >= 1) best = kPanelMaxC;
  }
  cudaGetLastError();  // a refused query leaves no error behind
  cache[dev] = best;
  return best;
}

// CTAs per front (C), threads (NT) and rows per thread (R) of the register panel for
// `rows` panel rows of nf fronts; false: too tall.  A step costs ~1000 cycles on one CTA
// and ~600 more through a cluster (32 columns: 24 us at 256 rows, 34 us at 1024 on one
// CTA and 36 us on a cluster of four).  FP32: one CTA up to 1024 rows; beyond, CTAs of
// 256 rows while the level leaves SMs free (2044 rows: 33 us on eight CTAs, 43 us on
// two), else up to 1536 rows per CTA.  FP64: the rank-1 updates run at two FMAs per SM
// cycle, so a level with few fronts splits each over as many SMs as there are, down to
// ~96 rows per CTA (2044 rows: 66 us on 16 CTAs; before the reciprocal was a division 61, and 80 on
// eight).
template <class T>
bool panel_shape(int nf, int rows, int* C, int* NT, int* R) {
  const int maxc = panel_max_cluster();
  int c = 1;
  const int most = sizeof(T) == 4 ? 1536 : 768;   // rows a CTA's registers hold
  const int aim = sizeof(T) == 4 ? 256 : 96;      // rows per CTA where SMs are free
  const bool spread = sizeof(T) == 8 || rows > 1024;
  while (rows > c * most || (spread && rows > c * aim && (long)nf * c * 2 <= 152 && c < maxc)) c *= 2;
  if (c > maxc) return false;
  const int rc = (rows + c - 1) / c;
  static const int s32[7][2] = {{32, 1}, {32, 2}, {64, 2}, {128, 2}, {256, 2}, {256, 4}, {256, 6}};
  // 513 .. 768 rows of many fronts: 128 x 6 leaves fewer idle rows (512 fronts of 729
  // rows: 82 us against 117 us as 256 x 4)
  if (sizeof(T) == 4 && rc > 512 && rc <= 768 && nf > 152) {
    *C = c;
    *NT = 128;
    *R = 6;
    return true;
  }
  static const int s64[6][2] = {{32, 1}, {64, 1}, {128, 1}, {128, 2}, {128, 3}, {256, 3}};
  const int (*sh)[2] = sizeof(T) == 4 ? s32 : s64;
  const int n = sizeof(T) == 4 ? 7 : 6;
  for (int i = 0; i < n; ++i)
    if (rc <= sh[i][0] * sh[i][1]) {
      *C = c;
      *NT = sh[i][0];
      *R = sh[i][1];
      return true;
    }
  return false;
}

// whether the level's panels are the register panel (decided by its tallest)
template <class T>
bool panel_in_registers(const DevLevel& L, const FactorWork& W) {
  int c, nt, r;
  if (W.grid_panel) return false;
  if (sizeof(T) == 4 && W.calu && grid_panel_front<T>(L.m)) return false;
  return panel_shape<T>(L.nf, L.m, &c, &nt, &r);
}

template <class T, int NT, int R>
void launch_panel_reg(DevLevel& L, T* F, int j0, int jb, int C, double ptol, int* status,
                      const FactorWork& W, cudaStream_t st) {
  auto kern = lu_panel_reg_kernel<T, NT, R>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(L.nf * C));
  cfg.blockDim = dim3(NT);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  if (C > 1) {
    static PerDevice attr;
    attr.run([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1); });
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
  cudaLaunchKernelEx(&cfg, kern, F, L.m, L.k, j0, jb, C, L.piv, L.pmap, L.perm, (const double*)L.scale, ptol,
                     status, W.wait_ns);
}

template <class T>
void panel_reg(DevLevel& L, T* F, int j0, int jb, double ptol, int* status, const FactorWork& W,
               cudaStream_t st) {
  int C, NT, R;
  if (!panel_shape<T>(L.nf, L.m - j0, &C, &NT, &R)) return;  // panel_in_registers: cannot happen
  auto go = [&](auto nt, auto r) {
    launch_panel_reg<T, decltype(nt)::value, decltype(r)::value>(L, F, j0, jb, C, ptol, status, W, st);
  };
  using std::integral_constant;
  if constexpr (sizeof(T) == 4) {
    if (NT == 32 && R == 1) go(integral_constant<int, 32>{}, integral_constant<int, 1>{});
    else if (NT == 32) go(integral_constant<int, 32>{}, integral_constant<int, 2>{});
    else if (NT == 64) go(integral_constant<int, 64>{}, integral_constant<int, 2>{});
    else if (NT == 128 && R == 2) go(integral_constant<int, 128>{}, integral_constant<int, 2>{});
    else if (NT == 128) go(integral_constant<int, 128>{}, integral_constant<int, 6>{});
    else if (R == 2) go(integral_constant<int, 256>{}, integral_constant<int, 2>{});
    else if (R == 4) go(integral_constant<int, 256>{}, integral_constant<int, 4>{});
    else go(integral_constant<int, 256>{}, integral_constant<int, 6>{});
  } else {
    if (NT == 32) go(integral_constant<int, 32>{}, integral_constant<int, 1>{});
    else if (NT == 64) go(integral_constant<int, 64>{}, integral_constant<int, 1>{});
    else if (NT == 128 && R == 1) go(integral_constant<int, 128>{}, integral_constant<int, 1>{});
    else if (NT == 128 && R == 2) go(integral_constant<int, 128>{}, integral_constant<int, 2>{});
    else if (NT == 128) go(integral_constant<int, 128>{}, integral_constant<int, 3>{});
    else go(integral_constant<int, 256>{}, integral_constant<int, 3>{});
  }
}

// Panel LU of columns [j0, j0+jb) followed by the interchanges and the row-block
// solve on the columns [c_lo, c_hi) outside the panel.
template <class T>
void panel_step(DevLevel& L, T* F, int j0, int jb, int c_lo, int c_hi, double ptol, int* status,
                const FactorWork& W, cudaStream_t st) {
  double pf = 0;
  for (int j = j0; j < j0 + jb; ++j) pf += (double)(L.m - j - 1) * (1.0 + 2.0 * (j0 + jb - j - 1));
  ProfScope pp(PROF_LU_PANEL, st);
  if (panel_in_registers<T>(L, W)) {
    panel_reg<T>(L, F, j0, jb, ptol, status, W, st);
  } else if (sizeof(T) == sizeof(float) && W.calu) {
    const int rows = L.m - j0;
    if (rows >= (1 << 20)) return;  // slot field of the pivot key; factor_level_t rejects it
    int nfl, G;
    calu_shape(L.nf, rows, &nfl, &G);
    const int chunk = (rows + G - 1) / G;
    for (int f0 = 0; f0 < L.nf; f0 += nfl) {
      const int nfg = std::min(nfl, L.nf - f0);
      // fresh publication tags for every launch (graph replays reuse the buffer)
      for (int fi = 0; fi < nfg; ++fi)
        cudaMemsetAsync(W.gpub + (size_t)(f0 + fi) * kCaluFrontWords, 0,
                        sizeof(unsigned long long) * kCaluTagWords, st);
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(nfg * G));
      cfg.blockDim = dim3(256);
      cfg.dynamicSmemBytes = calu_smem(chunk);
      cfg.stream = st;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeCooperative;
      at[0].val.cooperative = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      cudaLaunchKernelEx(&cfg, lu_panel_calu_kernel, (float*)F, L.m, L.k, j0, jb, f0, G, L.piv,
                         (const double*)L.scale, ptol, status, W.gpub, W.wait_ns);
    }
  } else {
    const int rows = L.m - j0;
    if (rows >= (1 << 20)) return;  // slot field of the pivot word; factor_level_t rejects it
    int nfl, G;
    grid_panel_shape<T>(L.nf, rows, &nfl, &G);
    const int chunk = (rows + G - 1) / G;
    const size_t sm = sizeof(T) * (size_t)chunk * jb + (size_t)chunk;
    for (int f0 = 0; f0 < L.nf; f0 += nfl) {
      const int nfg = std::min(nfl, L.nf - f0);
      // fresh publication tags for every launch (graph replays reuse the buffer)
      cudaMemsetAsync(W.gpub + (size_t)f0 * 2 * kGridPanelMaxG * kPubWords, 0,
                      sizeof(unsigned long long) * (size_t)nfg * 2 * kGridPanelMaxG * kPubWords,
                      st);
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(nfg * G));
      cfg.blockDim = dim3(256);
      cfg.dynamicSmemBytes = sm;
      cfg.stream = st;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeCooperative;
      at[0].val.cooperative = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      cudaLaunchKernelEx(&cfg, lu_panel_grid_kernel<T>, F, L.m, L.k, j0, jb, f0, G, L.piv,
                         (const double*)L.scale, ptol, status, W.gpub, W.wait_ns);
    }
  }
  if (!panel_in_registers<T>(L, W)) panel_map_kernel<<<L.nf, 32, 0, st>>>(L.piv, L.pmap, L.k, j0, jb);
  pp.done(pf * L.nf, 1, st);
  const int nleft = std::max(0, std::min(j0, c_hi) - c_lo);
  const int nright = std::max(0, c_hi - std::max(j0 + jb, c_lo));
  const int ncols = nleft + nright;
  if (ncols > 0) {
    dim3 gt((ncols + kTrsmCols - 1) / kTrsmCols, L.nf);
    ProfScope pt(PROF_LU_TRSM, st);
    lu_trsm_kernel<T><<<gt, 4 * kTrsmCols, 0, st>>>(F, L.m, L.k, j0, jb, L.pmap, c_lo, c_hi, 1);
    pt.done((double)nright * jb * (jb - 1) * L.nf, 1, st);
  }
}

// C -= A B on the fronts (M x N x K sub-blocks at the given offsets, leading
// dimension m, front stride m^2): SIMT tiles for K <= 32, else the general GEMM
// or, for the tensor-core form, TF32 tensor cores.
template <class T>
void schur_update(DevLevel& L, T* F, int M, int N, int K, long offA, long offB, long offC,
                  const FactorWork& W, int* status, cudaStream_t st) {
  if (M <= 0 || N <= 0 || K <= 0) return;
  const long mm = (long)L.m * L.m;
  const double fl = 2.0 * M * N * K * L.nf;
  if (K <= kNB) {
    ProfScope pg(PROF_LU_GEMM, st);
    gemm_sub<T>(M, N, K, F + offA, L.m, mm, F + offB, L.m, mm, F + offC, L.m, mm, L.nf, st,
                L.gemm_tile);
    pg.done(fl, 1, st);
    return;
  }
  if constexpr (sizeof(T) == sizeof(float)) {
    if (W.tc) {
      ProfScope pc(PROF_LU_TC, st);
      tc_schur_update(M, N, K, (const float*)(F + offA), L.m, mm, (const float*)(F + offB), L.m, mm,
                      (float*)(F + offC), L.m, mm, L.nf, W.packA, W.packB, W.tc_split, status, st,
                      W.tc_epi);
      pc.done(fl, 3, st);
      return;
    }
  }
  ProfScope pg(PROF_LU_GEMM, st);
  const GemmSide<T> g{M, N, K, F + offA, L.m, mm, 0, F + offB, L.m, mm, 0, F + offC, L.m, mm, 0, 0, 0};
  gemm_gen<T>(g, nullptr, true, true, L.nf, 1, 0, st);
  pg.done(fl, 1, st);
}

template <class T>
void front_scale(DevLevel& L, cudaStream_t st) {
  const long mm = (long)L.m * L.m;
  cudaMemsetAsync(L.scale, 0, sizeof(double) * L.nf, st);
  long chunks = std::min<long>(std::max<long>(1, mm / (256 * 16)), std::max<long>(1, 1216 / L.nf));
  dim3 gs((unsigned)chunks, L.nf);
  front_scale_kernel<T><<<gs, 256, 0, st>>>((const T*)L.front, mm, L.scale);
}

// LU of the fronts of a level and the inverses of their diagonal blocks, from the assembled
// fronts and their largest magnitudes L.scale.
template <class T>
cudaError_t lu_fronts(DevLevel& L, double ptol, int* status, const FactorWork& W, cudaStream_t st) {
  static PerDevice attr;
  const cudaError_t ea = attr.run([] {
    const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(lu_panel_grid_kernel<T>, at, (int)kGridPanelSmem + 1024);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(lu_panel_calu_kernel, at, (int)kGridPanelSmem + 1024);
  });
  if (ea != cudaSuccess) return ea;
  const int m = L.m, k = L.k;
  T* F = (T*)L.front;
  if (panel_in_registers<T>(L, W)) {
    const long np = (long)L.nf * k;
    perm_identity_kernel<<<(unsigned)((np + 255) / 256), 256, 0, st>>>(L.perm, k, np);
  }
  const int NB = panel_width<T>(m);
  if (NB == 0 || m >= (1 << 20)) return cudaErrorInvalidValue;
  const int OB = factor_outer_block(sizeof(T) == sizeof(float) ? SP_PREC_FP32 : SP_PREC_FP64, W.tc,
                                    m, k);
  if (OB == 0) {
    // right-looking LU with a Schur update after every 32-column panel
    for (int j0 = 0; j0 < k; j0 += NB) {
      const int jb = std::min(NB, k - j0);
      panel_step<T>(L, F, j0, jb, 0, m, ptol, status, W, st);
      const int base = j0 + jb, rem = m - base;
      schur_update<T>(L, F, rem, rem, jb, base + (long)j0 * m, j0 + (long)base * m,
                      base + (long)base * m, W, status, st);
    }
  } else {
    // Two-level blocked LU.  An outer block [J0, e1) of OB columns is factored in
    // sub-blocks [J1, e2) of IB columns; a sub-block is factored by 32-column
    // panel steps whose interchanges, row-block solves and updates stay inside it,
    // then its interchanges go to the rest of the outer block, its row band
    // [J1, e2) x [e2, e1) is solved and the outer block's remaining columns get
    // one update of depth IB.  After the outer block its interchanges go to the
    // other columns, the row band U12 = L11^{-1} A12 is solved in the same
    // sub-block pattern, and the trailing matrix gets one update of depth OB.
    // The updates of depth > 32 run on the tensor cores in the tensor-core forms.
    // block sizes from the outer block down to the panels: OB, 256, 32.  (A third
    // level of 128 columns, whose depth-128 updates would run on the tensor cores
    // too, leaves too much TF32 rounding in the columns next to the panels: at 3D
    // 128^3 one Helmholtz medium's preconditioner stalled GMRES at 0.42 with it.)
    const int IB = std::min(OB, kTcSubBlock);
    std::vector<int> bsz = {OB};
    if (IB < OB) bsz.push_back(IB);
    bsz.push_back(NB);
    auto laswp = [&](int p0, int cnt, int a0, int a1, int b0, int b1) {
      const int ncols = std::max(0, a1 - a0) + std::max(0, b1 - b0);
      if (ncols <= 0 || cnt <= 0) return;
      ProfScope pt(PROF_LU_TRSM, st);
      dim3 g((ncols + 7) / 8, L.nf);
      lu_laswp_kernel<T><<<g, 256, 0, st>>>(F, m, k, p0, cnt, L.pmap, a0, std::max(a0, a1), b0,
                                            std::max(b0, b1));
      pt.done(0, 1, st);
    };
    // row band [r0, r1) x [c0, c1) solved with the unit lower block at [r0, r1): the
    // rows split in blocks of bsz[lev] (recursively down to 32-row solve steps), each
    // block's update of the rows below it of depth bsz[lev]
    std::function<void(int, int, int, int, int)> band = [&](int r0, int r1, int c0, int c1,
                                                            int lev) {
      if (c1 <= c0 || r1 <= r0) return;
      const int bs = bsz[lev];
      if (bs == NB) {
        for (int j0 = r0; j0 < r1; j0 += NB) {
          const int jb = std::min(NB, r1 - j0);
          {
            const int ncol = c1 - c0;
            dim3 gt((ncol + kTrsmCols - 1) / kTrsmCols, L.nf);
            ProfScope pt(PROF_LU_TRSM, st);
            lu_trsm_kernel<T><<<gt, 4 * kTrsmCols, 0, st>>>(F, m, k, j0, jb, L.pmap, c0, c1, 0);
            pt.done((double)ncol * jb * (jb - 1) * L.nf, 1, st);
          }
          const int base = j0 + jb;
          schur_update<T>(L, F, r1 - base, c1 - c0, jb, base + (long)j0 * m, j0 + (long)c0 * m,
                          base + (long)c0 * m, W, status, st);
        }
        return;
      }
      for (int B0 = r0; B0 < r1; B0 += bs) {
        const int B1 = std::min(r1, B0 + bs);
        band(B0, B1, c0, c1, lev + 1);
        schur_update<T>(L, F, r1 - B1, c1 - c0, B1 - B0, B1 + (long)B0 * m, B0 + (long)c0 * m,
                        B1 + (long)c0 * m, W, status, st);
      }
    };
    // LU of the columns [J, e) (rows J .. m) whose width is at most bsz[lev]: sub-blocks
    // of bsz[lev + 1] columns factored in turn (32-column panel steps at the bottom),
    // each followed by its interchanges on the block's other columns, the row band of
    // the block's columns to its right and their update of depth bsz[lev + 1]
    std::function<void(int, int, int)> block = [&](int J, int e, int lev) {
      const int bs = bsz[lev + 1];
      if (bs == NB) {
        for (int j0 = J; j0 < e; j0 += NB) {
          const int jb = std::min(NB, e - j0);
          panel_step<T>(L, F, j0, jb, J, e, ptol, status, W, st);
          const int base = j0 + jb;
          schur_update<T>(L, F, m - base, e - base, jb, base + (long)j0 * m, j0 + (long)base * m,
                          base + (long)base * m, W, status, st);
        }
        return;
      }
      for (int J1 = J; J1 < e; J1 += bs) {
        const int e2 = std::min(e, J1 + bs);
        block(J1, e2, lev + 1);
        laswp(J1, e2 - J1, J, J1, e2, e);
        if (e2 < e) {
          band(J1, e2, e2, e, lev + 2);
          schur_update<T>(L, F, m - e2, e - e2, e2 - J1, e2 + (long)J1 * m, J1 + (long)e2 * m,
                          e2 + (long)e2 * m, W, status, st);
        }
      }
    };
    for (int J0 = 0; J0 < k; J0 += OB) {
      const int e1 = std::min(k, J0 + OB);
      block(J0, e1, 0);
      laswp(J0, e1 - J0, 0, J0, e1, m);
      if (e1 < m) {
        band(J0, e1, e1, m, 1);
        schur_update<T>(L, F, m - e1, m - e1, e1 - J0, e1 + (long)J0 * m, J0 + (long)e1 * m,
                        e1 + (long)e1 * m, W, status, st);
      }
    }
  }
  // the register panels keep the row permutation themselves
  if (!panel_in_registers<T>(L, W))
    lu_perm_kernel<<<(L.nf + 127) / 128, 128, 0, st>>>(L.piv, L.perm, L.k, L.nf);
  ProfScope pi(PROF_LU_TRINV, st);
  double bw = 0;
  if (L.inv) {
    invert_triangles<T>(L, (T*)W.inv, L.ib, st);
    const int Bz = L.ib < L.k ? L.ib : L.k;
    bw = (2.0 / 3.0) * (double)Bz * Bz * L.k * L.nf;
  } else {
    dim3 gd((L.k + kNB - 1) / kNB, L.nf);
    diag32_kernel<T><<<gd, 256, 0, st>>>(F, L.m, L.k, (T*)nullptr, (T*)nullptr, 0, 0L);
    bw = (2.0 / 3.0) * (double)kNB * kNB * L.k * L.nf;
  }
  pi.done(bw, 1, st);
  return cudaGetLastError();
}

template <class T>
cudaError_t factor_level_t(int d, DevLevel& L, const DevLevel* child, const double* Qcat,
                           const double* Ccat, const double* q, double ptol, int* status,
                           const FactorWork& W, cudaStream_t st) {
  const long mm = (long)L.m * L.m;
  T* F = (T*)L.front;
  ProfScope pa(PROF_ASSEMBLE, st);
  cudaError_t e = cudaMemsetAsync(F, 0, sizeof(T) * mm * L.nf, st);
  if (e != cudaSuccess) return e;
  int na = 1;
  if (L.nasm > 0) {
    dim3 g((L.nasm + 255) / 256, L.nf);
    assemble_kernel<T><<<g, 256, 0, st>>>(F, L.m, L.nasm, L.asm_row, L.asm_tidx, L.asm_cvar,
                                          L.gidx, Qcat, Ccat, q, L.nfp > 0 ? L.nfp : L.nf,
                                          W.tab_stride);
    ++na;
  }
  double abytes = (double)sizeof(T) * mm * L.nf;
  if (child) {
    const int nbd = L.mc - L.kc;
    long work = (long)nbd * nbd;
    dim3 g((unsigned)((work + 256 * kEaU - 1) / (256 * kEaU)), L.nf);
    for (int dl = 0; dl < (1 << d); ++dl)
      extend_add_kernel<T><<<g, 256, 0, st>>>(F, L.m, L.nb1, (const T*)child->front, L.mc, L.kc,
                                               L.ea_map + (long)dl * nbd, dl, d);
    na += 1 << d;
    abytes += (double)sizeof(T) * work * child->nf;
  }
  front_scale<T>(L, st);
  pa.done(abytes, na + 1, st);
  return lu_fronts<T>(L, ptol, status, W, st);
}

}  // namespace

cudaError_t factor_level(int prec, int d, DevLevel& L, const DevLevel* child, const double* Qcat,
                         const double* Ccat, const double* q, double pivot_tol, int* status,
                         const FactorWork& W, cudaStream_t st) {
  if (prec == SP_PREC_FP32)
    return factor_level_t<float>(d, L, child, Qcat, Ccat, q, pivot_tol, status, W, st);
  return factor_level_t<double>(d, L, child, Qcat, Ccat, q, pivot_tol, status, W, st);
}

cudaError_t front_lu_raw(int prec, int m, int k, int nf, int grid_panel, double pivot_tol,
                         unsigned long long wait_ns, void* fronts, int* piv, int* perm, int* status,
                         cudaStream_t st) {
  DevLevel L;
  FactorWork W;
  L.m = m;
  L.k = k;
  L.nf = nf;
  L.front = fronts;
  L.piv = piv;
  L.perm = perm;
  W.grid_panel = grid_panel;
  W.wait_ns = wait_ns;
  cudaError_t e = cudaMalloc(&L.scale, sizeof(double) * nf);
  if (e == cudaSuccess) e = cudaMalloc(&L.pmap, sizeof(int) * 2 * kNB * nf * ((k + kNB - 1) / kNB));
  if (e == cudaSuccess && (grid_panel || factor_grid_panel(prec, m)))
    e = cudaMalloc(&W.gpub, sizeof(unsigned long long) * grid_panel_pub_words(nf));
  if (e == cudaSuccess) e = cudaMemsetAsync(status, 0, sizeof(int), st);
  auto go = [&](auto t) {
    using T = decltype(t);
    front_scale<T>(L, st);
    return lu_fronts<T>(L, pivot_tol, status, W, st);
  };
  if (e == cudaSuccess) e = prec == SP_PREC_FP32 ? go(0.f) : go(0.0);
  const cudaError_t es = cudaStreamSynchronize(st);
  cudaFree(L.scale);
  cudaFree(L.pmap);
  cudaFree(W.gpub);
  return e != cudaSuccess ? e : es;
}

cudaError_t schur_update_raw(int prec, bool tc, bool split, int M, int N, int K, const void* A,
                             int lda, long sA, const void* B, int ldb, long sB, void* C, int ldc,
                             long sC, int batch, float* packA, float* packB, int* status,
                             cudaStream_t st) {
  if (M <= 0 || N <= 0 || K <= 0 || batch <= 0) return cudaSuccess;
  if (prec == SP_PREC_FP32 && tc)
    return tc_schur_update(M, N, K, (const float*)A, lda, sA, (const float*)B, ldb, sB, (float*)C,
                           ldc, sC, batch, packA, packB, split, status, st);
  auto go = [&](auto t) {
    using T = decltype(t);
    if (K <= kNB) {
      gemm_sub<T>(M, N, K, (const T*)A, lda, sA, (const T*)B, ldb, sB, (T*)C, ldc, sC, batch, st);
    } else {
      const GemmSide<T> g{M, N, K, (const T*)A, lda, sA, 0, (const T*)B, ldb, sB, 0, (T*)C, ldc, sC, 0, 0, 0};
      gemm_gen<T>(g, nullptr, true, true, batch, 1, 0, st);
    }
  };
  if (prec == SP_PREC_FP32) go(0.f);
  else go(0.0);
  return cudaGetLastError();
}

int factor_outer_block(int prec, bool tc, int m, int k) {
  // the tensor-core form blocks the fronts whose trailing updates are large
  // enough to fill the GPU with 128 x 128 tiles
  if (prec == SP_PREC_FP32 && tc && m >= kTcMinFront && k > kNB) return kTcMaxK;
  return 0;
}

size_t invert_scratch_elems(int nf, int k, int ib) {
  return (size_t)nf * ((size_t)2 * k * (ib + 1) + (size_t)2 * k * (ib / 2));
}

cudaError_t factor_copy16(DevLevel& L, cudaStream_t st) {
  if (!L.front16) return cudaSuccess;
  dim3 g((unsigned)((L.m + 7) / 8), L.nf);
  f16_copy_kernel<<<g, 256, 0, st>>>((const float*)L.front, L.m, L.k, (__half*)L.front16,
                                     L.fscale16);
  return cudaGetLastError();
}

size_t grid_panel_pub_words(int nf) {
  return (size_t)nf * std::max<size_t>((size_t)2 * kGridPanelMaxG * kPubWords, kCaluFrontWords);
}

bool factor_grid_panel(int prec, int m) {
  return prec == SP_PREC_FP32 ? grid_panel_front<float>(m) : grid_panel_front<double>(m);
}

int factor_panel_width(int prec, int m) {
  return prec == SP_PREC_FP32 ? panel_width<float>(m) : panel_width<double>(m);
}

}  // namespace sp
