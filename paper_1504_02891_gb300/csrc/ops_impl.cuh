// ops_impl.cuh -- kernel templates of libgpe, instantiated per precision by
// ops_f32.cu and ops_f64.cu.  See gpe_kernels.cuh for the design summary.
#pragma once
#include <math.h>
#include <stdint.h>
#include <algorithm>
#include <type_traits>
#include "gpe_kernels.cuh"
#include "gpe_internal.h"

namespace gpe {

// ----------------------------------------------------------------- value helpers
__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 operator-(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 operator*(float s, float2 a) { return make_float2(s * a.x, s * a.y); }
__device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 operator-(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 operator-(double2 a) { return make_double2(-a.x, -a.y); }
__device__ __forceinline__ double2 operator*(double s, double2 a) { return make_double2(s * a.x, s * a.y); }

template <typename T, bool CPLX> struct VT { using V = T; };
template <typename T> struct VT<T, true> { using V = typename C2t<T>::type; };

// Re(conj(a) b), |a|^2 in the working precision
__device__ __forceinline__ float tre(float a, float b) { return a * b; }
__device__ __forceinline__ double tre(double a, double b) { return a * b; }
__device__ __forceinline__ float tre(float2 a, float2 b) { return a.x * b.x + a.y * b.y; }
__device__ __forceinline__ double tre(double2 a, double2 b) { return a.x * b.x + a.y * b.y; }
// the same products accumulated in float64
__device__ __forceinline__ double dre(float a, float b) { return (double)a * (double)b; }
__device__ __forceinline__ double dre(double a, double b) { return a * b; }
__device__ __forceinline__ double dre(float2 a, float2 b) { return (double)a.x * b.x + (double)a.y * b.y; }
__device__ __forceinline__ double dre(double2 a, double2 b) { return a.x * b.x + a.y * b.y; }

template <typename V> __device__ __forceinline__ V vzero();
template <> __device__ __forceinline__ float vzero<float>() { return 0.f; }
template <> __device__ __forceinline__ double vzero<double>() { return 0.0; }
template <> __device__ __forceinline__ float2 vzero<float2>() { return make_float2(0.f, 0.f); }
template <> __device__ __forceinline__ double2 vzero<double2>() { return make_double2(0.0, 0.0); }

__device__ __forceinline__ float2 cmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
template <typename C> __device__ __forceinline__ C mk(double re, double im);
template <> __device__ __forceinline__ float2 mk<float2>(double re, double im) { return make_float2((float)re, (float)im); }
template <> __device__ __forceinline__ double2 mk<double2>(double re, double im) { return make_double2(re, im); }

// ----------------------------------------------------------------- accumulators
// Per-thread sums of the float64 reductions.  In float32 kernels they are kept
// as unevaluated float pairs (hi + lo, Knuth two-sum), so no float64 unit is
// touched per element (GB300's float64 rate is a small fraction of float32);
// the pairs become float64 once per warp.  Float64 kernels accumulate in
// double.
struct DF {
  float hi, lo;
};
__device__ __forceinline__ void acc_zero(DF& a) { a.hi = 0.f; a.lo = 0.f; }
__device__ __forceinline__ void acc_zero(double& a) { a = 0.0; }
__device__ __forceinline__ void acc_add(DF& a, float b) {
  const float s = a.hi + b;
  const float bb = s - a.hi;
  const float err = (a.hi - (s - bb)) + (b - bb);
  a.hi = s;
  a.lo += err;
}
__device__ __forceinline__ void acc_add(double& a, double b) { a += b; }
__device__ __forceinline__ void acc_add(float& a, float b) { a += b; }   // short float partials
__device__ __forceinline__ void acc_merge(DF& a, const DF& b) {
  acc_add(a, b.hi);
  a.lo += b.lo;
}
__device__ __forceinline__ void acc_merge(double& a, double b) { a += b; }
__device__ __forceinline__ double acc_value(const DF& a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ double acc_value(double a) { return a; }
__device__ __forceinline__ DF shfl_down(const DF& a, int o) {
  DF r;
  r.hi = __shfl_down_sync(0xffffffffu, a.hi, o);
  r.lo = __shfl_down_sync(0xffffffffu, a.lo, o);
  return r;
}
__device__ __forceinline__ double shfl_down(double a, int o) { return __shfl_down_sync(0xffffffffu, a, o); }
template <typename T> struct AccT { using type = double; };
template <> struct AccT<float> { using type = DF; };

// ----------------------------------------------------------------- tile geometry
// Base offset of data line l of a tile; false if the line lies outside the grid.
// ri receives the index into the rotation coordinate table.
template <typename T>
__device__ __forceinline__ bool line_base(const PassGeom<T>& G, int inst, int tile, int l,
                                          long long& base, int& ri) {
  if (G.axis == 0) {
    long long r = (long long)tile * G.LB + l;
    if (r >= (long long)G.n1 * G.n2) return false;
    base = inst * G.M + r * G.n0;
    ri = (int)(r % G.n1);
    return true;
  }
  int o = tile / G.xt;
  int x = (tile - o * G.xt) * G.LB + l;
  if (x >= G.n0) return false;
  base = inst * G.M + (long long)o * G.ostride + x;
  ri = x;
  return true;
}

// ----------------------------------------------------------------- FFT in shared memory
// Stockham autosort, radix 4 (and one radix-2 stage when log2 F is odd),
// forward sign e^{-2 pi i j p / F}, unnormalised.  nl lines of length F stored
// contiguously in `a`; `b` is scratch of the same size.  Returns the buffer that
// holds the result.  Ends with a barrier.
template <typename C>
__device__ C* fft_lines(C* a, C* b, int F, int nl, const C* __restrict__ tw, int P = 0) {
  if (P == 0) P = F;     // row pitch (>= F; padded rows avoid bank conflicts)
  C* src = a;
  C* dst = b;
  for (int Ns = 1; Ns < F;) {
    const int R = ((F / Ns) & 3) == 0 ? 4 : 2;
    const int nb = F / R;
    const int tot = nl * nb;
    const int twstep = F / (Ns * R);
    for (int t = threadIdx.x; t < tot; t += blockDim.x) {
      const int line = t / nb;
      const int j = t - line * nb;
      const int k = j & (Ns - 1);
      const C* s = src + line * P + j;
      C* d = dst + line * P + (j - k) * R + k;
      if (R == 4) {
        C v0 = s[0], v1 = s[nb], v2 = s[2 * nb], v3 = s[3 * nb];
        if (Ns > 1) {
          const int e = k * twstep;
          v1 = cmul(v1, tw[e]);
          v2 = cmul(v2, tw[2 * e]);
          v3 = cmul(v3, tw[3 * e]);
        }
        C s02 = v0 + v2, d02 = v0 - v2, s13 = v1 + v3, d13 = v1 - v3;
        d[0] = s02 + s13;
        d[Ns].x = d02.x + d13.y;  d[Ns].y = d02.y - d13.x;      // d02 - i d13
        d[2 * Ns] = s02 - s13;
        d[3 * Ns].x = d02.x - d13.y; d[3 * Ns].y = d02.y + d13.x;  // d02 + i d13
      } else {
        C v0 = s[0], v1 = s[nb];
        if (Ns > 1) v1 = cmul(v1, tw[k * twstep]);
        d[0] = v0 + v1;
        d[Ns] = v0 - v1;
      }
    }
    __syncthreads();
    C* t = src; src = dst; dst = t;
    Ns *= R;
  }
  return src;
}

// ----------------------------------------------------------------- register-radix FFT
// Mixed-radix Stockham FFT (radix 16/8/4/2 butterflies in registers, 2-3
// shared-memory stages for F <= 1024) on nl lines of length F with row pitch P
// and padded indexing pidx(i) = i + i/16 (one spare slot every 16 elements),
// which keeps the stride-16 scatter of the first stage free of bank conflicts.
// Forward sign, unnormalised.  `post(line, m, v)` is applied to every output of
// the last stage (m = frequency index), e.g. the spectral symbol.
__device__ __forceinline__ int pidx(int i) { return i + (i >> 4); }

template <typename C> __device__ __forceinline__ C cmulc(C v, double wr, double wi) {
  using T = decltype(v.x);
  C r;
  r.x = v.x * (T)wr - v.y * (T)wi;
  r.y = v.x * (T)wi + v.y * (T)wr;
  return r;
}
template <typename C> __device__ __forceinline__ C mul_mi(C v) {   // -i v
  C r;
  r.x = v.y;
  r.y = -v.x;
  return r;
}

// Complex sum and difference of the butterflies.  PK: in float32 one packed
// two-lane instruction each (a - b as fma(b, -1, a), exactly rounded); it
// trades issue slots for FMA-pipe throughput, which pays in the latency-bound
// cluster engine and not in the register-FFT line kernels (measured).
template <bool PK, typename C> __device__ __forceinline__ C cadd(C a, C b) {
  if constexpr (PK && std::is_same<C, float2>::value) return __fadd2_rn(a, b);
  else return a + b;
}
template <bool PK, typename C> __device__ __forceinline__ C csub(C a, C b) {
  if constexpr (PK && std::is_same<C, float2>::value) return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
  else return a - b;
}

template <typename C, bool PK = true> __device__ __forceinline__ void dft2(C& a, C& b) {
  const C t = a;
  a = cadd<PK>(t, b);
  b = csub<PK>(t, b);
}
template <typename C, bool PK = true> __device__ __forceinline__ void dft4(C& v0, C& v1, C& v2, C& v3) {
  const C s02 = cadd<PK>(v0, v2), d02 = csub<PK>(v0, v2), s13 = cadd<PK>(v1, v3), d13 = csub<PK>(v1, v3);
  v0 = cadd<PK>(s02, s13);
  v2 = csub<PK>(s02, s13);
  v1 = d02 + mul_mi(d13);
  v3 = d02 - mul_mi(d13);
}
// cos(pi/8), sin(pi/8), sqrt(2)/2
#define GPE_C8 0.92387953251128675613
#define GPE_S8 0.38268343236508977173
#define GPE_R2 0.70710678118654752440
template <typename C, bool PK = true> __device__ __forceinline__ void dft8(C* v) {
  C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4<C, PK>(e0, e1, e2, e3);
  dft4<C, PK>(o0, o1, o2, o3);
  o1 = cmulc(o1, GPE_R2, -GPE_R2);
  o2 = mul_mi(o2);
  o3 = cmulc(o3, -GPE_R2, -GPE_R2);
  v[0] = cadd<PK>(e0, o0); v[4] = csub<PK>(e0, o0);
  v[1] = cadd<PK>(e1, o1); v[5] = csub<PK>(e1, o1);
  v[2] = e2 + o2; v[6] = e2 - o2;
  v[3] = cadd<PK>(e3, o3); v[7] = csub<PK>(e3, o3);
}
template <typename C> __device__ __forceinline__ void dft16(C* v) {
  C e[8], o[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    e[i] = v[2 * i];
    o[i] = v[2 * i + 1];
  }
  dft8(e);
  dft8(o);
  o[1] = cmulc(o[1], GPE_C8, -GPE_S8);
  o[2] = cmulc(o[2], GPE_R2, -GPE_R2);
  o[3] = cmulc(o[3], GPE_S8, -GPE_C8);
  o[4] = mul_mi(o[4]);
  o[5] = cmulc(o[5], -GPE_S8, -GPE_C8);
  o[6] = cmulc(o[6], -GPE_R2, -GPE_R2);
  o[7] = cmulc(o[7], -GPE_C8, -GPE_S8);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    v[i] = cadd<true>(e[i], o[i]);
    v[i + 8] = csub<true>(e[i], o[i]);
  }
}
template <typename C, int R> __device__ __forceinline__ void dft_r(C* v) {
  if constexpr (R == 2) dft2(v[0], v[1]);
  else if constexpr (R == 4) dft4(v[0], v[1], v[2], v[3]);
  else if constexpr (R == 8) dft8(v);
  else dft16(v);
}

// One Stockham stage of radix R = 2^LR.
template <typename C, int LR, typename Post>
__device__ __forceinline__ void fft_stage(const C* __restrict__ src, C* __restrict__ dst, int logF, int logNs, int nl,
                                          int P, const C* __restrict__ tw, bool last, Post& post) {
  constexpr int R = 1 << LR;
  const int lognb = logF - LR;
  const int nb = 1 << lognb;
  const int Ns = 1 << logNs;
  const int tot = nl << lognb;
  const int logtw = logF - logNs - LR;        // twiddle step F / (Ns R)
  for (int t = threadIdx.x; t < tot; t += blockDim.x) {
    const int line = t >> lognb;
    const int j = t & (nb - 1);
    const int k = j & (Ns - 1);
    const C* s = src + line * P;
    C v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = s[pidx(j + (r << lognb))];
    if (Ns > 1) {
      // twiddles w^r, w = e^{-2 pi i k / (Ns R)}, from w, w^2, w^4, w^8 of the table
      const int e = k << logtw;
      C w[R];
      w[1] = tw[e];
      if constexpr (R >= 4) {
        w[2] = tw[2 * e];
        w[3] = cmul(w[1], w[2]);
      }
      if constexpr (R >= 8) {
        w[4] = tw[4 * e];
        w[5] = cmul(w[1], w[4]);
        w[6] = cmul(w[2], w[4]);
        w[7] = cmul(w[3], w[4]);
      }
      if constexpr (R >= 16) {
        w[8] = tw[8 * e];
#pragma unroll
        for (int r = 9; r < 16; ++r) w[r] = cmul(w[r - 8], w[8]);
      }
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], w[r]);
    }
    dft_r<C, R>(v);
    C* d = dst + line * P;
    const int mb = ((j - k) << LR) + k;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int m = mb + (r << logNs);
      d[pidx(m)] = last ? post(line, m, v[r]) : v[r];
    }
  }
}

struct PostNone {
  template <typename C> __device__ __forceinline__ C operator()(int, int, C v) const { return v; }
};

// Radix schedule: ceil(logF/4) stages with the bits spread evenly (16x16 for
// 256, 8x8x8 for 512, 16x8x8 for 1024, ...).  Ends with a barrier.
template <typename C, typename Post>
__device__ C* fft_run(C* a, C* b, int logF, int nl, int P, const C* tw, Post post) {
  const int S = (logF + 3) >> 2;
  const int base = S ? logF / S : 0, extra = S ? logF % S : 0;
  C* src = a;
  C* dst = b;
  int logNs = 0;
  for (int st = 0; st < S; ++st) {
    const int lr = base + (st < extra ? 1 : 0);
    const bool last = st == S - 1;
    switch (lr) {
      case 1: fft_stage<C, 1>(src, dst, logF, logNs, nl, P, tw, last, post); break;
      case 2: fft_stage<C, 2>(src, dst, logF, logNs, nl, P, tw, last, post); break;
      case 3: fft_stage<C, 3>(src, dst, logF, logNs, nl, P, tw, last, post); break;
      default: fft_stage<C, 4>(src, dst, logF, logNs, nl, P, tw, last, post); break;
    }
    __syncthreads();
    C* t = src;
    src = dst;
    dst = t;
    logNs += lr;
  }
  return src;
}

// Asynchronous global -> shared copies (cp.async, sm_80+): the whole tile is in
// flight at once instead of one dependent load per thread and iteration.
template <typename V>
__device__ __forceinline__ void cp_async(V* dst_smem, const V* src) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(dst_smem);
  if constexpr (sizeof(V) == 16) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(src) : "memory");
  } else if constexpr (sizeof(V) == 8) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(src) : "memory");
  } else {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(src) : "memory");
  }
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// ----------------------------------------------------------------- block reductions
// Partials are NQ slots of 8 bytes per CTA: float64 in float64 kernels, float
// pairs (hi, lo) in float32 kernels, so that a float32 reduction never touches
// the float64 pipe until its final NQ values.
__device__ __forceinline__ void df_max(DF& a, const DF& b) { a.hi = fmaxf(a.hi, b.hi); }

// The sums of a warp: at offsets 16, 8, 4, 2 a lane keeps one half of its
// quantities (chosen by its lane bit) and adds its partner's copy of that half,
// so after four steps lane l holds quantity (l >> 1) & 15 summed over the 16
// lanes of its parity, and offset 1 adds the other parity: 16 merges and 32
// shuffles per lane instead of a 5-level tree per quantity (75 merges).  The
// float64 trees were a quarter of the float64 instructions of whole kernels.
__device__ __forceinline__ DF shfl_xor(const DF& a, int o) {
  DF r;
  r.hi = __shfl_xor_sync(0xffffffffu, a.hi, o);
  r.lo = __shfl_xor_sync(0xffffffffu, a.lo, o);
  return r;
}
__device__ __forceinline__ double shfl_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
template <typename A> __device__ __forceinline__ A warp_reduce_scatter(A (&v)[16]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16, H = 8; o >= 2; o >>= 1, H >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const A keep = up ? v[i + H] : v[i];
      const A send = up ? v[i] : v[i + H];
      const A w = shfl_xor(send, o);
      v[i] = keep;
      acc_merge(v[i], w);
    }
  }
  // the two parities in a fixed order (even lane's sum first)
  const A w = shfl_xor(v[0], 1);
  A r = (lane & 1) ? w : v[0];
  acc_merge(r, (lane & 1) ? v[0] : w);
  return r;
}
__device__ __forceinline__ void acc_max(DF& a, const DF& b) { a.hi = fmaxf(a.hi, b.hi); }
__device__ __forceinline__ void acc_max(double& a, double b) { a = fmax(a, b); }

// Reduce the per-thread sums acc[0..nq) over the block and write this CTA's
// partials to out[0..NQ); the other slots are 0.  Slot Q_MAX, the largest |.|
// (amax2: its square), is reduced when all NQ slots are asked for.  Threads
// 0..NQ-1 return the sums (quantity = thread).  Ends with a barrier.
template <typename A, typename M>
static __device__ A block_partial(A (&acc)[NQ], M amax2, int nq, double* out) {
  constexpr bool F32ACC = !std::is_same<A, double>::value;
  __shared__ A red[NTHREADS / 32][16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  if (nq < NQ) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      if (q >= nq) continue;
      A v = acc[q];
      for (int o = 16; o > 0; o >>= 1) acc_merge(v, shfl_down(v, o));
      if (lane == 0) red[warp][q] = v;
    }
  } else {
    A v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      if (q < NQ && q != Q_MAX) v[q] = acc[q];
      else acc_zero(v[q]);
    }
    A r = warp_reduce_scatter(v);
    const int q = (lane >> 1) & 15;
    // the root of the largest |.|^2 in the working precision (correctly
    // rounded; a float64 root costs ~0.3 us and the float64 pipe)
    A m;
    if constexpr (F32ACC) {
      float x = sqrtf((float)amax2);
      for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
      m.hi = x;
      m.lo = 0.f;
    } else {
      double x = amax2;
      for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
      m = sqrt(x);
    }
    if (q == Q_MAX) r = m;
    if ((lane & 1) == 0 && q < NQ) red[warp][q] = r;
  }
  __syncthreads();
  A v;
  acc_zero(v);
  if (threadIdx.x < NQ) {
    const int q = threadIdx.x;
    if (q < nq) {
      v = red[0][q];
      for (int w = 1; w < nw; ++w) {
        if (q == Q_MAX) acc_max(v, red[w][q]);
        else acc_merge(v, red[w][q]);
      }
    }
    reinterpret_cast<A*>(out)[q] = v;
  }
  __syncthreads();
  return v;
}

// Fold `rows` rows of partials, `stride` rows apart, in a fixed order; called by
// one whole CTA.  Thread t takes quantity t mod 16 of the rows t / 16, t / 16 +
// (threads / 16), ..., eight loads in flight; then lanes l and l + 16 and the
// warps are joined.  Threads 0..NQ-1 return the sums (quantity = thread).
template <typename A>
static __device__ A fold_rows(const double* partials, int rows, int stride, int nq) {
  __shared__ A red[NTHREADS / 32][16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5, slices = blockDim.x >> 4;
  const int q = threadIdx.x & 15;
  A x;
  acc_zero(x);
  if (q < nq) {
    const A* pp = reinterpret_cast<const A*>(partials) + q;
    const size_t rs = (size_t)stride * NQ;
    for (int i0 = threadIdx.x >> 4; i0 < rows; i0 += 8 * slices) {
      A w[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = i0 + u * slices;
        acc_zero(w[u]);
        if (i < rows) {
          if constexpr (std::is_same<A, double>::value) {
            w[u] = __ldcg(pp + i * rs);
          } else {
            const float2 f = __ldcg(reinterpret_cast<const float2*>(pp + i * rs));
            w[u].hi = f.x;
            w[u].lo = f.y;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (q == Q_MAX) acc_max(x, w[u]);
        else acc_merge(x, w[u]);
      }
    }
  }
  {
    const A w = shfl_xor(x, 16);
    if (lane < 16) {
      if (q == Q_MAX) acc_max(x, w);
      else acc_merge(x, w);
      red[warp][q] = x;
    }
  }
  __syncthreads();
  A v;
  acc_zero(v);
  if (threadIdx.x < NQ) {
    const int k = threadIdx.x;
    v = red[0][k];
    for (int w = 1; w < nw; ++w) {
      if (k == Q_MAX) acc_max(v, red[w][k]);
      else acc_merge(v, red[w][k]);
    }
  }
  return v;
}

// The sums of `tiles` consecutive CTAs' partials as float64 in res[0..NQ)
// (shared memory) and out[0..NQ) (may be null).  Ends with a barrier.
template <typename A>
static __device__ void fold_partials(const double* partials, int tiles, int stride, int nq, double* out, double* res) {
  const A v = fold_rows<A>(partials, tiles, stride, nq);
  if (threadIdx.x < NQ) {
    const double d = acc_value(v);
    if (out) out[threadIdx.x] = d;
    res[threadIdx.x] = d;
  }
  __syncthreads();
}

// Tickets of a launch of `blocks` CTAs over nb instances: one per instance and
// one per group of FOLD_GROUP CTAs.
constexpr int FOLD_GROUP = 16;
static inline size_t fold_tickets(size_t blocks, size_t nb) { return 2 * nb + blocks / FOLD_GROUP + 1; }

// Block partial; the last CTA of an instance to finish (atomic tickets) folds
// the instance's partials into results[inst][q] and returns them (in shared
// memory); the others return null.  One last CTA for the whole batch folded the
// instances one after another, about 0.5 us for each sum: 64 us of the 82 us of
// a moments launch over 128 instances.  Instances of more than FOLD_GROUP CTAs
// are folded in two steps, each group by its own last CTA: one CTA of 64
// threads took 10 us over the rows of 900 CTAs.
template <typename A, typename M>
static __device__ const double* reduce_partials(A (&acc)[NQ], M amax2, int nq, double* partials, double* results,
                                                unsigned int* ticket, int tiles) {
  __shared__ int s_last;
  __shared__ double s_res[NQ];
  const int inst = blockIdx.x / tiles, tile = blockIdx.x - inst * tiles;
  double* base = partials + (size_t)inst * tiles * NQ;
  const A own = block_partial(acc, amax2, nq, base + (size_t)tile * NQ);
  if (tiles == 1) {   // nobody to wait for
    if (threadIdx.x < NQ) results[(size_t)inst * NQ + threadIdx.x] = s_res[threadIdx.x] = acc_value(own);
    __syncthreads();
    return s_res;
  }
  // called after a barrier: thread 0's fences cover the CTA's writes and reads
  auto last_of = [&](unsigned int* t, int n) -> bool {
    if (threadIdx.x == 0) {
      __threadfence();
      s_last = atomicAdd(t, 1u) == (unsigned)n - 1u;
      if (s_last) {
        *t = 0u;
        __threadfence();
      }
    }
    __syncthreads();
    return s_last != 0;
  };
  int rows = tiles, stride = 1;
  if (tiles > FOLD_GROUP) {
    const int ngroups = (tiles + FOLD_GROUP - 1) / FOLD_GROUP, g = tile / FOLD_GROUP;
    const int n = min(FOLD_GROUP, tiles - g * FOLD_GROUP);
    double* grow = base + (size_t)g * FOLD_GROUP * NQ;
    if (!last_of(ticket + gridDim.x / tiles + inst * ngroups + g, n)) return nullptr;
    const A v = fold_rows<A>(grow, n, 1, nq);
    if (threadIdx.x < NQ) reinterpret_cast<A*>(grow)[threadIdx.x] = v;
    __syncthreads();
    rows = ngroups;
    stride = FOLD_GROUP;
  }
  if (!last_of(ticket + inst, rows)) return nullptr;
  fold_partials<A>(base, rows, stride, nq, results + (size_t)inst * NQ, s_res);
  return s_res;
}

// Grid-wide barrier for a cooperative (co-resident) launch: arrival counter
// bar[0] and generation bar[1].  Every wait is bounded: after max_polls polls
// (2^22 by default, about a second) the CTA sets *err and returns false, and
// so does every CTA that later sees *err set.
static __device__ bool grid_barrier(unsigned int* bar, int* err, long long max_polls) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    volatile unsigned int* vgen = bar + 1;
    volatile int* verr = err;
    const unsigned int gen = *vgen;
    __threadfence();
    if (atomicAdd(bar, 1u) == gridDim.x - 1) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      long long polls = 0;
      while (*vgen == gen) {
        if (*verr) { ok = 0; break; }
        if (++polls > max_polls) {
          atomicExch(err, 1);
          ok = 0;
          break;
        }
        __nanosleep(100);
      }
    }
    __threadfence();
    if (*verr) ok = 0;
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// ----------------------------------------------------------------- solver control
// The control of Algorithm 1 is one thread's serial chain of scalar
// operations once per trial; it runs in the arithmetic type R of the run.
// Float64 runs keep float64 (R = double).  Float32 runs (R = float) take their
// sums from float32 data, and use the step coefficients, theta and tau as
// float32 values, so float32 arithmetic loses nothing they can use, and on
// this hardware a float64 division or square root has a latency of hundreds
// of nanoseconds against tens for float32.  The block keeps float64 storage.

// Cayley coefficients of Theorem 3.3 for the current point and step tau, with
// the §4 renormalisation folded in as the scale s.
template <typename R, typename CT>
static __device__ __forceinline__ void set_coef(CT* c) {
  const R t = (R)c->tau, nX = (R)c->nX, XG = (R)c->XG, GG = (R)c->GG, PP = (R)c->PP;
  const R nxpp = nX * PP;                            // nX*GG - XG^2, cancellation-free
  R a, b, am1;
  if (sizeof(R) == 4 && t > R(1) && !(nxpp > R(0))) {
    // float32, A(X)X = 0 to float32 accuracy: the curve stays at X
    a = R(1);
    b = R(0);
    am1 = R(0);
  } else if (sizeof(R) == 4 && t > R(1)) {
    // float32: numerator and denominator divided by tau^2 (u = 1/tau), so
    // that steps up to the 1e20 clamp do not overflow
    const R u = R(1) / t;
    const R inv = R(1) / (u * u + nxpp);
    a = (u * u + R(2) * u * XG - nxpp) * inv;
    b = R(-2) * u * nX * inv;
    am1 = (R(2) * u * XG - R(2) * nxpp) * inv;
  } else {
    const R inv = R(1) / (R(1) + t * t * nxpp);      // one division for a, b and a - 1
    a = (R(1) + R(2) * t * XG - t * t * nxpp) * inv;
    b = R(-2) * t * nX * inv;
    am1 = (R(2) * t * XG - R(2) * t * t * nxpp) * inv;
  }
  // |Y|^2: float64 evaluates a^2 nX + 2ab XG + b^2 GG; in float32 those terms
  // cancel to rounding noise for large tau, so the identity |Y|^2 = |X|^2 of
  // Theorem 3.3 (the Cayley curve keeps the norm) is used instead
  const R ny = sizeof(R) == 4 ? nX : a * a * nX + R(2) * a * b * XG + b * b * GG;
  R s = R(1) / sqrt(ny);
  if (!c->always_renorm && fabs(ny - R(1)) <= (R)c->renorm_tol) s = R(1);
  c->a = a;
  c->b = b;
  c->s = s;
  c->am1 = am1;   // a - 1
}

// Algorithm 1 after an evaluation at the trial point: the nonmonotone test of
// Eq. NMLS-Armijo, backtracking, the reference value update (C, Q), Eq. crit1,
// and the next Barzilai-Borwein step of Eq. bb-1 (alternating tau^{k,1} on even
// k and tau^{k,2} on odd k, clamped), then the coefficients of the next trial.
// The objective value itself is kept in float64 (reported, never tested).
template <typename R, typename CT>
static __device__ __forceinline__ void alg1_control_impl(CT* c, const double* r) {
  const double obj = (c->objective == 0) ? r[Q_E2] + c->alpha * r[Q_E4] : r[Q_E2] + r[Q_WX];
  const R nY = (R)r[Q_NY], YG = (R)r[Q_YG];
  c->obj_last = obj;
  c->nfe += 1;
  if (!isfinite(obj) || !isfinite(r[Q_GG]) || !(nY > R(0))) {
    c->done = 1;
    c->status = 4;  // GPE_ENONFINITE
    return;
  }
  // Eq. NMLS-Armijo relative to the current point: with Cg = C - F(X_cur),
  // F(Y) <= C - rho1 tau res^2 reads dF <= Cg - rho1 tau res^2, dF formed
  // pointwise (no cancellation of two nearly equal objective values)
  const R dF = (R)r[Q_DF];
  const R tau = (R)c->tau, res = (R)c->res;
  bool accept = true;
  if (c->phase != 0) {
    const R thr = (R)c->Cg - (R)c->rho1 * tau * res * res;
    accept = (dF <= thr) || (c->m >= c->max_bt);
  }
  if (!accept) {
    c->tau = tau * (R)c->delta_bt;
    c->m += 1;
    c->accepted_last = 0;
    set_coef<R>(c);
    return;
  }
  const R thY = YG / nY;
  const R dth = thY - (R)(c->has_cur ? c->theta_c : c->theta_hint);
  R PPn = (R)r[Q_Q] - R(2) * dth * (R)r[Q_QY] + dth * dth * nY;
  if (PPn < R(0)) PPn = R(0);
  const R SS = (R)r[Q_SS];
  const R SW = (R)r[Q_SV] - dth * (R)r[Q_SY];
  const R WW = (R)r[Q_VV] - R(2) * dth * (R)r[Q_VY] + dth * dth * nY;
  if (c->two_slots) {
    const int oc = c->has_cur ? c->cur : 1 - c->trial;
    c->cur = c->trial;
    c->trial = oc;
    c->prev = oc;
  } else if (c->has_cur) {
    const int oc = c->cur, op = c->prev, tr = c->trial;
    c->prev = oc;
    c->cur = tr;
    c->trial = op;
  } else {
    const int tr = c->trial;
    c->cur = tr;
    c->prev = (tr + 1) % 3;
    c->trial = (tr + 2) % 3;
  }
  const R resn = nY * sqrt(PPn);
  c->F_cur = obj;
  c->theta_c = thY;
  c->nX = nY;
  c->XG = YG;
  c->GG = r[Q_GG];
  c->PP = PPn;
  c->res = resn;
  c->smax = r[Q_MAX];
  if (c->phase == 0) {
    c->Cg = 0.0;
    c->Q = 1.0;
    c->k = 0;
    c->tau = c->monotone ? c->alpha_hat : c->tau0;
    c->phase = 1;
    c->has_cur = 1;
  } else {
    if (c->monotone) {
      // Eq. Armijo1: the reference value is F(X^(k+1)) itself
      c->Cg = 0.0;
    } else {
      // C+ = (eta Q C + F(Y)) / Q+  =>  C+ - F(Y) = eta Q (Cg - dF) / Q+
      const R eta = (R)c->eta, Q = (R)c->Q;
      const R Qn = eta * Q + R(1);
      c->Cg = eta * Q * ((R)c->Cg - dF) / Qn;
      c->Q = Qn;
    }
    c->k += 1;
    c->tau_last = c->tau;
    if (c->eps0 > 0.0 && (R)r[Q_MAX] <= (R)c->eps0 * tau) { c->done = 1; c->status = 0; }   // Eq. crit1, tau > 0
    if (c->monotone) {
      c->tau = c->alpha_hat;   // Remark after Theorem 3.4: every search starts at alpha_hat
    } else {
      R tb;
      if ((c->k & 1) == 0) tb = fabs(SW) > R(0) ? SS / fabs(SW) : R(1e20);
      else tb = WW > R(0) ? fabs(SW) / WW : R(1e20);
      if (!isfinite(tb)) tb = R(1e20);
      tb = fmin(fmax(tb, R(1e-20)), R(1e20));
      c->tau = R(0.5) * tb;
    }
  }
  c->m = 0;
  c->accepted_last = 1;
  if (c->res_tol > 0.0 && resn <= (R)c->res_tol) { c->done = 1; c->status = 0; }
  if (c->res_rel > 0.0 && resn <= (R)c->res_rel * fabs(thY)) { c->done = 1; c->status = 0; }
  // precision floor: no new smallest residual (by 10%) for stall_iters steps
  if (c->phase == 1 && (c->k == 0 || resn < R(0.9) * (R)c->best_res)) {
    c->best_res = resn;
    c->k_best = c->k;
  } else if (c->stall_iters > 0 && c->k - c->k_best >= c->stall_iters) {
    // the precision floor: stopped, not converged (GPE_ENOCONV)
    c->done = 1;
    c->status = 5;
  }
  if (!c->done && c->k >= c->max_iter) { c->done = 1; c->status = 5; }
  set_coef<R>(c);
}

// The control on a register copy of the block and of the sums: the fields are
// read and written back once instead of one dependent shared- or global-memory
// access per use (the control is a single thread's serial chain).
template <typename R, typename CT>
static __device__ void alg1_control(CT* cp, const double* rp) {
  CT c = *cp;
  double r[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) r[q] = rp[q];
  alg1_control_impl<R>(&c, r);
  *cp = c;
}

// Eq. TR-ratio with both reductions in difference form, Eq. update-X and
// Eq. tau-up (gamma1, gamma2 factors), on the ratio pass's sums.
static __device__ void rn_control(RNCtl* c, const double* r) {
  const double a = c->alpha, d = c->delta;
  const double ared = r[R_AXD] + 0.5 * r[R_DAD] + a * r[R_QD];
  const double pred = r[R_GD] + 0.5 * (r[R_DAD] + 4.0 * a * (r[R_X2D2] + 2.0 * r[R_R2])) + 0.5 * d * r[R_DD];
  double rho;
  if (fabs(pred) <= 1e-15 * fmax(fabs(c->F_k), 1.0)) rho = 1.0;
  else rho = ared / pred;
  c->ared = ared;
  c->pred = pred;
  c->rho = rho;
  c->dmax = r[Q_MAX];
  c->accepted = (rho >= c->eta1) ? 1 : 0;
  double nd = d;
  if (rho > c->eta2) nd = d / c->gamma1;
  else if (rho >= c->eta1) nd = d;
  else nd = d * c->gamma2;
  c->delta = fmin(fmax(nd, c->delta_min), c->delta_max);
}

// ----------------------------------------------------------------- dependent launches
// The kernels of one operator application follow one another on a stream, each
// a few microseconds long, and a launch costs one to two.  They are launched
// with programmatic stream serialisation: a kernel may be made resident while
// the one before it drains, loads its constant tables, and waits
// (griddepcontrol.wait) for that kernel's completion and memory before it
// touches anything else.  Every CTA of every such kernel executes the wait
// before it can return, so completion is transitive along the stream.  The wait
// orders ordinary loads (ld, ld.cg, cp.async).  The read-only path is for data
// that nobody writes while the kernel is resident, and that is longer than its
// own work here: fields, accumulators and sums are never read through it, only
// the tables and potentials of a plan (ld_const).  Launches
// being captured keep plain edges: the solver's graphs of 16 iterations ran 2%
// slower with programmatic ones (64^3: 14.9 against 14.6 ms a solve).  Measured:
// 127^3 Hessian-vector float32 59 -> 50 us, 64^3 -> 128^3 transfer 32 -> 24 us,
// 512^2 complex128 Hessian-vector 36.9 -> 34.5 us.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Let the next kernel be made resident (once every CTA has got here or ended).
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
static cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = stream_capturing(st) ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// ----------------------------------------------------------------- coherent loads
// Inside a persistent launch, data written by other CTAs during the same launch
// must bypass the (non-coherent) L1: ld.global.cg.
template <int COH, typename X> __device__ __forceinline__ X ldv(const X* p) {
  static_assert(COH == 0 || COH == 1, "plain or coherent in L2");
  if constexpr (COH == 1) return __ldcg(p);
  else return *p;
}
// The read-only path: potentials and tables, written when a plan or a level is
// set up and by no kernel.
template <typename X> __device__ __forceinline__ X ld_const(const X* p) { return __ldg(p); }
template <int COH, typename X> __device__ __forceinline__ X rdc(const X& r) {
  if constexpr (COH == 1) return *(const volatile X*)&r;
  else return r;
}

// ----------------------------------------------------------------- pointwise epilogue
template <typename T, bool CPLX>
struct EpiCtx {
  using V = typename VT<T, CPLX>::V;
  V* out;
  const V* xc;
  const V* gc;
  const V* base;
  const V* gk;
  T nl, shift, lin_scale, th_c, delta, thk;
};

// The vectors an epilogue reads at a point besides x and its linear part: HESS
// psi; F X_cur, G_cur; W those and X^k; WS those and P_k; RATIO X^k, G_k.  They
// are values here, so that a kernel can load those of several points before
// the first store (the compiler has to keep a load behind a store that may
// alias it, so each point would wait for the one before).
constexpr __host__ __device__ int epi_nops(int epi) {
  return epi == EPI_HESS ? 1 : (epi == EPI_F || epi == EPI_RATIO) ? 2 : epi == EPI_W ? 3 : epi == EPI_WS ? 4 : 0;
}
template <typename V, int EPI> struct EpiOps {
  V v[epi_nops(EPI) > 0 ? epi_nops(EPI) : 1];
};
// Points whose operands are held together: at most 16 registers.
template <typename V, int EPI> constexpr __host__ __device__ int epi_batch(int nv) {
  int n = nv;
  while (n > 1 && n * epi_nops(EPI) * (int)sizeof(V) > 64) n /= 2;
  return n;
}
template <typename T, bool CPLX, int EPI, int COH>
__device__ __forceinline__ void epilogue_load(EpiOps<typename VT<T, CPLX>::V, EPI>& o, const EpiCtx<T, CPLX>& E,
                                              long long gi) {
  using V = typename VT<T, CPLX>::V;
  if constexpr (EPI == EPI_HESS) {
    o.v[0] = ldv<COH>(E.base + gi);
  } else if constexpr (EPI == EPI_RATIO) {
    o.v[0] = ldv<COH>(E.base + gi);
    o.v[1] = ldv<COH>(E.gk + gi);
  } else if constexpr (epi_nops(EPI) > 0) {
    o.v[0] = E.xc ? ldv<COH>(E.xc + gi) : vzero<V>();
    o.v[1] = E.gc ? ldv<COH>(E.gc + gi) : vzero<V>();
    if constexpr (EPI == EPI_W || EPI == EPI_WS) o.v[2] = ldv<COH>(E.base + gi);
    if constexpr (EPI == EPI_WS) o.v[3] = ldv<COH>(E.gk + gi);
  }
}

// One point: the output, handed to put, and the sums.  diff (objective passes): there is a current
// point.  A run's first evaluation has none and its control reads no difference
// sum (slots Q_SS.. and Q_MAX); in float64 they are half of the 36 operations a
// point, of which an SM sub-partition issues one warp's in 64 clocks: they were
// 37 of the 80 thousand cycles of the 256^2 real x-kernel (49 -> 44.5 us without
// the differences).
template <typename T, bool CPLX, int EPI, typename A, typename Put>
__device__ __forceinline__ void epilogue_put(const EpiCtx<T, CPLX>& E, typename VT<T, CPLX>::V x,
                                             typename VT<T, CPLX>::V lin,
                                             const EpiOps<typename VT<T, CPLX>::V, EPI>& o, A (&acc)[NQ], T& amax,
                                             bool diff, Put&& put) {
  using V = typename VT<T, CPLX>::V;
  if constexpr (EPI == EPI_GRAD) {
    const T x2 = tre(x, x);
    if (E.out) put(lin + (E.nl * x2) * x);
    acc_add(acc[0], tre(x, lin));
    acc_add(acc[1], x2 * x2);
    acc_add(acc[2], x2);
  } else if constexpr (EPI == EPI_HESS) {
    const V p = o.v[0];
    const T p2 = tre(p, p);
    const T R = tre(p, x);
    // gathered by x and p: 12 operations a complex point instead of 18 (float64 issues 2 a clock)
    put(lin + (E.nl * p2 + E.shift) * x + (T(2) * E.nl * R) * p);
  } else if constexpr (EPI == EPI_RATIO) {
    const V d = x;
    const V xk = o.v[0], gk = o.v[1];
    const T x2 = tre(xk, xk);
    const V ax = gk - (T(4) * E.nl * x2) * xk;
    const V z = xk + d;
    const T R = tre(xk, d), d2 = tre(d, d);
    acc_add(acc[R_AXD], tre(ax, d));
    acc_add(acc[R_DAD], T(2) * tre(d, lin));
    acc_add(acc[R_QD], (T(2) * R + d2) * (tre(z, z) + x2));
    acc_add(acc[R_X2D2], x2 * d2);
    acc_add(acc[R_R2], R * R);
    acc_add(acc[R_DD], d2);
    acc_add(acc[R_GD], tre(gk, d));
    amax = fmax(amax, d2);
  } else if constexpr (EPI == EPI_F || EPI == EPI_W) {
    const V y = x;
    V g;
    if constexpr (EPI == EPI_F) {
      g = E.lin_scale * lin + (T(4) * E.nl * tre(y, y)) * y;
    } else {
      const V xk = o.v[2];
      const V dd = y - xk;
      const T x2 = tre(xk, xk);
      const T R = tre(xk, dd);
      g = E.lin_scale * lin + (T(4) * E.nl * x2) * y + (T(8) * E.nl * R) * xk + E.delta * dd;
      const T d2 = tre(dd, dd);
      acc_add(acc[Q_WX], T(4) * E.nl * x2 * R + T(2) * E.nl * (x2 * d2 + T(2) * R * R) + T(0.5) * E.delta * d2);
    }
    put(g);
    const T y2 = tre(y, y);
    acc_add(acc[Q_E2], tre(y, lin));
    acc_add(acc[Q_E4], y2 * y2);
    acc_add(acc[Q_NY], y2);
    acc_add(acc[Q_YG], tre(y, g));
    acc_add(acc[Q_GG], tre(g, g));
    const V q = g - E.th_c * y;
    acc_add(acc[Q_Q], tre(q, q));
    acc_add(acc[Q_QY], tre(q, y));
    if (!diff) return;
    const V xc = o.v[0], gc = o.v[1];
    const V s = y - xc;
    const V v = (g - gc) - E.th_c * s;
    const T s2 = tre(s, s);
    acc_add(acc[Q_SS], s2);
    acc_add(acc[Q_SV], tre(s, v));
    acc_add(acc[Q_VV], tre(v, v));
    acc_add(acc[Q_VY], tre(v, y));
    acc_add(acc[Q_SY], tre(s, y));
    // objective(y) - objective(x_c) by the trapezoid rule on the theta-shifted
    // gradients (q + q_c = 2q - v); exact for the quadratic part, the quartic
    // term of F adds -alpha Re<s, y + x_c> |s|^2.  The dropped real multiple
    // of y + x_c changes the objective only off the unit sphere.
    T df = tre(s, q) - T(0.5) * tre(s, v);
    if (EPI == EPI_F) df -= E.nl * tre(s, y + xc) * s2;
    acc_add(acc[Q_DF], df);
    amax = fmax(amax, s2);
  } else if constexpr (EPI == EPI_WS) {
    // difference form (the unknown y is D = X - X^k): G^ = P_k + H_k D +
    // (delta - theta_k) D, objective Re<P_k, D> + theta_k Re<X^k, D> +
    // 1/2 Re<D, H_k D> + delta/2 |D|^2, moments of X = X^k + D
    const V y = x;
    const V xc = o.v[0], gc = o.v[1], xk = o.v[2], pk = o.v[3];
    const T x2 = tre(xk, xk), R = tre(xk, y);
    const V hD = E.lin_scale * lin + (T(4) * E.nl) * (x2 * y + (T(2) * R) * xk);
    const V gh = pk + hD + (E.delta - E.thk) * y;
    put(gh);
    const V X = xk + y;
    acc_add(acc[Q_WX], tre(pk, y) + E.thk * R + T(0.5) * tre(y, hD) + T(0.5) * E.delta * tre(y, y));
    acc_add(acc[Q_NY], tre(X, X));
    acc_add(acc[Q_YG], tre(X, gh));
    acc_add(acc[Q_GG], tre(gh, gh));
    const V q = gh - E.th_c * X;
    acc_add(acc[Q_Q], tre(q, q));
    acc_add(acc[Q_QY], tre(q, X));
    const V s = y - xc;
    const V v = (gh - gc) - E.th_c * s;
    const T s2 = tre(s, s);
    acc_add(acc[Q_SS], s2);
    acc_add(acc[Q_SV], tre(s, v));
    acc_add(acc[Q_VV], tre(v, v));
    acc_add(acc[Q_VY], tre(v, X));
    acc_add(acc[Q_SY], tre(s, X));
    acc_add(acc[Q_DF], tre(s, q) - T(0.5) * tre(s, v));   // the model is quadratic: trapezoid exact
    amax = fmax(amax, s2);
  }
}
// The output stored at once.
template <typename T, bool CPLX, int EPI, typename A>
__device__ __forceinline__ void epilogue_apply(const EpiCtx<T, CPLX>& E, long long gi, typename VT<T, CPLX>::V x,
                                               typename VT<T, CPLX>::V lin,
                                               const EpiOps<typename VT<T, CPLX>::V, EPI>& o, A (&acc)[NQ], T& amax,
                                               bool diff) {
  epilogue_put<T, CPLX, EPI>(E, x, lin, o, acc, amax, diff, [&](typename VT<T, CPLX>::V g) { E.out[gi] = g; });
}

// The first evaluation of a float64 run leaves out the difference sums.
template <typename T, bool CPLX> __device__ __forceinline__ bool epilogue_diff(const EpiCtx<T, CPLX>& E) {
  return sizeof(T) == 4 || E.xc != nullptr;
}
template <typename T, bool CPLX, int EPI, int COH = 0, typename A>
__device__ __forceinline__ void epilogue_point(const EpiCtx<T, CPLX>& E, long long gi, typename VT<T, CPLX>::V x,
                                               typename VT<T, CPLX>::V lin, A (&acc)[NQ], T& amax) {
  EpiOps<typename VT<T, CPLX>::V, EPI> o;
  epilogue_load<T, CPLX, EPI, COH>(o, E, gi);
  epilogue_apply<T, CPLX, EPI>(E, gi, x, lin, o, acc, amax, epilogue_diff(E));
}

template <typename T, bool CPLX, int EPI, int COH = 0>
__device__ __forceinline__ void make_ctx(EpiCtx<T, CPLX>& E, const PassData<T>& D) {
  using V = typename VT<T, CPLX>::V;
  E.out = (V*)D.out;
  E.xc = nullptr;
  E.gc = nullptr;
  E.base = (const V*)D.base;
  E.gk = (const V*)D.gk;
  E.nl = (T)D.nl;
  E.shift = (T)D.shift;
  E.lin_scale = (T)D.lin_scale;
  E.th_c = T(0);
  E.delta = T(0);
  if (D.ctl) {
    const Alg1Ctl* c = D.ctl;
    E.nl = (T)rdc<COH>(c->alpha);
    E.delta = (T)rdc<COH>(c->delta);
    if (D.use_slots) {
      E.out = (V*)D.gs[rdc<COH>(c->trial)];
      if (rdc<COH>(c->has_cur)) {
        E.xc = (const V*)D.xs[rdc<COH>(c->cur)];
        E.gc = (const V*)D.gs[rdc<COH>(c->cur)];
        E.th_c = (T)rdc<COH>(c->theta_c);
      } else {
        E.th_c = (T)rdc<COH>(c->theta_hint);
      }
    }
  }
  E.thk = D.ctl ? (T)rdc<COH>(D.ctl->theta_ref) : T(0);
  if (D.rn) E.nl = (T)D.rn->alpha;
}

template <typename T>
__device__ __forceinline__ void run_control(const PassData<T>& D, const double* r) {
  if (threadIdx.x == 0 && r) {
    if (D.control == 1) alg1_control<T>(D.ctl, r);
    else if (D.control == 2) rn_control(D.rn, r);
  }
}

// ----------------------------------------------------------------- the axis pass
// Visit the data elements (line l, position j, global offset) of this CTA's
// tile with a coalesced thread mapping and no integer division: axis-0 lines
// are contiguous (tpl threads per line); strided lines are read as LB
// consecutive x positions per row.
template <typename T, typename Fn>
__device__ __forceinline__ void visit_tile(const PassGeom<T>& G, const long long* s_off, Fn&& fn) {
  const int nt = blockDim.x, tid = threadIdx.x;
  if (G.axis == 0) {
    const int lps = nt >> G.ltpl;
    for (int l = tid >> G.ltpl; l < G.LB; l += lps) {
      const long long off = s_off[l];
      if (off < 0) continue;
      for (int j = tid & (G.tpl - 1); j < G.len; j += G.tpl) fn(l, j, off + j);
    }
  } else {
    const int nval = G.LB * G.len;
    for (int f = tid; f < nval; f += nt) {
      const int l = f & (G.LB - 1);
      const int j = f >> G.logLB;
      const long long off = s_off[l];
      if (off < 0) continue;
      fn(l, j, off + (long long)j * G.stride);
    }
  }
}

// One tile of one axis pass: load (asynchronous copies, or L2-coherent loads
// inside a persistent launch), forward FFT with the fused symbol, inverse FFT,
// epilogue into acc/amax.  blk = instance * tiles + tile.  Ends with a barrier.
template <typename T, bool CPLX, int EPI, bool COH, typename A>
__device__ __forceinline__ void pass_tile(const PassGeom<T>& G, const PassData<T>& D, int blk,
                                          unsigned char* smem_raw, long long* s_off, T* s_rc, A (&acc)[NQ],
                                          T& amax,
                                          const typename C2t<T>::type* tw_pre = nullptr) {
  using C = typename C2t<T>::type;
  using V = typename VT<T, CPLX>::V;
  const int F = G.F, Pt = G.P;
  const int nt = blockDim.x, tid = threadIdx.x;
  const int inst = blk / G.tiles;
  const int tile = blk - inst * G.tiles;

  // operands: src0 (input, or X_cur for the Cayley step), src1 (x_sub or G_cur), acc_in
  const V* xin = (const V*)D.x;
  V* yst = nullptr;
  const V* src1 = (const V*)D.xsub;
  T sa = 0, sb = 0;
  if (D.use_slots) {
    const Alg1Ctl* c = D.ctl;
    const int trial = rdc<COH>(c->trial);
    xin = (const V*)D.xs[trial];
    if (D.step_on_load) {
      const int cur = rdc<COH>(c->cur);
      yst = (V*)D.xs[trial];
      xin = (const V*)D.xs[cur];
      src1 = (const V*)D.gs[cur];
      const double cs = rdc<COH>(c->s);
      sa = (T)(cs * rdc<COH>(c->a));
      sb = (T)(cs * rdc<COH>(c->b));
    }
  }
  const V* accin = (const V*)D.acc_in;
  const int tile_n = G.LB * G.len;
  C* tw_s = reinterpret_cast<C*>(smem_raw);
  C* buf0 = tw_s + F;
  C* buf1 = buf0 + G.LC * Pt;
  V* st0 = reinterpret_cast<V*>(buf1 + G.LC * Pt);
  V* st1 = st0 + tile_n;
  V* st2 = st1 + (src1 ? tile_n : 0);
  // potential of the tile (final passes only), staged with the other operands
  T* stv = reinterpret_cast<T*>(st2 + (accin ? tile_n : 0));
  const bool want_v = EPI != EPI_ACC;
  const long long vbase = (long long)inst * G.M;

  for (int l = tid; l < G.LB; l += nt) {
    long long b;
    int ri;
    const bool ok = line_base(G, inst, tile, l, b, ri);
    s_off[l] = ok ? b : -1;
    if (G.rcoord) s_rc[l] = G.rcoord[ok ? ri : 0];
  }
  // twiddle table (read-only): preloaded by the caller, or an asynchronous
  // copy, or plain loads when the tile loads below are not asynchronous
  if (!tw_pre) {
    for (int i = tid; i < F; i += nt) {
      if constexpr (COH) tw_s[i] = G.tw[i];
      else cp_async(tw_s + i, G.tw + i);
    }
  }
  const C* twx = tw_pre ? tw_pre : tw_s;
  __syncthreads();
  // the whole tile (and the operands the epilogue needs) in flight at once
  visit_tile(G, s_off, [&](int l, int j, long long gi) {
    const int q = G.axis == 0 ? l * G.len + j : j * G.LB + l;
    if constexpr (COH) {
      st0[q] = __ldcg(xin + gi);
      if (src1) st1[q] = __ldcg(src1 + gi);
      if (accin) st2[q] = __ldcg(accin + gi);
      if (want_v) stv[q] = D.V[gi - vbase];
    } else {
      cp_async(st0 + q, xin + gi);
      if (src1) cp_async(st1 + q, src1 + gi);
      if (accin) cp_async(st2 + q, accin + gi);
      if (want_v) cp_async(stv + q, D.V + (gi - vbase));
    }
  });
  for (int i = tid; i < G.LC * Pt; i += nt) buf0[i] = mk<C>(0.0, 0.0);
  if constexpr (!COH) cp_async_wait_all();
  __syncthreads();

  visit_tile(G, s_off, [&](int l, int j, long long gi) {
    const int q = G.axis == 0 ? l * G.len + j : j * G.LB + l;
    V v = st0[q];
    if (src1) {
      v = yst ? sa * v + sb * st1[q] : v - st1[q];
      st0[q] = v;
      if (yst) yst[gi] = v;
    }
    const int m = G.odd_ext ? j + 1 : j;
    if constexpr (CPLX) {
      C* row = buf0 + l * Pt;
      row[pidx(m)] = v;
      if (G.odd_ext) row[pidx(F - m)] = -v;
    } else {
      T* row = reinterpret_cast<T*>(buf0 + (l >> 1) * Pt);
      const int comp = l & 1;
      row[2 * pidx(m) + comp] = v;
      if (G.odd_ext) row[2 * pidx(F - m) + comp] = -v;
    }
  });
  __syncthreads();

  // forward FFT with the line symbol (and the conjugation that turns the
  // next forward FFT into the inverse) fused into its last stage
  const T c2 = G.c2, c1 = G.c1, dlam = G.dlam;
  const bool rot = G.rcoord != nullptr;
  auto symbol = [&](int line, int m, C v) -> C {
    const T lm = dlam * (T)(m < (F >> 1) ? m : m - F);
    T sym = c2 * lm * lm;
    if (rot) sym += c1 * s_rc[line] * lm;
    C r;
    r.x = sym * v.x;
    r.y = -sym * v.y;
    return r;
  };
  C* r = fft_run<C>(buf0, buf1, G.logF, G.LC, Pt, twx, symbol);
  C* o = fft_run<C>(r, r == buf0 ? buf1 : buf0, G.logF, G.LC, Pt, twx, PostNone());

  EpiCtx<T, CPLX> E;
  if (EPI != EPI_ACC) make_ctx<T, CPLX, EPI, COH>(E, D);
  const long long ibase = inst * G.M;
  visit_tile(G, s_off, [&](int l, int j, long long gi) {
    const int q = G.axis == 0 ? l * G.len + j : j * G.LB + l;
    const int m = G.odd_ext ? j + 1 : j;
    V kin;
    if constexpr (CPLX) {
      const C ov = o[l * Pt + pidx(m)];
      kin.x = ov.x;
      kin.y = -ov.y;
    } else {
      const C ov = o[(l >> 1) * Pt + pidx(m)];
      kin = (l & 1) ? -ov.y : ov.x;
    }
    if (accin) kin = kin + st2[q];
    if (EPI == EPI_ACC) {
      ((V*)D.out)[gi] = kin;
      return;
    }
    const V x = st0[q];
    const V lin = kin + stv[q] * x;
    epilogue_point<T, CPLX, EPI, COH>(E, gi, x, lin, acc, amax);
  });
  __syncthreads();
}

template <typename T, bool CPLX, int EPI>
__global__ void __launch_bounds__(NTHREADS) k_pass(PassGeom<T> G, PassData<T> D) {
  pdl_next();
  pdl_wait();
  if (D.ctl && D.ctl->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ long long s_off[MAXLB];
  __shared__ T s_rc[MAXLB];
  using A = typename AccT<T>::type;
  A acc[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) acc_zero(acc[q]);
  T amax = T(0);
  pass_tile<T, CPLX, EPI, false>(G, D, blockIdx.x, smem_raw, s_off, s_rc, acc, amax);
  if (EPI == EPI_ACC || EPI == EPI_HESS || D.nq == 0) return;
  run_control<T>(D, reduce_partials(acc, amax, D.nq, D.partials, D.results, D.ticket, G.tiles));
}

// One launch runs a whole Algorithm 1 run (until the control block says done).
// Every iteration executes the axis passes over all tiles (CTAs loop over
// tiles) separated by bounded grid barriers; then EVERY CTA folds the last
// pass's tile partials in the same fixed order and runs the step-size control
// on its own shared-memory copy of the control block, so all CTAs hold
// bit-identical state without a third barrier.  CTA 0 writes the state back.
// The slot pointers and the twiddle tables stay in shared memory for the whole
// launch.  Must be launched cooperatively (all CTAs co-resident).
template <typename T, bool CPLX, int EPI>
__global__ void __launch_bounds__(NTHREADS) k_alg1_persist(PersistArgs<T> P) {
  using C = typename C2t<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ long long s_off[MAXLB];
  __shared__ T s_rc[MAXLB];
  __shared__ Alg1Ctl s_ctl;
  __shared__ void* s_xs[3];
  __shared__ void* s_gs[3];
  __shared__ double s_res[NQ];
  using A = typename AccT<T>::type;
  // twiddle tables of all axes at the front of dynamic shared memory
  C* s_tw[3] = {nullptr, nullptr, nullptr};
  {
    C* tp = reinterpret_cast<C*>(smem_raw);
    for (int a = 0; a < P.dim; ++a) {
      s_tw[a] = tp;
      for (int i = threadIdx.x; i < P.G[a].F; i += blockDim.x) tp[i] = P.G[a].tw[i];
      tp += P.G[a].F;
    }
  }
  unsigned char* work = smem_raw + P.tw_bytes;
  if (threadIdx.x == 0) {
    s_ctl = *P.D.ctl;
    for (int i = 0; i < 3; ++i) {
      s_xs[i] = P.D.xs[i];
      s_gs[i] = P.D.gs[i];
    }
  }
  __syncthreads();
  PassData<T> D0 = P.D;
  D0.ctl = &s_ctl;
  D0.xs = s_xs;
  D0.gs = s_gs;
  auto stamp = [&](int loop, int k) {
    if (P.dbg && blockIdx.x == 0 && threadIdx.x == 0 && loop < P.dbg_n) {
      unsigned long long t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      P.dbg[loop * 4 + k] = t;
    }
  };
  auto writeback = [&]() {
    if (blockIdx.x == 0 && threadIdx.x == 0) *P.D.ctl = s_ctl;
  };
  for (int loop = 0; loop < P.max_loops; ++loop) {
    if (s_ctl.done) {
      writeback();
      return;
    }
    stamp(loop, 0);
    for (int a = 0; a < P.dim; ++a) {
      const bool last = a == P.dim - 1;
      PassData<T> Da = D0;
      Da.step_on_load = a == 0 ? 1 : 0;
      Da.acc_in = a > 0 ? P.acc : nullptr;
      if (!last) {
        Da.out = P.acc;
        Da.nq = 0;
      }
      for (int blk = blockIdx.x; blk < P.blocks[a]; blk += gridDim.x) {
        A acc[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) acc_zero(acc[q]);
        T amax = T(0);
        if (!last) {
          pass_tile<T, CPLX, EPI_ACC, true>(P.G[a], Da, blk, work, s_off, s_rc, acc, amax, s_tw[a]);
        } else {
          pass_tile<T, CPLX, EPI, true>(P.G[a], Da, blk, work, s_off, s_rc, acc, amax, s_tw[a]);
          block_partial(acc, amax, NQ, P.D.partials + (size_t)blk * NQ);
        }
      }
      if (!grid_barrier(P.bar, P.err, P.max_polls)) {
        writeback();
        return;
      }
      stamp(loop, 1 + (a < 1 ? a : 1));
    }
    fold_partials<A>(P.D.partials, P.blocks[P.dim - 1], 1, NQ, nullptr, s_res);
    if (threadIdx.x == 0) alg1_control<T>(&s_ctl, s_res);
    __syncthreads();
    stamp(loop, 3);
  }
  writeback();
}

// ----------------------------------------------------------------- finite differences
// H_lin of §2.1 per axis (3/5/7-point, zero Dirichlet values outside) with the
// central-difference rotation term, then the same epilogue as the spectral pass.
// Float64 is bound by the float64 pipe (2 operations a clock and SM): each axis
// is one addition and two multiply-adds, (x - (x- + x+)/2) / h^2, and the CTAs
// are few (two per SM) because a warp's reduction costs as much as two of its
// points.  The difference is taken before it is scaled: its rounding is that of
// the neighbours' sum alone.  With one diagonal (V + sum 1/h^2) x for all axes
// the kernel was two operations a point and 4 us shorter (149 x 100 x 76: 71.2
// against 76 us), but its error 2 to 2.5 times as large on smooth states of
// two and three dimensions (against extended precision; scaling each x and
// neighbours' sum by itself lies between).
template <typename T, bool CPLX, int EPI>
__global__ void __launch_bounds__(NTHREADS) k_fd(FDGeom G, const T* __restrict__ rx, const T* __restrict__ ry,
                                                PassData<T> D) {
  using V = typename VT<T, CPLX>::V;
  pdl_next();
  pdl_wait();
  if (D.ctl && D.ctl->done) return;
  const int inst = blockIdx.x / G.tiles;
  const int tb = blockIdx.x - inst * G.tiles;
  const V* xin = (const V*)D.x;
  if (D.use_slots) xin = (const V*)D.xs[D.ctl->trial];
  const V* xsub = (const V*)D.xsub;
  EpiCtx<T, CPLX> E;
  make_ctx<T, CPLX, EPI>(E, D);
  using A = typename AccT<T>::type;
  A acc[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) acc_zero(acc[q]);
  T amax = T(0);
  const long long base = inst * G.M;
  xin += base;
  if (xsub) xsub += base;
  const T a0 = (T)G.ih2[0], a1 = (T)G.ih2[1], a2 = (T)G.ih2[2];
  constexpr bool F64 = sizeof(T) == 8;
  const unsigned int n0 = G.n0, n1 = G.n1, n2 = G.n2, s2 = n0 * n1, M = (unsigned int)G.M;
  const unsigned int step = (unsigned int)G.tiles * blockDim.x;
  for (unsigned int li = (unsigned int)tb * blockDim.x + threadIdx.x; li < M; li += step) {
    const unsigned int row = li / n0, i0 = li - row * n0;
    const unsigned int i2 = row / n1, i1 = row - i2 * n1;
    auto ld = [&](unsigned int k) -> V {
      V v = xin[k];
      if (xsub) v = v - xsub[k];
      return v;
    };
    const V x = ld(li);
    V xm = i0 > 0 ? ld(li - 1) : vzero<V>();
    V xp = i0 < n0 - 1 ? ld(li + 1) : vzero<V>();
    V dx = vzero<V>(), dy = vzero<V>(), lin;
    if constexpr (F64) {
      lin = a0 * (x + T(-0.5) * (xm + xp));
      if constexpr (CPLX) dx = xp - xm;
      if (G.dim >= 2) {
        V ym = i1 > 0 ? ld(li - n0) : vzero<V>();
        V yp = i1 < n1 - 1 ? ld(li + n0) : vzero<V>();
        lin = lin + a1 * (x + T(-0.5) * (ym + yp));
        if constexpr (CPLX) dy = yp - ym;
      }
      if (G.dim >= 3) {
        V zm = i2 > 0 ? ld(li - s2) : vzero<V>();
        V zp = i2 < n2 - 1 ? ld(li + s2) : vzero<V>();
        lin = lin + a2 * (x + T(-0.5) * (zm + zp));
      }
    } else {
      lin = (a0) * x - (T(0.5) * a0) * (xm + xp);
      dx = xp - xm;
      if (G.dim >= 2) {
        V ym = i1 > 0 ? ld(li - n0) : vzero<V>();
        V yp = i1 < n1 - 1 ? ld(li + n0) : vzero<V>();
        lin = lin + (a1) * x - (T(0.5) * a1) * (ym + yp);
        dy = yp - ym;
      }
      if (G.dim >= 3) {
        V zm = i2 > 0 ? ld(li - s2) : vzero<V>();
        V zp = i2 < n2 - 1 ? ld(li + s2) : vzero<V>();
        lin = lin + (a2) * x - (T(0.5) * a2) * (zm + zp);
      }
    }
    if constexpr (CPLX) {
      if (G.omega != 0.0) {
        // -Omega L_z psi = i Omega (x d_y psi - y d_x psi)
        const T cx = (T)(G.omega * G.ih2c[0]), cy = (T)(G.omega * G.ih2c[1]);
        const T xv = rx[i0], yv = ry[i1];
        const V w = (xv * cy) * dy - (yv * cx) * dx;
        V iw;
        iw.x = -w.y;
        iw.y = w.x;
        lin = lin + iw;
      }
    }
    lin = lin + D.V[li] * x;
    epilogue_point<T, CPLX, EPI>(E, base + li, x, lin, acc, amax);
  }
  if (EPI == EPI_HESS || D.nq == 0) return;
  run_control<T>(D, reduce_partials(acc, amax, D.nq, D.partials, D.results, D.ticket, G.tiles));
}

// ----------------------------------------------------------------- elementwise kernels
// Cayley step of Theorem 3.3 into the trial slot (FD path; the spectral path
// forms it while loading the first pass).
template <typename T, bool CPLX>
__global__ void k_step(void* const* xs, void* const* gs, const Alg1Ctl* c, long long n, const void* xkv) {
  using V = typename VT<T, CPLX>::V;
  pdl_next();
  pdl_wait();
  if (c->done) return;
  const V* X = (const V*)xs[c->cur];
  const V* Gv = (const V*)gs[c->cur];
  V* Y = (V*)xs[c->trial];
  const T a = (T)(c->s * c->a), b = (T)(c->s * c->b);
  if (xkv) {
    // difference form: D+ = (a - 1) X^k + a D + b G^ (no renormalisation)
    const V* xk = (const V*)xkv;
    const T am1 = (T)c->am1, a1 = (T)c->a, b1 = (T)c->b;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
      Y[i] = am1 * xk[i] + a1 * X[i] + b1 * Gv[i];
    return;
  }
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    Y[i] = a * X[i] + b * Gv[i];
}

// What the last CTA of an instance makes of its moments: nothing, the Cayley
// coefficients of gpe_feasible_step (grid units in, unified units inside:
// X = sqrt(h) psi, G = 2 sqrt(h) hpsi), or the scale to unit discrete norm.
struct MomentCoef {
  int mode;        // 0: none, 1: step, 2: norm
  double h, tau;
  double* coef;    // [nbatch][2] (step) or [nbatch] (norm)
};
static __device__ void moment_coef(const MomentCoef& mc, int b, const double* r) {
  if (mc.mode == 1) {
    const double h = mc.h;
    const double nX = h * r[0], XG = 2.0 * h * r[1], GG = 4.0 * h * r[2];
    double PP = GG - XG * XG / nX;
    if (PP < 0.0) PP = 0.0;
    const double t = mc.tau, nxpp = nX * PP, den = 1.0 + t * t * nxpp;
    const double a = (1.0 + 2.0 * t * XG - t * t * nxpp) / den;
    const double bb = -2.0 * t * nX / den;
    const double ny = a * a * nX + 2.0 * a * bb * XG + bb * bb * GG;
    const double s = 1.0 / sqrt(ny);
    // psi_out = (s a X + s b G) / sqrt(h) = s a psi + 2 s b hpsi
    mc.coef[(size_t)b * 2 + 0] = s * a;
    mc.coef[(size_t)b * 2 + 1] = 2.0 * s * bb;
  } else if (mc.mode == 2) {
    mc.coef[b] = 1.0 / sqrt(mc.h * r[0]);
  }
}

// Re(conj(a) b) of the moments with a fixed rounding, whatever the compiler
// would contract: the step's float32 coefficients depend on it.
__device__ __forceinline__ float mre(float a, float b) { return a * b; }
__device__ __forceinline__ double mre(double a, double b) { return a * b; }
__device__ __forceinline__ float mre(float2 a, float2 b) { return __fmaf_rn(a.x, b.x, __fmul_rn(a.y, b.y)); }
__device__ __forceinline__ double mre(double2 a, double2 b) { return a.x * b.x + a.y * b.y; }

// Several values of a field as one 16-byte access (field arrays that start on
// 16 bytes for every instance), or one value.
template <typename V, int W> struct alignas(sizeof(V) * W) Pack {
  V v[W];
};

// Per-instance sums |x|^2, Re conj(x) g, |g|^2 (g may be null), W values per
// access.  A few CTAs per SM stride over their instance: with one value per
// thread the block reductions cost several times the reading.  128 x 128^2
// complex64: 82 us with one value per thread and one fold for the batch.
template <typename T, bool CPLX, int W>
__global__ void __launch_bounds__(NTHREADS) k_moments(const void* xv, const void* gv, long long M, int tiles,
                                                      double* partials, double* results, unsigned int* ticket,
                                                      MomentCoef mc) {
  using V = typename VT<T, CPLX>::V;
  using P = Pack<V, W>;
  pdl_next();
  pdl_wait();
  const int inst = blockIdx.x / tiles;
  const int tb = blockIdx.x - inst * tiles;
  const P* x = reinterpret_cast<const P*>((const V*)xv + inst * M);
  const P* g = gv ? reinterpret_cast<const P*>((const V*)gv + inst * M) : nullptr;
  using A = typename AccT<T>::type;
  A acc[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) acc_zero(acc[q]);
  const long long n = M / W;
#pragma unroll 4
  for (long long i = (long long)tb * blockDim.x + threadIdx.x; i < n; i += (long long)tiles * blockDim.x) {
    const P xi = x[i];
    P gi;
    if (g) gi = g[i];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      acc_add(acc[0], mre(xi.v[w], xi.v[w]));
      if (g) {
        acc_add(acc[1], mre(xi.v[w], gi.v[w]));
        acc_add(acc[2], mre(gi.v[w], gi.v[w]));
      }
    }
  }
  const double* r = reduce_partials(acc, T(0), 3, partials, results, ticket, tiles);
  if (r && threadIdx.x == 0) moment_coef(mc, inst, r);
}

// s a and s a + c with one rounding per operation whatever the compiler would
// contract: the float32 energy of a step depends on them in its 8th digit.
__device__ __forceinline__ float scaled(float s, float a) { return __fmul_rn(s, a); }
__device__ __forceinline__ double scaled(double s, double a) { return __dmul_rn(s, a); }
__device__ __forceinline__ float fused_add(float s, float a, float c) { return __fmaf_rn(s, a, c); }
__device__ __forceinline__ double fused_add(double s, double a, double c) { return __fma_rn(s, a, c); }
template <typename T, typename C> __device__ __forceinline__ C scaled(T s, C a) {
  a.x = scaled(s, a.x);
  a.y = scaled(s, a.y);
  return a;
}
template <typename T, typename C> __device__ __forceinline__ C fused_add(T s, C a, C c) {
  c.x = fused_add(s, a.x, c.x);
  c.y = fused_add(s, a.y, c.y);
  return c;
}

// out_b = ca[b] * x_b + cb[b] * g_b  (g may be null), W values per access; the
// CTAs of row blockIdx.y take the instances y, y + gridDim.y, ...
template <typename T, bool CPLX, int W>
__global__ void __launch_bounds__(NTHREADS) k_axpby(const void* xv, const void* gv, const double* coef,
                                                    int stride_coef, long long M, int nbatch, void* outv) {
  using V = typename VT<T, CPLX>::V;
  using P = Pack<V, W>;
  const long long n = M / W;
  pdl_next();
  pdl_wait();
  for (int b = blockIdx.y; b < nbatch; b += gridDim.y) {
    const P* x = reinterpret_cast<const P*>((const V*)xv + b * M);
    const P* g = gv ? reinterpret_cast<const P*>((const V*)gv + b * M) : nullptr;
    P* out = reinterpret_cast<P*>((V*)outv + b * M);
    const T ca = (T)coef[(size_t)b * stride_coef];
    const T cb = g ? (T)coef[(size_t)b * stride_coef + 1] : T(0);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
      const P xi = x[i];
      P r, gi;
      if (g) gi = g[i];
#pragma unroll
      for (int w = 0; w < W; ++w) {
        r.v[w] = g ? fused_add(ca, xi.v[w], scaled(cb, gi.v[w])) : scaled(ca, xi.v[w]);
      }
      out[i] = r;
    }
  }
}

// Values per 16-byte access, 1 if an instance does not start on 16 bytes.
static inline int pack_width(size_t vsz, long long M, const void* a, const void* b, const void* c) {
  const int w = (int)(16 / vsz);
  const uintptr_t bits = (uintptr_t)a | (uintptr_t)b | (uintptr_t)c;
  return (w > 1 && M % w == 0 && (bits & 15) == 0) ? w : 1;
}
template <typename T, bool CPLX>
static void run_moments(const void* x, const void* g, long long M, int nbatch, int tiles, double* partials,
                        double* results, unsigned int* ticket, const MomentCoef& mc, cudaStream_t st) {
  using V = typename VT<T, CPLX>::V;
  constexpr int W = (int)(16 / sizeof(V));
  if (pack_width(sizeof(V), M, x, g, nullptr) > 1)
    launch_pdl(k_moments<T, CPLX, W>, tiles * nbatch, NTHREADS, 0, st, x, g, M, tiles, partials, results, ticket, mc);
  else
    launch_pdl(k_moments<T, CPLX, 1>, tiles * nbatch, NTHREADS, 0, st, x, g, M, tiles, partials, results, ticket, mc);
}
template <typename T, bool CPLX>
static void run_axpby(const void* x, const void* g, const double* coef, int stride, long long M, int nbatch, void* out,
                      cudaStream_t st) {
  using V = typename VT<T, CPLX>::V;
  constexpr int W = (int)(16 / sizeof(V));
  const int w = pack_width(sizeof(V), M, x, g, out);
  // about eight CTAs per SM in all, one value (pack) per thread and pass
  const int gy = std::min(nbatch, 65535);
  const long long full = (M / w + NTHREADS - 1) / NTHREADS;
  const int gx = (int)std::max<long long>(1, std::min<long long>(full, std::max(1, 152 * 8 / gy)));
  if (w > 1) launch_pdl(k_axpby<T, CPLX, W>, dim3(gx, gy), NTHREADS, 0, st, x, g, coef, stride, M, nbatch, out);
  else launch_pdl(k_axpby<T, CPLX, 1>, dim3(gx, gy), NTHREADS, 0, st, x, g, coef, stride, M, nbatch, out);
}

// Shifted subproblem inputs in float32: X^k and P_k = G_k - theta_k X^k
// (interleaved real components; theta_k is real).
static __global__ void k_to_shifted_f32(const double* xk, const double* gk, double th, float* xk32, float* pk32,
                                 long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double x = xk[i];
    xk32[i] = (float)x;
    pk32[i] = (float)(gk[i] - th * x);
  }
}

// Z = X^k + D (D from the float32 subproblem), float64.
static __global__ void k_add_f32_to_f64(const double* xk, const float* d, double* z, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    z[i] = xk[i] + (double)d[i];
}

template <typename Ti, typename To>
__global__ void k_convert(const Ti* in, To* out, long long n, double scale) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = (To)((double)in[i] * scale);
}

// fine -> coarse: values at the coarse nodes (Algorithm 3 initial guess).  The
// fine mesh is r = 2^k times finer; coarse index i sits at fine index r*i
// (periodic grids, node 0 shared) or r*(i+1)-1 (interior nodes of Dirichlet
// grids).
template <typename T, bool CPLX>
__global__ void k_inject(const void* fv, void* cv, int dim, int f0, int f1, int c0, int c1, int r, int dirichlet,
                         long long Mf, long long Mc, int nbatch) {
  using V = typename VT<T, CPLX>::V;
  const V* f = (const V*)fv;
  V* c = (V*)cv;
  const long long n = Mc * nbatch;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int b = (int)(i / Mc);
    const long long li = i - b * Mc;
    const int i0 = (int)(li % c0);
    const long long rr = li / c0;
    const int i1 = (int)(rr % c1);
    const int i2 = (int)(rr / c1);
    auto fine = [&](int ic) -> long long { return dirichlet ? (long long)r * (ic + 1) - 1 : (long long)r * ic; };
    const long long j0 = fine(i0);
    const long long j1 = dim >= 2 ? fine(i1) : 0;
    const long long j2 = dim >= 3 ? fine(i2) : 0;
    c[i] = f[b * Mf + (j2 * f1 + j1) * f0 + j0];
  }
}

// Spectral prolongation along one axis (Algorithm 3 transfer): each line of
// length Nc (Fourier) or Nc-1 (sine, odd extension to 2Nc) is transformed,
// zero-padded to Ff = 2 Fc with the Fourier Nyquist coefficient split evenly
// between +-Nc/2, and transformed back on the fine line.  Lines are enumerated
// like the axis pass (coarse extents along this axis, current extents along the
// others).
template <typename T, bool CPLX>
__global__ void __launch_bounds__(NTHREADS) k_prolong_axis(PassGeom<T> G, int Ff, int logFf, const typename C2t<T>::type* twf,
                                                           int len_f, long long stride_f, long long ostride_f,
                                                           long long Mf, const void* inv, void* outv) {
  using C = typename C2t<T>::type;
  using V = typename VT<T, CPLX>::V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Fc = G.F;
  C* b0 = reinterpret_cast<C*>(smem_raw);
  C* b1 = b0 + G.LC * Ff;
  const int inst = blockIdx.x / G.tiles;
  const int tile = blockIdx.x - inst * G.tiles;
  const V* in = (const V*)inv;
  V* out = (V*)outv;
  for (int i = threadIdx.x; i < 2 * G.LC * Ff; i += blockDim.x) b0[i] = mk<C>(0.0, 0.0);
  __syncthreads();
  const int nval = G.LB * G.len;
  for (int f = threadIdx.x; f < nval; f += blockDim.x) {
    int l, j;
    if (G.axis == 0) { l = f / G.len; j = f - l * G.len; }
    else { j = f / G.LB; l = f - j * G.LB; }
    long long b;
    int ri;
    if (!line_base(G, inst, tile, l, b, ri)) continue;
    const V v = in[b + (long long)j * G.stride];
    const int m = G.odd_ext ? j + 1 : j;
    if constexpr (CPLX) {
      C* row = b0 + l * Fc;
      row[m] = v;
      if (G.odd_ext) row[Fc - m] = -v;
    } else {
      T* row = reinterpret_cast<T*>(b0 + (l >> 1) * Fc);
      row[2 * m + (l & 1)] = v;
      if (G.odd_ext) row[2 * (Fc - m) + (l & 1)] = -v;
    }
  }
  __syncthreads();
  // coarse forward FFTs use the first LC*Fc entries of b0/b1
  C* r = fft_lines<C>(b0, b1, Fc, G.LC, G.tw);
  C* dst = (r == b0) ? b1 : b0;
  for (int i = threadIdx.x; i < G.LC * Ff; i += blockDim.x) dst[i] = mk<C>(0.0, 0.0);
  __syncthreads();
  const T inv_n = T(1) / T(Fc);
  for (int t = threadIdx.x; t < G.LC * Fc; t += blockDim.x) {
    const int c = t / Fc;
    const int m = t - c * Fc;
    C v = r[t];
    v.x *= inv_n;
    v.y *= inv_n;
    // conjugate now so that the forward FFT below acts as the inverse
    v.y = -v.y;
    C* row = dst + c * Ff;
    if (m < Fc / 2) {
      row[m] = v;
    } else if (m > Fc / 2) {
      row[Ff - (Fc - m)] = v;
    } else {
      // Nyquist p = -Fc/2: zero for the sine extension; split for Fourier
      v.x *= T(0.5);
      v.y *= T(0.5);
      row[Fc / 2] = v;
      row[Ff - Fc / 2] = v;
    }
  }
  __syncthreads();
  C* o = fft_lines<C>(dst, r, Ff, G.LC, twf);
  const int nvf = G.LB * len_f;
  for (int f = threadIdx.x; f < nvf; f += blockDim.x) {
    int l, j;
    if (G.axis == 0) { l = f / len_f; j = f - l * len_f; }
    else { j = f / G.LB; l = f - j * G.LB; }
    // output line base on the fine-along-axis array
    long long bo;
    if (G.axis == 0) {
      long long rr = (long long)tile * G.LB + l;
      if (rr >= (long long)G.n1 * G.n2) continue;
      bo = inst * Mf + rr * len_f;
    } else {
      int oo = tile / G.xt;
      int x = (tile - oo * G.xt) * G.LB + l;
      if (x >= G.n0) continue;
      bo = inst * Mf + (long long)oo * ostride_f + x;
    }
    const int m = G.odd_ext ? j + 1 : j;
    V val;
    if constexpr (CPLX) {
      const C ov = o[l * Ff + m];
      val.x = ov.x;
      val.y = -ov.y;
    } else {
      const C ov = o[(l >> 1) * Ff + m];
      val = (l & 1) ? -ov.y : ov.x;
    }
    out[bo + (long long)j * stride_f] = val;
  }
  (void)logFf;
}

// FD prolongation along one axis: linear interpolation with zero Dirichlet ends.
template <typename T, bool CPLX>
__global__ void k_prolong_fd_axis(const void* inv, void* outv, int axis, int e0, int e1, int e2, int lc, int lf,
                                  long long Mc, long long Mf, int nbatch) {
  using V = typename VT<T, CPLX>::V;
  const V* in = (const V*)inv;
  V* out = (V*)outv;
  // output extents: along `axis` lf, others e*
  int o0 = e0, o1 = e1, o2 = e2;
  if (axis == 0) o0 = lf; else if (axis == 1) o1 = lf; else o2 = lf;
  const long long n = Mf * nbatch;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int b = (int)(i / Mf);
    const long long li = i - b * Mf;
    int idx[3];
    idx[0] = (int)(li % o0);
    const long long r = li / o0;
    idx[1] = (int)(r % o1);
    idx[2] = (int)(r / o1);
    const int jf = idx[axis] + 1;                     // fine node number 1..lf
    const int jc = jf >> 1;                            // coarse node left of it
    const bool odd = jf & 1;
    auto at = [&](int node) -> V {                     // coarse node value (0 at the ends)
      if (node < 1 || node > lc) return vzero<V>();
      int id[3] = {idx[0], idx[1], idx[2]};
      id[axis] = node - 1;
      int c0 = e0, c1 = e1;
      if (axis == 0) c0 = lc; else if (axis == 1) c1 = lc;
      return in[b * Mc + ((long long)id[2] * c1 + id[1]) * c0 + id[0]];
    };
    V v;
    if (!odd) v = at(jc);
    else v = T(0.5) * (at(jc) + at(jc + 1));
    out[i] = v;
  }
}

}  // namespace gpe
