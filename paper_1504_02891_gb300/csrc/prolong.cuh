// prolong.cuh -- spectral prolongation along one axis (Algorithm 3 transfer) by
// the register line transforms, for complex and real Fourier lines and real
// sine lines (lines3.cuh) of 32 to 512 transform points on the coarse mesh.
//
// The zero-padded spectrum's interpolant passes through the coarse values, so
// only the midpoints are computed: the coarse line is transformed (length F),
// its mode p is multiplied by e^{i pi p / F} (half a coarse cell; the Nyquist
// coefficient, split evenly between +-F/2, vanishes there) and transformed
// back (length F).  A padded inverse transform of length 2F would recompute
// the coarse values too.  The midpoint operator is real, so two real lines
// still share one complex line.  64^3 -> 128^3 sine float32, per axis kernel:
// 27 us for the shared-memory transforms of length F and 2F with a division
// per element.
#pragma once
#include "lines3.cuh"

namespace gpe {

// Midpoint values of a line: forward transform, phase, inverse transform (as
// the conjugate of the forward transform of the conjugate); 1/F in `scale`.
// fine: twiddles e^{-2 pi i k / (2F)}.
template <int LF, typename Ex>
__device__ __forceinline__ void midpoints(const LineFFT<float, LF>& fft, float2 (&v)[8], const Ex& ex, int& par,
                                          const float2* __restrict__ fine) {
  constexpr int F = 1 << LF, TPL = F / 8;
  fft.forward(v, ex, par);
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int m = fft.j + s * TPL;
    const int p = m < (F >> 1) ? m : m - F;
    // conj(v e^{i pi p / F}) / F = conj(v) e^{-2 pi i p / (2F)} / F
    const float2 w = ld_const(fine + (p & (2 * F - 1)));
    const float sc = m == (F >> 1) ? 0.f : 1.f / F;
    v[s] = cmul(make_float2(sc * v[s].x, -sc * v[s].y), w);
  }
  fft.forward(v, ex, par);
#pragma unroll
  for (int s = 0; s < 8; ++s) v[s].y = -v[s].y;
}
template <int LF, typename Ex>
__device__ __forceinline__ void midpoints(const LineFFT<double, LF>& fft, double2 (&v)[8], const Ex& ex, int& par,
                                          const int4* __restrict__ fine) {
  fft.midpoints(v, ex, par, fine);
}

template <typename T> struct ProlongArgs {
  PassGeom<T> G;          // the coarse line geometry (extents of the array read)
  const void* in;
  void* out;
  const double* coef;     // scale applied to the output (null: 1), per instance
  const typename C2t<T>::type* twf;   // fine table, float32
  const int4* twf_fix;                // fine table, float64
  int width, tiles;       // strided kernel: inner width, tiles per plane
  int planes_per_inst;
};

template <typename T, int LF> __device__ __forceinline__ auto fine_table(const ProlongArgs<T>& A) {
  if constexpr (sizeof(T) == 4) return A.twf;
  else return A.twf_fix;
}

// Strided axis: plane p of the input has G.len rows of `width` values, of the
// output 2 len (Fourier) or 2 len + 1 (sine) rows.
template <typename T, int KIND, int LF>
__global__ void __launch_bounds__(axs_threads<T>(LF)) k_prolong_s(ProlongArgs<T> A) {
  using FFT = LineFFT<T, LF>;
  using C = typename FFT::C;
  using X = typename FFT::X;
  using V = typename VT<T, KIND == LK_CPLX>::V;
  constexpr int F = FFT::F, TPL = FFT::TPL, CW = axs_cw<T>(LF), NT = axs_threads<T>(LF);
  constexpr int NP = KIND == LK_SINE ? 4 : 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  typename FFT::Tw* tws = reinterpret_cast<typename FFT::Tw*>(smem_raw);
  X* xb = reinterpret_cast<X*>(tws + F);
  __shared__ long long s_red[(NT + 31) / 32 * CW];
  const PassGeom<T>& G = A.G;
  const int tid = threadIdx.x, cl = tid & (CW - 1), j = tid / CW;
  const int plane = blockIdx.x / A.tiles, tile = blockIdx.x - plane * A.tiles;
  const int width = A.width;
  const int c0 = KIND == LK_CPLX ? tile * CW + cl : (KIND == LK_REAL ? 2 * (tile * CW + cl) : 2 * tile * CW + cl);
  const int c1 = KIND == LK_REAL ? c0 + 1 : c0 + CW;
  const bool in0 = c0 < width, in1 = KIND != LK_CPLX && c1 < width;
  load_table(tws, line_table<FFT>(G), F);
  FFT fft;
  fft.init(j, tws);
  pdl_next();
  pdl_wait();
  const V* in = (const V*)A.in + (long long)plane * G.len * width;
  const int flen = KIND == LK_SINE ? 2 * G.len + 1 : 2 * G.len;
  V* out = (V*)A.out + (long long)plane * flen * width;
  auto has = [&](int s) -> bool { return KIND != LK_SINE || s > 0 || j > 0; };
  C v[8], x[NP];
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    const long long o = (long long)(j + s * TPL - (KIND == LK_SINE ? 1 : 0)) * width;
    const V p = has(s) && in0 ? in[o + c0] : vzero<V>();
    if constexpr (KIND == LK_CPLX) {
      v[s] = p;
    } else {
      v[s].x = p;
      v[s].y = has(s) && in1 ? in[o + c1] : vzero<V>();
    }
    x[s] = v[s];
  }
  int par = 0;
  ExCols<X, CW> ex{xb + cl, F * CW, s_red};
  if constexpr (KIND == LK_SINE) mirror_odd<T, LF>(v, ex, par, j);
  midpoints<LF>(fft, v, ex, par, fine_table<T, LF>(A));
  const T sc = A.coef ? (T)A.coef[plane / A.planes_per_inst] : T(1);
  // coarse node m is fine row 2m (sine: 2m - 1), its right midpoint the next row
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    const long long o = (long long)(2 * (j + s * TPL) - (KIND == LK_SINE ? 1 : 0)) * width;
    if constexpr (KIND == LK_CPLX) {
      if (in0) out[o + c0] = sc * x[s];
      if (in0) out[o + width + c0] = sc * v[s];
    } else {
      if (has(s) && in0) out[o + c0] = sc * x[s].x;
      if (has(s) && in1) out[o + c1] = sc * x[s].y;
      if (in0) out[o + width + c0] = sc * v[s].x;
      if (in1) out[o + width + c1] = sc * v[s].y;
    }
  }
}

// x axis: rows of G.len values, one group of lines per CTA.
template <typename T, int KIND, int LF>
__global__ void __launch_bounds__(axx_threads<T>(LF)) k_prolong_x(ProlongArgs<T> A) {
  using FFT = LineFFT<T, LF>;
  using C = typename FFT::C;
  using X = typename FFT::X;
  constexpr bool CPLX = KIND == LK_CPLX;
  using V = typename VT<T, CPLX>::V;
  constexpr int F = FFT::F, TPL = FFT::TPL, NT = axx_threads<T>(LF), NL = NT / TPL;
  constexpr int NP = KIND == LK_SINE ? 4 : 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  typename FFT::Tw* tws = reinterpret_cast<typename FFT::Tw*>(smem_raw);
  X* xb = reinterpret_cast<X*>(tws + F);
  __shared__ long long s_red[(NT + 31) / 32];
  const PassGeom<T>& G = A.G;
  const int tid = threadIdx.x, l = tid / TPL, j = tid & (TPL - 1);
  const int inst = blockIdx.x / A.tiles, grp = blockIdx.x - inst * A.tiles;
  const int rows = (int)(G.M / G.len);
  const int r0 = CPLX ? grp * NL + l : 2 * (grp * NL + l);
  const bool in0 = r0 < rows, in1 = !CPLX && r0 + 1 < rows;
  load_table(tws, line_table<FFT>(G), F);
  FFT fft;
  fft.init(j, tws);
  pdl_next();
  pdl_wait();
  const V* in = (const V*)A.in + (long long)inst * G.M + (long long)r0 * G.len;
  const int flen = KIND == LK_SINE ? 2 * G.len + 1 : 2 * G.len;
  V* out = (V*)A.out + ((long long)inst * rows + r0) * flen;
  auto has = [&](int s) -> bool { return KIND != LK_SINE || s > 0 || j > 0; };
  C v[8], x[NP];
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    const int o = j + s * TPL - (KIND == LK_SINE ? 1 : 0);
    const V p = has(s) && in0 ? in[o] : vzero<V>();
    if constexpr (CPLX) {
      v[s] = p;
    } else {
      v[s].x = p;
      v[s].y = has(s) && in1 ? in[o + G.len] : vzero<V>();
    }
    x[s] = v[s];
  }
  int par = 0;
  ExRow<X, FFT::P> ex{xb + l * FFT::P, NL * FFT::P, 1 + l, TPL, s_red};
  if constexpr (KIND == LK_SINE) mirror_odd<T, LF>(v, ex, par, j);
  midpoints<LF>(fft, v, ex, par, fine_table<T, LF>(A));
  const T sc = A.coef ? (T)A.coef[inst] : T(1);
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    const int o = 2 * (j + s * TPL) - (KIND == LK_SINE ? 1 : 0);
    if constexpr (CPLX) {
      if (in0) out[o] = sc * x[s];
      if (in0) out[o + 1] = sc * v[s];
    } else {
      if (has(s) && in0) out[o] = sc * x[s].x;
      if (in0) out[o + 1] = sc * v[s].x;
      if (has(s) && in1) out[flen + o] = sc * x[s].y;
      if (in1) out[flen + o + 1] = sc * v[s].y;
    }
  }
}

template <typename T, int KIND, int LF>
static gpe_status launch_prolong_line_t(int axis, ProlongArgs<T> A, int nbatch, cudaStream_t st) {
  using FFT = LineFFT<T, LF>;
  const PassGeom<T>& G = A.G;
  if (axis == 0) {
    constexpr int NT = axx_threads<T>(LF), NL = NT / FFT::TPL;
    const size_t smem = (size_t)FFT::F * sizeof(typename FFT::Tw) + 2 * (size_t)NL * FFT::P * sizeof(typename FFT::X);
    static KernelShape shape;
    int occ = 0;
    GPE_CUDA(kernel_shape(shape, (const void*)k_prolong_x<T, KIND, LF>, NT, smem, &occ));
    const long long rows = G.M / G.len, lines = KIND == LK_CPLX ? rows : (rows + 1) / 2;
    A.tiles = (int)((lines + NL - 1) / NL);
    GPE_CUDA(launch_pdl(k_prolong_x<T, KIND, LF>, nbatch * A.tiles, NT, smem, st, A));
  } else {
    constexpr int CW = axs_cw<T>(LF), NT = axs_threads<T>(LF);
    const size_t smem = (size_t)FFT::F * sizeof(typename FFT::Tw) + 2 * (size_t)FFT::F * CW * sizeof(typename FFT::X);
    static KernelShape shape;
    int occ = 0;
    GPE_CUDA(kernel_shape(shape, (const void*)k_prolong_s<T, KIND, LF>, NT, smem, &occ));
    A.width = axis == 1 ? G.n0 : G.n0 * G.n1;
    A.planes_per_inst = axis == 1 ? G.n2 : 1;
    const int cols = KIND == LK_CPLX ? CW : 2 * CW;
    A.tiles = (A.width + cols - 1) / cols;
    GPE_CUDA(launch_pdl(k_prolong_s<T, KIND, LF>, nbatch * A.planes_per_inst * A.tiles, NT, smem, st, A));
  }
  return GPE_OK;
}

template <typename T, int KIND>
static gpe_status launch_prolong_line_k(int axis, const ProlongArgs<T>& A, int nbatch, cudaStream_t st) {
  switch (A.G.logF) {
    case 5: return launch_prolong_line_t<T, KIND, 5>(axis, A, nbatch, st);
    case 6: return launch_prolong_line_t<T, KIND, 6>(axis, A, nbatch, st);
    case 7: return launch_prolong_line_t<T, KIND, 7>(axis, A, nbatch, st);
    case 8: return launch_prolong_line_t<T, KIND, 8>(axis, A, nbatch, st);
    case 9: return launch_prolong_line_t<T, KIND, 9>(axis, A, nbatch, st);
  }
  return fail(GPE_EINVAL, "unsupported line length");
}

template <typename T>
gpe_status launch_prolong_line(const GridHost& gc, int axis, const PassGeom<T>& G, const void* in, void* out,
                               const double* coef, const GridDev<T>& df, cudaStream_t st) {
  ProlongArgs<T> A{};
  A.G = G;
  A.in = in;
  A.out = out;
  A.coef = coef;
  A.twf = df.tw[axis];
  A.twf_fix = df.geom[axis].twf;
  if (gc.disc == GPE_SINE) return launch_prolong_line_k<T, LK_SINE>(axis, A, gc.nbatch, st);
  if (gc.is_complex) return launch_prolong_line_k<T, LK_CPLX>(axis, A, gc.nbatch, st);
  return launch_prolong_line_k<T, LK_REAL>(axis, A, gc.nbatch, st);
}

}  // namespace gpe
