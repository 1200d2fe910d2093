// lines3.cuh -- the operator on 1D and 3D Fourier grids and on real sine grids
// of any dimension, one kernel per axis, with every line transform in registers
// (linefft.cuh in float32, fixfft.cuh in float64).
//
// A line of F points (Fourier: the grid line; sine: its odd extension to 2N
// points, Eq. tpll) belongs to F/8 threads, 8 points each.  Real grids pack two
// lines into one complex line.  The strided axes go first (z, then y), each
// adding its kinetic part to the accumulator; the x-kernel comes last, adds the
// accumulator and V X and runs the pointwise epilogue, the reduction and the
// control.
//
//   k_axis_s (y, z): a CTA owns CW complex columns of one plane; consecutive
//     lanes hold consecutive columns.  Sine grids have odd row lengths, so
//     their pairs are columns x and x + CW of a tile (coalesced single values)
//     instead of adjacent ones (misaligned pairs).
//   k_axis_x: NL lines per CTA, the threads of a line consecutive.
//
// The odd half of a sine line is mirrored through the exchange buffer, so each
// value is read from memory once.  The accumulator and V are fetched (registers
// in float32, cp.async slots in float64) before the transforms, or on large
// float64 grids after them (see launch_axis_x_t); the other vectors of the
// epilogue after them, ahead of the line's stores.
//
// What bounds them: on 128^3 grids the arrays stay in L2 and the integer and
// float32 issue counts (half of the cycles of the strided kernels, with 32% of
// the warps resident in float32 and 23% in float64); on 64^3 a kernel is a
// chain of a few latencies.
// Measured against the general passes (a shared-memory tile per axis): 127^3
// sine gradient float64 1039 -> 208 us, Hessian-vector float32 117 -> 40.8 us
// (245 and 59 before the register budget below, the two-level folds and the
// programmatic launches; 45.6 with the stores between the epilogue's loads),
// energy of 512 points float64 52 -> 27.6 us (with the pinned sums).
#pragma once
#include "lines2d.cuh"

namespace gpe {

// What a line holds: a complex Fourier line, two real Fourier lines, two real
// sine lines.
enum LineKind { LK_CPLX = 0, LK_REAL = 1, LK_SINE = 2 };

// Complex columns per CTA of the strided kernel: 64-byte row segments, at most
// 512 threads (float64: 256).
template <typename T> __host__ __device__ constexpr int axs_cw(int lf) {
  return sizeof(T) == 4 ? (lf <= 9 ? 8 : 4) : (lf <= 6 ? 8 : (lf <= 9 ? 4 : 2));
}
template <typename T> __host__ __device__ constexpr int axs_threads(int lf) { return axs_cw<T>(lf) * (1 << lf) / 8; }
// Resident CTAs the strided kernel's registers are sized for: 24 warps per SM in
// float32 (85 registers) and 16 in float64 (128), where the compiler's own
// choice (92 and 168) left room for 16 and 12 (127^3: Hessian-vector float32
// 48.5 -> 45.6 us, gradient float64 217 -> 208; measured there, on 256-point
// transforms, only).  CTAs of 512 (float64: 256) threads, the longest lines, are
// left to the compiler.
template <typename T> __host__ __device__ constexpr int axs_minb(int lf) {
  const int warps = sizeof(T) == 4 ? 24 : 16, w = axs_threads<T>(lf) / 32;
  return axs_threads<T>(lf) >= (sizeof(T) == 4 ? 512 : 256) ? 1 : warps / w;
}
// Threads of the x-kernel's CTA: 128 in float32, 64 in float64 (which lowers
// the tail of small grids), or one line's.
template <typename T> __host__ __device__ constexpr int axx_threads(int lf) {
  const int base = sizeof(T) == 4 ? 128 : 64;
  return (1 << lf) / 8 > base ? (1 << lf) / 8 : base;
}
// registers: at most 128 per thread
template <typename T> __host__ __device__ constexpr int axx_minb(int lf) { return 65536 / (axx_threads<T>(lf) * 128); }

// Mirror a sine line: this thread's points s < 4 (m = j + s F/8 in [0, N), the
// point m = 0 is not data) into points F - m, then read s >= 4.
template <typename T, int LF, typename Ex, typename C>
__device__ __forceinline__ void mirror_odd(C (&v)[8], const Ex& ex, int& par, int j) {
  constexpr int F = 1 << LF, TPL = F / 8;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int m = j + s * TPL;
    if (m == 0) v[s].x = v[s].y = T(0);
    *reinterpret_cast<C*>(ex(par, m == 0 ? F / 2 : F - m)) = -v[s];
  }
  ex.sync();
#pragma unroll
  for (int s = 4; s < 8; ++s) v[s] = *reinterpret_cast<C*>(ex(par, j + s * TPL));
  par ^= 1;
}

// Strided axis: out = (acc_in or 0) + T_a X over the tiles of all planes.
template <typename T, int KIND, int LF>
__global__ void __launch_bounds__(axs_threads<T>(LF), axs_minb<T>(LF)) k_axis_s(PassGeom<T> G, PassData<T> D, int width, int tiles) {
  using FFT = LineFFT<T, LF>;
  using C = typename FFT::C;
  using X = typename FFT::X;
  using V = typename VT<T, KIND == LK_CPLX>::V;
  constexpr int F = FFT::F, TPL = FFT::TPL, CW = axs_cw<T>(LF), NT = axs_threads<T>(LF);
  constexpr int NP = KIND == LK_SINE ? 4 : 8;    // data points per thread and line
  extern __shared__ __align__(16) unsigned char smem_raw[];
  typename FFT::Tw* tws = reinterpret_cast<typename FFT::Tw*>(smem_raw);
  X* xb = reinterpret_cast<X*>(tws + F);         // [2][F][CW]
  __shared__ long long s_red[(NT + 31) / 32 * CW];
  const int tid = threadIdx.x;
  const int cl = tid & (CW - 1), j = tid / CW;
  const int plane = blockIdx.x / tiles, tile = blockIdx.x - plane * tiles;
  load_table(tws, line_table<FFT>(G), F);
  FFT fft;
  fft.init(j, tws);
  pdl_next();
  pdl_wait();
  if (D.ctl && D.ctl->done) return;
  const V* x0 = (const V*)D.x;
  const V* x1 = (const V*)D.xsub;
  V* yst = nullptr;
  const V* xk = nullptr;
  T sa = 0, sb = 0, sk = 0;
  if (D.use_slots) {
    const Alg1Ctl* c = D.ctl;
    x0 = (const V*)D.xs[c->trial];
    if (D.step_on_load) {
      yst = (V*)D.xs[c->trial];
      x0 = (const V*)D.xs[c->cur];
      x1 = (const V*)D.gs[c->cur];
      sa = (T)(c->s * c->a);
      sb = (T)(c->s * c->b);
      if (D.step_on_load == 2) {
        xk = (const V*)D.base;
        sk = (T)c->am1;
        sa = (T)c->a;
        sb = (T)c->b;
      }
    }
  }
  const V* acc = (const V*)D.acc_in;
  V* out = (V*)D.out;
  // columns of this lane: one complex, or the two real ones of its pair
  const int c0 = KIND == LK_CPLX ? tile * CW + cl : (KIND == LK_REAL ? 2 * (tile * CW + cl) : 2 * tile * CW + cl);
  const int c1 = KIND == LK_REAL ? c0 + 1 : c0 + CW;
  const bool in0 = c0 < width, in1 = KIND != LK_CPLX && c1 < width;
  const long long pbase = (long long)plane * G.len * width;
  // offset of data point s of column c
  auto off = [&](int s, int c) -> long long {
    const int m = j + s * TPL - (KIND == LK_SINE ? 1 : 0);
    return pbase + (long long)m * width + c;
  };
  auto has = [&](int s) -> bool { return KIND != LK_SINE || s > 0 || j > 0; };
  C v[8];
  V a0[NP], a1[KIND == LK_CPLX ? 1 : NP];
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    V p = vzero<V>(), q = vzero<V>();
    if (has(s)) {
      if (in0) p = x0[off(s, c0)];
      if (in1) q = x0[off(s, c1)];
      if (x1) {
        const V p1 = in0 ? x1[off(s, c0)] : vzero<V>(), q1 = in1 ? x1[off(s, c1)] : vzero<V>();
        if (xk) {
          p = (in0 ? sk * xk[off(s, c0)] : vzero<V>()) + sa * p + sb * p1;
          q = (in1 ? sk * xk[off(s, c1)] : vzero<V>()) + sa * q + sb * q1;
        } else {
          p = yst ? sa * p + sb * p1 : p - p1;
          q = yst ? sa * q + sb * q1 : q - q1;
        }
      }
    }
    if constexpr (KIND == LK_CPLX) {
      v[s] = p;
    } else {
      v[s].x = p;
      v[s].y = q;
    }
  }
  // the earlier axes' part, on its way while the line is transformed
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    a0[s] = vzero<V>();
    if (acc && in0 && has(s)) a0[s] = acc[off(s, c0)];
    if constexpr (KIND != LK_CPLX) {
      a1[s] = vzero<V>();
      if (acc && in1 && has(s)) a1[s] = acc[off(s, c1)];
    }
  }
  if (yst) {
#pragma unroll
    for (int s = 0; s < NP; ++s) {
      if (!has(s)) continue;
      if constexpr (KIND == LK_CPLX) {
        if (in0) yst[off(s, c0)] = v[s];
      } else {
        if (in0) yst[off(s, c0)] = v[s].x;
        if (in1) yst[off(s, c1)] = v[s].y;
      }
    }
  }
  int par = 0;
  ExCols<X, CW> ex{xb + cl, F * CW, s_red};
  if constexpr (KIND == LK_SINE) mirror_odd<T, LF>(v, ex, par, j);
  LineSym<T, F> sym;
  sym.c2 = G.c2;
  sym.dl = G.dlam;
  sym.c1c = (KIND == LK_CPLX && G.rcoord && in0) ? G.c1 * G.rcoord[c0] : T(0);
  fft.apply(v, ex, par, sym);
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    if (!has(s)) continue;
    if constexpr (KIND == LK_CPLX) {
      if (in0) out[off(s, c0)] = a0[s] + v[s];
    } else {
      if (in0) out[off(s, c0)] = a0[s] + v[s].x;
      if (in1) out[off(s, c1)] = a1[s] + v[s].y;
    }
  }
}

// x axis: lines are contiguous rows; epilogue, reduction, control.  CTA `tile`
// of an instance takes the line groups tile, tile + tiles_per_inst, ...
template <typename T, int KIND, int EPI, int LF>
__global__ void __launch_bounds__(axx_threads<T>(LF), axx_minb<T>(LF)) k_axis_x(PassGeom<T> G, PassData<T> D,
                                                                              int tiles_per_inst, int groups,
                                                                              int slots) {
  using FFT = LineFFT<T, LF>;
  using C = typename FFT::C;
  using X = typename FFT::X;
  constexpr bool CPLX = KIND == LK_CPLX;
  using V = typename VT<T, CPLX>::V;
  using A = typename AccT<T>::type;
  constexpr int F = FFT::F, TPL = FFT::TPL, NT = axx_threads<T>(LF), NL = NT / TPL;
  constexpr int NP = KIND == LK_SINE ? 4 : 8;    // data points per thread and row
  constexpr int NV = CPLX ? NP : 2 * NP;         // values per thread
  constexpr bool REGS = sizeof(T) == 4;          // epilogue operands in registers
  extern __shared__ __align__(16) unsigned char smem_raw[];
  typename FFT::Tw* tws = reinterpret_cast<typename FFT::Tw*>(smem_raw);
  X* xb = reinterpret_cast<X*>(tws + F);         // [2][NL][P]
  V* es = reinterpret_cast<V*>(xb + 2 * NL * FFT::P);   // float64: [NV][NT] input, with slots [2] (accumulator)
  T* ev = reinterpret_cast<T*>(es + 2 * NV * NT);       // with slots: [NV][NT] potential
  __shared__ long long s_red[(NT + 31) / 32];
  load_table(tws, line_table<FFT>(G), F);
  const int tid = threadIdx.x;
  const int l = tid / TPL, j = tid & (TPL - 1);
  FFT fft;
  fft.init(j, tws);
  pdl_next();
  pdl_wait();
  if (D.ctl && D.ctl->done) return;
  int par = 0;
  const int inst = blockIdx.x / tiles_per_inst;
  const int tile = blockIdx.x - inst * tiles_per_inst;
  const V* xin = (const V*)D.x;
  const V* xsub = (const V*)D.xsub;
  V* yst = nullptr;
  const V* xk = nullptr;
  T sa = 0, sb = 0, sk = 0;
  if (D.use_slots) {
    const Alg1Ctl* c = D.ctl;
    xin = (const V*)D.xs[c->trial];
    if (D.step_on_load) {   // 1D: this is the first pass too
      yst = (V*)D.xs[c->trial];
      xin = (const V*)D.xs[c->cur];
      xsub = (const V*)D.gs[c->cur];
      sa = (T)(c->s * c->a);
      sb = (T)(c->s * c->b);
      if (D.step_on_load == 2) {
        xk = (const V*)D.base;
        sk = (T)c->am1;
        sa = (T)c->a;
        sb = (T)c->b;
      }
    }
  }
  const V* accin = (const V*)D.acc_in;
  EpiCtx<T, CPLX> E;
  make_ctx<T, CPLX, EPI, false>(E, D);
  A acc[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) acc_zero(acc[q]);
  T amax = T(0);
  const long long ibase = (long long)inst * G.M;
  const T* Vp = D.V;
  const int rows = (int)(G.M / G.len);
  LineSym<T, F> sym;
  sym.c2 = G.c2;
  sym.dl = G.dlam;
  static_assert(TPL < 32 || (TPL % 32 == 0 && NL <= 15), "named barriers per line");
  ExRow<X, FFT::P> ex{xb + l * FFT::P, NL * FFT::P, 1 + l, TPL, s_red};
  for (int grp = tile; grp < groups; grp += tiles_per_inst) {
    const int line = grp * NL + l;
    const int r0 = CPLX ? line : 2 * line;
    // value q: point q % NP of row r0 (q < NP) or r0 + 1
    auto has = [&](int q) -> bool {
      return r0 + q / NP < rows && (KIND != LK_SINE || q % NP > 0 || j > 0);
    };
    auto at = [&](int q) -> int {   // offset within the instance
      return (r0 + q / NP) * G.len + j + (q % NP) * TPL - (KIND == LK_SINE ? 1 : 0);
    };
    V xv[NV], av[REGS ? NV : 1];
    T vv[REGS ? NV : 1];
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      xv[q] = vzero<V>();
      if (has(q)) {
        xv[q] = xin[ibase + at(q)];
        if (xsub) {
          const V b = xsub[ibase + at(q)];
          if (xk) xv[q] = sk * xk[ibase + at(q)] + sa * xv[q] + sb * b;
          else xv[q] = yst ? sa * xv[q] + sb * b : xv[q] - b;
        }
      }
    }
    ex.sync();   // the line's exchange rows are reused
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      if constexpr (REGS) {
        av[q] = vzero<V>();
        vv[q] = T(0);
        if (has(q)) {
          if (accin) av[q] = accin[ibase + at(q)];
          vv[q] = Vp[at(q)];
        }
      } else {
        if (slots && has(q)) {
          if (accin) cp_async(es + (NV + q) * NT + tid, accin + ibase + at(q));
          cp_async(ev + q * NT + tid, Vp + at(q));
        }
        es[q * NT + tid] = xv[q];
      }
    }
    if (yst) {
#pragma unroll
      for (int q = 0; q < NV; ++q)
        if (has(q)) yst[ibase + at(q)] = xv[q];
    }
    C v[8];
#pragma unroll
    for (int s = 0; s < NP; ++s) {
      if constexpr (CPLX) {
        v[s] = xv[s];
      } else {
        v[s].x = xv[s];
        v[s].y = xv[s + NP];
      }
    }
    if constexpr (KIND == LK_SINE) mirror_odd<T, LF>(v, ex, par, j);
    sym.c1c = (CPLX && G.rcoord && r0 < rows) ? G.c1 * G.rcoord[r0 % G.n1] : T(0);
    fft.apply(v, ex, par, sym);
    // v becomes the linear part: + accumulator + V x
    auto part = [&](int q) -> V& {
      if constexpr (CPLX) return v[q];
      else return q < NP ? v[q % NP].x : v[q % NP].y;
    };
    auto value = [&](int q) -> V {
      if constexpr (REGS) return xv[q];
      else return es[q * NT + tid];
    };
    auto add_lin = [&](int q, V aq, T pv) {
      V kin = part(q);
      if (REGS || accin) kin = kin + aq;
      part(q) = kin + pv * value(q);
    };
    if constexpr (REGS) {
#pragma unroll
      for (int q = 0; q < NV; ++q)
        if (has(q)) add_lin(q, av[q], vv[q]);
    } else if (slots) {
      cp_async_wait_all();
#pragma unroll
      for (int q = 0; q < NV; ++q)
        if (has(q)) add_lin(q, accin ? es[(NV + q) * NT + tid] : vzero<V>(), ev[q * NT + tid]);
    } else {
      constexpr int NE = NV < 8 ? NV : 8;   // values whose operands are in flight together
#pragma unroll
      for (int q0 = 0; q0 < NV; q0 += NE) {
        V ac[NE];
        T pc[NE];
#pragma unroll
        for (int u = 0; u < NE; ++u) {
          ac[u] = vzero<V>();
          pc[u] = T(0);
          if (!has(q0 + u)) continue;
          if (accin) ac[u] = __ldcg(accin + ibase + at(q0 + u));
          pc[u] = ld_const(Vp + at(q0 + u));
        }
#pragma unroll
        for (int u = 0; u < NE; ++u)
          if (has(q0 + u)) add_lin(q0 + u, ac[u], pc[u]);
      }
    }
    const bool diff = epilogue_diff(E);
    // with other vectors to load, the results take the linear part's place and
    // are stored last: a load must not wait for the store of the value before
    // it, and gathering the loads of several values ahead of their stores spills
    // (64^2 real float32 F 22.1 us gathered, 19.0 stored last; 64^3 sine 21.7 and
    // 19.8; 128 x 64 x 32 float64 F 47 and 45.3, its first evaluation, which loads
    // nothing, 38.9 and 40.9)
    constexpr bool LATE = epi_nops(EPI) > 0;
#pragma unroll
    for (int q = 0; q < NV; ++q)
      if (has(q)) {
        EpiOps<V, EPI> o;
        epilogue_load<T, CPLX, EPI, 0>(o, E, ibase + at(q));
        if constexpr (LATE)
          epilogue_put<T, CPLX, EPI>(E, value(q), part(q), o, acc, amax, diff, [&](V g) { part(q) = g; });
        else
          epilogue_apply<T, CPLX, EPI>(E, ibase + at(q), value(q), part(q), o, acc, amax, diff);
      }
    if constexpr (LATE && EPI != EPI_RATIO) {
#pragma unroll
      for (int q = 0; q < NV; ++q)
        if (has(q)) E.out[ibase + at(q)] = part(q);
    }
  }
  if (EPI == EPI_HESS || D.nq == 0) return;
  run_control<T>(D, reduce_partials(acc, amax, D.nq, D.partials, D.results, D.ticket, tiles_per_inst));
}

static inline int line_kind(const GridHost& g) {
  return g.disc == GPE_FOURIER ? (g.is_complex ? LK_CPLX : LK_REAL) : LK_SINE;
}
template <typename T, int KIND, int LF>
static gpe_status launch_axis_s_t(const GridDev<T>& d, int axis, const PassData<T>& D, int nbatch, cudaStream_t st) {
  using FFT = LineFFT<T, LF>;
  const PassGeom<T>& G = d.geom[axis];
  constexpr int CW = axs_cw<T>(LF), NT = axs_threads<T>(LF);
  const size_t smem = (size_t)FFT::F * sizeof(typename FFT::Tw) + 2 * (size_t)FFT::F * CW * sizeof(typename FFT::X);
  static KernelShape shape;
  int occ = 0;
  GPE_CUDA(kernel_shape(shape, (const void*)k_axis_s<T, KIND, LF>, NT, smem, &occ));
  const int width = axis == 1 ? G.n0 : G.n0 * G.n1;
  const int planes = nbatch * (axis == 1 ? G.n2 : 1);
  const int cols = KIND == LK_CPLX ? CW : 2 * CW;
  const int tiles = (width + cols - 1) / cols;
  ProfScope ps(kernel_name("axis_s", sizeof(T) == 8, KIND == LK_CPLX, EPI_ACC, G.M * nbatch), st);
  GPE_CUDA(launch_pdl(k_axis_s<T, KIND, LF>, planes * tiles, NT, smem, st, G, D, width, tiles));
  return GPE_OK;
}

template <typename T, int KIND, int EPI, int LF>
static gpe_status launch_axis_x_t(const GridDev<T>& d, const PassData<T>& D, int nbatch, cudaStream_t st) {
  using FFT = LineFFT<T, LF>;
  const PassGeom<T>& G = d.geom[0];
  constexpr int NT = axx_threads<T>(LF), NL = NT / FFT::TPL;
  constexpr int NV = KIND == LK_REAL ? 16 : 8;
  const size_t vsz = sizeof(T) * (KIND == LK_CPLX ? 2 : 1);
  const size_t base = (size_t)FFT::F * sizeof(typename FFT::Tw) + 2 * (size_t)NL * FFT::P * sizeof(typename FFT::X);
  const size_t few = base + (sizeof(T) == 8 ? (size_t)NV * NT * vsz : 0);
  const size_t all = base + (sizeof(T) == 8 ? (size_t)NV * NT * (2 * vsz + sizeof(T)) : 0);
  static KernelShape sf, sa;
  int occ_few = 0, occ_all = 0;
  GPE_CUDA(kernel_shape(sf, (const void*)k_axis_x<T, KIND, EPI, LF>, NT, few, &occ_few));
  GPE_CUDA(kernel_shape(sa, (const void*)k_axis_x<T, KIND, EPI, LF>, NT, all, &occ_all));
  const long long rows = G.M / G.len;
  const long long lines = KIND == LK_CPLX ? rows : (rows + 1) / 2;
  const int groups = (int)((lines + NL - 1) / NL);
  // float64: shared-memory slots for the epilogue's operands hide their latency
  // behind the transforms, but cost resident CTAs.  With more than two and a half
  // waves of groups the operands are loaded after the transforms instead (128^3
  // real Fourier gradient 165 -> 147.5 us, 127^3 sine gradient 209.8 -> 207.0 and
  // Hessian-vector 187.5 -> 182.1; at 2.2 waves, four 64^3 complex gradients,
  // 151 with and without, at 1.6, three 64^3 sine gradients, 116 against 124)
  const int slots = sizeof(T) == 8 && 2LL * groups * nbatch <= 5LL * occ_all * num_sms();
  const size_t smem = slots ? all : few;
  // one resident wave (each CTA pays its tables and a reduction of its sums; a
  // CTA per group took 47.8 us for the 127^3 Hessian-vector product, this 45.6
  // then),
  // within the reduction scratch
  long long cap = std::min<long long>((long long)(slots ? occ_all : occ_few) * num_sms(), d.max_blocks);
  const int tiles = (int)std::max<long long>(1, std::min<long long>(groups, std::max<long long>(cap / nbatch, 1)));
  if ((long long)tiles * nbatch > d.max_blocks) return fail(GPE_EINVAL, "reduction scratch too small");
  ProfScope ps(kernel_name("axis_x", sizeof(T) == 8, KIND == LK_CPLX, EPI, G.M * nbatch), st);
  GPE_CUDA(launch_pdl(k_axis_x<T, KIND, EPI, LF>, nbatch * tiles, NT, smem, st, G, D, tiles, groups, slots));
  return GPE_OK;
}

#define GPE_LF_SWITCH(lf, CALL)                    \
  switch (lf) {                                    \
    case 5: return CALL(5);                        \
    case 6: return CALL(6);                        \
    case 7: return CALL(7);                        \
    case 8: return CALL(8);                        \
    case 9: return CALL(9);                        \
    case 10: return CALL(10);                      \
  }                                                \
  return fail(GPE_EINVAL, "unsupported line length")

template <typename T>
gpe_status launch_axis_s(const GridHost& g, const GridDev<T>& d, int axis, const PassData<T>& D, cudaStream_t st) {
  const int lf = ilog2(g.F[axis]), nb = g.nbatch;
  const int kind = line_kind(g);
  if (kind == LK_CPLX) {
#define GPE_CALL(L) launch_axis_s_t<T, LK_CPLX, L>(d, axis, D, nb, st)
    GPE_LF_SWITCH(lf, GPE_CALL);
#undef GPE_CALL
  }
  if (kind == LK_REAL) {
#define GPE_CALL(L) launch_axis_s_t<T, LK_REAL, L>(d, axis, D, nb, st)
    GPE_LF_SWITCH(lf, GPE_CALL);
#undef GPE_CALL
  }
#define GPE_CALL(L) launch_axis_s_t<T, LK_SINE, L>(d, axis, D, nb, st)
  GPE_LF_SWITCH(lf, GPE_CALL);
#undef GPE_CALL
}

template <typename T, int EPI>
gpe_status launch_axis_x(const GridHost& g, const GridDev<T>& d, const PassData<T>& D, cudaStream_t st) {
  const int lf = ilog2(g.F[0]), nb = g.nbatch;
  const int kind = line_kind(g);
  if (kind == LK_CPLX) {
#define GPE_CALL(L) launch_axis_x_t<T, LK_CPLX, EPI, L>(d, D, nb, st)
    GPE_LF_SWITCH(lf, GPE_CALL);
#undef GPE_CALL
  }
  if (kind == LK_REAL) {
#define GPE_CALL(L) launch_axis_x_t<T, LK_REAL, EPI, L>(d, D, nb, st)
    GPE_LF_SWITCH(lf, GPE_CALL);
#undef GPE_CALL
  }
#define GPE_CALL(L) launch_axis_x_t<T, LK_SINE, EPI, L>(d, D, nb, st)
  GPE_LF_SWITCH(lf, GPE_CALL);
#undef GPE_CALL
}

}  // namespace gpe
