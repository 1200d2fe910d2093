// persist_lines.cuh -- one cooperative launch runs a whole float32 Algorithm 1
// run (objective F, or the difference-form model of the subproblem) on square
// 2D and cubic 3D grids, with the register line transforms of lines3.cuh.
//
// Why: on these grids an iteration is a chain of latencies.  As kernels (one per
// axis, the last with the reduction and the control, queued in graphs of 16) it
// took 21-24 us on 64^2 to 256^2 complex grids and 28 us on 32^3 and 64^3
// grids, whatever the size; here a grid barrier stands between the axes, every
// CTA folds the partials and runs the control on its own copy (identical
// inputs, identical state, no broadcast), and tables and launches are paid
// once: 14-15 us and 20 us with everything else of a solve.  127^3 grids, where
// the passes themselves count, take the same time both ways (81 against 84 us).
//
// Every value that another CTA writes during the launch is read from L2
// (ld.global.cg); X^k, P_k, V and the tables are constant while it is resident
// (a cooperative launch has plain edges).  CTAs of 256 threads (128 on 256-point
// lines: chosen on 256^2 grids, where it gives 64 CTAs; 127^3 sine grids, whose
// lines are as long, were only measured with it) hold their threads / (F/8)
// complex lines, so 64^3 grids take one tile per CTA and axis.
#pragma once
#include "lines3.cuh"

namespace gpe {

struct PersistLinesArgs {
  PassGeom<float> G[3];
  int dim;
  PassData<float> D;        // slots, control block, partials
  float* acc;               // kinetic accumulator
  unsigned long long* bar;  // arrivals so far (zero at launch)
  int* err;                 // set when a barrier wait gave up
  long long max_polls;
  int max_loops;
  int width[3], tiles[3];   // strided axes: inner width, tiles per plane
  int total[3];             // tiles of all planes (axis 0: line groups)
};

template <int LF> __host__ __device__ constexpr int pl_threads() { return LF == 8 ? 128 : 256; }

// Grid barrier number n (from 1): every CTA adds one to the arrival count and
// waits until n times the grid has arrived.  Bounded: after max_polls polls the
// CTA sets *err and returns false, and so does every CTA that sees *err.
__device__ __forceinline__ bool pl_barrier(const PersistLinesArgs& P, unsigned long long n) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long want = n * gridDim.x;
    asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(P.bar) : "memory");
    int ok = 1;
    long long polls = 0;
    for (;;) {
      unsigned long long have;
      asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(have) : "l"(P.bar) : "memory");
      if (have >= want) break;
      if (*(volatile int*)P.err) {
        ok = 0;
        break;
      }
      if (++polls > P.max_polls) {
        atomicExch(P.err, 1);
        ok = 0;
        break;
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

template <int KIND, int EPI, int LF>
__global__ void __launch_bounds__(pl_threads<LF>()) k_alg1_lines(PersistLinesArgs P) {
  using T = float;
  using FFT = LineFFT<T, LF>;
  using C = float2;
  constexpr bool CPLX = KIND == LK_CPLX;
  using V = typename VT<T, CPLX>::V;
  constexpr int F = FFT::F, TPL = FFT::TPL, NT = pl_threads<LF>(), NL = NT / TPL, CW = NL;
  constexpr int NP = KIND == LK_SINE ? 4 : 8;    // data points per thread and line
  constexpr int NV = CPLX ? NP : 2 * NP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tws = reinterpret_cast<C*>(smem_raw);
  C* xb = tws + F;                               // exchange: [2][F][CW] or [2][NL][P]
  __shared__ Alg1CtlT<float> s_ctl;
  __shared__ double s_res[NQ];
  const int tid = threadIdx.x;
  load_table(tws, P.G[0].tw, F);                 // equal lines: one table for every axis
  if (tid == 0) ctl_copy(s_ctl, *P.D.ctl);
  __syncthreads();
  unsigned long long nbar = 0;
  auto writeback = [&]() {
    if (blockIdx.x == 0 && tid == 0) ctl_copy(*P.D.ctl, s_ctl);
  };
  const T* Vp = P.D.V;
  const V* xk = (const V*)P.D.base;
  V* acc = reinterpret_cast<V*>(P.acc);
  for (int loop = 0; loop < P.max_loops; ++loop) {
    if (s_ctl.done) break;
    const V* xc = (const V*)P.D.xs[s_ctl.cur];
    const V* gc = (const V*)P.D.gs[s_ctl.cur];
    V* yt = (V*)P.D.xs[s_ctl.trial];
    // the step: s(a X + b G), or in difference form (a - 1) X^k + a D + b G^
    const T sk = EPI == EPI_WS ? s_ctl.am1 : T(0);
    const T sa = EPI == EPI_WS ? s_ctl.a : s_ctl.s * s_ctl.a, sb = EPI == EPI_WS ? s_ctl.b : s_ctl.s * s_ctl.b;
    auto step_at = [&](long long i) -> V {
      V v = sa * __ldcg(xc + i) + sb * __ldcg(gc + i);
      if constexpr (EPI == EPI_WS) v = v + sk * __ldg(xk + i);
      return v;
    };
    for (int a = P.dim - 1; a > 0; --a) {
      const PassGeom<T>& G = P.G[a];
      const bool first = a == P.dim - 1;
      const int cl = tid & (CW - 1), j = tid / CW;
      FFT fft;
      fft.init(j, tws);
      int par = 0;
      ExCols<C, CW> ex{xb + cl, F * CW, nullptr};
      LineSym<T, F> sym;
      sym.c2 = G.c2;
      sym.dl = G.dlam;
      const int width = P.width[a];
      for (int t = blockIdx.x; t < P.total[a]; t += gridDim.x) {
        const int plane = t / P.tiles[a], tile = t - plane * P.tiles[a];
        const int c0 = CPLX ? tile * CW + cl : (KIND == LK_REAL ? 2 * (tile * CW + cl) : 2 * tile * CW + cl);
        const int c1 = KIND == LK_REAL ? c0 + 1 : c0 + CW;
        const bool in0 = c0 < width, in1 = !CPLX && c1 < width;
        const long long pbase = (long long)plane * G.len * width;
        auto off = [&](int s, int c) -> long long {
          return pbase + (long long)(j + s * TPL - (KIND == LK_SINE ? 1 : 0)) * width + c;
        };
        auto has = [&](int s) -> bool { return KIND != LK_SINE || s > 0 || j > 0; };
        C v[8];
        V a0[NP], a1[CPLX ? 1 : NP];
#pragma unroll
        for (int s = 0; s < NP; ++s) {
          V p = vzero<V>(), q = vzero<V>();
          if (has(s) && in0) p = first ? step_at(off(s, c0)) : __ldcg(yt + off(s, c0));
          if (has(s) && in1) q = first ? step_at(off(s, c1)) : __ldcg(yt + off(s, c1));
          if constexpr (CPLX) {
            v[s] = p;
          } else {
            v[s].x = p;
            v[s].y = q;
          }
          a0[s] = vzero<V>();
          if (!first && has(s) && in0) a0[s] = __ldcg(acc + off(s, c0));
          if constexpr (!CPLX) {
            a1[s] = vzero<V>();
            if (!first && has(s) && in1) a1[s] = __ldcg(acc + off(s, c1));
          }
        }
        if (first) {
#pragma unroll
          for (int s = 0; s < NP; ++s) {
            if (!has(s)) continue;
            if constexpr (CPLX) {
              if (in0) yt[off(s, c0)] = v[s];
            } else {
              if (in0) yt[off(s, c0)] = v[s].x;
              if (in1) yt[off(s, c1)] = v[s].y;
            }
          }
        }
        __syncthreads();   // the exchange buffers are reused
        if constexpr (KIND == LK_SINE) mirror_odd<T, LF>(v, ex, par, j);
        sym.c1c = (CPLX && G.rcoord && in0) ? G.c1 * G.rcoord[c0] : T(0);
        fft.apply(v, ex, par, sym);
#pragma unroll
        for (int s = 0; s < NP; ++s) {
          if (!has(s)) continue;
          if constexpr (CPLX) {
            if (in0) acc[off(s, c0)] = a0[s] + v[s];
          } else {
            if (in0) acc[off(s, c0)] = a0[s] + v[s].x;
            if (in1) acc[off(s, c1)] = a1[s] + v[s].y;
          }
        }
      }
      if (!pl_barrier(P, ++nbar)) {
        writeback();
        return;
      }
    }
    // x lines, epilogue, sums
    const PassGeom<T>& G = P.G[0];
    const int l = tid / TPL, j = tid & (TPL - 1);
    FFT fft;
    fft.init(j, tws);
    int par = 0;
    ExRow<C, FFT::P> ex{xb + l * FFT::P, NL * FFT::P, 1 + l, TPL, nullptr};
    EpiCtx<T, CPLX> E;
    E.out = (V*)P.D.gs[s_ctl.trial];
    E.xc = s_ctl.has_cur ? xc : nullptr;
    E.gc = s_ctl.has_cur ? gc : nullptr;
    E.base = xk;
    E.gk = (const V*)P.D.gk;
    E.nl = (T)s_ctl.alpha;
    E.shift = T(0);
    E.lin_scale = T(2);
    E.th_c = s_ctl.has_cur ? s_ctl.theta_c : s_ctl.theta_hint;
    E.delta = s_ctl.delta;
    E.thk = s_ctl.theta_ref;
    DF sums[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc_zero(sums[q]);
    T amax = T(0);
    const int rows = (int)(G.M / G.len);
    LineSym<T, F> sym;
    sym.c2 = G.c2;
    sym.dl = G.dlam;
    static_assert(TPL < 32 || (TPL % 32 == 0 && NL <= 15), "named barriers per line");
    for (int grp = blockIdx.x; grp < P.total[0]; grp += gridDim.x) {
      const int r0 = CPLX ? grp * NL + l : 2 * (grp * NL + l);
      auto has = [&](int q) -> bool { return r0 + q / NP < rows && (KIND != LK_SINE || q % NP > 0 || j > 0); };
      auto at = [&](int q) -> long long {
        return (long long)(r0 + q / NP) * G.len + j + (q % NP) * TPL - (KIND == LK_SINE ? 1 : 0);
      };
      V xv[NV], av[NV];
      T vv[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        xv[q] = vzero<V>();
        av[q] = vzero<V>();
        vv[q] = T(0);
        if (has(q)) {
          xv[q] = __ldcg(yt + at(q));
          av[q] = __ldcg(acc + at(q));
          vv[q] = ld_const(Vp + at(q));
        }
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
      ex.sync();   // the line's exchange rows are reused
      if constexpr (KIND == LK_SINE) mirror_odd<T, LF>(v, ex, par, j);
      sym.c1c = (CPLX && G.rcoord && r0 < rows) ? G.c1 * G.rcoord[r0 % G.n1] : T(0);
      fft.apply(v, ex, par, sym);
      // the point's other vectors, ahead of the stores of the epilogue
      V xcv[NV], gcv[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        xcv[q] = vzero<V>();
        gcv[q] = vzero<V>();
        if (has(q)) {
          xcv[q] = __ldcg(xc + at(q));
          gcv[q] = __ldcg(gc + at(q));
        }
      }
      E.xc = E.gc = nullptr;
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        if (!has(q)) continue;
        V kin;
        if constexpr (CPLX) kin = v[q];
        else kin = q < NP ? v[q % NP].x : v[q % NP].y;
        const V lin = (kin + av[q]) + vv[q] * xv[q];
        EpiOps<V, EPI> o;
        o.v[0] = xcv[q];
        o.v[1] = gcv[q];
        if constexpr (EPI == EPI_WS) {   // constant during the launch
          o.v[2] = __ldg(E.base + at(q));
          o.v[3] = __ldg(E.gk + at(q));
        }
        epilogue_apply<T, CPLX, EPI>(E, at(q), xv[q], lin, o, sums, amax, true);
      }
    }
    block_partial(sums, amax, NQ, P.D.partials + (size_t)blockIdx.x * NQ);
    if (!pl_barrier(P, ++nbar)) {
      writeback();
      return;
    }
    // every CTA folds the same rows in the same order and takes the same decisions
    fold_partials<DF>(P.D.partials, gridDim.x, 1, NQ, nullptr, s_res);
    if (tid == 0) alg1_control<float>(&s_ctl, s_res);
    // (the rows are rewritten only after the next iteration's first barrier)
    __syncthreads();
  }
  writeback();
}

template <int KIND, int EPI, int LF>
static gpe_status launch_alg1_lines_t(PersistLinesArgs& P, int* grid_only, cudaStream_t st) {
  using FFT = LineFFT<float, LF>;
  constexpr int NT = pl_threads<LF>(), NL = NT / FFT::TPL, CW = NL;
  const size_t smem = ((size_t)FFT::F + 2 * std::max((size_t)FFT::F * CW, (size_t)NL * FFT::P)) * sizeof(float2);
  static KernelShape shape;
  int occ = 0;
  GPE_CUDA(kernel_shape(shape, (const void*)k_alg1_lines<KIND, EPI, LF>, NT, smem, &occ));
  int most = 1;
  for (int a = 0; a < P.dim; ++a) {
    const PassGeom<float>& G = P.G[a];
    if (a == 0) {
      const long long rows = G.M / G.len, lines = KIND == LK_CPLX ? rows : (rows + 1) / 2;
      P.total[0] = (int)((lines + NL - 1) / NL);
    } else {
      const int cols = KIND == LK_CPLX ? CW : 2 * CW;
      P.width[a] = a == 1 ? G.n0 : G.n0 * G.n1;
      P.tiles[a] = (P.width[a] + cols - 1) / cols;
      P.total[a] = P.tiles[a] * (a == 1 ? G.n2 : 1);
    }
    most = std::max(most, P.total[a]);
  }
  const int grid = std::min(most, occ * num_sms());
  if (grid_only) {
    *grid_only = grid;
    return GPE_OK;
  }
  GPE_CUDA(cudaMemsetAsync(P.bar, 0, sizeof(unsigned long long), st));
  GPE_CUDA(cudaMemsetAsync(P.err, 0, sizeof(int), st));
  void* args[] = {&P};
  ProfScope ps(kernel_name("alg1_lines", 0, KIND == LK_CPLX, EPI, P.G[0].M), st);
  GPE_CUDA(cudaLaunchCooperativeKernel((const void*)k_alg1_lines<KIND, EPI, LF>, dim3(grid), dim3(NT), args, smem, st));
  return GPE_OK;
}

template <int KIND, int EPI>
static gpe_status launch_alg1_lines_k(PersistLinesArgs& P, int* grid_only, cudaStream_t st) {
  switch (P.G[0].logF) {
    case 6: return launch_alg1_lines_t<KIND, EPI, 6>(P, grid_only, st);
    case 7: return launch_alg1_lines_t<KIND, EPI, 7>(P, grid_only, st);
    case 8: return launch_alg1_lines_t<KIND, EPI, 8>(P, grid_only, st);
    case 9: return launch_alg1_lines_t<KIND, EPI, 9>(P, grid_only, st);
  }
  return fail(GPE_EINVAL, "unsupported line length");
}

// 2D and 3D grids whose lines have 64 to 512 transform points, the same on every
// axis.
bool alg1_lines_ok(const GridHost& g) {
  for (int a = 0; a < g.dim; ++a)
    if (!line_axis_ok(g, a) || g.F[a] != g.F[0] || g.F[a] < 64 || g.F[a] > 512) return false;
  return g.nbatch == 1 && g.dim >= 2;
}

gpe_status launch_alg1_lines(const GridHost& g, const GridDev<float>& d, const PassData<float>& D, void* acc,
                             unsigned int* bar, int* err, int max_loops, int epi, size_t cap_blocks, bool* launched,
                             cudaStream_t st) {
  *launched = false;
  if (!alg1_lines_ok(g)) return GPE_OK;
  PersistLinesArgs P{};
  for (int a = 0; a < g.dim; ++a) P.G[a] = d.geom[a];
  P.dim = g.dim;
  P.D = D;
  P.acc = static_cast<float*>(acc);
  P.bar = reinterpret_cast<unsigned long long*>(bar);
  P.err = err;
  P.max_loops = max_loops;
  P.max_polls = wait_limit(1LL << 22);
  const int kind = line_kind(g);
  auto go = [&](int* grid_only) -> gpe_status {
    if (epi == EPI_F) {
      if (kind == LK_CPLX) return launch_alg1_lines_k<LK_CPLX, EPI_F>(P, grid_only, st);
      if (kind == LK_REAL) return launch_alg1_lines_k<LK_REAL, EPI_F>(P, grid_only, st);
      return launch_alg1_lines_k<LK_SINE, EPI_F>(P, grid_only, st);
    }
    if (kind == LK_CPLX) return launch_alg1_lines_k<LK_CPLX, EPI_WS>(P, grid_only, st);
    if (kind == LK_REAL) return launch_alg1_lines_k<LK_REAL, EPI_WS>(P, grid_only, st);
    return launch_alg1_lines_k<LK_SINE, EPI_WS>(P, grid_only, st);
  };
  int grid = 0;
  gpe_status s = go(&grid);
  if (s != GPE_OK || (size_t)grid > cap_blocks) return s;
  s = go(nullptr);
  if (s == GPE_OK) *launched = true;
  return s;
}

}  // namespace gpe
