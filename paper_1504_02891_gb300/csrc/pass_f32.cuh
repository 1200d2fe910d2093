// pass_f32.cuh -- the general axis pass (ops_impl.cuh) of float32 gradients, one
// kernel per transform length and line direction.
//
// Float32 gradients keep the arithmetic of the general pass to the last bit
// (see axis_x_takes), so what can be saved is around it: the general kernel
// carries every radix, both line directions and the solver's operands, and its
// warps wait for instruction fetches first of all.  Here the length and the
// direction are constants, the radix schedule is unrolled, only the gradient's
// operands are left, and the constant part comes before the wait for the kernel
// ahead.  64^3 rotating complex gradient: 36 -> 17 us (46 with its reduction
// and plain launches), the same bits.
#pragma once
#include "ops_launch.cuh"

namespace gpe {

// fft_run with the length known: the same stages in the same order.
template <int LOGF, int LOGNS, int ST, typename C, typename Post>
__device__ __forceinline__ C* fft_run_s(C* src, C* dst, int nl, int P, const C* tw, Post& post) {
  constexpr int S = (LOGF + 3) >> 2, base = LOGF / S, extra = LOGF % S;
  if constexpr (ST == S) {
    return src;
  } else {
    constexpr int lr = base + (ST < extra ? 1 : 0);
    fft_stage<C, lr>(src, dst, LOGF, LOGNS, nl, P, tw, ST == S - 1, post);
    __syncthreads();
    return fft_run_s<LOGF, LOGNS + lr, ST + 1>(dst, src, nl, P, tw, post);
  }
}

template <bool CPLX, int EPI, int LOGF, bool AX0>
__global__ void __launch_bounds__(NTHREADS) k_pass_s(PassGeom<float> G, PassData<float> D) {
  using T = float;
  using C = float2;
  using V = typename VT<T, CPLX>::V;
  constexpr int F = 1 << LOGF;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ long long s_off[MAXLB];
  __shared__ T s_rc[MAXLB];
  const int Pt = G.P, nt = blockDim.x, tid = threadIdx.x, len = G.len, LB = G.LB;
  const int inst = blockIdx.x / G.tiles;
  const int tile = blockIdx.x - inst * G.tiles;
  C* tw_s = reinterpret_cast<C*>(smem_raw);
  C* buf0 = tw_s + F;
  C* buf1 = buf0 + G.LC * Pt;
  V* st0 = reinterpret_cast<V*>(buf1 + G.LC * Pt);
  V* st2 = st0 + LB * len;
  const V* xin = (const V*)D.x;
  const V* accin = (const V*)D.acc_in;
  T* stv = reinterpret_cast<T*>(st2 + (accin ? LB * len : 0));
  const long long vbase = (long long)inst * G.M;
  // constants first: line offsets, rotation coordinates, twiddles, zeroed rows
  for (int l = tid; l < LB; l += nt) {
    long long b;
    int ri;
    bool ok;
    if constexpr (AX0) {
      const long long r = (long long)tile * LB + l;
      ok = r < (long long)G.n1 * G.n2;
      b = inst * G.M + r * G.n0;
      ri = (int)(r % G.n1);
    } else {
      const int o = tile / G.xt, x = (tile - o * G.xt) * LB + l;
      ok = x < G.n0;
      b = inst * G.M + (long long)o * G.ostride + x;
      ri = x;
    }
    s_off[l] = ok ? b : -1;
    if (G.rcoord) s_rc[l] = G.rcoord[ok ? ri : 0];
  }
  for (int i = tid; i < F; i += nt) cp_async(tw_s + i, G.tw + i);
  for (int i = tid; i < G.LC * Pt; i += nt) buf0[i] = make_float2(0.f, 0.f);
  pdl_next();
  pdl_wait();
  __syncthreads();
  // the data of the tile: fn(line, point, offset, staging slot)
  auto visit = [&](auto&& fn) {
    if constexpr (AX0) {
      const int lps = nt >> G.ltpl;
      for (int l = tid >> G.ltpl; l < LB; l += lps) {
        const long long off = s_off[l];
        if (off < 0) continue;
        for (int j = tid & (G.tpl - 1); j < len; j += G.tpl) fn(l, j, off + j, l * len + j);
      }
    } else {
      const int nval = LB * len;
      for (int f = tid; f < nval; f += nt) {
        const int l = f & (LB - 1), j = f >> G.logLB;
        const long long off = s_off[l];
        if (off < 0) continue;
        fn(l, j, off + (long long)j * G.stride, f);
      }
    }
  };
  visit([&](int, int, long long gi, int q) {
    cp_async(st0 + q, xin + gi);
    if (accin) cp_async(st2 + q, accin + gi);
    if (EPI != EPI_ACC) cp_async(stv + q, D.V + (gi - vbase));
  });
  cp_async_wait_all();
  __syncthreads();
  const int odd = G.odd_ext;
  visit([&](int l, int j, long long, int q) {
    const V v = st0[q];
    const int m = odd ? j + 1 : j;
    if constexpr (CPLX) {
      C* row = buf0 + l * Pt;
      row[pidx(m)] = v;
      if (odd) row[pidx(F - m)] = -v;
    } else {
      T* row = reinterpret_cast<T*>(buf0 + (l >> 1) * Pt);
      const int comp = l & 1;
      row[2 * pidx(m) + comp] = v;
      if (odd) row[2 * pidx(F - m) + comp] = -v;
    }
  });
  __syncthreads();
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
  PostNone none;
  C* r = fft_run_s<LOGF, 0, 0>(buf0, buf1, G.LC, Pt, tw_s, symbol);
  C* o = fft_run_s<LOGF, 0, 0>(r, r == buf0 ? buf1 : buf0, G.LC, Pt, tw_s, none);
  EpiCtx<T, CPLX> E;
  if (EPI != EPI_ACC) make_ctx<T, CPLX, EPI, false>(E, D);
  DF acc[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) acc_zero(acc[q]);
  T amax = T(0);
  visit([&](int l, int j, long long gi, int q) {
    const int m = odd ? j + 1 : j;
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
    epilogue_point<T, CPLX, EPI, false>(E, gi, x, lin, acc, amax);
  });
  if (EPI == EPI_ACC || D.nq == 0) return;
  run_control<T>(D, reduce_partials(acc, amax, D.nq, D.partials, D.results, D.ticket, G.tiles));
}

template <bool CPLX, int EPI, int LOGF, bool AX0>
static gpe_status launch_pass_s_t(const PassGeom<float>& G, int blocks, const PassData<float>& D, size_t smem,
                                  cudaStream_t st) {
  GPE_CUDA(raise_smem((const void*)k_pass_s<CPLX, EPI, LOGF, AX0>, smem));
  ProfScope ps(kernel_name("pass", 0, CPLX, EPI, G.M * (blocks / G.tiles)), st);
  GPE_CUDA(launch_pdl(k_pass_s<CPLX, EPI, LOGF, AX0>, blocks, G.nthreads, smem, st, G, D));
  return GPE_OK;
}

template <bool CPLX, int EPI>
gpe_status launch_pass_s(const PassGeom<float>& G, int blocks, const PassData<float>& D, size_t smem,
                         cudaStream_t st) {
#define GPE_CASE(L)                                                                          \
  case L:                                                                                    \
    return G.axis == 0 ? launch_pass_s_t<CPLX, EPI, L, true>(G, blocks, D, smem, st)         \
                       : launch_pass_s_t<CPLX, EPI, L, false>(G, blocks, D, smem, st);
  switch (G.logF) {
    GPE_CASE(5)
    GPE_CASE(6)
    GPE_CASE(7)
    GPE_CASE(8)
    GPE_CASE(9)
    GPE_CASE(10)
  }
#undef GPE_CASE
  return fail(GPE_EINVAL, "unsupported line length");
}

}  // namespace gpe
