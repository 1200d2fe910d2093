// fixfft.cuh -- the float64 line operator of the line kernels, carried out in
// 64-bit fixed point on the integer units (the Eq. fftp36 / Eq. fftp35
// transforms with the line symbol of Eq. energy-discrete-FP in between).
//
// Why: a GB300 SM issues 2 float64 operations per clock, 64 widening 32-bit
// multiply-adds and 64 64-bit additions (measured: 0.57, 17.4 and 18.5 T/s).
// A 512-point line operator costs 2 x 45 float64 operations per point, 45
// clocks of an SM; in fixed point about 540 instructions, 4.5 clocks.  The
// Hessian-vector product on one 512^2 complex grid went from 90 to 37 us (y
// kernel 38 -> 13, x kernel 46 -> 21: its pointwise part stays float64 and
// takes 40% of the kernel's float64 issue slots); what is left is the latency
// of 7 warps per SM, issuing in a quarter to a third of the cycles.  Errors
// against extended-precision sums (sampled points, 64^2 to 1024^2, smooth,
// noisy and spiky fields) are 0.06 to 1.0 of the float64 transforms'.
//
// Scaling (units are powers of two per line; every bound below is on moduli).
// A product by a twiddle of a radix-8 stage drops 2 bits (the top 64 of the
// 126-bit product: no shifts), and so do its untwiddled partners.  Forward: a
// value after n of the line's points have been summed is at most n max and at
// most the line's sum(|re| + |im|) = L1, so the input level m (max < 2^m) is
// the highest that keeps every stage and the spectrum X below 2^62.  Symbol: a
// 62-bit fraction of a power of two 2^es >= max |symbol|, lowered by k bits.
// Inverse: a partial sum of symbol X over n frequencies, every F/n-th one, is
// the line's product with the sum of symbol(p) e^{-2 pi i p m / F} over them, by
// Cauchy-Schwarz at most
//   sqrt(n F) sigma_n ||x||_2,   ||x||_2^2 <= max(|re|, |im|) L1,
// sigma_n the root mean square of the symbol a p^2 + c p over those frequencies
// (p in [-1, 1)).  k keeps this below 2^62 with a common
// sigma^2 = 0.21 a^2 + 0.34 c^2 for all of them.  sigma_n^2 is at most 1.03 (n >=
// 64), 1.09 (32), 1.5 (8) and 2.17 (4) times that, all with a c < 0 and the
// Nyquist frequency among the n (over all offsets, F = 32 to 1024), so values
// stay below 2^62.3 between stages, and a sum of the two parts of a four-term
// sum inside a radix-8 butterfly below 2^62.6; sums, halves and products hold
// up to 2^63.
// Rounding happens where bits are dropped, so it is about one unit of the
// largest spectrum value (2^-61 L1) per spectrum value, where float64
// transforms round every operation to 2^-53 of its own size.  Data and factor
// of a product are split into signed 32-bit halves; low x low (2^-62 of the
// result's bound) is dropped.  Lines that hold a NaN or an infinity return
// NaN.
#pragma once
#include "linefft.cuh"

namespace gpe {

// Complex fixed-point value.
using I2 = longlong2;
__device__ __forceinline__ I2 mkI2(long long x, long long y) {
  I2 r;
  r.x = x;
  r.y = y;
  return r;
}

// v = hi 2^32 + lo with lo a signed 32-bit number.
__device__ __forceinline__ void split_balanced(long long v, int& hi, int& lo) {
  lo = (int)v;
  hi = (int)(v >> 32) + (int)((unsigned int)lo >> 31);
}
// a b + c, one widening multiply-add
__device__ __forceinline__ long long madw(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ long long mulw(int a, int b) { return (long long)a * (long long)b; }

// a w / 2^62, w = (wh, wl) in balanced halves; |a| < 2^62.6.
__device__ __forceinline__ long long fix_mul(long long a, int wh, int wl) {
  int ah, al;
  split_balanced(a, ah, al);
  const long long mid = madw(ah, wl, madw(al, wh, 1LL << 29));
  return (long long)((unsigned long long)mulw(ah, wh) << 2) + (mid >> 30);
}
// Complex product by a twiddle w = (re hi, re lo, im hi, im lo); LOWER: a
// quarter of it.
template <bool LOWER>
__device__ __forceinline__ I2 fix_cmul(I2 a, int4 w) {
  int xh, xl, yh, yl;
  split_balanced(a.x, xh, xl);
  split_balanced(a.y, yh, yl);
  const int nz = -w.z, nw = -w.w;   // (the tables hold no -2^31)
  constexpr long long rnd = LOWER ? 1LL << 31 : 1LL << 29;
  const long long mr = madw(yl, nz, madw(yh, nw, madw(xl, w.x, madw(xh, w.y, rnd))));
  const long long mi = madw(yl, w.x, madw(yh, w.y, madw(xl, w.z, madw(xh, w.w, rnd))));
  if (LOWER) {
    return mkI2(madw(yh, nz, madw(xh, w.x, mr >> 32)), madw(yh, w.x, madw(xh, w.z, mi >> 32)));
  } else {
    const long long hr = madw(yh, nz, mulw(xh, w.x));
    const long long hi = madw(yh, w.x, mulw(xh, w.z));
    return mkI2((long long)((unsigned long long)hr << 2) + (mr >> 30),
                (long long)((unsigned long long)hi << 2) + (mi >> 30));
  }
}
// v / 4, rounded
__device__ __forceinline__ I2 fix_lower(I2 v) { return I2{(v.x + 2) >> 2, (v.y + 2) >> 2}; }

__device__ __forceinline__ I2 operator+(I2 a, I2 b) { return mkI2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ I2 operator-(I2 a, I2 b) { return mkI2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ I2 mul_mi(I2 v) { return mkI2(v.y, -v.x); }   // -i v

__device__ __forceinline__ void fix_dft2(I2& a, I2& b) {
  const I2 t = a;
  a = t + b;
  b = t - b;
}
__device__ __forceinline__ void fix_dft4(I2& v0, I2& v1, I2& v2, I2& v3) {
  const I2 s02 = v0 + v2, d02 = v0 - v2, s13 = v1 + v3, d13 = v1 - v3;
  v0 = s02 + s13;
  v2 = s02 - s13;
  v1 = mkI2(d02.x + d13.y, d02.y - d13.x);
  v3 = mkI2(d02.x - d13.y, d02.y + d13.x);
}
__device__ __forceinline__ void fix_dft8(I2* v) {
  // sqrt(1/2) as a 62-bit fraction in balanced halves
  constexpr long long R2 = 3260954456333195553LL;
  constexpr int R2H = (int)((R2 + 0x80000000LL) >> 32), R2L = (int)(unsigned int)(R2 & 0xffffffffLL);
  constexpr int NR2H = (int)((-R2 + 0x80000000LL) >> 32), NR2L = (int)(unsigned int)(-R2 & 0xffffffffLL);
  I2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  fix_dft4(e0, e1, e2, e3);
  fix_dft4(o0, o1, o2, o3);
  o1 = mkI2(fix_mul(o1.x + o1.y, R2H, R2L), fix_mul(o1.y - o1.x, R2H, R2L));
  o2 = mul_mi(o2);
  o3 = mkI2(fix_mul(o3.y - o3.x, R2H, R2L), fix_mul(o3.x + o3.y, NR2H, NR2L));
  v[0] = e0 + o0; v[4] = e0 - o0;
  v[1] = e1 + o1; v[5] = e1 - o1;
  v[2] = e2 + o2; v[6] = e2 - o2;
  v[3] = e3 + o3; v[7] = e3 - o3;
}

// Biased exponent of a double (1 for zero and subnormal values).
__device__ __forceinline__ int dexp(double v) {
  const int E = (__double2hiint(v) >> 20) & 0x7ff;
  return E > 0 ? E : 1;
}
// v 2^(base - Eref) of a finite v whose biased exponent is <= Eref, in units of
// its 53-bit mantissa's last place (base <= 9), rounded to the nearest integer.
__device__ __forceinline__ long long d2fix(double v, int Eref, int base) {
  const int hi = __double2hiint(v);
  const int E = (hi >> 20) & 0x7ff;
  const unsigned int mh = (unsigned int)(hi & 0xfffff) | (E > 0 ? 0x100000u : 0u);
  const unsigned long long m = (((unsigned long long)mh << 32) | (unsigned int)__double2loint(v)) << 10;
  const int r = min(10 - base + Eref - (E > 0 ? E : 1), 63);   // >= 1
  const long long f = (long long)((m + (1ull << (r - 1))) >> r);
  return hi < 0 ? -f : f;
}
// z 2^e rounded to double (|z| < 2^63).  Built in integer registers: two
// float64 additions and a multiplication would cost 1.5 clocks of the SM, this
// about 0.2.
__device__ __forceinline__ double fix2d(long long z, int e) {
  const int sgn = (int)(z >> 63);
  const unsigned long long a = (unsigned long long)((z ^ (long long)sgn) - (long long)sgn);
  const unsigned int ah = (unsigned int)(a >> 32), al = (unsigned int)a;
  const int lz = __clz((int)ah) - 1;                   // shift that brings the leading bit to bit 62
  const int E = 62 - lz + e + 1023;
  if (ah == 0u || (unsigned)(E - 1) > 2043u) return ldexp((double)z, e);   // small, subnormal or near overflow
  const unsigned int nh = __funnelshift_l(al, ah, lz), nl = al << lz;
  const unsigned long long n = (((unsigned long long)nh << 32) | nl) + 512ull;
  // bits 62..10 rounded to nearest: 53 bits with the leading one; a carry raises the exponent by itself
  const unsigned int lo = __funnelshift_r((unsigned int)n, (unsigned int)(n >> 32), 10);
  const unsigned int hi = (unsigned int)(n >> 42) + ((unsigned int)(E - 1) << 20);
  return __hiloint2double((int)(hi | ((unsigned int)sgn & 0x80000000u)), (int)lo);
}

// The largest biased exponent of a line's values and the sum of their
// magnitudes in units of 2^(Emax - 1023 - 19), rounded up.
struct LineMag {
  unsigned int E, S;
};
__device__ __forceinline__ LineMag mag_join(LineMag a, LineMag b) {
  LineMag r;
  r.E = max(a.E, b.E);
  const unsigned int da = min(r.E - a.E, 31u), db = min(r.E - b.E, 31u);
  r.S = (a.S >> da) + (b.S >> db) + (da | db ? 1u : 0u);
  return r;
}
__device__ __forceinline__ LineMag mag_shfl_xor(LineMag a, int o) {
  LineMag r;
  r.E = __shfl_xor_sync(0xffffffffu, a.E, o);
  r.S = __shfl_xor_sync(0xffffffffu, a.S, o);
  return r;
}

template <int LF>
struct LineFFT<double, LF> {
  using C = double2;
  using X = I2;                     // what the exchanges move
  using Tw = int4;                  // twiddle table entry
  static constexpr int F = 1 << LF;
  static constexpr int TPL = F / 8;
  static constexpr int N8 = LF / 3;
  static constexpr int TAIL = LF % 3;
  static constexpr int P = ((F + F / 16 + 15) & ~15) + 8;
  const Tw* tws;
  int j;

  __device__ __forceinline__ void init(int jj, const Tw* table) {
    j = jj;
    tws = table;
  }
  // 32-bit shared-memory addresses: generic pointers cost two instructions more per access
  static __device__ __forceinline__ void sts(unsigned int a, I2 v) {
    asm volatile("st.shared.v2.s64 [%0], {%1, %2};" ::"r"(a), "l"(v.x), "l"(v.y) : "memory");
  }
  static __device__ __forceinline__ I2 lds(unsigned int a) {
    I2 v;
    asm volatile("ld.shared.v2.s64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(a) : "memory");
    return v;
  }
  // bits a transform drops: 2 before every radix-8 stage but the first
  static constexpr int LOW = 2 * (N8 - 1);
  // The stages of the float32 transform (linefft.cuh).  One copy of the code
  // serves every radix-8 stage (and both transforms of apply()): unrolled, the
  // line operator was 95 KB of instructions that each warp runs once, and the
  // warps waited for instruction fetches (2/3 of the stalls).
  template <typename Ex>
  __device__ __forceinline__ void forward(I2 (&v)[8], const Ex& ex, int& par) const {
#pragma unroll 1
    for (int st = 0; st < N8; ++st) {
      const int k = j & ((1 << (3 * st)) - 1);
      if (st > 0) {
        const int kt = k << (LF - 3 - 3 * st);
        v[0] = fix_lower(v[0]);
#pragma unroll
        for (int r = 1; r < 8; ++r) v[r] = fix_cmul<true>(v[r], tws[r * kt]);
      }
      fix_dft8(v);
      if (st + 1 < N8 || TAIL) {
        const int mb = ((j - k) << 3) + k;
#pragma unroll
        for (int r = 0; r < 8; ++r) sts(ex.addr(par, mb + (r << (3 * st))), v[r]);
        ex.sync();
#pragma unroll
        for (int s = 0; s < 8; ++s) v[s] = lds(ex.addr(par, j + s * TPL));
        par ^= 1;
      }
    }
    if constexpr (TAIL == 2) {
#pragma unroll
      for (int r = 1; r < 4; ++r) {
        v[2 * r] = fix_cmul<false>(v[2 * r], tws[r * j]);
        v[2 * r + 1] = fix_cmul<false>(v[2 * r + 1], tws[r * (j + TPL)]);
      }
      fix_dft4(v[0], v[2], v[4], v[6]);
      fix_dft4(v[1], v[3], v[5], v[7]);
    } else if constexpr (TAIL == 1) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        v[u + 4] = fix_cmul<false>(v[u + 4], tws[j + u * TPL]);
        fix_dft2(v[u], v[u + 4]);
      }
    }
  }

  // A line in fixed point: its level (max < 2^m and L1 < 2^(m + l) in units of
  // 2^(E - 1075 - (m - 53))) and whether it is finite.
  struct Level {
    int E, m, l;
    bool finite;
  };
  template <typename Ex>
  __device__ __forceinline__ Level to_fixed(const double2 (&v)[8], I2 (&z)[8], const Ex& ex) const {
    LineMag mg;
    mg.E = 1;
#pragma unroll
    for (int s = 0; s < 8; ++s) mg.E = max(mg.E, (unsigned)max(dexp(v[s].x), dexp(v[s].y)));
    mg.S = 0;
    auto top = [&](double x) -> unsigned int {   // |x| in units of 2^(E - 1023 - 19), rounded up
      const int hi = __double2hiint(x);
      const unsigned int m = (((unsigned int)hi & 0xfffffu) | 0x100000u) >> 1;
      return (m >> min((int)mg.E - dexp(x), 31)) + 1u;
    };
#pragma unroll
    for (int s = 0; s < 8; ++s) mg.S += top(v[s].x) + top(v[s].y);
    mg = ex.join(mg);
    Level L;
    L.finite = mg.E < 2047;
    L.E = L.finite ? (int)mg.E : 1;
    const int b = 32 - __clz((int)mg.S);         // L1 < 2^(b + E - 1023 - 19)
    // a value is below 2^62 after one stage, after two, and in the spectrum
    L.l = b - 20;
    L.m = min(61, min(62 - min(4, L.l), 62 + LOW - L.l));
    if (N8 > 1) L.m = min(L.m, 64 - min(7, L.l));
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      z[s].x = L.finite ? d2fix(v[s].x, L.E, L.m - 53) : 0;
      z[s].y = L.finite ? d2fix(v[s].y, L.E, L.m - 53) : 0;
    }
    return L;
  }
  // Back to double, conjugated; the value of one unit is 2^e.
  static __device__ __forceinline__ void from_fixed(const I2 (&z)[8], double2 (&v)[8], int e, bool finite) {
    const double bad = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      v[s].x = finite ? fix2d(z[s].x, e) : bad;
      v[s].y = finite ? -fix2d(z[s].y, e) : bad;
    }
  }

  // T applied to the line (as LineFFT<float>::apply); ex.join(m) joins the
  // line's magnitudes over its threads.
  template <typename Ex>
  __device__ __forceinline__ void apply(double2 (&v)[8], const Ex& ex, int& par, const LineSym<double, F>& sym) const {
    I2 z[8];
    const Level L = to_fixed(v, z, ex);
    // symbol (a p^2 + c p) 2^es with |a| + |c| <= 1, p in units of F/2
    const double pm = (double)(F / 2);
    const double a = sym.c2 * (sym.dl * pm) * (sym.dl * pm), c = sym.c1c * (sym.dl * pm);
    const bool rot = c != 0.0;
    const int es = dexp(fabs(a) + fabs(c)) - 1022;
    // F sigma^2 ||x||_2^2 <= 2^R2 in the spectrum's units; sigma^2 is a^2/5 + c^2/3
    // (the mean square over p in [-1, 1)) and a little more.  Later radix-8
    // stages grow by 1.5 bits and drop 2
    const int R2 = LF + (L.m - LOW) + (L.m + L.l - LOW) + dexp(0.21 * a * a + 0.34 * c * c) - 1022 - 2 * es;
    const int k = max(0, max((R2 + 4) >> 1, ((R2 + LF + 1) >> 1) - LOW) - 62);
    // a, c as fractions of 2^(62 - k): mantissas shifted from 2^(E - 1075)
    int ah, al, ch, cl;
    split_balanced(d2fix(a, es + 1022, 9 - k), ah, al);
    split_balanced(d2fix(c, es + 1022, 9 - k), ch, cl);
    constexpr int S2 = 2 * LF - 2, S1 = LF - 1;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      forward(z, ex, par);
      if (pass == 0) {
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          const int m = j + s * TPL;
          const int p = m < (F >> 1) ? m : m - F;
          const int p2 = p * p;
          long long f = (long long)((unsigned long long)mulw(ah, p2) << (32 - S2)) + (mulw(al, p2) >> S2);
          if (rot)
            f += (long long)((unsigned long long)mulw(ch, p) << (32 - S1)) + (mulw(cl, p) >> S1);
          int fh, fl;
          split_balanced(f, fh, fl);
          z[s].x = fix_mul(z[s].x, fh, fl);
          z[s].y = -fix_mul(z[s].y, fh, fl);
        }
      }
    }
    // value of one unit: the line's, the bits dropped, the symbol's 2^es
    from_fixed(z, v, L.E - 1075 - (L.m - 53) + 2 * LOW + es + k, L.finite);
  }

  // The line's midpoint values (prolong.cuh): forward transform, mode p times
  // e^{i pi p / F}, inverse transform; fine: the table of 2F points.
  template <typename Ex>
  __device__ __forceinline__ void midpoints(double2 (&v)[8], const Ex& ex, int& par, const Tw* __restrict__ fine) const {
    I2 z[8];
    const Level L = to_fixed(v, z, ex);
    const int R2 = LF + (L.m - LOW) + (L.m + L.l - LOW);   // unit symbol
    const int k = max(0, max((R2 + 4) >> 1, ((R2 + LF + 1) >> 1) - LOW) - 62);
    const long long h = (1LL << k) >> 1;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      forward(z, ex, par);
      if (pass == 0) {
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          const int m = j + s * TPL;
          const int p = m < (F >> 1) ? m : m - F;
          const I2 c = fix_cmul<false>(mkI2(z[s].x, -z[s].y), ld_const(fine + (p & (2 * F - 1))));
          const bool nyq = m == (F >> 1);
          z[s] = mkI2(nyq ? 0 : (c.x + h) >> k, nyq ? 0 : (c.y + h) >> k);
        }
      }
    }
    from_fixed(z, v, L.E - 1075 - (L.m - 53) + 2 * LOW + k - LF, L.finite);
  }
};

}  // namespace gpe
