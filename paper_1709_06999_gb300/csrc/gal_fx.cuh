// 64-bit fixed-point arithmetic of the double-precision path.
//
// GB300 issues two FP64 operations per clock and SM (measured: 0.62e12 fused
// multiply-adds per second), but 64 integer additions and 32 multiply-adds of
// 32 x 32 -> 64 bits (7.6e12 per second measured).  A double transform is
// therefore done on integers: the values of one sequence share one power of
// two (a block exponent), chosen from the sum of their magnitudes so that no
// partial sum of the transform can overflow, and keep 60 bits below that sum.
// A double keeps 53 bits below each value, so this is no less precise: every
// rounding of the transform is at 2^-60 of a bound on its outputs.  Inputs and
// outputs in memory stay doubles.
//
// A complex product by a unit-modulus factor takes 12 multiply-adds (three
// 32 x 32 products per real product: high x high and the two cross terms, the
// low x low term being below the last bit).
#pragma once

#include "gal_common.cuh"
#include "gal_fft2.cuh"
#include "gal_fft3.cuh"

namespace gal {

// A factor of modulus at most 1: each component is h 2^32 + l in units of
// 2^-62, with a signed low digit l > -2^31 (so that digits can be negated).
struct __align__(16) fxtw {
  int xh, xl, yh, yl;
};

__host__ __device__ __forceinline__ void fx_digits(long long q, int& h, int& l) {
  l = (int)q;
  if (l == (int)0x80000000) {  // one unit of 2^-62 off: the digit must be negatable
    q += 1;
    l += 1;
  }
  h = (int)((q - l) >> 32);
}
__device__ __forceinline__ fxtw fx_factor(double x, double y) {  // |x|, |y| <= 1
  constexpr double k62 = 4611686018427387904.0;
  fxtw w;
  fx_digits(__double2ll_rn(x * k62), w.xh, w.xl);
  fx_digits(__double2ll_rn(y * k62), w.yh, w.yl);
  return w;
}

__device__ __forceinline__ long long madw(int a, int b, long long c) {
  return (long long)a * (long long)b + c;
}
// a = h 2^32 + l with a signed low digit
__device__ __forceinline__ void fx_split(long long a, int& h, int& l) {
  l = (int)a;
  h = (int)(a >> 32) + (int)((unsigned)l >> 31);
}
constexpr long long kFxHalf = 0x80000000ll;  // rounds the cross terms to nearest

// hi 64 bits of a w (a |a| < 2^61, w in units of 2^-62): a w / 4
__device__ __forceinline__ long long fx_mul_q(long long a, int wh, int wl) {
  int h, l;
  fx_split(a, h, l);
  const long long c = madw(h, wl, madw(l, wh, kFxHalf));
  return madw(h, wh, c >> 32);
}
__device__ __forceinline__ long long fx_mul(long long a, int wh, int wl) {
  return fx_mul_q(a, wh, wl) << 2;
}

// a w / 4 for complex a (components below 2^62, modulus below 2^61.5)
__device__ __forceinline__ fx2 fx_cmul_q(fx2 a, const fxtw& w) {
  int xh, xl, yh, yl;
  fx_split(a.x, xh, xl);
  fx_split(a.y, yh, yl);
  const long long cr = madw(yh, -w.yl, madw(yl, -w.yh, madw(xh, w.xl, madw(xl, w.xh, kFxHalf))));
  const long long ci = madw(yh, w.xl, madw(yl, w.xh, madw(xh, w.yl, madw(xl, w.yh, kFxHalf))));
  return fx2{madw(yh, -w.yh, madw(xh, w.xh, cr >> 32)), madw(yh, w.xh, madw(xh, w.yh, ci >> 32))};
}
__device__ __forceinline__ fx2 cmul(fx2 a, const fxtw& w) {
  const fx2 p = fx_cmul_q(a, w);
  return fx2{p.x << 2, p.y << 2};
}
__device__ __forceinline__ fxtw cconj(const fxtw& w) { return fxtw{w.xh, w.xl, -w.yh, -w.yl}; }
__device__ __forceinline__ fxtw ldg_tw(const fxtw* p) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(p));
  return fxtw{v.x, v.y, v.z, v.w};
}
// x / sqrt 2 (bfly8): 2^61.5 to the nearest, in digits
template <> __device__ __forceinline__ long long mul_sqrt_half<long long>(long long x) {
  return fx_mul(x, 0x2D413CCD, -25716447);
}

// ---------------------------------------------------------------------------
// doubles to a common power of two and back
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned shr_clamp(unsigned v, int n) {  // 0 for n >= 32
  unsigned r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
  return r;
}
__device__ __forceinline__ unsigned long long shr64_clamp(unsigned long long v, int n) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}
__device__ __forceinline__ unsigned long long shl64_clamp(unsigned long long v, int n) {
  unsigned long long r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}
// biased exponent (at least 1) and the 53-bit significand of |x| = m 2^(e - 1075)
__device__ __forceinline__ unsigned long long fx_mant(double x, int& e) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int be = (int)((hi >> 20) & 0x7ffu);
  const unsigned mh = (hi & 0xfffffu) + ((unsigned)min(be, 1) << 20);
  e = max(be, 1);
  return ((unsigned long long)mh << 32) | lo;
}
__device__ __forceinline__ long long fx_sign(long long v, double x) {
  const long long s = (long long)(__double2hiint(x) >> 31);
  return (v ^ s) - s;
}
// bits of |x| that order like its exponent
__device__ __forceinline__ unsigned fx_ebits(double x) {
  return (unsigned)__double2hiint(x) & 0x7fffffffu;
}
// |x| rounded up, in units of 2^(E - 1040), E >= its exponent: at most 2^18 + 1
__device__ __forceinline__ unsigned fx_ceil_units(double x, int E) {
  const unsigned hi = (unsigned)__double2hiint(x);
  const int be = (int)((hi >> 20) & 0x7ffu);
  const unsigned mh = (hi & 0xfffffu) + ((unsigned)min(be, 1) << 20);
  return shr_clamp(mh, E - max(be, 1) + 3) + 1u;
}

// Block exponent of a sequence: E is its largest biased exponent (>= 1), T the
// sum of fx_ceil_units over its real values.  The sum of magnitudes is then
// below 2^(bits + E - 1040); fixed-point value f stands for f 2^q, with every
// partial sum of the transform below 2^60.
struct FxScale {
  int D;     // right shift of a 63-bit significand of exponent e: D - e
  int q;     // exponent of one unit
  bool bad;  // the sequence holds an infinity or a NaN
};
__device__ __forceinline__ FxScale fx_scale(int E, unsigned T) {
  const int bits = max(32 - __clz((int)T), 16);
  return FxScale{bits + E - 15, bits + E - 1100, E >= 0x7ff};
}
__device__ __forceinline__ long long fx_from(double x, const FxScale& s) {
  int e;
  const unsigned long long m = fx_mant(x, e);
  return fx_sign((long long)((shr64_clamp(m << 10, s.D - e - 1) + 1ull) >> 1), x);
}
// v 2^q, rounded once (twice only where the result is subnormal)
__device__ __forceinline__ double fx_to(long long v, int q) {
  const double y = __ll2double_rn(v);
  if (q >= -1021 && q <= 959)  // 1 <= |y| < 2^63 or y = 0: the exponent cannot leave its field
    return v ? __hiloint2double(__double2hiint(y) + (q << 20), __double2loint(y)) : 0.0;
  const int a = q / 2, b = q - a;
  return y * __hiloint2double((1023 + a) << 20, 0) * __hiloint2double((1023 + b) << 20, 0);
}
__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

// ---------------------------------------------------------------------------
// The transform: the Stockham plan of gal_fft3.cuh at radix 8, with its staged
// factors in digits.  TAB: those of the stages before the last come from a copy in
// shared memory (the first fx_ntab entries of the table); otherwise through L1.
// The copy pays for rows of 1024 points and more, whose blocks have many (4096^2
// image 277 against 281 us a call, 2048^2 98.6 against 100.6), and for columns of
// 2048 and more, where it is made while the row pass ends (4096^2 277.6 against
// 280.3); shorter ones do without (256 image 26.4 against 24.6, 1024 profile 82.4
// against 81.7).
// ---------------------------------------------------------------------------
template <int L, int LMIN> constexpr int fx_ntab() {
  return L >= LMIN ? ipowc(8, P3<L, 8>::nstage - 1) - 8 : 0;
}

template <int L, int ST, bool TAB> struct FxHead {
  using P = P3<L, 8>;
  static __device__ __forceinline__ void run(fx2 (&v)[8], fx2* A, fx2* B, int t,
                                             const fxtw* tws) {
    if constexpr (ST < P::nstage - 1) {
      constexpr int T = P::T, Ns = ipowc(8, ST);
      fx2* in = (ST % 2 == 1) ? A : B;
      fx2* out = (ST % 2 == 0) ? A : B;
      const int k = t & (Ns - 1);
      if constexpr (ST > 0) {
        const fxtw* w = tws + (Ns - 8) + k;
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = in[pad3<8>(t + r * T)];
        if constexpr (TAB) {
#pragma unroll
          for (int r = 1; r < 8; ++r) v[r] = cmul(v[r], w[(r - 1) * Ns]);
        } else {
#pragma unroll
          for (int r = 1; r < 8; ++r) v[r] = cmul(v[r], ldg_tw(w + (r - 1) * Ns));
        }
      }
      bfly8(v);
      const int base = ST == 0 ? 9 * t : pad3<8>((t - k) * 8 + k);
#pragma unroll
      for (int r = 0; r < 8; ++r) out[ST == 0 ? base + r : base + r * pad_step<8>(Ns)] = v[r];
      __syncthreads();
      FxHead<L, ST + 1, TAB>::run(v, A, B, t, tws);
    }
  }
};

// last stage, complete: v[q R + r] <- X[t + q T + r L / R]
template <int L>
__device__ __forceinline__ void fx_last_full(fx2 (&v)[8], const fx2* in, int t,
                                             const fxtw* __restrict__ tws) {
  using P = P3<L, 8>;
  constexpr int R = P::rlast, T = P::T;
  if constexpr (P::nstage == 1) {
    bflyR<8>(v);
  } else {
#pragma unroll
    for (int q = 0; q < 8 / R; ++q) {
      const int b = t + q * T;
#pragma unroll
      for (int r = 0; r < R; ++r) v[q * R + r] = in[pad3<8>(b + r * (L / R))];
#pragma unroll
      for (int r = 1; r < R; ++r) 
        v[q * R + r] = cmul(v[q * R + r], ldg_tw(tws + (P::Nsl - 8) + (r - 1) * P::Nsl + b));
      bflyR<R>(&v[q * R]);
    }
  }
}

// X[j] and X[L - j] only (pruned_pair3)
template <int L>
__device__ __forceinline__ void fx_pruned_pair(const fx2* in, int j, const fxtw* __restrict__ tws,
                                               fx2& xj, fx2& xmj) {
  using P = P3<L, 8>;
  constexpr int R = P::rlast, Ns = P::Nsl;
  const int jb = j == 0 ? Ns : j;
  const int ba = pad3<8>(j), bb = -jb + ((-jb) >> P::lv);
  fx2 a = in[ba], b = in[bb + pad_step<8>(Ns)];
#pragma unroll
  for (int r = 1; r < R; ++r) {
    const fxtw w = ldg_tw(tws + (Ns - 8) + (r - 1) * Ns + j);
    a = cadd(a, cmul(in[ba + r * pad_step<8>(Ns)], w));
    b = cadd(b, cmul(in[bb + (r + 1) * pad_step<8>(Ns)], cconj(w)));
  }
  xj = a;
  xmj = j == 0 ? a : b;
}

// 2 X_k of a real row from the bins Z_k, Z_{M-k} of its packed transform
// (r2c_unpack without the halving, which goes into the exponent)
__device__ __forceinline__ fx2 fx_r2c_unpack2(fx2 zk, fx2 zmk, const fxtw& w) {
  const fx2 b = cconj(zmk);
  return cadd(cadd(zk, b), cmul(cmul_mi(csub(zk, b)), w));
}

// Largest and sum over the TT threads of one sequence (threads t0 .. t0+TT-1
// of the block, TT a power of two); `red` holds one value per warp.  Every
// thread of the block calls it; it synchronises when a sequence spans warps.
template <int TT, bool MAX> __device__ __forceinline__ unsigned fx_group(unsigned x, unsigned* red) {
  auto op = [](unsigned a, unsigned b) { return MAX ? max(a, b) : a + b; };
  if constexpr (TT >= 32) {
    x = MAX ? __reduce_max_sync(0xffffffffu, x) : __reduce_add_sync(0xffffffffu, x);
    if constexpr (TT > 32) {
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
      __syncthreads();
      const int w0 = (threadIdx.x / TT) * (TT / 32);
      x = red[w0];
#pragma unroll
      for (int i = 1; i < TT / 32; ++i) x = op(x, red[w0 + i]);
    }
  } else {
#pragma unroll
    for (int o = TT / 2; o > 0; o >>= 1) x = op(x, __shfl_xor_sync(0xffffffffu, x, o));
  }
  return x;
}

// The values z of this thread's sequence to fixed point; returns its scale.
template <int TT>
__device__ __forceinline__ FxScale fx_load(const double2 (&z)[8], fx2 (&v)[8], unsigned* red_max,
                                           unsigned* red_sum) {
  unsigned h = 0;
#pragma unroll
  for (int r = 0; r < 8; ++r) h = max(h, max(fx_ebits(z[r].x), fx_ebits(z[r].y)));
  const int E = max((int)(fx_group<TT, true>(h, red_max) >> 20), 1);
  unsigned s = 0;
#pragma unroll
  for (int r = 0; r < 8; ++r) s += fx_ceil_units(z[r].x, E) + fx_ceil_units(z[r].y, E);
  const FxScale sc = fx_scale(E, fx_group<TT, false>(s, red_sum));
#pragma unroll
  for (int r = 0; r < 8; ++r) v[r] = fx2{fx_from(z[r].x, sc), fx_from(z[r].y, sc)};
  return sc;
}

// ---------------------------------------------------------------------------
// Sampling: grid positions, phases and the bilinear stencil on integers, so
// that a point costs the FP64 pipe only its rotation, its phase argument and
// its chi-square term.
// ---------------------------------------------------------------------------
constexpr int kSinCos = 1024;  // table of W_1024^k = cos - i sin at k / 1024 turns
constexpr int kPosBits = 50;   // fraction bits of a grid position

// grid offset x in units of 2^-50, to nearest; |x| >= 4096 (beyond every grid) saturates
__device__ __forceinline__ long long fx_pos(double x) {
  int e;
  const unsigned long long m = fx_mant(x, e);
  const int d = 1035 - e;
  const long long f =
      d >= 1 ? (long long)((shr64_clamp(m << 10, d - 1) + 1ull) >> 1) : (1ll << 62);
  return fx_sign(f, x);
}
// x in turns modulo 1, in units of 2^-64
__device__ __forceinline__ unsigned long long fx_turns(double x) {
  int e;
  const unsigned long long m = fx_mant(x, e);
  const int s = e - 1011;
  return (unsigned long long)fx_sign(
      (long long)(s >= 0 ? shl64_clamp(m, s) : shr64_clamp(m, -s)), x);
}
__device__ __forceinline__ bool fx_isnan(double x) {  // results of arithmetic: quiet NaNs
  return fx_ebits(x) > 0x7ff00000u;
}
__device__ __forceinline__ bool fx_nonfinite(double x) { return fx_ebits(x) >= 0x7ff00000u; }

// cos and sin of p turns in units of 2^-62: the table entry nearest to p turned
// by the rest r, |r| <= pi / 1024, with 1 - cos r = r^2/2 - r^4/24 and sin r =
// r - r^3/6 + r^5/120 (the next terms are below 2^-59)
__device__ __forceinline__ fx2 fx_cos_sin(unsigned long long p, const fxtw* tab) {
  const unsigned i = (unsigned)((p + (1ull << 53)) >> 54);
  const long long R = (long long)(p - ((unsigned long long)i << 54)) << 9;
  const long long rho = fx_mul(R, 0x3243F6A9, -2007355251);  // r 2^70: times pi / 4
  int rh, rl;
  fx_split(rho, rh, rl);
  const long long q = madw(rh, rh, madw(rh, rl, 0) >> 31);  // r^2 2^76
  const unsigned z = (unsigned)(q >> 28);                   // r^2 2^48
  const unsigned z2 = __umulhi(z, z);                       // r^4 2^64
  const long long kap = (q - ((long long)__umulhi(z2, 178956971u) << 13)) >> 7;  // (1 - cos r) 2^70
  const unsigned g = (unsigned)(((unsigned long long)z * 715827883u) >> 29) -
                     (__umulhi(z2, 35791394u) >> 13);       // (r^2/6 - r^4/120) 2^51
  const long long sig = rho - (madw(rh, (int)(g >> 1), 0) >> 18);  // sin r 2^70
  const fxtw w = tab[i];
  const fx2 d = fx_cmul_q(fx2{kap, sig}, w);  // (kap C + sig S, sig C - kap S) 2^-2
  const long long C = ((long long)w.xh << 32) + w.xl, nS = ((long long)w.yh << 32) + w.yl;
  return fx2{C - ((d.x + 32) >> 6), ((d.y + 32) >> 6) - nS};
}

// Nodes of one cell at the power of two of the largest of their 8 values, E its
// biased exponent: 2^59 <= |largest| < 2^60, one unit 2^(E - 1082).
__device__ __forceinline__ long long fx_node(double x, int E) {
  int e;
  const unsigned long long m = fx_mant(x, e);
  return fx_sign((long long)shr64_clamp(m << 7, E - e), x);
}
__device__ __forceinline__ fx2 fx_lerp(fx2 a, fx2 b, int fh, int fl) {
  return fx2{a.x + fx_mul(b.x - a.x, fh, fl), a.y + fx_mul(b.y - a.y, fh, fl)};
}

}  // namespace gal
