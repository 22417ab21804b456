// 64-bit fixed-point arithmetic of the double-precision path.
//
// GB300 issues two FP64 operations per clock and SM (measured: 0.62e12 fused
// multiply-adds per second), but 64 integer additions and 32 multiply-adds of
// 32 x 32 -> 64 bits (7.6e12 per second measured).  A double transform is
// therefore done on integers: the values of one sequence share one power of
// two (a block exponent) that grows with the transform.  After s stages of radix
// 8 a value is at most min(8^s largest modulus, sum of magnitudes), both known
// at the load; the values enter each stage below 2^60 of that bound, grow by up
// to 8 in its butterflies, and are shifted back, by as many bits as the bound
// grew, inside the next product.  Each stage thus rounds at 2^-60 of what the
// values can be at that stage: the largest inputs keep all 53 bits, and the
// roundings of the early stages are far below those of the last.  Inputs and
// outputs in memory stay doubles.
//
// Error against 64 bits, root mean square over the rms spectrum, after row and
// column pass within 24 cells of the origin (the same steps on a CPU against an
// extended-precision transform; the FP64 plan in brackets): noise 1.0e-16
// (2.9e-16) at 512^2, 1.2e-16 (3.3e-16) at 2048^2, 1.4e-16 (3.5e-16) at 4096^2;
// a smooth source 6.0e-17 (1.3e-16), 6.0e-17 (1.3e-16), 6.1e-17 (1.5e-16);
// positive random pixels 8.0e-17 (8.9e-17), 8.9e-17 (9.0e-17), 4.3e-17
// (4.4e-17).  One scale for all stages, taken from the sum, had 8.4e-16, 7.6e-15
// and 2.9e-14 for the noise, growing with the side.
//
// A complex product by a unit-modulus factor takes 12 multiply-adds (three
// 32 x 32 products per real product: high x high and the two cross terms, the
// low x low term being a quarter of the last bit at most where the values use
// all 63 bits, as in the stages).
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
// The staged factors of the transforms: the same in units of 2^-61, and 1 is one
// unit short.  A product by 1 is a shift, whose ties are frequent; rounded up
// like all others they would bias every value the same way, which adds up in the
// sums (24 times the other errors at the origin of a 4096^2 spectrum).  One unit
// less makes them round towards zero.
__device__ __forceinline__ fxtw fx_stage_factor(double x, double y) {
  constexpr long long one = 1ll << 61;
  auto units = [](double a) {
    const long long q = __double2ll_rn(a * (double)one);
    return q == one ? q - 1 : q == -one ? q + 1 : q;
  };
  fxtw w;
  fx_digits(units(x), w.xh, w.xl);
  fx_digits(units(y), w.yh, w.yl);
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

// hi 64 bits of a w (|a| < 2^62.5): a w / 4 for w in units of 2^-62
__device__ __forceinline__ long long fx_mul_q(long long a, int wh, int wl) {
  int h, l;
  fx_split(a, h, l);
  const long long c = madw(h, wl, madw(l, wh, kFxHalf));
  return madw(h, wh, c >> 32);
}
__device__ __forceinline__ long long fx_mul(long long a, int wh, int wl) {
  return fx_mul_q(a, wh, wl) << 2;
}

// a w / 4 for complex a (modulus below 2^62); for a staged factor (fx_stage_factor)
// a w / 8 (modulus below 2^63): the cross terms' sum stays below 2^63 either way
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
// x / sqrt 2 (bfly8), |x| < 2^62: 2^62.5 to the nearest, in digits
template <> __device__ __forceinline__ long long mul_sqrt_half<long long>(long long x) {
  return fx_mul_q(x << 1, 0x5A82799A, -51432894);
}
// a w 2^(p - 3) for a staged factor w; the modulus of a is below 2^(63 - p)
__device__ __forceinline__ fx2 fx_stage_mul(fx2 a, const fxtw& w, int p) {
  return fx_cmul_q(fx2{(long long)((unsigned long long)a.x << p), (long long)((unsigned long long)a.y << p)}, w);
}
// a / 2^g to the nearest, ties towards zero (see fx_stage_factor), 0 <= g <= 3
__device__ __forceinline__ long long fx_shr(long long a, int g) {
  const unsigned up = (unsigned)((unsigned long long)a >> 63) & (g > 0 ? 1u : 0u);
  return (long long)((unsigned long long)a + (unsigned)((((1 << g) - 1) >> 1) + up)) >> g;
}
__device__ __forceinline__ fx2 fx_shr(fx2 a, int g) { return fx2{fx_shr(a.x, g), fx_shr(a.y, g)}; }

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
// the double of high word hi rounded up, in units of 2^(E - 1040), E >= its
// exponent: at most 2^18 + 1
__device__ __forceinline__ unsigned fx_ceil_units(unsigned hi, int E) {
  const int be = (int)((hi >> 20) & 0x7ffu);
  const unsigned mh = (hi & 0xfffffu) + ((unsigned)min(be, 1) << 20);
  return shr_clamp(mh, E - max(be, 1) + 3) + 1u;
}

// Block exponent of a sequence: E is its largest biased exponent (>= 1), C the
// largest and T the sum of fx_ceil_units over its real values.  The moduli are
// below 2^mb and their sum below 2^bits in the same units; fixed-point value f
// stands for f 2^q.
struct FxScale {
  int D;     // right shift of a 63-bit significand of exponent e: D - e
  int q;     // exponent of one unit: moduli start below 2^60 units
  int left;  // bits by which the transform's values can grow beyond that
  bool bad;  // the sequence holds an infinity or a NaN
  // The shift before a stage whose inputs were just stored: as much as the values
  // may have grown in the stage before (3 bits: radix 8).
  __device__ __forceinline__ int stage() {
    const int g = min(3, left);
    left -= g;
    q += g;
    return g;
  }
};
__device__ __forceinline__ FxScale fx_scale(int E, unsigned C, unsigned T) {
  const int bits = max(32 - __clz((int)T), 16);
  const int mb = max(32 - __clz((int)(C + (C >> 1))), 16);  // 3/2 > sqrt 2: modulus from components
  const int s0 = min(mb, bits);
  return FxScale{s0 + E - 15, s0 + E - 1100, bits - s0, E >= 0x7ff};
}
__device__ __forceinline__ long long fx_from(double x, const FxScale& s) {
  int e;
  const unsigned long long m = fx_mant(x, e);
  return fx_sign((long long)((shr64_clamp(m << 10, s.D - e - 1) + 1ull) >> 1), x);
}
__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

// v 2^q as doubles, |v.x|, |v.y| < 2^63, each rounded once (twice only where the
// result is subnormal); NaN for q = kFxBad.  One branch for exponents that could
// leave their field (two, one to a component: 4096^2 image 284.3 against 282.2 us,
// 1024 profile 82.4 against 81.1).
constexpr int kFxBad = 4096;
__device__ __forceinline__ double2 fx_to(fx2 v, int q) {
  const double x = __ll2double_rn(v.x), y = __ll2double_rn(v.y);
  if ((unsigned)(q + 1021) > 1980u) {
    if (q == kFxBad) return make_double2(fx_nan(), fx_nan());
    const int a = q / 2, b = q - a;
    const double f = __hiloint2double((1023 + a) << 20, 0), g = __hiloint2double((1023 + b) << 20, 0);
    return make_double2(x * f * g, y * f * g);
  }
  // 1 <= |x| <= 2^63 or x = 0
  auto scaled = [&](double d) {
    const int h = __double2hiint(d);
    return __hiloint2double(h + (h ? q << 20 : 0), __double2loint(d));
  };
  return make_double2(scaled(x), scaled(y));
}

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
                                             const fxtw* tws, FxScale& sc) {
    if constexpr (ST < P::nstage - 1) {
      constexpr int T = P::T, Ns = ipowc(8, ST);
      fx2* in = (ST % 2 == 1) ? A : B;
      fx2* out = (ST % 2 == 0) ? A : B;
      const int k = t & (Ns - 1);
      if constexpr (ST > 0) {
        const fxtw* w = tws + (Ns - 8) + k;
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = in[pad3<8>(t + r * T)];
        const int g = sc.stage(), p = 3 - g;
        v[0] = fx_shr(v[0], g);
        if constexpr (TAB) {
#pragma unroll
          for (int r = 1; r < 8; ++r) v[r] = fx_stage_mul(v[r], w[(r - 1) * Ns], p);
        } else {
#pragma unroll
          for (int r = 1; r < 8; ++r) v[r] = fx_stage_mul(v[r], ldg_tw(w + (r - 1) * Ns), p);
        }
      }
      bfly8(v);
      const int base = ST == 0 ? 9 * t : pad3<8>((t - k) * 8 + k);
#pragma unroll
      for (int r = 0; r < 8; ++r) out[ST == 0 ? base + r : base + r * pad_step<8>(Ns)] = v[r];
      __syncthreads();
      FxHead<L, ST + 1, TAB>::run(v, A, B, t, tws, sc);
    }
  }
};

// The last stage's shift g of its inputs (FxScale::stage; none if it is the only
// stage) and the bits r its outputs may exceed 2^60 by.
struct FxLast {
  int g, r;
};
template <int L> __device__ __forceinline__ FxLast fx_last(FxScale& sc) {
  using P = P3<L, 8>;
  const int g = P::nstage > 1 ? sc.stage() : 0;
  return FxLast{g, min(ilog2c(P::rlast), sc.left)};
}
// last stage, complete: v[q R + r] <- X[t + q T + r L / R]
template <int L>
__device__ __forceinline__ void fx_last_full(fx2 (&v)[8], const fx2* in, int t,
                                             const fxtw* __restrict__ tws, int g) {
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
      v[q * R] = fx_shr(v[q * R], g);
#pragma unroll
      for (int r = 1; r < R; ++r)
        v[q * R + r] = fx_stage_mul(v[q * R + r], ldg_tw(tws + (P::Nsl - 8) + (r - 1) * P::Nsl + b), 3 - g);
      bflyR<R>(&v[q * R]);
    }
  }
}

// X[j] and X[L - j] only (pruned_pair3)
template <int L>
__device__ __forceinline__ void fx_pruned_pair(const fx2* in, int j, const fxtw* __restrict__ tws,
                                               int g, fx2& xj, fx2& xmj) {
  using P = P3<L, 8>;
  constexpr int R = P::rlast, Ns = P::Nsl;
  const int jb = j == 0 ? Ns : j;
  const int ba = pad3<8>(j), bb = -jb + ((-jb) >> P::lv);
  fx2 a = fx_shr(in[ba], g), b = fx_shr(in[bb + pad_step<8>(Ns)], g);
#pragma unroll
  for (int r = 1; r < R; ++r) {
    const fxtw w = ldg_tw(tws + (Ns - 8) + (r - 1) * Ns + j);
    a = cadd(a, fx_stage_mul(in[ba + r * pad_step<8>(Ns)], w, 3 - g));
    b = cadd(b, fx_stage_mul(in[bb + (r + 1) * pad_step<8>(Ns)], cconj(w), 3 - g));
  }
  xj = a;
  xmj = j == 0 ? a : b;
}

// 2 X_k of a real row from the bins Z_k, Z_{M-k} of its packed transform
// (r2c_unpack without the halving, which goes into the exponent); the bins below
// 2^60, w in units of 2^-62
__device__ __forceinline__ fx2 fx_r2c_unpack2(fx2 zk, fx2 zmk, const fxtw& w) {
  const fx2 b = cconj(zmk);
  const fx2 d = cmul_mi(csub(zk, b));
  const fx2 p = fx_cmul_q(fx2{d.x << 1, d.y << 1}, w);
  return cadd(cadd(zk, b), fx2{p.x << 1, p.y << 1});
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
  h = fx_group<TT, true>(h, red_max);
  const int E = max((int)(h >> 20), 1);
  auto units = [&](double x) { return fx_ceil_units((unsigned)__double2hiint(x), E); };
  unsigned s = 0;
#pragma unroll
  for (int r = 0; r < 8; ++r) s += units(z[r].x) + units(z[r].y);
  const FxScale sc = fx_scale(E, fx_ceil_units(h, E), fx_group<TT, false>(s, red_sum));
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

// grid offset x in units of 2^-50, to nearest; |x| >= 4096 (beyond every grid)
// saturates.  Coarser than the double itself within 4 cells of the origin, by
// 2^-51 of the step between two nodes at most.
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
// biased exponent: 2^59 <= |largest| < 2^60, one unit 2^(E - 1082); a smaller node
// is cut at that unit, 2^-59 of the largest.
__device__ __forceinline__ long long fx_node(double x, int E) {
  int e;
  const unsigned long long m = fx_mant(x, e);
  return fx_sign((long long)shr64_clamp(m << 7, E - e), x);
}
__device__ __forceinline__ fx2 fx_lerp(fx2 a, fx2 b, int fh, int fl) {
  return fx2{a.x + fx_mul(b.x - a.x, fh, fl), a.y + fx_mul(b.y - a.y, fh, fl)};
}

}  // namespace gal
