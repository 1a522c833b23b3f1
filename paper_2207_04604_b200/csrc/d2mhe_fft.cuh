// Exact ring products by double-precision FFT.
//
// A product of a residue polynomial c (below a prime p = 2^b - d < 2^56) with a polynomial s of small random
// coefficients is needed modulo X^N + 1 and p.  Both are integer polynomials, so the product can be formed over
// the integers and reduced afterwards: c is centred and split, c = c_lo + 2^h c_hi, each part is multiplied with
// s by a complex FFT of n = N/2 points in double precision, and the two integer results are rounded and
// recombined modulo p.  The double-precision pipe of this GPU has as many lanes as its integer multiplier (64 per SM), but
// a complex radix-2 butterfly (two points = four coefficients, six fused multiply-adds) stands for two modular
// butterflies of 15 multiplier slots each.
//
// Exactness.  X^N + 1 = (X^n - i)(X^n + i), so with z_j = a_j + i a_(j+n) and psi = e^(i pi / 2n) the transform
// is Z_k = sum_j z_j psi^j e^(2 pi i j k / n), and z_j = psi^-j / n sum_k Z_k e^(-2 pi i j k / n) recovers a product.
// The result has to be off by less than 1/2 minus the rounding below for EVERY residue polynomial c, so what is relied
// on is the 2-norm only; with u = 2^-53:
//   A stage's error is at most 2.94 u times the 2-norm of its outputs, plus the error of its twiddle factors: for a
//     butterfly (X, Y) -> (X + wY = U, X - wY = V) as computed below, U is off by at most u ((1 + a) |U| + b |V|) and V by
//     u |V| more, a = |3 + e^(2i arg w)| / 4, b = |1 - e^(2i arg w)| / 4.  Stages with w = 1 and i: u.
//   All steps but these are unitary up to scaling, so relative errors in the 2-norm add up (Higham, Accuracy and Stability
//     of Numerical Algorithms, ch. 24).  With the errors that the twiddle factors of this file have (0.6 to 2.6 u, computed
//     and compared in the tests), forward, product and inverse together come to fft_error_units(log2 N) u.
//   The two norms multiply as |C S|_2 <= |C|_2 max_k |S_k|.  That takes a bound for every single point of the key's
//     transform and of its error.  A 2-norm bound gives none (n points share the error, one may have it all), so the
//     transforms of keys are made in double-double arithmetic (kern_fft_keys.cu): every point is good to 1.2 u.
//   |c|_2 <= 2^(m-1) sqrt(N) for a part of m bits, |u|_2 <= sqrt(N) for the ternary u of an encryption.
//   max_k |S_k| < FFT_KEY_MAX sqrt(N) for a ternary s, but for a share of 2^-137 of all keys (uniform ternary
//     coefficients are sub-Gaussian with variance 2/3; 32 directions, n points; there are 2^83 keys at most, for
//     every seed and party).  max_k |P_k| < FFT_PK_MAX 2^m sqrt(N) for a uniform part of m bits of a public key, but for
//     2^-111.  |mu|_2 < FFT_MU_NORM sqrt(N) for the Gaussian mu of Conversion, but for 2^-300.
// fft_error, fft_error_pk and fft_error_conv below are these bounds; the host admits what stays below 1/2 with the
// rounding, which keeps f >= 4 fraction bits and rounds once or twice (2^-f at most).  Shares and BFV.Decrypt: 0.22 + 1/16 at
// N = 16384, smaller rings half of that; encryption 0.14; 32-bit words 0.44; Conversion 0.41 with parts of 27 bits.
// (Seen: 2^-14 with random and with extreme c, 2^-10 with s = all ones.)
// The low part has h <= 40 - log2 N bits, so that its product with a ternary factor fits 40 bits for any c.  Conversion
// adds the product of the recipient's public key with mu, up to four times larger by the norms above: its low results
// are kept in 44 bits, and its parts are halves, ceil(b / 2) bits each.
//
// Organisation.  A group of 16 R threads (R = 8 or 16) transforms 256 R points, 16 of them in a thread's registers.
// Index digits k = kC + R kB + 16 R kA, j = jA + 16 jB + 256 jC:
//   inverse   pass A: over kA (radix 16) in thread (kC, kB); exchange inside the 16 threads of kC;
//             pass B: over kB (radix 16) in thread (kC, jA); exchange across the group;
//             pass C: over kC (radix R) in thread r = jA + 16 jB: coefficients r + 256 jC.
//   forward   the same digits the other way round.
// Every pass evaluates a polynomial at points t w^j (decimation in time): the twiddle factors between passes are
// folded into the butterflies.  n = 2048 and 4096 take one group.  n = 8192 takes two: with X^8192 - i =
// (X^4096 - q)(X^4096 + q), q = e^(i pi / 4), group g works modulo X^4096 -+ q (a twist of its own), and one more
// exchange with its butterfly joins the two results.  (One group of 256 threads with 32 points each: eight warps
// per SM hide too little of the latencies.)
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>
#include <utility>

#ifndef D2MHE_HD
#ifdef __CUDACC__
#define D2MHE_HD __host__ __device__ __forceinline__
#else
#define D2MHE_HD inline
#endif
#endif

// f(integral_constant<int, 0>) .. f(integral_constant<int, N - 1>): loops over registers whose indices must be
// constants before the optimiser runs (arrays indexed by an unrolled loop variable ended up in local memory)
template <class F, int... I>
D2MHE_HD void static_for_seq(F& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
D2MHE_HD void static_for(F f) {
  static_for_seq(f, std::make_integer_sequence<int, N>{});
}

struct cpx {
  double r, i;
};

// cos(pi m / 64), m = 0 .. 32
D2MHE_HD constexpr double cos64(int m) {
  switch (m) {
    case 0: return 1.0;
    case 1: return 0.9987954562051724;
    case 2: return 0.9951847266721969;
    case 3: return 0.989176509964781;
    case 4: return 0.9807852804032304;
    case 5: return 0.970031253194544;
    case 6: return 0.9569403357322088;
    case 7: return 0.9415440651830208;
    case 8: return 0.9238795325112867;
    case 9: return 0.9039892931234433;
    case 10: return 0.881921264348355;
    case 11: return 0.8577286100002721;
    case 12: return 0.8314696123025452;
    case 13: return 0.8032075314806449;
    case 14: return 0.773010453362737;
    case 15: return 0.7409511253549591;
    case 16: return 0.7071067811865476;
    case 17: return 0.6715589548470184;
    case 18: return 0.6343932841636455;
    case 19: return 0.5956993044924334;
    case 20: return 0.5555702330196022;
    case 21: return 0.5141027441932218;
    case 22: return 0.47139673682599764;
    case 23: return 0.4275550934302821;
    case 24: return 0.3826834323650898;
    case 25: return 0.33688985339222005;
    case 26: return 0.2902846772544624;
    case 27: return 0.2429801799032639;
    case 28: return 0.19509032201612828;
    case 29: return 0.14673047445536175;
    case 30: return 0.0980171403295606;
    case 31: return 0.049067674327418015;
    default: return 0.0;
  }
}
#ifdef __CUDACC__
// the same values for the kernels: operands read through the constant bank (as literals they were kept in uniform
// registers across the loop, and spilled)
static __device__ __constant__ double c_cos64[33] = {
    1.0, 0.9987954562051724, 0.9951847266721969, 0.989176509964781,
    0.9807852804032304, 0.970031253194544, 0.9569403357322088, 0.9415440651830208,
    0.9238795325112867, 0.9039892931234433, 0.881921264348355, 0.8577286100002721,
    0.8314696123025452, 0.8032075314806449, 0.773010453362737, 0.7409511253549591,
    0.7071067811865476, 0.6715589548470184, 0.6343932841636455, 0.5956993044924334,
    0.5555702330196022, 0.5141027441932218, 0.47139673682599764, 0.4275550934302821,
    0.3826834323650898, 0.33688985339222005, 0.2902846772544624, 0.2429801799032639,
    0.19509032201612828, 0.14673047445536175, 0.0980171403295606, 0.049067674327418015,
    0.0};
#endif
// cos and sin of pi M / 64
template <int M>
D2MHE_HD double root_c() {
  constexpr int m = (M & 127) > 64 ? 128 - (M & 127) : (M & 127);
  if constexpr (m == 0) return 1.0;
  if constexpr (m == 32) return 0.0;
  if constexpr (m == 64) return -1.0;
#ifdef __CUDA_ARCH__
  if constexpr (m < 32) return c_cos64[m];
  return -c_cos64[m < 32 ? 0 : 64 - m];
#else
  return m < 32 ? cos64(m) : -cos64(64 - m);
#endif
}
template <int M>
D2MHE_HD double root_s() {
  return root_c<M - 32>();
}

// bit reversal of an index below R (R = 4, 8, 16), without a loop so that it folds early
template <int R>
D2MHE_HD constexpr int brev_c(int i) {
  return R == 4 ? ((i & 1) << 1) | ((i >> 1) & 1)
         : R == 8 ? ((i & 1) << 2) | (i & 2) | ((i >> 2) & 1)
                  : ((i & 1) << 3) | ((i & 2) << 1) | ((i & 4) >> 1) | ((i >> 3) & 1);
}

#ifdef __CUDA_ARCH__
#define D2MHE_FMA(a, b, c) __fma_rn((a), (b), (c))
#else
#define D2MHE_FMA(a, b, c) std::fma((a), (b), (c))
#endif

// Error bounds (see above).
#define FFT_KEY_MAX 8.5
#define FFT_PK_MAX 2.75
#define FFT_MU_NORM 4.0
// |V| <= FFT_CONV_V N 2^(m-1) for a result of Conversion on parts of m bits: 1 for c s, FFT_MU_NORM for mu p
#define FFT_CONV_V 5
constexpr double fft_error_units(int logn) { return logn == 12 ? 91.0 : logn == 13 ? 101.0 : 107.0; }
constexpr double fft_pow2(int e) { return e < 0 ? 1.0 / (double)(1ull << -e) : (double)(1ull << e); }
// a part of m bits times a key; u times a part of a public key; the sum of Conversion (its product stage loses 5 u more on
// c s and 3 u on mu p)
constexpr double fft_error(int logn, int m) { return fft_error_units(logn) * FFT_KEY_MAX * fft_pow2(m - 1 + logn - 53); }
constexpr double fft_error_pk(int logn, int m) { return fft_error_units(logn) * FFT_PK_MAX * fft_pow2(m + logn - 53); }
constexpr double fft_error_conv(int logn, int m) {
  return (fft_error_units(logn) + 5.0) * FFT_KEY_MAX * fft_pow2(m - 1 + logn - 53) +
         (fft_error_units(logn) + 3.0) * FFT_MU_NORM * FFT_PK_MAX * fft_pow2(m + logn - 53);
}

// (X, Y) -> (X + w Y, X - w Y)
D2MHE_HD void fft_bfly(double& xr, double& xi, double& yr, double& yi, double wr, double wi) {
  const double ur = D2MHE_FMA(-wi, yi, D2MHE_FMA(wr, yr, xr));
  const double ui = D2MHE_FMA(wi, yr, D2MHE_FMA(wr, yi, xi));
  yr = D2MHE_FMA(2.0, xr, -ur);
  yi = D2MHE_FMA(2.0, xi, -ui);
  xr = ur;
  xi = ui;
}
D2MHE_HD void fft_bfly_one(double& xr, double& xi, double& yr, double& yi) {  // w = 1
  const double tr = yr, ti = yi;
  yr = xr - tr;
  yi = xi - ti;
  xr += tr;
  xi += ti;
}
template <int SGN>
D2MHE_HD void fft_bfly_i(double& xr, double& xi, double& yr, double& yi) {  // w = SGN i
  const double tr = SGN > 0 ? -yi : yi, ti = SGN > 0 ? yr : -yr;
  yr = xr - tr;
  yi = xi - ti;
  xr += tr;
  xi += ti;
}
D2MHE_HD cpx cmul(cpx a, cpx b) {
  return cpx{D2MHE_FMA(a.r, b.r, -(a.i * b.i)), D2MHE_FMA(a.r, b.i, a.i * b.r)};
}

// Twiddle factors of a pass that evaluates at t w_R^j.  The stage that merges blocks of L/2 into blocks
// of L uses t^(R/L) w_L^m, m < L/4 (the others are these times i; L = 2: m = 0).
// Derived from t and t^4: the powers between by squaring, the rotations by constants.
template <int R, int SGN>
struct TwDerived {
  static constexpr int LG = R == 8 ? 3 : 4;
  cpx pw[LG];  // pw[s] = t^(R / 2^(s+1)): stage L = 2^(s+1)
  D2MHE_HD explicit TwDerived(const cpx (&t)[2]) {
    static_for<LG>([&](auto i_) {
      constexpr int i = decltype(i_)::value;
      pw[LG - 1 - i] = i % 2 ? cmul(t[i / 2], t[i / 2]) : t[i / 2];
    });
  }
  template <int lg, int m>
  D2MHE_HD cpx get() const {  // L = 2^lg
    if constexpr (m == 0) {
      return pw[lg - 1];
    } else {
      constexpr int a = SGN * (m * 128 >> lg);
      return cmul(pw[lg - 1], cpx{root_c<a>(), root_s<a>()});
    }
  }
};
struct TwNone {};

// y_j = sum_k x_k (t w^j)^k, w = e^(SGN 2 pi i / R): inputs in natural order, y_j left in x[brev(j)].
// TwNone: t = 1.  FIRST: stages done already (2 = the stages L = 2 and L = 4).
template <int R, int SGN, int FIRST, class TW>
D2MHE_HD void fft_eval(double* xr, double* xi, const TW& tw) {
  constexpr int LG = R == 8 ? 3 : 4;
  constexpr bool TRIV = std::is_same<TW, TwNone>::value;
  static_for<LG - FIRST>([&](auto s_) {
    constexpr int lg = FIRST + 1 + decltype(s_)::value, L = 1 << lg;
    static_for<(L >= 4 ? L / 4 : 1)>([&](auto m_) {
      constexpr int m = decltype(m_)::value;
      auto both = [&](double wr, double wi) {
        static_for<R / L>([&](auto b_) {
          constexpr int b = decltype(b_)::value * L;
          {
            constexpr int p = brev_c<R>(b + m), q = brev_c<R>(b + m + L / 2);
            if constexpr (TRIV && m == 0)
              fft_bfly_one(xr[p], xi[p], xr[q], xi[q]);
            else
              fft_bfly(xr[p], xi[p], xr[q], xi[q], wr, wi);
          }
          if constexpr (L >= 4) {
            constexpr int p = brev_c<R>(b + m + L / 4), q = brev_c<R>(b + m + L / 4 + L / 2);
            if constexpr (TRIV && m == 0)
              fft_bfly_i<SGN>(xr[p], xi[p], xr[q], xi[q]);
            else if constexpr (SGN > 0)
              fft_bfly(xr[p], xi[p], xr[q], xi[q], -wi, wr);
            else
              fft_bfly(xr[p], xi[p], xr[q], xi[q], wi, -wr);
          }
        });
      };
      if constexpr (TRIV) {
        both(root_c<SGN * m * 128 / L>(), root_s<SGN * m * 128 / L>());
      } else {
        const cpx w = tw.template get<lg, m>();
        both(w.r, w.i);
      }
    });
  });
}

// Pointwise products of four points (k, k + 8, k + 4, k + 12 of a radix-16 pass without twiddles) and the
// two stages L = 2, L = 4 of that pass.  x: in = second factor, out = values; c: first factor.
template <int SGN>
D2MHE_HD void fft_product4(double* xr, double* xi, int k, const cpx (&c)[4]) {
  const int i0 = k, i1 = k + 8, i2 = k + 4, i3 = k + 12;
  const cpx x0 = cmul(c[0], cpx{xr[i0], xi[i0]}), x2 = cmul(c[2], cpx{xr[i2], xi[i2]});
  const double y1r = xr[i1], y1i = xi[i1], y3r = xr[i3], y3i = xi[i3];
  xr[i0] = D2MHE_FMA(-c[1].i, y1i, D2MHE_FMA(c[1].r, y1r, x0.r));
  xi[i0] = D2MHE_FMA(c[1].i, y1r, D2MHE_FMA(c[1].r, y1i, x0.i));
  xr[i2] = D2MHE_FMA(-c[3].i, y3i, D2MHE_FMA(c[3].r, y3r, x2.r));
  xi[i2] = D2MHE_FMA(c[3].i, y3r, D2MHE_FMA(c[3].r, y3i, x2.i));
  xr[i1] = D2MHE_FMA(2.0, x0.r, -xr[i0]);
  xi[i1] = D2MHE_FMA(2.0, x0.i, -xi[i0]);
  xr[i3] = D2MHE_FMA(2.0, x2.r, -xr[i2]);
  xi[i3] = D2MHE_FMA(2.0, x2.i, -xi[i2]);
  fft_bfly_one(xr[i0], xi[i0], xr[i2], xi[i2]);
  fft_bfly_i<SGN>(xr[i1], xi[i1], xr[i3], xi[i3]);
}

// cos(pi m / 64) for any m
D2MHE_HD constexpr double cos64_any(int m) {
  const int k = m & 127, h = k > 64 ? 128 - k : k;
  return h <= 32 ? cos64(h) : -cos64(64 - h);
}
// The factor of digit j in psi^-j of the columns of group g (two groups): what fft_twist multiplies by, as a table entry.
D2MHE_HD constexpr cpx fft_digit(int g, int j) {
  const int a = g ? 3 * j : -j;
  return cpx{cos64_any(a), cos64_any(a - 32)};
}

// psi^-j of digit jC = JC of a column: tw * e^(-i pi JC / 2R) (one group), e^(-i pi JC / 4R) (first of two) or
// e^(3 i pi JC / 4R) (second of two; psi_1 = e^(-3 i pi / 4 NG)).
template <int R, int GR, int JC>
D2MHE_HD cpx fft_twist(const cpx tw, unsigned group) {
  if constexpr (JC == 0) return tw;
  if constexpr (GR == 1) {
    constexpr int a = -32 * JC / R;
    return cmul(tw, cpx{root_c<a>(), root_s<a>()});
  } else {
    const cpx r0{root_c<-JC>(), root_s<-JC>()}, r1{root_c<3 * JC>(), root_s<3 * JC>()};
    return cmul(tw, group ? r1 : r0);
  }
}

D2MHE_HD cpx cmul_add(cpx a, cpx b, cpx c) {
  return cpx{D2MHE_FMA(-a.i, b.i, D2MHE_FMA(a.r, b.r, c.r)), D2MHE_FMA(a.i, b.r, D2MHE_FMA(a.r, b.i, c.i))};
}
// The same for the sums c x + a b of two products each.
template <int SGN>
D2MHE_HD void fft_product4_sum(double* xr, double* xi, int k, const cpx (&c)[4], const cpx (&a)[4], const cpx (&b)[4]) {
  const int at[4] = {k, k + 8, k + 4, k + 12};
#pragma unroll
  for (int h = 0; h < 4; h += 2) {
    const int i = at[h], j = at[h + 1];
    const cpx x = cmul_add(a[h], b[h], cmul(c[h], cpx{xr[i], xi[i]}));
    const cpx y = cmul_add(a[h + 1], b[h + 1], cmul_add(c[h + 1], cpx{xr[j], xi[j]}, x));
    xr[i] = y.r;
    xi[i] = y.i;
    xr[j] = D2MHE_FMA(2.0, x.r, -y.r);
    xi[j] = D2MHE_FMA(2.0, x.i, -y.i);
  }
  fft_bfly_one(xr[k], xi[k], xr[k + 4], xi[k + 4]);
  fft_bfly_i<SGN>(xr[k + 8], xi[k + 8], xr[k + 12], xi[k + 12]);
}

// Double-double numbers h + l, |l| <= u |h| (Dekker; Knuth's sum, a fused product): relative errors of a few u^2.  The
// single operations are spelled out: a sum that was contracted with the product before it would not be that sum.
#ifdef __CUDA_ARCH__
#define D2MHE_ADD(a, b) __dadd_rn((a), (b))
#define D2MHE_MUL(a, b) __dmul_rn((a), (b))
#else
#define D2MHE_ADD(a, b) ((a) + (b))
#define D2MHE_MUL(a, b) ((a) * (b))
#endif
struct alignas(16) dd {
  double h, l;
};
struct ddc {
  dd r, i;
};
D2MHE_HD dd dd_norm(double a, double b) {  // |a| >= |b|
  const double s = D2MHE_ADD(a, b);
  return dd{s, D2MHE_ADD(b, -D2MHE_ADD(s, -a))};
}
D2MHE_HD dd dd_add(dd a, dd b) {
  const double s = D2MHE_ADD(a.h, b.h), t = D2MHE_ADD(s, -a.h);
  const double e = D2MHE_ADD(D2MHE_ADD(a.h, -D2MHE_ADD(s, -t)), D2MHE_ADD(b.h, -t));
  return dd_norm(s, D2MHE_ADD(e, D2MHE_ADD(a.l, b.l)));
}
D2MHE_HD dd dd_sub(dd a, dd b) { return dd_add(a, dd{-b.h, -b.l}); }
D2MHE_HD dd dd_mul(dd a, dd b) {
  const double p = D2MHE_MUL(a.h, b.h);
  return dd_norm(p, D2MHE_FMA(a.h, b.l, D2MHE_FMA(a.l, b.h, D2MHE_FMA(a.h, b.h, -p))));
}
D2MHE_HD ddc dd_cadd(ddc a, ddc b) { return ddc{dd_add(a.r, b.r), dd_add(a.i, b.i)}; }
D2MHE_HD ddc dd_csub(ddc a, ddc b) { return ddc{dd_sub(a.r, b.r), dd_sub(a.i, b.i)}; }
D2MHE_HD ddc dd_cmul(ddc a, ddc b) {
  return ddc{dd_sub(dd_mul(a.r, b.r), dd_mul(a.i, b.i)), dd_add(dd_mul(a.r, b.i), dd_mul(a.i, b.r))};
}
// e^(2 pi i k / order) for any k, from coarse[k / 256] and fine[k mod 256]; order: a power of two
#define FFT_ROOT_FINE 256
D2MHE_HD ddc dd_root(const ddc* coarse, const ddc* fine, unsigned order, unsigned k) {
  k &= order - 1;
  return dd_cmul(coarse[k / FFT_ROOT_FINE], fine[k % FFT_ROOT_FINE]);
}
// The table entry e^(2 pi i k / order), 64 bits of each part: the angle is brought below pi / 4 in whole numbers.
inline ddc dd_root_entry(unsigned order, unsigned k) {
  const unsigned quarter = order / 4, q = k / quarter, r = k % quarter;
  const bool swap = r > quarter / 2;
  const long double a = 6.283185307179586476925286766559005768L * (long double)(swap ? quarter - r : r) / (long double)order;
  const long double c = swap ? sinl(a) : cosl(a), s = swap ? cosl(a) : sinl(a);
  const long double x = q == 0 ? c : q == 1 ? -s : q == 2 ? -c : s, y = q == 0 ? s : q == 1 ? c : q == 2 ? -s : -c;
  const double xh = (double)x, yh = (double)y;
  return ddc{dd{xh, (double)(x - xh)}, dd{yh, (double)(y - yh)}};
}

// The split of a residue c in [0, p): centred, low part in [-2^(h-1), 2^(h-1)), high part the rest.
D2MHE_HD void fft_split(unsigned long long c, unsigned long long p, unsigned h, int& lo, int& hi) {
  const long long v = (long long)c - (c > (p >> 1) ? (long long)p : 0ll);
  const int l = (int)((unsigned)(unsigned long long)v << (32 - h)) >> (32 - h);
  lo = l;
  hi = (int)((v - l) >> h);
}

// How a launch's products are dealt out: `rows` fixed factors (a limb of a unit's c_1), each with the products of all
// parties.  The first `whole` rows get a block each, the others `split` blocks, each of which transforms the fixed factor for
// itself.
struct FftDeal {
  unsigned whole, split, blocks;
};
// Part transforms of a block: of its fixed factor, and for each of its parties.  A 64-bit residue has two parts, a 32-bit one
// is one (taken for two there, 176 rows of ten at N = 8192 stayed whole: 71.4 us, in five blocks a row 57.7; 88 rows at
// N = 16384 79.4 and 68.1; 455 rows of twenty at N = 4096 121.8 and 108.1).
struct FftWork {
  unsigned fixed, per_party;
};
constexpr FftWork FFT_WORK_SHARE = {2, 2}, FFT_WORK_SHARE32 = {1, 1}, FFT_WORK_BOOT = {2, 2}, FFT_WORK_CONVERT = {2, 4};
// The deal with the shortest schedule, counted in part transforms over waves of `places` blocks: whole rows for as many full
// waves as there are and the rest split over one wave, or all rows split alike.
// (594 rows of nine on 296 places: three blocks to a row took seven waves of three parties; 592 whole rows and two rows split
// nine ways take two waves of nine and one of one: 320 -> 264 us at N = 8192.)
inline FftDeal fft_deal(unsigned places, unsigned rows, unsigned n_parties, FftWork work) {
  const unsigned full = rows / places * places, rest = rows - full, all = work.fixed + work.per_party * n_parties;
  FftDeal deal = {0, 1, rows};
  unsigned long long best = (unsigned long long)((rows + places - 1) / places) * all;
  auto consider = [&](unsigned whole, unsigned split, unsigned long long waves) {
    const unsigned long long cost =
        (unsigned long long)(whole / places) * all + waves * (work.fixed + work.per_party * ((n_parties + split - 1) / split));
    if (cost < best) best = cost, deal = FftDeal{whole, split, whole + (rows - whole) * split};
  };
  if (full && rest) consider(full, std::max(1u, std::min(n_parties, places / rest)), 1);
  for (unsigned c = 2; c <= n_parties && c <= 16u; ++c) consider(0, c, ((unsigned long long)rows * c + places - 1) / places);
  if (!full) consider(0, std::max(1u, std::min(n_parties, places / std::max(rows, 1u))), 1);
  return deal;
}
// A block's row and its part of the parties: first, first + step, ..  MIXED: some rows are whole, others not (an
// instance of its own, with a step that is not a launch constant: as the only one it made the refresh shares of 2960 rows of
// ten at N = 8192, which are not mixed, 1702 us instead of 1574).
template <bool MIXED>
D2MHE_HD unsigned fft_dealt(const FftDeal& deal, unsigned block, unsigned& first, unsigned& step) {
  if (MIXED && block < deal.whole) {
    first = 0, step = 1;
    return block;
  }
  const unsigned b = MIXED ? block - deal.whole : block;
  first = b % deal.split, step = deal.split;
  return (MIXED ? deal.whole : 0u) + b / deal.split;
}
