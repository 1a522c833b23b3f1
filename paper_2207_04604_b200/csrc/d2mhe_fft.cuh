// Exact ring products by double-precision FFT.
//
// A product of a residue polynomial c (below a prime p = 2^b - d < 2^56) with a polynomial s of small random
// coefficients is needed modulo X^N + 1 and p.  Both are integer polynomials, so the product can be formed over
// the integers and reduced afterwards: c is centred and split, c = c_lo + 2^h c_hi, each part is multiplied with
// s by a complex FFT of n = N/2 points in double precision, and the two integer results are rounded and
// recombined modulo p.  The double-precision pipe of this GPU issues as many lanes per clock as its integer
// multiplier (62 of 64 measured), but a complex radix-2 butterfly (two points = four coefficients, six fused
// multiply-adds) stands for two modular butterflies of 15 multiplier slots each.
//
// Exactness.  X^N + 1 = (X^n - i)(X^n + i), so with z_j = a_j + i a_(j+n) and psi = e^(i pi / 2n) the transform
// is Z_k = sum_j z_j psi^j e^(2 pi i j k / n), and z_j = psi^-j / n sum_k Z_k e^(-2 pi i j k / n) recovers a product.
// With u = 2^-53, a butterfly (X, Y) -> (X + wY, X - wY) computed as below has an error of at most 3.02 u times
// the 2-norm of its outputs, plus the error of w (1 u for a table value or a constant, 4 u for its square, 3 u
// more for a rotation by a constant); the rest of the operations are unitary up to scaling, so relative errors in
// the 2-norm add up (Higham, Accuracy and Stability of Numerical Algorithms, ch. 24).  Counted over the stages:
// 88 u per forward transform, 78 u for product and inverse, 254 u for a product.  A result coefficient is then
// off by less than 256 u |c|_2 max_k |S_k|.
//   |c|_2 <= 2^(m-1) sqrt(N) for EVERY part of m bits;
//   max_k |S_k| < 6.5 sqrt(N) for a ternary s, except with probability below 2^-70 over the key (uniform ternary
//   coefficients are sub-Gaussian with variance 2/3; 16 directions, n points).
// Parts of at most 28 bits at N = 16384 stay below 0.41 (smaller rings: below 0.21); the rounding keeps at least
// four fraction bits and rounds twice (1/16), and 0.41 + 1/16 < 1/2: the rounded value IS the integer.  (Seen:
// 2^-14 with random and with extreme c, 2^-10 with s = all ones.)  The low part has h <= 40 - log2 N bits, so that
// its product fits 40 bits for any c and s.
// Conversion adds the product of a public key (uniform: |p|_2 is sqrt(3) smaller) with a Gaussian mu (|M_k| 3.9 times
// larger): there the 2-norm bound is 1.4, and what is relied on is that the error is spread, as rounding errors are: it
// would take a tenth of its square on one of the 16384 coefficients to reach 1/2 (seen: 2^-13).
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

// The split of a residue c in [0, p): centred, low part in [-2^(h-1), 2^(h-1)), high part the rest.
D2MHE_HD void fft_split(unsigned long long c, unsigned long long p, unsigned h, int& lo, int& hi) {
  const long long v = (long long)c - (c > (p >> 1) ? (long long)p : 0ll);
  const int l = (int)((unsigned)(unsigned long long)v << (32 - h)) >> (32 - h);
  lo = l;
  hi = (int)((v - l) >> h);
}
