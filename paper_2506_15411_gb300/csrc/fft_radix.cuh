// fft_radix.cuh -- small in-register DFTs ("codelets") for the mixed-radix FFT passes.
//
// The 3D FFTs of the CBS iteration (the "N log N" cost of Fig. 1(b) of arXiv 2506.15411)
// are built from the DFTs below, applied to R values held in registers: two steps of compile-time
// radices (xrow.cuh, colpass.cuh), or in-place DIF / DIT stages (fft_ip.cuh) of 1 (identity) to 13
// and 16 for axes that do not split so.  The two steps also use 14, 15, 18, 20, 21, 22, 24 to 28,
// 30, 32, 35 and 36.
//   - odd primes: symmetric-pair form, X[k] and X[R-k] share the sums over the pairs
//     x[m] +- x[R-m] with real cos/sin constants;
//   - composites: one Cooley-Tukey split R = R1 * R2 (decimation in time) with the inner
//     twiddles as compile-time constants; quarter and eighth turns become swaps/negations.
// Constants come from a constexpr Taylor series in double precision, rounded to float.
#pragma once
#include <cuda_runtime.h>
#include <utility>

// The codelets also compile for the host (the tests run the FFT stages on the CPU).
#ifndef CBS_HD
#if defined(__CUDACC__)
#define CBS_HD __host__ __device__ __forceinline__
#else
#define CBS_HD inline
#endif
#endif

namespace cbs {

// Twiddle tables of a two-step axis, one for every kTwiddlePhases-th iteration (axis_plan.h).
constexpr int kTwiddlePhases = 8;

// ---------------------------------------------------------------- complex helpers
// The device code adds complex values with the packed FP32x2 instructions of sm_100+ (one
// instruction for both parts; the same IEEE results as two scalar adds; CBS_SCALAR_ADD turns
// them off).
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000 && !defined(CBS_SCALAR_ADD)
#define CBS_USE_PACKED 1
#else
#define CBS_USE_PACKED 0
#endif
CBS_HD float2 cadd(float2 a, float2 b) {
#if CBS_USE_PACKED
  return __fadd2_rn(a, b);
#else
  return make_float2(a.x + b.x, a.y + b.y);
#endif
}
CBS_HD float2 csub(float2 a, float2 b) {
#if CBS_USE_PACKED
  return __fadd2_rn(a, make_float2(-b.x, -b.y));
#else
  return make_float2(a.x - b.x, a.y - b.y);
#endif
}
// a + c b for real c, both parts
CBS_HD float2 cfma_r(float c, float2 b, float2 a) {
#if CBS_USE_PACKED
  return __ffma2_rn(make_float2(c, c), b, a);
#else
  return make_float2(fmaf(c, b.x, a.x), fmaf(c, b.y, a.y));
#endif
}
CBS_HD float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
CBS_HD float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
CBS_HD float2 mul_i(float2 a) { return make_float2(-a.y, a.x); }      //  i a
CBS_HD float2 mul_mi(float2 a) { return make_float2(a.y, -a.x); }     // -i a

// ---------------------------------------------------------------- compile-time loops
template <class F, int... I>
CBS_HD void static_for_impl(F&& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
CBS_HD void static_for(F&& f) {
  static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// ---------------------------------------------------------------- constexpr trigonometry
// cos and sin of 2 pi m / R from their Taylor series on [-pi, pi] (30 terms: the
// truncation error is far below double rounding there).
constexpr double kPi = 3.14159265358979323846264338327950288;
constexpr double ct_angle(int m, int R) {
  int mm = ((m % R) + R) % R;
  double a = 2.0 * kPi * (double)mm / (double)R;
  return a > kPi ? a - 2.0 * kPi : a;
}
constexpr double ct_sin(double x) {
  double term = x, sum = x;
  for (int n = 1; n < 30; ++n) {
    term *= -x * x / ((2.0 * n) * (2.0 * n + 1.0));
    sum += term;
  }
  return sum;
}
constexpr double ct_cos(double x) {
  double term = 1.0, sum = 1.0;
  for (int n = 1; n < 30; ++n) {
    term *= -x * x / ((2.0 * n - 1.0) * (2.0 * n));
    sum += term;
  }
  return sum;
}

// The float next to f = (float)x on the other side of x.
constexpr float ct_other(double x) {
  const float f = (float)x;
  if (x == 0.0) return f;
  double p = 1.0;
  while (p > (x < 0 ? -x : x)) p *= 0.5;
  const double ulp = p / (1 << 23);
  return (float)((double)f + ((double)f < x ? ulp : -ulp));
}
constexpr float ct_low(double x) { return (float)(x - (double)(float)x); }
constexpr double ct_abs(double x) { return x < 0 ? -x : x; }

// cos and sin of 2 pi m / R as the floats beside them whose squares add up closest to 1 (a tenth of
// the error of the angle counted in).  A transform and its inverse use the same constants,
// conjugated: an error of the angle cancels in the pair, an error of the modulus is there twice, in
// every iteration again.  The nearest floats have a modulus up to 4e-8 off; 2e-8 on the
// twiddles of one axis moved a gradient by 9e-7 in 32 iterations (65 x 56 x 48).
struct CosSin {
  float c, s;
};
constexpr CosSin unit_pair(double c, double s) {
  const float cc[2] = {(float)c, ct_other(c)}, ss[2] = {(float)s, ct_other(s)};
  CosSin best{cc[0], ss[0]};
  double least = 1e300;
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      const double dc = (double)cc[i] - c, ds = (double)ss[j] - s;
      const double cost = ct_abs(c * dc + s * ds) + 0.1 * ct_abs(c * ds - s * dc);
      if (cost < least) {
        least = cost;
        best = CosSin{cc[i], ss[j]};
      }
    }
  return best;
}
constexpr CosSin ct_pair(int m, int R) { return unit_pair(ct_cos(ct_angle(m, R)), ct_sin(ct_angle(m, R))); }

// The constants cos(2 pi k / R) and sin(2 pi k / R), k <= H = (R - 1) / 2, of an odd prime's
// transform: each one of the two floats around it, chosen together so that the transform's even
// part (on x_m + x_{R-m}) and odd part (x_m - x_{R-m}) come closest to orthogonal, for the reason
// given at unit_pair.
template <int R>
struct OddConstants {
  static constexpr int H = (R - 1) / 2;
  float c[H], s[H];

  static constexpr OddConstants make() {
    double co[R] = {}, si[R] = {};
    for (int k = 0; k < R; ++k) {
      co[k] = ct_cos(ct_angle(k, R));
      si[k] = ct_sin(ct_angle(k, R));
    }
    OddConstants r{};
    for (int part = 0; part < 2; ++part) {
      const bool even = part == 0;
      float f[H][2] = {};
      double d[H][2] = {};
      for (int k = 0; k < H; ++k) {
        const double x = even ? co[k + 1] : si[k + 1];
        f[k][0] = (float)x;
        f[k][1] = ct_other(x);
        for (int i = 0; i < 2; ++i) d[k][i] = (double)f[k][i] - x;
      }
      double least = 1e300;
      for (int pick = 0; pick < 1 << H; ++pick) {
        double e[R] = {};   // the error of each entry's constant, by its angle's multiple
        for (int k = 0; k < H; ++k) {
          e[k + 1] = d[k][pick >> k & 1];
          e[R - k - 1] = even ? e[k + 1] : -e[k + 1];
        }
        // sum of squares of M dM^T + dM M^T; row and vector 0 of the even part are the plain sums
        double dev = 0.0;
        for (int i = even ? 0 : 1; i <= H; ++i)
          for (int j = even ? 0 : 1; j <= i; ++j) {
            double g = 0.0;
            for (int m = 1; m <= H; ++m)
              g += (even ? co : si)[i * m % R] * e[j * m % R] + e[i * m % R] * (even ? co : si)[j * m % R];
            dev += (i == j ? 1.0 : 2.0) * (i ? 1.0 : 0.5) * (j ? 1.0 : 0.5) * g * g;
          }
        if (dev < least) {
          least = dev;
          for (int k = 0; k < H; ++k) (even ? r.c : r.s)[k] = f[k][pick >> k & 1];
        }
      }
    }
    return r;
  }
  constexpr float cos(int m) const { return m % R == 0 ? 1.f : (m % R <= H ? c[m % R - 1] : c[R - m % R - 1]); }
  constexpr float sin(int m) const { return m % R == 0 ? 0.f : (m % R <= H ? s[m % R - 1] : -s[R - m % R - 1]); }
};

// a * w_R^M with w_R = exp(-2 pi i / R) (forward) or exp(+2 pi i / R) (inverse).
template <int M, int R, bool INV>
CBS_HD float2 twc(float2 a) {
  constexpr int m = ((M % R) + R) % R;
  if constexpr (m == 0) {
    return a;
  } else if constexpr (2 * m == R) {
    return make_float2(-a.x, -a.y);
  } else if constexpr (4 * m == R) {
    return INV ? mul_i(a) : mul_mi(a);
  } else if constexpr (4 * m == 3 * R) {
    return INV ? mul_mi(a) : mul_i(a);
  } else {
    constexpr CosSin w = ct_pair(m, R);
    constexpr float c = w.c, s = INV ? w.s : -w.s;
    return make_float2(fmaf(a.x, c, -a.y * s), fmaf(a.x, s, a.y * c));
  }
}

// ---------------------------------------------------------------- DFT codelets
template <int R, bool INV>
struct DFT;

template <bool INV>
struct DFT<1, INV> {
  static CBS_HD void run(float2*) {}
};

template <bool INV>
struct DFT<2, INV> {
  static CBS_HD void run(float2* v) {
    float2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};

// Odd prime R: X[k] = A_k - i B_k, X[R-k] = A_k + i B_k (forward), with
// A_k = x0 + sum_m cos(2 pi k m / R)(x_m + x_{R-m}), B_k = sum_m sin(2 pi k m / R)(x_m - x_{R-m}).
// R = 3 and 5 need one constant beyond FP32 each: sin 60 for 3, sqrt(5) / 4 of
// A_{1,2} = x0 - (a_1 + a_2) / 4 +- sqrt(5) / 4 (a_1 - a_2) for 5; its low part is multiplied first, as
// added to a rounded product it would be lost.  (All the constants so split: the gradients' errors a
// tenth lower, z of 336 = 28 x 12 1.35 -> 1.52 ms at 640 x 640 x 336.)
template <int R, bool INV>
struct DFTOdd {
  static CBS_HD void run(float2* v) {
    constexpr int H = (R - 1) / 2;
    constexpr OddConstants<R> t = OddConstants<R>::make();
    float2 a[H], b[H];
    const float2 x0 = v[0];
    static_for<H>([&](auto mi) {
      constexpr int m = decltype(mi)::value + 1;
      a[m - 1] = cadd(v[m], v[R - m]);
      b[m - 1] = csub(v[m], v[R - m]);
    });
    float2 sum = a[0];
    static_for<H - 1>([&](auto mi) { sum = cadd(sum, a[decltype(mi)::value + 1]); });
    v[0] = cadd(x0, sum);
    float2 mean, part;   // R = 5
    if constexpr (R == 5) {
      constexpr double r = 0.55901699437494742410;   // sqrt(5) / 4
      const float2 e = csub(a[0], a[1]);
      mean = cfma_r(-0.25f, sum, x0);
      part = cfma_r((float)r, e, cscale(e, ct_low(r)));
    }
    static_for<H>([&](auto ki) {
      constexpr int k = decltype(ki)::value + 1;
      float2 A, B;
      if constexpr (R == 3) {
        constexpr double s = ct_sin(ct_angle(1, 3));
        A = cfma_r(-0.5f, sum, x0);
        B = cfma_r((float)s, b[0], cscale(b[0], ct_low(s)));
      } else {
        if constexpr (R == 5) A = k == 1 ? cadd(mean, part) : csub(mean, part);
        else A = x0;
        static_for<H>([&](auto mi) {
          constexpr int m = decltype(mi)::value + 1;
          constexpr float c = t.cos(k * m), s = t.sin(k * m);
          if constexpr (R != 5) A = cfma_r(c, a[m - 1], A);
          B = m == 1 ? cscale(b[0], s) : cfma_r(s, b[m - 1], B);
        });
      }
      // forward: X[k] = A - iB = (A.x + B.y, A.y - B.x); X[R-k] = A + iB
      if constexpr (!INV) {
        v[k] = make_float2(A.x + B.y, A.y - B.x);
        v[R - k] = make_float2(A.x - B.y, A.y + B.x);
      } else {
        v[k] = make_float2(A.x - B.y, A.y + B.x);
        v[R - k] = make_float2(A.x + B.y, A.y - B.x);
      }
    });
  }
};

template <bool INV> struct DFT<3, INV> : DFTOdd<3, INV> {};
template <bool INV> struct DFT<5, INV> : DFTOdd<5, INV> {};
template <bool INV> struct DFT<7, INV> : DFTOdd<7, INV> {};
template <bool INV> struct DFT<11, INV> : DFTOdd<11, INV> {};
template <bool INV> struct DFT<13, INV> : DFTOdd<13, INV> {};

constexpr int ct_inverse(int a, int m) {   // of a modulo m
  int x = 1;
  while (a * x % m != 1 % m) ++x;
  return x;
}
constexpr int ct_gcd(int a, int b) { return b ? ct_gcd(b, a % b) : a; }

// Composite R = R1 * R2.  Coprime factors: input index n = R2 n1 + R1 n2 and output index k with
// k = k1 mod R1, k = k2 mod R2 (the prime-factor map), two independent transforms and no products
// between them.  Else input index n = R2 n1 + n2, output index k = k1 + R1 k2,
// X[k1 + R1 k2] = sum_n2 w_R2^{n2 k2} w_R^{n2 k1} sum_n1 x[R2 n1 + n2] w_R1^{n1 k1}.
template <int R1, int R2, bool INV>
struct DFTSplit {
  static constexpr int R = R1 * R2;
  static constexpr bool kPrimeFactor = ct_gcd(R1, R2) == 1;
  static CBS_HD void run(float2* v) {
    float2 y[R];
    static_for<R2>([&](auto n2i) {
      constexpr int n2 = decltype(n2i)::value;
      float2 t[R1];
      static_for<R1>([&](auto n1i) {
        constexpr int n1 = decltype(n1i)::value;
        t[n1] = v[kPrimeFactor ? (R2 * n1 + R1 * n2) % R : R2 * n1 + n2];
      });
      DFT<R1, INV>::run(t);
      static_for<R1>([&](auto k1i) {
        constexpr int k1 = decltype(k1i)::value;
        y[R2 * k1 + n2] = twc<kPrimeFactor ? 0 : n2 * k1, R, INV>(t[k1]);
      });
    });
    static_for<R1>([&](auto k1i) {
      constexpr int k1 = decltype(k1i)::value;
      float2 u[R2];
      static_for<R2>([&](auto n2i) {
        constexpr int n2 = decltype(n2i)::value;
        u[n2] = y[R2 * k1 + n2];
      });
      DFT<R2, INV>::run(u);
      static_for<R2>([&](auto k2i) {
        constexpr int k2 = decltype(k2i)::value;
        constexpr int k = kPrimeFactor
                              ? (R2 * ct_inverse(R2 % R1, R1) * k1 + R1 * ct_inverse(R1 % R2, R2) * k2) % R
                              : k1 + R1 * k2;
        v[k] = u[k2];
      });
    });
  }
};

template <bool INV> struct DFT<4, INV> : DFTSplit<2, 2, INV> {};
template <bool INV> struct DFT<6, INV> : DFTSplit<2, 3, INV> {};
template <bool INV> struct DFT<8, INV> : DFTSplit<2, 4, INV> {};
template <bool INV> struct DFT<9, INV> : DFTSplit<3, 3, INV> {};
template <bool INV> struct DFT<10, INV> : DFTSplit<2, 5, INV> {};
template <bool INV> struct DFT<12, INV> : DFTSplit<3, 4, INV> {};
template <bool INV> struct DFT<14, INV> : DFTSplit<2, 7, INV> {};
template <bool INV> struct DFT<15, INV> : DFTSplit<3, 5, INV> {};
template <bool INV> struct DFT<16, INV> : DFTSplit<4, 4, INV> {};
template <bool INV> struct DFT<18, INV> : DFTSplit<2, 9, INV> {};
template <bool INV> struct DFT<20, INV> : DFTSplit<4, 5, INV> {};
template <bool INV> struct DFT<21, INV> : DFTSplit<3, 7, INV> {};
template <bool INV> struct DFT<22, INV> : DFTSplit<2, 11, INV> {};
template <bool INV> struct DFT<24, INV> : DFTSplit<3, 8, INV> {};
template <bool INV> struct DFT<25, INV> : DFTSplit<5, 5, INV> {};
template <bool INV> struct DFT<26, INV> : DFTSplit<2, 13, INV> {};
template <bool INV> struct DFT<27, INV> : DFTSplit<3, 9, INV> {};
template <bool INV> struct DFT<28, INV> : DFTSplit<4, 7, INV> {};
template <bool INV> struct DFT<30, INV> : DFTSplit<5, 6, INV> {};
template <bool INV> struct DFT<32, INV> : DFTSplit<4, 8, INV> {};
template <bool INV> struct DFT<35, INV> : DFTSplit<5, 7, INV> {};
template <bool INV> struct DFT<36, INV> : DFTSplit<4, 9, INV> {};

// Calls f(std::integral_constant<int, R>) for the runtime radix r (uniform across the block).
// The stages' radices: 1 to 13 and 16.  Those above MAXR are not compiled in (a plan whose axes
// need them uses a MAXR = 16 kernel); leaving them out keeps the register allocation to what the smaller radices need.
template <int MAXR = 16, class F>
CBS_HD void radix_dispatch(int r, F&& f) {
  switch (r) {
    case 1: f(std::integral_constant<int, 1>{}); break;
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    case 6: f(std::integral_constant<int, 6>{}); break;
    case 7: f(std::integral_constant<int, 7>{}); break;
    case 8: f(std::integral_constant<int, 8>{}); break;
    case 9: if constexpr (MAXR >= 9) f(std::integral_constant<int, 9>{}); break;
    case 10: if constexpr (MAXR >= 10) f(std::integral_constant<int, 10>{}); break;
    case 11: if constexpr (MAXR >= 11) f(std::integral_constant<int, 11>{}); break;
    case 12: if constexpr (MAXR >= 12) f(std::integral_constant<int, 12>{}); break;
    case 13: if constexpr (MAXR >= 13) f(std::integral_constant<int, 13>{}); break;
    case 16: if constexpr (MAXR >= 16) f(std::integral_constant<int, 16>{}); break;
    default: break;
  }
}

}  // namespace cbs
