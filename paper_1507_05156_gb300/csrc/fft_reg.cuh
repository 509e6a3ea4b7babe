// fft_reg.cuh - fully unrolled mixed-radix (2, 3, 4, 5) complex DFT of a pencil held in
// registers (prime-factor algorithm across coprime factors, Cooley-Tukey within prime powers).  Used by every 3-D transform of the Fock-like term (Sec. II C, Eq. "Fock":
// the pair density is transformed, multiplied by the kernel and transformed back).
//
// Convention: fft<N, -1> computes X[k] = sum_n x[n] exp(-2 pi i n k / N) (no scaling);
// fft<N, +1> the same with exp(+...).  Input and output are in natural order.
//
// All loops are compile-time (static_for), so every twiddle factor is a constant folded
// into the instruction stream and trivial twiddles (1, -1, +-i) cost nothing.
#pragma once

#include <type_traits>
#include <utility>

namespace hse {

template <typename T>
struct cpx {
  T x, y;
};

// ---------------------------------------------------------------------------
// compile-time trigonometry: cos/sin(2 pi j / n) from the Taylor series of sin and
// cos on an argument reduced exactly (integer arithmetic) to [0, pi/4].
// ---------------------------------------------------------------------------
constexpr double kPi = 3.141592653589793238462643383279502884;

__host__ __device__ constexpr double taylor_sin(double x) {
  double term = x, sum = x;
  for (int k = 1; k < 16; ++k) {
    term *= -x * x / double((2 * k) * (2 * k + 1));
    sum += term;
  }
  return sum;
}

__host__ __device__ constexpr double taylor_cos(double x) {
  double term = 1.0, sum = 1.0;
  for (int k = 1; k < 16; ++k) {
    term *= -x * x / double((2 * k - 1) * (2 * k));
    sum += term;
  }
  return sum;
}

// returns cos (which = 0) or sin (which = 1) of 2 pi j / n
__host__ __device__ constexpr double trig2pi(int j, int n, int which) {
  j %= n;
  if (j < 0) j += n;
  const int q = (4 * j) / n;        // quarter turns
  const int rnum = 4 * j - q * n;   // remainder: angle = pi/2 * (q + rnum / n)
  double c = 0.0, s = 0.0;
  if (2 * rnum <= n) {
    const double r = (kPi / 2) * double(rnum) / double(n);
    c = taylor_cos(r);
    s = taylor_sin(r);
  } else {
    const double r = (kPi / 2) * double(n - rnum) / double(n);
    c = taylor_sin(r);
    s = taylor_cos(r);
  }
  double cc = c, ss = s;
  if (q == 1) { cc = -s; ss = c; }
  if (q == 2) { cc = -c; ss = -s; }
  if (q == 3) { cc = s; ss = -c; }
  return which == 0 ? cc : ss;
}

template <int B, int E, typename F>
__host__ __device__ __forceinline__ void static_for(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(static_cast<F&&>(f));
  }
}

template <typename T>
__host__ __device__ __forceinline__ cpx<T> cadd(cpx<T> a, cpx<T> b) { return {a.x + b.x, a.y + b.y}; }
template <typename T>
__host__ __device__ __forceinline__ cpx<T> csub(cpx<T> a, cpx<T> b) { return {a.x - b.x, a.y - b.y}; }
// (DIR * i) * a
template <int DIR, typename T>
__host__ __device__ __forceinline__ cpx<T> mul_i(cpx<T> a) {
  if constexpr (DIR > 0) return {-a.y, a.x};
  else return {a.y, -a.x};
}

// a * exp(DIR * 2 pi i J / N)
template <int N, int J, int DIR, typename T>
__host__ __device__ __forceinline__ cpx<T> twiddle(cpx<T> a) {
  constexpr int j = ((J % N) + N) % N;
  if constexpr (j == 0) {
    return a;
  } else if constexpr (2 * j == N) {
    return {-a.x, -a.y};
  } else if constexpr (4 * j == N) {
    return mul_i<DIR>(a);
  } else if constexpr (4 * j == 3 * N) {
    return mul_i<-DIR>(a);
  } else {
    constexpr T c = T(trig2pi(j, N, 0));
    constexpr T s = T(DIR * trig2pi(j, N, 1));
    return {a.x * c - a.y * s, a.x * s + a.y * c};
  }
}

// ---------------------------------------------------------------------------
// radix butterflies: y_s = sum_r x_r exp(DIR 2 pi i r s / R)
// ---------------------------------------------------------------------------
template <int R, int DIR, typename T>
struct Butterfly;

template <int DIR, typename T>
struct Butterfly<2, DIR, T> {
  static __host__ __device__ __forceinline__ void run(cpx<T>* a) {
    const cpx<T> t = a[0];
    a[0] = cadd(t, a[1]);
    a[1] = csub(t, a[1]);
  }
};

template <int DIR, typename T>
struct Butterfly<3, DIR, T> {
  static __host__ __device__ __forceinline__ void run(cpx<T>* a) {
    constexpr T h = T(0.5);
    constexpr T s = T(DIR * 0.866025403784438646763723170752936183);  // DIR sin(2 pi / 3)
    const cpx<T> t1 = cadd(a[1], a[2]);
    const cpx<T> t2 = csub(a[1], a[2]);
    const cpx<T> m = {a[0].x - h * t1.x, a[0].y - h * t1.y};
    const cpx<T> r = {-s * t2.y, s * t2.x};  // i s t2
    a[0] = cadd(a[0], t1);
    a[1] = cadd(m, r);
    a[2] = csub(m, r);
  }
};

template <int DIR, typename T>
struct Butterfly<4, DIR, T> {
  static __host__ __device__ __forceinline__ void run(cpx<T>* a) {
    const cpx<T> a0 = cadd(a[0], a[2]);
    const cpx<T> a1 = csub(a[0], a[2]);
    const cpx<T> b0 = cadd(a[1], a[3]);
    const cpx<T> b1 = mul_i<DIR>(csub(a[1], a[3]));
    a[0] = cadd(a0, b0);
    a[2] = csub(a0, b0);
    a[1] = cadd(a1, b1);
    a[3] = csub(a1, b1);
  }
};

// 32 operations: the cosine sums through t1 + t2 and t1 - t2 (c1 + c2 = -1/2, c1 - c2 = sqrt(5)/2),
// the sine sums as s2 (g t3 + t4) and s2 (t3 - g t4), g = s1 / s2, with the factor s2 in the last
// multiply-adds (36 with the four products written out).  Rounded to FP32, s2 and g change a plane
// wave by 6e-10 through a transform and its inverse; s1 and s2 / s1 would by 4e-8, the four sines
// and cosines by 2e-8.
template <int DIR, typename T>
struct Butterfly<5, DIR, T> {
  static __host__ __device__ __forceinline__ void run(cpx<T>* a) {
    constexpr T hr5 = T(0.559016994374947424102293417182819059);  // sqrt(5) / 4
    constexpr T s2 = T(DIR * trig2pi(2, 5, 1));
    constexpr T g = T(trig2pi(1, 5, 1) / trig2pi(2, 5, 1));
    const cpx<T> t1 = cadd(a[1], a[4]);
    const cpx<T> t2 = cadd(a[2], a[3]);
    const cpx<T> t3 = csub(a[1], a[4]);
    const cpx<T> t4 = csub(a[2], a[3]);
    const cpx<T> t = cadd(t1, t2), u = csub(t1, t2);
    const cpx<T> m = {a[0].x - T(0.25) * t.x, a[0].y - T(0.25) * t.y};
    const cpx<T> p1 = {m.x + hr5 * u.x, m.y + hr5 * u.y};
    const cpx<T> p2 = {m.x - hr5 * u.x, m.y - hr5 * u.y};
    const cpx<T> q1 = {g * t3.x + t4.x, g * t3.y + t4.y};
    const cpx<T> q2 = {t3.x - g * t4.x, t3.y - g * t4.y};
    a[0] = cadd(a[0], t);
    a[1] = {p1.x - s2 * q1.y, p1.y + s2 * q1.x};
    a[4] = {p1.x + s2 * q1.y, p1.y - s2 * q1.x};
    a[2] = {p2.x - s2 * q2.y, p2.y + s2 * q2.x};
    a[3] = {p2.x + s2 * q2.y, p2.y - s2 * q2.x};
  }
};

// Last butterfly of a 4-point column whose twiddles are folded in: s0, s1 are the sum and the
// difference of the even inputs, the odd inputs are c u1 and c u3 with one real c, which rides on
// the multiply-adds.
template <int DIR, typename T>
__host__ __device__ __forceinline__ void fold_column(cpx<T>* a, cpx<T> s0, cpx<T> s1, cpx<T> u1, cpx<T> u3, T c) {
  const cpx<T> t0 = cadd(u1, u3), t1 = mul_i<DIR>(csub(u1, u3));
  a[0] = {s0.x + c * t0.x, s0.y + c * t0.y};
  a[2] = {s0.x - c * t0.x, s0.y - c * t0.y};
  a[1] = {s1.x + c * t1.x, s1.y + c * t1.y};
  a[3] = {s1.x - c * t1.x, s1.y - c * t1.y};
}
// x (1 + DIR i t) and x (t + DIR i)
template <int DIR, typename T>
__host__ __device__ __forceinline__ cpx<T> mul_1t(cpx<T> x, T t) {
  const T s = DIR * t;
  return {x.x - s * x.y, x.y + s * x.x};
}
template <int DIR, typename T>
__host__ __device__ __forceinline__ cpx<T> mul_t1(cpx<T> x, T t) {
  if constexpr (DIR > 0) return {t * x.x - x.y, t * x.y + x.x};
  else return {t * x.x + x.y, t * x.y - x.x};
}
// x (1 + DIR i) and x (DIR i - 1)
template <int DIR, typename T>
__host__ __device__ __forceinline__ cpx<T> mul_11(cpx<T> x) {
  if constexpr (DIR > 0) return {x.x - x.y, x.y + x.x};
  else return {x.x + x.y, x.y - x.x};
}
template <int DIR, typename T>
__host__ __device__ __forceinline__ cpx<T> mul_i1(cpx<T> x) {
  if constexpr (DIR > 0) return {-x.x - x.y, x.x - x.y};
  else return {x.y - x.x, -x.x - x.y};
}

// 8 and 16 points, 4-point columns with folded twiddles: 52 and 144 operations instead of 56 and
// 164 with a complex multiplication per twiddle.
template <int DIR, typename T>
__host__ __device__ __forceinline__ void fft8_fold(cpx<T>* a) {
  constexpr T h = T(trig2pi(1, 8, 0));
  cpx<T> s[4], d[4];
  static_for<0, 4>([&](auto rc) {
    constexpr int r = decltype(rc)::value;
    s[r] = cadd(a[r], a[r + 4]);
    d[r] = csub(a[r], a[r + 4]);
  });
  Butterfly<4, DIR, T>::run(s);
  cpx<T> o[4];
  const cpx<T> e = mul_i<DIR>(d[2]);
  fold_column<DIR, T>(o, cadd(d[0], e), csub(d[0], e), mul_11<DIR, T>(d[1]), mul_i1<DIR, T>(d[3]), h);
  static_for<0, 4>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    a[2 * k] = s[k];
    a[2 * k + 1] = o[k];
  });
}

template <int DIR, typename T>
__host__ __device__ __forceinline__ void fft16_fold(cpx<T>* a) {
  constexpr T h = T(trig2pi(2, 16, 0)), c1 = T(trig2pi(1, 16, 0));
  constexpr T t = T(trig2pi(1, 16, 1) / trig2pi(1, 16, 0));
  cpx<T> m[4][4];  // m[k][r]: output k of the DFT over a[r], a[4 + r], a[8 + r], a[12 + r]
  static_for<0, 4>([&](auto rc) {
    constexpr int r = decltype(rc)::value;
    cpx<T> c[4] = {a[r], a[4 + r], a[8 + r], a[12 + r]};
    Butterfly<4, DIR, T>::run(c);
    static_for<0, 4>([&](auto kc) { m[decltype(kc)::value][r] = c[decltype(kc)::value]; });
  });
  Butterfly<4, DIR, T>::run(m[0]);
  {  // W = c1 (1 +- i t), W^2 = h (1 +- i), W^3 = c1 (t +- i)
    const cpx<T> u = mul_11<DIR, T>(m[1][2]);
    fold_column<DIR, T>(m[1], {m[1][0].x + h * u.x, m[1][0].y + h * u.y}, {m[1][0].x - h * u.x, m[1][0].y - h * u.y},
                        mul_1t<DIR, T>(m[1][1], t), mul_t1<DIR, T>(m[1][3], t), c1);
  }
  {  // W^2, W^4 = +- i, W^6 = h (+- i - 1)
    const cpx<T> u = mul_i<DIR>(m[2][2]);
    fold_column<DIR, T>(m[2], cadd(m[2][0], u), csub(m[2][0], u), mul_11<DIR, T>(m[2][1]), mul_i1<DIR, T>(m[2][3]), h);
  }
  {  // W^3, W^6, W^9 = -c1 (1 +- i t)
    const cpx<T> u = mul_i1<DIR, T>(m[3][2]);
    const cpx<T> w = mul_1t<DIR, T>(m[3][3], t);
    fold_column<DIR, T>(m[3], {m[3][0].x + h * u.x, m[3][0].y + h * u.y}, {m[3][0].x - h * u.x, m[3][0].y - h * u.y},
                        mul_t1<DIR, T>(m[3][1], t), {-w.x, -w.y}, c1);
  }
  static_for<0, 4>([&](auto kc) {
    static_for<0, 4>([&](auto sc) { a[decltype(kc)::value + 4 * decltype(sc)::value] = m[decltype(kc)::value][decltype(sc)::value]; });
  });
}

__host__ __device__ constexpr int pick_radix(int n) {
  return (n % 4 == 0) ? 4 : (n % 2 == 0) ? 2 : (n % 3 == 0) ? 3 : (n % 5 == 0) ? 5 : n;
}

__host__ __device__ constexpr bool radix_ok(int n) {
  if (n < 1) return false;
  while (n % 2 == 0) n /= 2;
  while (n % 3 == 0) n /= 3;
  while (n % 5 == 0) n /= 5;
  return n == 1;
}

__host__ __device__ constexpr int gcd_c(int a, int b) { return b == 0 ? a : gcd_c(b, a % b); }

// Coprime split N = N1 * N2 for the prime-factor algorithm: N1 = the power-of-two part, or
// the power-of-three part when N is odd; 0 when N is a prime power (no split exists).
__host__ __device__ constexpr int pfa_n1(int n) {
  int p2 = 1;
  while (n % (p2 * 2) == 0) p2 *= 2;
  if (p2 > 1 && p2 < n) return p2;
  int p3 = 1;
  while (n % (p3 * 3) == 0) p3 *= 3;
  if (p3 > 1 && p3 < n) return p3;
  return 0;
}

// k in [0, n1*n2) with k = k1 (mod n1) and k = k2 (mod n2)  (Chinese remainder theorem)
__host__ __device__ constexpr int crt_index(int k1, int k2, int n1, int n2) {
  int k = 0;
  while (k % n1 != k1 || k % n2 != k2) ++k;
  return k;
}

template <int N, int DIR, typename T>
__host__ __device__ __forceinline__ void fft(cpx<T>* a);

// Cooley-Tukey (decimation in time) for prime powers: N = R * M with twiddles (FOLD: the folded
// forms of 8 and 16).
template <int N, int DIR, typename T, bool FOLD = true>
__host__ __device__ __forceinline__ void fft_ct(cpx<T>* a) {
  constexpr int R = pick_radix(N);
  if constexpr (R == N) {
    Butterfly<N, DIR, T>::run(a);
  } else if constexpr (FOLD && N == 8) {
    fft8_fold<DIR, T>(a);
  } else if constexpr (FOLD && N == 16) {
    fft16_fold<DIR, T>(a);
  } else {
    constexpr int M = N / R;
    cpx<T> sub[R][M];
    static_for<0, R>([&](auto rc) {
      static_for<0, M>([&](auto mc) {
        sub[decltype(rc)::value][decltype(mc)::value] = a[decltype(mc)::value * R + decltype(rc)::value];
      });
    });
    static_for<0, R>([&](auto rc) { fft<M, DIR, T>(sub[decltype(rc)::value]); });
    static_for<0, M>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      cpx<T> t[R];
      static_for<0, R>([&](auto rc) {
        constexpr int r = decltype(rc)::value;
        t[r] = twiddle<N, r * k, DIR, T>(sub[r][k]);
      });
      Butterfly<R, DIR, T>::run(t);
      static_for<0, R>([&](auto sc) {
        constexpr int s = decltype(sc)::value;
        a[k + M * s] = t[s];
      });
    });
  }
}

// Prime-factor (Good-Thomas) algorithm for N = N1 * N2 with gcd(N1, N2) = 1: input index
// n = (N2 n1 + N1 n2) mod N, output index k = CRT(k1, k2); the 2-D DFT of size N1 x N2 that
// remains needs no twiddle factors.
template <int N, int DIR, typename T>
__host__ __device__ __forceinline__ void fft_pfa(cpx<T>* a) {
  constexpr int N1 = pfa_n1(N);
  constexpr int N2 = N / N1;
  static_assert(N1 > 1 && N2 > 1 && gcd_c(N1, N2) == 1, "prime-factor split");
  cpx<T> m[N1][N2];
  static_for<0, N1>([&](auto c1) {
    static_for<0, N2>([&](auto c2) {
      constexpr int n1 = decltype(c1)::value, n2 = decltype(c2)::value;
      constexpr int src = (N2 * n1 + N1 * n2) % N;
      m[n1][n2] = a[src];
    });
  });
  static_for<0, N1>([&](auto c1) { fft<N2, DIR, T>(m[decltype(c1)::value]); });
  static_for<0, N2>([&](auto c2) {
    constexpr int k2 = decltype(c2)::value;
    cpx<T> col[N1];
    static_for<0, N1>([&](auto c1) { col[decltype(c1)::value] = m[decltype(c1)::value][k2]; });
    // FP32 24 points: the 24^3 kernel has no registers to spare for the folded 8-point form
    // (24^3, 64 k, 32 sampled, 16 + 32 bands: 51.2 -> 52.1 ms with it)
    if constexpr (N1 == 8 && sizeof(T) == 4) fft_ct<N1, DIR, T, false>(col);
    else fft<N1, DIR, T>(col);
    static_for<0, N1>([&](auto c1) {
      constexpr int k1 = decltype(c1)::value;
      constexpr int k = crt_index(k1, k2, N1, N2);
      a[k] = col[k1];
    });
  });
}

// In-place DFT of length N on a register array: prime-factor split when N has two coprime
// factors, Cooley-Tukey otherwise.
template <int N, int DIR, typename T>
__host__ __device__ __forceinline__ void fft(cpx<T>* a) {
  static_assert(radix_ok(N), "axis length must factor into 2, 3, 5");
  if constexpr (N == 1) {
    return;
  } else if constexpr (pfa_n1(N) != 0) {
    fft_pfa<N, DIR, T>(a);
  } else {
    fft_ct<N, DIR, T>(a);
  }
}

}  // namespace hse
