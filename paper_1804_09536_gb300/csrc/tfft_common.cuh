// Host/device shared definitions of the CUDA path: layout addressing on the
// virtual process grid, radix butterflies and the Stockham index schedule.
// Compiled by nvcc for the kernels and by the host compiler for the plan code.
#pragma once

#include <stdint.h>
#include <vector_types.h>
#include <vector_functions.h>

#if defined(__CUDACC__)
#define TFFT_HD __host__ __device__ __forceinline__
#else
#define TFFT_HD inline
#endif

namespace tfft {

constexpr int MAXD = 4;        // array dimensions
constexpr int MAXG = 3;        // grid dimensions
constexpr int MAXSTAGES = 12;  // radix stages of one 1-D FFT
constexpr int MAXLEN = 4096;   // longest transformed axis

// One alignment ("stage") of a d-D global array on the virtual grid.  Axis m
// is cut in Mx[m] parts by one grid direction (Mx[m] = 1 when the stage holds
// it whole) with the balanced block decomposition of Eq. decompose; the part
// index along that direction contributes part * rs[m] to the rank.  A rank's
// local array is C ordered and sits at element offset[rank] of the stage
// buffer.
struct DevLayout {
  int d;
  int64_t N[MAXD];
  int64_t Mx[MAXD];
  int64_t rs[MAXD];
  int32_t q[MAXD], r[MAXD];  // N / Mx and N mod Mx
  const int64_t* offset;  // nranks entries and the total (device memory in kernels)
  int64_t pitch;          // > 0: the innermost axis is stored `pitch` apart (a padded internal layout)
};

// Inverse of Eq. decompose: which part (coord) of N split in M holds global
// index g, g's index inside that part, and the part's length.  Extents are
// below 2^31, so 32-bit division suffices.
TFFT_HD void locate(int64_t N64, int64_t M64, int64_t g64, int64_t& coord, int64_t& local,
                    int64_t& n) {
  const uint32_t N = (uint32_t)N64, M = (uint32_t)M64, g = (uint32_t)g64;
  const uint32_t q = N / M, r = N - q * M;
  const uint32_t big = r * (q + 1);
  if (g < big) {
    const uint32_t c = g / (q + 1);
    coord = c;
    local = g - c * (q + 1);
    n = q + 1;
  } else {
    const uint32_t h = g - big;  // q >= 1 here because g < N
    const uint32_t c = h / q;
    coord = r + c;
    local = h - c * q;
    n = q;
  }
}

// ------------------------------------------------------------ complex math

TFFT_HD float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
TFFT_HD float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// The rounding order is spelled out on the device, so every kernel that
// applies the same twiddle gets the same bits, however the compiler would
// otherwise contract the products into FMAs.
TFFT_HD float2 cmul(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
#else
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
#endif
}
TFFT_HD float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// multiply by -i (the forward quarter turn)
TFFT_HD float2 mul_mi(float2 a) { return make_float2(a.y, -a.x); }

// Forward (sign -1) DFTs of size R on v[0..R-1], in place, natural order out.
template <int R>
struct Dft;

template <>
struct Dft<2> {
  TFFT_HD static void run(float2* v) {
    const float2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};

template <>
struct Dft<3> {
  TFFT_HD static void run(float2* v) {
    const float c = -0.5f, s = 0.86602540378443864676f;  // cos, sin of 2 pi / 3
    const float2 t = cadd(v[1], v[2]), u = csub(v[1], v[2]);
    const float2 a = v[0];
    const float2 m = make_float2(a.x + c * t.x, a.y + c * t.y);
    const float2 su = make_float2(s * u.y, -s * u.x);  // -i s u
    v[0] = cadd(a, t);
    v[1] = cadd(m, su);
    v[2] = csub(m, su);
  }
};

template <>
struct Dft<4> {
  TFFT_HD static void run(float2* v) {
    const float2 t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
    const float2 t2 = cadd(v[1], v[3]), t3 = mul_mi(csub(v[1], v[3]));
    v[0] = cadd(t0, t2);
    v[2] = csub(t0, t2);
    v[1] = cadd(t1, t3);
    v[3] = csub(t1, t3);
  }
};

template <>
struct Dft<5> {
  TFFT_HD static void run(float2* v) {
    const float c1 = 0.30901699437494742410f;   // cos(2 pi / 5)
    const float c2 = -0.80901699437494742410f;  // cos(4 pi / 5)
    const float s1 = 0.95105651629515357212f;   // sin(2 pi / 5)
    const float s2 = 0.58778525229247312917f;   // sin(4 pi / 5)
    const float2 a = v[0];
    const float2 t1 = cadd(v[1], v[4]), u1 = csub(v[1], v[4]);
    const float2 t2 = cadd(v[2], v[3]), u2 = csub(v[2], v[3]);
    const float2 m1 = make_float2(a.x + c1 * t1.x + c2 * t2.x, a.y + c1 * t1.y + c2 * t2.y);
    const float2 m2 = make_float2(a.x + c2 * t1.x + c1 * t2.x, a.y + c2 * t1.y + c1 * t2.y);
    // -i (s1 u1 + s2 u2) and -i (s2 u1 - s1 u2)
    const float2 p1 = mul_mi(make_float2(s1 * u1.x + s2 * u2.x, s1 * u1.y + s2 * u2.y));
    const float2 p2 = mul_mi(make_float2(s2 * u1.x - s1 * u2.x, s2 * u1.y - s1 * u2.y));
    v[0] = make_float2(a.x + t1.x + t2.x, a.y + t1.y + t2.y);
    v[1] = cadd(m1, p1);
    v[4] = csub(m1, p1);
    v[2] = cadd(m2, p2);
    v[3] = csub(m2, p2);
  }
};

template <>
struct Dft<8> {
  TFFT_HD static void run(float2* v) {
    const float h = 0.70710678118654752440f;  // sqrt(1/2)
    float2 e[4] = {v[0], v[2], v[4], v[6]};
    float2 o[4] = {v[1], v[3], v[5], v[7]};
    Dft<4>::run(e);
    Dft<4>::run(o);
    // o[k] *= exp(-2 pi i k / 8)
    o[1] = make_float2(h * (o[1].x + o[1].y), h * (o[1].y - o[1].x));
    o[2] = mul_mi(o[2]);
    o[3] = make_float2(h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = cadd(e[k], o[k]);
      v[k + 4] = csub(e[k], o[k]);
    }
  }
};

template <>
struct Dft<16> {
  TFFT_HD static void run(float2* v) {
    // 16 = 4 x 4: inner DFT4 over n2 for each n1 (n = 4 n2 + n1), twiddle
    // exp(-2 pi i n1 k1 / 16), outer DFT4 over n1; output k = k1 + 4 k2.
    const float c = 0.92387953251128675613f;  // cos(pi / 8)
    const float s = 0.38268343236508977173f;  // sin(pi / 8)
    const float h = 0.70710678118654752440f;
    float2 y[4][4];
#pragma unroll
    for (int n1 = 0; n1 < 4; ++n1) {
      y[n1][0] = v[n1];
      y[n1][1] = v[4 + n1];
      y[n1][2] = v[8 + n1];
      y[n1][3] = v[12 + n1];
      Dft<4>::run(y[n1]);
    }
    // twiddles w16^(n1 k1) for n1, k1 in 1..3
    const float2 w1 = make_float2(c, -s), w2 = make_float2(h, -h), w3 = make_float2(s, -c);
    const float2 w6 = make_float2(-h, -h), w9 = make_float2(-c, s);
    y[1][1] = cmul(y[1][1], w1);
    y[1][2] = cmul(y[1][2], w2);
    y[1][3] = cmul(y[1][3], w3);
    y[2][1] = cmul(y[2][1], w2);
    y[2][2] = mul_mi(y[2][2]);
    y[2][3] = cmul(y[2][3], w6);
    y[3][1] = cmul(y[3][1], w3);
    y[3][2] = cmul(y[3][2], w6);
    y[3][3] = cmul(y[3][3], w9);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      float2 z[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
      Dft<4>::run(z);
      v[k1] = z[0];
      v[k1 + 4] = z[1];
      v[k1 + 8] = z[2];
      v[k1 + 12] = z[3];
    }
  }
};

// exp(-2 pi i m / 32) for 0 <= m < 32, from cos(pi j / 16), j = 0..8, by
// the symmetries of the circle.
TFFT_HD float2 w32(int m) {
  const float c[9] = {1.0f,
                      0.98078528040323044913f,
                      0.92387953251128675613f,
                      0.83146961230254523708f,
                      0.70710678118654752440f,
                      0.55557023301960222474f,
                      0.38268343236508977173f,
                      0.19509032201612826785f,
                      0.0f};
  // cos and sin of pi m / 16 for m in [0, 32)
  const int q = m & 7, oct = m >> 3;  // m = 8 oct + q
  float cs, sn;
  switch (oct) {
    case 0: cs = c[q]; sn = c[8 - q]; break;
    case 1: cs = -c[8 - q]; sn = c[q]; break;
    case 2: cs = -c[q]; sn = -c[8 - q]; break;
    default: cs = c[8 - q]; sn = -c[q]; break;
  }
  return make_float2(cs, -sn);
}

template <>
struct Dft<32> {
  TFFT_HD static void run(float2* v) {
    // 32 = 4 x 8: inner DFT8 over n2 for each n1 (n = 4 n2 + n1), twiddle
    // exp(-2 pi i n1 k1 / 32), outer DFT4 over n1; output k = k1 + 8 k2.
    float2 y[4][8];
#pragma unroll
    for (int n1 = 0; n1 < 4; ++n1) {
#pragma unroll
      for (int n2 = 0; n2 < 8; ++n2) y[n1][n2] = v[4 * n2 + n1];
      Dft<8>::run(y[n1]);
    }
#pragma unroll
    for (int n1 = 1; n1 < 4; ++n1)
#pragma unroll
      for (int k1 = 1; k1 < 8; ++k1) y[n1][k1] = cmul(y[n1][k1], w32(n1 * k1));
#pragma unroll
    for (int k1 = 0; k1 < 8; ++k1) {
      float2 z[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
      Dft<4>::run(z);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) v[k1 + 8 * k2] = z[k2];
    }
  }
};

// ------------------------------------------------------------ composed DFTs
//
// The other radices: odd primes by their cosine / sine sums, composite ones
// by the prime factor map (coprime factors, no twiddles) or a Cooley-Tukey
// step with constant twiddles.  Every constant is formed in double precision
// at compile time.

// cos and sin of 2 pi m / n: m reduced to the first octant as an integer,
// then the Taylor series on [0, pi / 4] (below 2^-60 after these terms).
struct CosSin {
  double c, s;
};
constexpr CosSin cos_sin(int m, int n) {
  m %= n;
  // angle = (pi / 4) (8 m / n): octant, and the remainder's distance
  const int o = 8 * m / n;
  const int up = (o & 1) ? (o + 1) * n - 8 * m : 8 * m - o * n;  // distance to the even octant edge, in n-ths of pi / 4
  const double x = 0.78539816339744830961566 * (double)up / (double)n;
  double c = 0.0, s = 0.0, t = 1.0;
  for (int k = 0; k < 24; ++k) {  // t = x^k / k!
    if (k & 1) s += (k & 2) ? -t : t;
    else c += (k & 2) ? -t : t;
    t = t * x / (double)(k + 1);
  }
  // edge e = ((o + 1) / 2) quarter turns; x is measured from it, forward for even octants, backward for odd ones
  if (o & 1) s = -s;
  switch (((o + 1) / 2) & 3) {
    case 0: return CosSin{c, s};
    case 1: return CosSin{-s, c};
    case 2: return CosSin{-c, -s};
    default: return CosSin{s, -c};
  }
}

// exp(-2 pi i M / N) as a pair of compile-time floats.
template <int N, int M>
struct Root {
  static constexpr float re = (float)cos_sin(M % N, N).c;
  static constexpr float im = (float)-cos_sin(M % N, N).s;
};

template <int I>
struct IntC {
  static constexpr int value = I;
};
template <int I, int N, class F>
TFFT_HD void unrolled(F&& f) {
  if constexpr (I < N) {
    f(IntC<I>{});
    unrolled<I + 1, N>(f);
  }
}

// Odd prime P: with t_k = v_k + v_{P-k}, u_k = v_k - v_{P-k}, k <= (P - 1) / 2,
// X_j, X_{P-j} = v_0 + sum t_k cos(2 pi j k / P) -+ i sum u_k sin(2 pi j k / P).
template <int P>
struct DftPrime {
  TFFT_HD static void run(float2* v) {
    constexpr int H = (P - 1) / 2;
    float2 t[H], u[H];
    const float2 a = v[0];
#pragma unroll
    for (int k = 0; k < H; ++k) {
      t[k] = cadd(v[k + 1], v[P - 1 - k]);
      u[k] = csub(v[k + 1], v[P - 1 - k]);
    }
    float2 sum = a;
#pragma unroll
    for (int k = 0; k < H; ++k) sum = cadd(sum, t[k]);
    v[0] = sum;
    unrolled<1, H + 1>([&](auto J) {
      constexpr int j = decltype(J)::value;
      float2 m = a, s = make_float2(0.f, 0.f);
      unrolled<1, H + 1>([&](auto K) {
        constexpr int k = decltype(K)::value;
        constexpr float c = Root<P, (j * k) % P>::re, sn = -Root<P, (j * k) % P>::im;
        m = make_float2(m.x + c * t[k - 1].x, m.y + c * t[k - 1].y);
        s = make_float2(s.x + sn * u[k - 1].x, s.y + sn * u[k - 1].y);
      });
      const float2 q = mul_mi(s);
      v[j] = cadd(m, q);
      v[P - j] = csub(m, q);
    });
  }
};
template <>
struct Dft<7> : DftPrime<7> {};

constexpr int gcd_of(int a, int b) { return b == 0 ? a : gcd_of(b, a % b); }
constexpr int inverse_mod(int a, int m) {
  for (int x = 1; x < m; ++x)
    if (a * x % m == 1) return x;
  return 1;
}

// N = A B.  Coprime: n = (B n1 + A n2) mod N, k = (B (1/B mod A) k1 +
// A (1/A mod B) k2) mod N turns the DFT into A x B DFTs without twiddles.
// Otherwise n = A n2 + n1, k = k1 + B k2: size-B DFTs over n2, twiddles
// exp(-2 pi i n1 k1 / N), size-A DFTs over n1.
template <int A, int B>
struct DftPair {
  TFFT_HD static void run(float2* v) {
    constexpr int N = A * B;
    constexpr bool coprime = gcd_of(A, B) == 1;
    float2 y[A][B];
    unrolled<0, A>([&](auto N1) {
      constexpr int n1 = decltype(N1)::value;
#pragma unroll
      for (int n2 = 0; n2 < B; ++n2) y[n1][n2] = v[coprime ? (B * n1 + A * n2) % N : A * n2 + n1];
      Dft<B>::run(y[n1]);
      if constexpr (!coprime && n1 > 0)
        unrolled<1, B>([&](auto K1) {
          constexpr int k1 = decltype(K1)::value;
          y[n1][k1] = cmul(y[n1][k1], make_float2(Root<N, n1 * k1>::re, Root<N, n1 * k1>::im));
        });
    });
#pragma unroll
    for (int k1 = 0; k1 < B; ++k1) {
      float2 z[A];
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) z[n1] = y[n1][k1];
      Dft<A>::run(z);
#pragma unroll
      for (int k2 = 0; k2 < A; ++k2)
        v[coprime ? (A * inverse_mod(A % B, B) * k1 + B * inverse_mod(B % A, A) * k2) % N : k1 + B * k2] = z[k2];
    }
  }
};
template <>
struct Dft<6> : DftPair<2, 3> {};
template <>
struct Dft<9> : DftPair<3, 3> {};
template <>
struct Dft<10> : DftPair<2, 5> {};
template <>
struct Dft<12> : DftPair<3, 4> {};
template <>
struct Dft<14> : DftPair<2, 7> {};
template <>
struct Dft<15> : DftPair<3, 5> {};
template <>
struct Dft<18> : DftPair<2, 9> {};
template <>
struct Dft<20> : DftPair<4, 5> {};
template <>
struct Dft<21> : DftPair<3, 7> {};
template <>
struct Dft<24> : DftPair<3, 8> {};
template <>
struct Dft<25> : DftPair<5, 5> {};
template <>
struct Dft<27> : DftPair<3, 9> {};
template <>
struct Dft<28> : DftPair<4, 7> {};
template <>
struct Dft<30> : DftPair<2, 15> {};

// ------------------------------------------------------------ Stockham schedule
//
// A length-L FFT with radices R_0, R_1, ... (product L).  Stage s has span
// Ns = R_0 ... R_{s-1}.  Work item j (0 <= j < L / R) of a stage reads
// x[j + r L / R] (r < R), multiplies input r by exp(-2 pi i r k / (Ns R)),
// k = j mod Ns, runs a size-R DFT and writes output r to
// (j / Ns) Ns R + k + r Ns.  After the last stage the result is in natural
// order (self-sorting).  Twiddles are read from one table of the L roots
// exp(-2 pi i m / L), index m = r k L / (Ns R) < L.

TFFT_HD int stockham_out_index(int j, int Ns, int R, int r) {
  const int k = j % Ns;
  return (j / Ns) * Ns * R + k + r * Ns;
}

TFFT_HD int stockham_tw_index(int j, int Ns, int R, int r, int L) {
  const int k = j % Ns;
  return r * k * (L / (Ns * R));
}

// FFT plan of one axis length, shared by host planning and device kernels.
// The radices are also packed 5 bits per stage in `code` so that kernels read
// stage s's radix with a shift instead of an indexed load.  The struct goes by
// value into every kernel, ahead of the geometry and the tensor maps: one more
// int moved those and cost the TMA-staged passes 0.6 % (512^3 1948 -> 1960 us).
struct AxisPlan {
  int L;           // transform length
  int E;           // runtime-radix kernels: elements per thread (every radix divides E), 0 = generic;
                   // compiled rows: ceil(L / T), but a thread holds emax<L, T, radices>() values
  int T;           // threads per line
  int nst;         // number of radix stages
  uint64_t code;   // radix of stage s = (code >> 5 s) & 31
  int spec;        // 1: a compile-time specialised kernel exists for this plan
  int width;       // lines per CTA (contiguous) or tile width W (strided)
  int radix[MAXSTAGES];
  int blue_m;      // > 0: length without a 2/3/5 plan, done by Bluestein with this convolution length
  int blue_spec;   // 1: that convolution length has compile-time specialised kernels (width is theirs);
                   // 2: strided passes of a prime length by Rader's convolution (width is theirs)
};

TFFT_HD int stage_radix(uint64_t code, int s) { return (int)((code >> (5 * s)) & 31); }

}  // namespace tfft
