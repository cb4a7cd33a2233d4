// Compile-time specialised real-line passes (r2c / c2r along the innermost
// axis) for the lengths of tfft_spec_table.h (the complex half-length).
#include "tfft_internal.h"
#include "tfft_spec_table.h"
#include "tfft_tiles.cuh"

namespace tfft {

namespace {

using namespace tiles;

// ------------------------------------------------------------ real lines
//
// Real-to-complex along the innermost axis (footnote to Eq. multifft: the
// Hermitian half k = 0 .. N/2).  A real line of N = 2L values is read as L
// complex values z[n] = x[2n] + i x[2n+1]; Z = FFT_L(z); then with
// w = exp(-2 pi i / N):  X[k] = (Z[k] + conj Z[L-k]) / 2
//                              - (i / 2) w^k (Z[k] - conj Z[L-k]),  k = 0 .. L.
// Complex-to-real inverts it: Z[k] = (X[k] + conj X[L-k])
//                              + i w^-k (X[k] - conj X[L-k]),  k < L,
// z = backward FFT_L(Z), x[2n] = Re z[n], x[2n+1] = Im z[n]; the imaginary
// parts of X[0] and X[L] are ignored (taken as zero).

// How the lines' Hermitian halves are spread over threads: the threads that
// synchronise together (a warp with 32 / T lines, or a line's T > 32 threads)
// take the pairs (k, L - k), k < L/2, of their lines in order, so that a warp
// reads or writes 32 consecutive elements of one row each way.  With T = 8
// threads a row, four rows per request in 64-byte pieces, the L1 was the
// bound (85 % busy in the c2r pass of 256^3, 45 % of its shared wavefronts
// bank conflicts).
template <int L, int T>
struct RealGroup {
  static constexpr int G = T > 32 ? T : 32;  // threads of a group
  static constexpr int LINES = G / T;
  static constexpr int NPAIR = (LINES * (L / 2) + G - 1) / G;
  static_assert(L % 2 == 0 && G % T == 0, "even lengths, whole lines");
  int lane, first;  // thread in the group, the group's first line in the CTA
  __device__ __forceinline__ RealGroup(int ly, int jt) {
    const unsigned tid = (unsigned)(ly * T + jt);
    lane = (int)(tid % G);
    first = (int)(tid / G) * LINES;
  }
  // Pair n of this thread: line i of the group and k; false past the end.
  __device__ __forceinline__ bool pair(int n, int& i, int& k) const {
    const unsigned u = (unsigned)(lane + n * G);
    i = (int)(u / (L / 2));
    k = (int)(u % (L / 2));
    return LINES * (L / 2) % G == 0 || u < (unsigned)(LINES * (L / 2));
  }
};

template <int L, int T, int B, int MB, bool CHAIN, int... Rs>
__global__ void __launch_bounds__(T * B, MB)
    k_r2c_spec(const RealArgs a) {
  constexpr int NST = sizeof...(Rs);
  constexpr int LP = line_pitch<L, Rs...>();
  constexpr int P = pad_every<Rs...>();
  extern __shared__ float2 smem[];
  const int ly = threadIdx.y;
  float2* sl = smem + ly * LP;
  if constexpr (CHAIN) {
    chain_next();
    chain_wait();
  }
  for (int64_t base = (int64_t)blockIdx.x * B; base < a.nlines; base += (int64_t)gridDim.x * B) {
    const int64_t line = base + ly;
    const bool act = line < a.nlines;
    const float2* src = reinterpret_cast<const float2*>(a.rin) + line * L;
    const int jt = opaque_tid_x();
    float2 v[emax<L, T, Rs...>()];
    static_for<0, NST>([&](auto S) {
      constexpr int s = decltype(S)::value;
      constexpr int R = radix_at<s, Rs...>();
      constexpr int Ns = span_at<s, Rs...>();
      if constexpr (s == 0) {
#pragma unroll
        for (int q = 0; q < nbf<L, T, R>(); ++q)
#pragma unroll
          for (int r = 0; r < R; ++r)
            v[q * R + r] = (act && bf_exists<L, T, R>(jt, q)) ? src[jt + q * T + r * (L / R)] : make_float2(0.f, 0.f);
      } else {
        constexpr int Rp = radix_at<s - 1, Rs...>();
        constexpr int Nsp = Ns / Rp;
        line_sync<T>();
#pragma unroll
        for (int q = 0; q < nbf<L, T, Rp>(); ++q)
          if (bf_exists<L, T, Rp>(jt, q))
#pragma unroll
            for (int r = 0; r < Rp; ++r) sl[padp<P>(stockham_out_index(jt + q * T, Nsp, Rp, r))] = v[q * Rp + r];
        line_sync<T>();
#pragma unroll
        for (int q = 0; q < nbf<L, T, R>(); ++q)
          if (bf_exists<L, T, R>(jt, q))
#pragma unroll
            for (int r = 0; r < R; ++r) v[q * R + r] = sl[padp<P>(jt + q * T + r * (L / R))];
      }
      constexpr int OFF = stage_table_off<s, Rs...>();
      spec_stage<L, T, R, Ns, OFF>(v, jt, OFF < 0 ? a.tw : a.tws);
    });
    constexpr int RL = radix_at<NST - 1, Rs...>();
    line_sync<T>();
#pragma unroll
    for (int q = 0; q < nbf<L, T, RL>(); ++q)
      if (bf_exists<L, T, RL>(jt, q))
#pragma unroll
        for (int r = 0; r < RL; ++r) sl[padp<P>(jt + q * T + r * (L / RL))] = v[q * RL + r];
    line_sync<T>();
    // outputs k and L - k together: with e, o of k, X[k] = e + o and, as
    // w^(L-k) = -conj(w^k) and the roles of Z[k], Z[L-k] swap,
    // X[L-k] = conj(e - o) -- one pair of shared loads and one twiddle for two
    // outputs (k = 0 gives X[0] and X[L]; k = L/2 is its own partner)
    const RealGroup<L, T> g(ly, jt);
    const int64_t gline = base + g.first;
    auto pair = [&](int i, int k, float2& lo, float2& hi) {
      const float2* z = smem + (g.first + i) * LP;
      const float2 zk = z[padp<P>(k)];
      const float2 zm = z[padp<P>(k == 0 ? 0 : L - k)];
      const float2 e = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));   // (Z[k] + conj Z[L-k]) / 2
      const float2 d = make_float2(0.5f * (zk.x - zm.x), 0.5f * (zk.y + zm.y));   // (Z[k] - conj Z[L-k]) / 2
      const float2 o = cmul(__ldg(&a.tw2[k]), mul_mi(d));                          // -i w^k d
      lo = cscale(cadd(e, o), a.scale);
      hi = cscale(make_float2(e.x - o.x, o.y - e.y), a.scale);
    };
#pragma unroll
    for (int n = 0; n < g.NPAIR; ++n) {
      int i, k;
      if (!g.pair(n, i, k)) continue;
      float2 lo, hi;
      pair(i, k, lo, hi);
      if (gline + i < a.nlines) {
        float2* row = a.cout + (gline + i) * a.cpitch;
        row[k] = lo;
        row[L - k] = hi;
      }
    }
    if (g.lane < g.LINES && gline + g.lane < a.nlines) {
      float2 lo, hi;
      pair(g.lane, L / 2, lo, hi);
      a.cout[(gline + g.lane) * a.cpitch + L / 2] = lo;
    }
  }
}

template <int L, int T, int B, int MB, bool CHAIN, int... Rs>
__global__ void __launch_bounds__(T * B, MB)
    k_c2r_spec(const RealArgs a) {
  constexpr int NST = sizeof...(Rs);
  constexpr int LP = line_pitch<L, Rs...>() + 1;
  constexpr int P = pad_every<Rs...>();
  extern __shared__ float2 smem[];
  const int ly = threadIdx.y;
  float2* sl = smem + ly * LP;
  if constexpr (CHAIN) {
    chain_next();
    chain_wait();
  }
  for (int64_t base = (int64_t)blockIdx.x * B; base < a.nlines; base += (int64_t)gridDim.x * B) {
    const int64_t line = base + ly;
    const bool act = line < a.nlines;
    float2* dst = reinterpret_cast<float2*>(a.rout) + line * L;
    const int jt = opaque_tid_x();
    // the L + 1 inputs as the pairs (X[k], X[L-k]), k < L/2 (k = 0 pairs X[0]
    // with X[L]), and X[L/2]: every load issued before the first shared store,
    // so that they are all in flight together
    const RealGroup<L, T> g(ly, jt);
    const int64_t gline = base + g.first;
    float2 xa[g.NPAIR], xb[g.NPAIR];
#pragma unroll
    for (int n = 0; n < g.NPAIR; ++n) {
      int i, k;
      const bool ok = g.pair(n, i, k) && gline + i < a.nlines;
      const float2* row = a.cin + (gline + i) * a.cpitch;
      xa[n] = ok ? row[k] : make_float2(0.f, 0.f);
      xb[n] = ok ? row[L - k] : make_float2(0.f, 0.f);
    }
    const bool mid = g.lane < g.LINES;
    float2 xmid = make_float2(0.f, 0.f);
    if (mid && gline + g.lane < a.nlines) xmid = a.cin[(gline + g.lane) * a.cpitch + L / 2];
    line_sync<T>();  // the previous line group is done with sl
    // Z[k] and Z[L-k] of each pair: with e, q = i w^-k d of k, Z[k] = e + q
    // and (w^-(L-k) = -w^k, the roles of X[k], X[L-k] swap) Z[L-k] =
    // conj(e - q); stored conjugated (backward = conj o forward o conj).
    // The imaginary parts of X[0] and X[L] are ignored; k = L/2 is its own
    // partner.
    auto store = [&](int i, int k, float2 xk, float2 xm) {
      float2* z = smem + (g.first + i) * LP;
      if (k == 0) {
        xk.y = 0.f;
        xm.y = 0.f;
      }
      const float2 e = make_float2(xk.x + xm.x, xk.y - xm.y);      // X[k] + conj X[L-k]
      const float2 d = make_float2(xk.x - xm.x, xk.y + xm.y);      // X[k] - conj X[L-k]
      const float2 w = __ldg(&a.tw2[k]);
      const float2 od = cmul(make_float2(w.x, -w.y), d);           // w^-k d
      const float2 qv = make_float2(-od.y, od.x);                  // i w^-k d
      z[padp<P>(k)] = make_float2(e.x + qv.x, -(e.y + qv.y));      // conj Z[k]
      if (k > 0 && 2 * k != L) z[padp<P>(L - k)] = make_float2(e.x - qv.x, e.y - qv.y);  // conj Z[L-k]
    };
#pragma unroll
    for (int n = 0; n < g.NPAIR; ++n) {
      int i, k;
      if (g.pair(n, i, k)) store(i, k, xa[n], xb[n]);
    }
    if (mid) store(g.lane, L / 2, xmid, xmid);
    line_sync<T>();
    float2 v[emax<L, T, Rs...>()];
    static_for<0, NST>([&](auto S) {
      constexpr int s = decltype(S)::value;
      constexpr int R = radix_at<s, Rs...>();
      constexpr int Ns = span_at<s, Rs...>();
      if constexpr (s == 0) {
#pragma unroll
        for (int q = 0; q < nbf<L, T, R>(); ++q)
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int k = bf_exists<L, T, R>(jt, q) ? jt + q * T + r * (L / R) : 0;
            v[q * R + r] = sl[padp<P>(k)];
          }
      } else {
        constexpr int Rp = radix_at<s - 1, Rs...>();
        constexpr int Nsp = Ns / Rp;
        line_sync<T>();
#pragma unroll
        for (int q = 0; q < nbf<L, T, Rp>(); ++q)
          if (bf_exists<L, T, Rp>(jt, q))
#pragma unroll
            for (int r = 0; r < Rp; ++r) sl[padp<P>(stockham_out_index(jt + q * T, Nsp, Rp, r))] = v[q * Rp + r];
        line_sync<T>();
#pragma unroll
        for (int q = 0; q < nbf<L, T, R>(); ++q)
          if (bf_exists<L, T, R>(jt, q))
#pragma unroll
            for (int r = 0; r < R; ++r) v[q * R + r] = sl[padp<P>(jt + q * T + r * (L / R))];
      }
      constexpr int OFF = stage_table_off<s, Rs...>();
      spec_stage<L, T, R, Ns, OFF>(v, jt, OFF < 0 ? a.tw : a.tws);
    });
    constexpr int RL = radix_at<NST - 1, Rs...>();
#pragma unroll
    for (int q = 0; q < nbf<L, T, RL>(); ++q)
#pragma unroll
      for (int r = 0; r < RL; ++r) {
        const float2 z = v[q * RL + r];
        if (act && bf_exists<L, T, RL>(jt, q)) dst[jt + q * T + r * (L / RL)] = make_float2(z.x * a.scale, -z.y * a.scale);
      }
  }
}

// the kernel's shared-memory limit raised to 227 KB, once per device
#define TFFT_ALLOW_SMEM(kernel)                          \
  static PerDevice<cudaError_t> attr_cache;              \
  const cudaError_t attr = smem_attr_once(attr_cache, kernel, 227 * 1024)

constexpr int64_t kMaxGrid = 1 << 20;

template <int L, int T, int B, int MB, bool CHAIN, int... Rs>
cudaError_t run_real(const RealArgs& a, cudaStream_t s) {
  if constexpr (!CHAIN && chainable(L))
    if (a.chained) return run_real<L, T, B, MB, true, Rs...>(a, s);
  const int64_t grid0 = (a.nlines + B - 1) / B;
  const int64_t grid = grid0 > kMaxGrid ? kMaxGrid : grid0;
  if (grid < 1) return cudaSuccess;
  if (a.dir < 0) {
    TFFT_ALLOW_SMEM((k_r2c_spec<L, T, B, MB, CHAIN, Rs...>));
    if (attr != cudaSuccess) return attr;
    const size_t smem = (size_t)B * line_pitch<L, Rs...>() * sizeof(float2);
    return launch_chained(k_r2c_spec<L, T, B, MB, CHAIN, Rs...>, dim3((unsigned)grid), dim3(T, B), smem, s, CHAIN ? a.chained : 0, a);
  } else {
    TFFT_ALLOW_SMEM((k_c2r_spec<L, T, B, MB, CHAIN, Rs...>));
    if (attr != cudaSuccess) return attr;
    const size_t smem = (size_t)B * (line_pitch<L, Rs...>() + 1) * sizeof(float2);
    return launch_chained(k_c2r_spec<L, T, B, MB, CHAIN, Rs...>, dim3((unsigned)grid), dim3(T, B), smem, s, CHAIN ? a.chained : 0, a);
  }
}

}  // namespace

namespace {

constexpr bool real_length(int L) {
#define X(LL) \
  if (L == LL) return true;
  TFFT_REAL_LENGTHS(X)
#undef X
  return false;
}

// the row of each real length (a template, so that the other rows are not
// instantiated)
template <class Args>
cudaError_t launch_real_row(const Args& a, cudaStream_t s) {
#define X(LL, T, B, MB, ...)                                              \
  if constexpr (real_length(LL) && std::is_same<Args, RealArgs>::value) \
    if (a.ap.L == LL) return run_real<LL, T, B, MB, false, __VA_ARGS__>(a, s);
  TFFT_CONTIG_LINES(X)
#undef X
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_real_spec(const RealArgs& a, cudaStream_t s) { return launch_real_row(a, s); }

}  // namespace tfft
