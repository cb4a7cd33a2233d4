// Bluestein passes with compile-time specialised convolution lengths.
//
// A line of length N with no compiled factorisation (the paper only needs some
// serial 1-D FFT per axis; App. A's 42 x 127 x 256 has one such axis) is
// transformed as a circular convolution: with the chirp c[n] = exp(-i pi
// (n^2 mod 2N) / N),  X[k] = c[k] sum_n (x[n] c[n]) conj(c[k - n]),  i.e.
// y = x c zero-padded to M >= 2N - 1 (even), Y = FFT_M(y) bhat with
// bhat = FFT_M(b) / M for the wrapped filter b[m] = b[M - m] = conj(c[m]),
// X = c IFFT_M(Y), the inverse taken as conj o FFT_M o conj.  Both length-M
// FFTs run as register-resident Stockham stages.  The second one takes the
// radices in reverse order: its first stage then wants exactly the values its
// thread holds after the first FFT's last stage (both at j + r M / R), so the
// filter is applied in registers and nothing is exchanged between the two.
// N <= M / 2, so the upper half of the first stage's inputs is zero and the
// upper half of the last stage's outputs is not needed: neither is loaded,
// multiplied or stored.  One read and one write of every element, as in the
// other passes.  The chirp and filter tables are built on the host in double
// precision and rounded once.
#pragma once

#include "tfft_tiles.cuh"

namespace tfft {
namespace blue {

using namespace tiles;

__device__ __forceinline__ float2 conjf2(float2 a) { return make_float2(a.x, -a.y); }

template <int... Rs>
struct Radices {};
template <class Done, int... Rs>
struct Reverse;
template <int... D>
struct Reverse<Radices<D...>> {
  using type = Radices<D...>;
};
template <int... D, int R, int... Rs>
struct Reverse<Radices<D...>, R, Rs...> : Reverse<Radices<R, D...>, Rs...> {};

// Pitch of a line's shared slot: the padding differs between the two orders of
// the radices.
template <int M, int... Rs>
__host__ __device__ constexpr int rev_pitch(Radices<Rs...>) {
  return line_pitch<M, Rs...>();
}
template <int M, int... Rs>
__host__ __device__ constexpr int blue_line_pitch() {
  constexpr int a = line_pitch<M, Rs...>(), b = rev_pitch<M>(typename Reverse<Radices<>, Rs...>::type{});
  return a > b ? a : b;
}

// Inputs of a first stage (outputs of a last stage) of radix R that can be
// non-zero (are needed): r < (R + 1) / 2, as the others lie at or above M / 2.
template <int R>
__host__ __device__ constexpr int half_of() {
  return (R + 1) / 2;
}

// Filter on the values held after the first FFT, conjugated for the inverse.
template <int M, int T, int RL, int EM>
__device__ __forceinline__ void apply_filter(float2 (&v)[EM], int jt, const float2* __restrict__ bhat) {
#pragma unroll
  for (int q = 0; q < nbf<M, T, RL>(); ++q)
    if (bf_exists<M, T, RL>(jt, q))
#pragma unroll
      for (int r = 0; r < RL; ++r)
        v[q * RL + r] = conjf2(cmul(v[q * RL + r], __ldg(&bhat[jt + q * T + r * (M / RL)])));
}

// One of the two FFTs of a line, in its column of a tile or its own slot.
template <int M, int T, int W, bool STRIDED, int EM, int... Rs>
__device__ __forceinline__ void stages(Radices<Rs...>, float2 (&v)[EM], float2* sl, int cx, int jt,
                                       const float2* __restrict__ tw) {
  if constexpr (STRIDED) strided_stages<M, T, W, Rs...>(v, sl, cx, jt, tw);
  else line_stages<M, T, Rs...>(v, sl, jt, tw);
}

// ------------------------------------------------------------ contiguous lines

// B lines per CTA, thread jt of line ly; lines are N long in memory.
template <int M, int T, int B, int MB, int... Rs>
__global__ void __launch_bounds__(T * B, MB) k_blue_contig_spec(const ContigArgs a, const BlueArgs b) {
  constexpr int NST = sizeof...(Rs);
  constexpr int R0 = radix_at<0, Rs...>(), RL = radix_at<NST - 1, Rs...>();
  using Rev = typename Reverse<Radices<>, Rs...>::type;
  constexpr int LP = blue_line_pitch<M, Rs...>();
  extern __shared__ float2 smem[];
  const int N = b.N;
  const int ly = threadIdx.y;
  float2* sl = smem + ly * LP;
  const bool inv = a.sign > 0;
  chain_next();
  chain_wait();
  const float oscale = contig_scale(a);
  for (int64_t base = (int64_t)blockIdx.x * B; base < a.nlines; base += (int64_t)gridDim.x * B) {
    const int64_t line = base + ly;
    const bool act = line < a.nlines;
    const float2* src = a.in + line * N;
    float2* dst = a.out + line * N;
    const int jt = opaque_tid_x();
    float2 v[emax<M, T, Rs...>()];
#pragma unroll
    for (int q = 0; q < nbf<M, T, R0>(); ++q)
#pragma unroll
      for (int r = 0; r < R0; ++r) {
        const int pos = jt + q * T + r * (M / R0);
        float2 x = make_float2(0.f, 0.f);
        if (r < half_of<R0>() && act && pos < N && bf_exists<M, T, R0>(jt, q)) {
          x = src[pos];
          if (inv) x.y = -x.y;
          x = cmul(x, __ldg(&b.chirp[pos]));
        }
        v[q * R0 + r] = x;
      }
    stages<M, T, 0, false>(Radices<Rs...>{}, v, sl, 0, jt, b.tws_f);
    apply_filter<M, T, RL>(v, jt, b.bhat);
    stages<M, T, 0, false>(Rev{}, v, sl, 0, jt, b.tws_r);
#pragma unroll
    for (int q = 0; q < nbf<M, T, R0>(); ++q)
#pragma unroll
      for (int r = 0; r < half_of<R0>(); ++r) {
        const int p = jt + q * T + r * (M / R0);
        if (act && p < N && bf_exists<M, T, R0>(jt, q)) {
          float2 y = cscale(cmul(conjf2(v[q * R0 + r]), __ldg(&b.chirp[p])), oscale);
          if (inv) y.y = -y.y;
          dst[p] = y;
        }
      }
    line_sync<T>();  // the line slot is free for the next group
  }
}

// ------------------------------------------------------------ strided lines

// Tile = the N rows of W columns, held as M x W in shared memory between the
// stages; row tables of the input and output layouts (tile_fold /
// row_offset) and a per-CTA table of every row's part and index.
template <int M, int W>
__host__ __device__ constexpr size_t blue_strided_smem(int N) {
  return (size_t)M * W * sizeof(float2) + 2 * (size_t)N * sizeof(int) + sizeof(TileShared) +
         2 * (size_t)N * sizeof(uint32_t) + 16;
}

template <int M, int T, int W, int MB, int... Rs>
__global__ void __launch_bounds__(W * T, MB) k_blue_strided_spec(const StridedArgs a, const BlueArgs b) {
  constexpr int NST = sizeof...(Rs);
  constexpr int R0 = radix_at<0, Rs...>(), RL = radix_at<NST - 1, Rs...>();
  using Rev = typename Reverse<Radices<>, Rs...>::type;
  static_assert(W * T > 32, "the two layouts' folds are computed by threads 0 and 32");
  extern __shared__ float2 smem[];
  const int N = b.N;
  TileShared* ts = reinterpret_cast<TileShared*>(smem + M * W);
  int* rin = reinterpret_cast<int*>(ts + 1);
  int* rout = rin + N;
  uint32_t* rp = reinterpret_cast<uint32_t*>(rout + N);
  const int cx = threadIdx.x;
  const int tid = threadIdx.y * W + cx;
  const bool inv = a.sign > 0;
  const int64_t ntiles = a.nouter * a.ncolblocks;
  chain_next();
  // part and index of every row of both layouts, once per CTA
  for (int i = tid; i < 2 * N; i += W * T) {
    const bool out = i >= N;
    const int row = out ? i - N : i;
    const int64_t NN = out ? a.lout.N[a.axis] : a.lin.N[a.axis];
    const int64_t MM = out ? a.lout.Mx[a.axis] : a.lin.Mx[a.axis];
    int64_t c = 0, l = row, n = NN;
    if (MM > 1) locate(NN, MM, row, c, l, n);
    rp[i] = ((uint32_t)c << 16) | (uint32_t)l;
  }
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    __syncthreads();  // the previous tile is done with the tables, the scalars and smem
    if (tid == 0) {
      const StridedTilePos tp(a, tile);
      tile_fold(a, a.lin, tp, ts, 0);
      ts->blk = tp.blk;
    } else if (tid == 32) {
      const StridedTilePos tp(a, tile);
      tile_fold(a, a.lout, tp, ts, 1);
    }
    __syncthreads();
    for (int i = tid; i < 2 * N; i += W * T) {
      const bool out = i >= N;
      const int row = out ? i - N : i;
      const int64_t c = rp[i] >> 16, l = rp[i] & 0xFFFF;
      if (out)
        rout[row] = row_offset(a.lout, a.axis, ts, 1, c, l);
      else
        rin[row] = row_offset(a.lin, a.axis, ts, 0, c, l);
    }
    __syncthreads();
    const int2 blk = ts->blk;
    const bool act = cx < blk.y;
    const int jt = opaque_tid_y();
    if (tile == blockIdx.x) chain_wait();
    float2 v[emax<M, T, Rs...>()];
#pragma unroll
    for (int q = 0; q < nbf<M, T, R0>(); ++q)
#pragma unroll
      for (int r = 0; r < R0; ++r) {
        const int pos = jt + q * T + r * (M / R0);
        float2 x = make_float2(0.f, 0.f);
        if (r < half_of<R0>() && act && pos < N && bf_exists<M, T, R0>(jt, q)) {
          x = a.in[rin[pos] + cx];
          if (inv) x.y = -x.y;
          x = cmul(x, __ldg(&b.chirp[pos]));
        }
        v[q * R0 + r] = x;
      }
    stages<M, T, W, true>(Radices<Rs...>{}, v, smem, cx, jt, b.twm);
    apply_filter<M, T, RL>(v, jt, b.bhat);
    stages<M, T, W, true>(Rev{}, v, smem, cx, jt, b.twm);
#pragma unroll
    for (int q = 0; q < nbf<M, T, R0>(); ++q)
#pragma unroll
      for (int r = 0; r < half_of<R0>(); ++r) {
        const int p = jt + q * T + r * (M / R0);
        if (act && p < N && bf_exists<M, T, R0>(jt, q)) {
          float2 y = cscale(cmul(conjf2(v[q * R0 + r]), __ldg(&b.chirp[p])), a.scale);
          if (inv) y.y = -y.y;
          a.out[rout[p] + cx] = y;
        }
      }
  }
}

// ------------------------------------------------------------ prime lengths
//
// Rader's form for a prime N whose M = N - 1 has compiled stages: with a
// primitive root g, X[g^-k] = x[0] + sum_q x[g^q] w^(g^(q - k)) is a cyclic
// convolution of length N - 1 itself, against Bluestein's 2N - 1 or more, and
// the permutations cost nothing where rows are read and written through
// tables: position q of the tile is row g^q on the way in and row g^-q on the
// way out.  Y = FFT_M(x[g^q]) bhat with bhat = FFT_M(w^(g^-q)) / M; x[0] added
// to Y[0] reaches every output of the inverse, and X[0] is x[0] plus bin 0 of
// the first FFT, both in the hands of one thread.
template <int M, int W>
__host__ __device__ constexpr size_t rader_strided_smem() {
  return (size_t)M * W * sizeof(float2) + 2 * (size_t)(M + 1) * sizeof(int) + sizeof(TileShared) +
         2 * (size_t)(M + 1) * sizeof(uint32_t) + 16;
}

template <int M, int T, int W, int MB, int... Rs>
__global__ void __launch_bounds__(W * T, MB) k_rader_strided(const StridedArgs a, const BlueArgs b) {
  constexpr int NST = sizeof...(Rs), N = M + 1;
  constexpr int R0 = radix_at<0, Rs...>(), RL = radix_at<NST - 1, Rs...>();
  using Rev = typename Reverse<Radices<>, Rs...>::type;
  static_assert(W * T > 32, "the two layouts' folds are computed by threads 0 and 32");
  extern __shared__ float2 smem[];
  TileShared* ts = reinterpret_cast<TileShared*>(smem + M * W);
  int* rin = reinterpret_cast<int*>(ts + 1);
  int* rout = rin + N;
  uint32_t* rp = reinterpret_cast<uint32_t*>(rout + N);
  const int cx = threadIdx.x;
  const int tid = threadIdx.y * W + cx;
  const bool inv = a.sign > 0;
  const int64_t ntiles = a.nouter * a.ncolblocks;
  chain_next();
  // part and index of every position's row in both layouts, once per CTA:
  // position i < M is row perm[i], position M is row 0
  for (int i = tid; i < 2 * N; i += W * T) {
    const bool out = i >= N;
    const int pos = out ? i - N : i;
    const int row = pos < M ? __ldg(&b.perm[out ? M + pos : pos]) : 0;
    const int64_t NN = out ? a.lout.N[a.axis] : a.lin.N[a.axis];
    const int64_t MM = out ? a.lout.Mx[a.axis] : a.lin.Mx[a.axis];
    int64_t c = 0, l = row, n = NN;
    if (MM > 1) locate(NN, MM, row, c, l, n);
    rp[i] = ((uint32_t)c << 16) | (uint32_t)l;
  }
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    __syncthreads();  // the previous tile is done with the tables, the scalars and smem
    if (tid == 0) {
      const StridedTilePos tp(a, tile);
      tile_fold(a, a.lin, tp, ts, 0);
      ts->blk = tp.blk;
    } else if (tid == 32) {
      const StridedTilePos tp(a, tile);
      tile_fold(a, a.lout, tp, ts, 1);
    }
    __syncthreads();
    for (int i = tid; i < 2 * N; i += W * T) {
      const bool out = i >= N;
      const int64_t c = rp[i] >> 16, l = rp[i] & 0xFFFF;
      if (out)
        rout[i - N] = row_offset(a.lout, a.axis, ts, 1, c, l);
      else
        rin[i] = row_offset(a.lin, a.axis, ts, 0, c, l);
    }
    __syncthreads();
    const int2 blk = ts->blk;
    const bool act = cx < blk.y;
    const int jt = opaque_tid_y();
    if (tile == blockIdx.x) chain_wait();
    float2 v[emax<M, T, Rs...>()];
#pragma unroll
    for (int q = 0; q < nbf<M, T, R0>(); ++q)
#pragma unroll
      for (int r = 0; r < R0; ++r) {
        float2 x = make_float2(0.f, 0.f);
        if (act && bf_exists<M, T, R0>(jt, q)) x = a.in[rin[jt + q * T + r * (M / R0)] + cx];
        if (inv) x.y = -x.y;
        v[q * R0 + r] = x;
      }
    // x[0], for the thread that holds bin 0 of the convolution
    float2 x0 = make_float2(0.f, 0.f);
    if (act && jt == 0) {
      x0 = a.in[rin[M] + cx];
      if (inv) x0.y = -x0.y;
    }
    stages<M, T, W, true>(Radices<Rs...>{}, v, smem, cx, jt, b.twr);
    const float2 sum = v[0];
    apply_filter<M, T, RL>(v, jt, b.rhat);
    if (jt == 0) {
      v[0] = cadd(v[0], conjf2(x0));
      if (act) {
        float2 y = cscale(cadd(sum, x0), a.scale);
        if (inv) y.y = -y.y;
        a.out[rout[M] + cx] = y;
      }
    }
    stages<M, T, W, true>(Rev{}, v, smem, cx, jt, b.twr);
#pragma unroll
    for (int q = 0; q < nbf<M, T, R0>(); ++q)
#pragma unroll
      for (int r = 0; r < R0; ++r)
        if (act && bf_exists<M, T, R0>(jt, q)) {
          float2 y = cscale(conjf2(v[q * R0 + r]), a.scale);
          if (inv) y.y = -y.y;
          a.out[rout[jt + q * T + r * (M / R0)] + cx] = y;
        }
  }
}

// Compiled M = N - 1: threads per column, tile width, CTAs per SM, radices.
#define TFFT_RADER_STRIDED(X) \
  X(28, 2, 32, 12, 14, 2)     \
  X(30, 2, 32, 12, 15, 2)     \
  X(36, 3, 32, 8, 6, 6)       \
  X(40, 2, 32, 10, 2, 20)     \
  X(42, 3, 32, 8, 14, 3)      \
  X(60, 4, 32, 6, 15, 4)      \
  X(70, 5, 32, 4, 14, 5)      \
  X(72, 6, 16, 8, 6, 12)      \
  X(96, 4, 32, 4, 8, 12)      \
  X(100, 5, 32, 4, 20, 5)     \
  X(108, 6, 16, 6, 18, 6)     \
  X(112, 8, 16, 6, 8, 14)     \
  X(126, 7, 16, 4, 21, 6)     \
  X(150, 5, 16, 6, 5, 30)     \
  X(162, 9, 16, 4, 9, 18)     \
  X(180, 15, 16, 3, 15, 12)   \
  X(192, 16, 16, 3, 16, 12)   \
  X(196, 14, 16, 3, 14, 14)   \
  X(210, 15, 16, 3, 15, 14)   \
  X(240, 16, 16, 3, 16, 15)   \
  X(250, 13, 16, 2, 25, 10)   \
  X(256, 16, 16, 3, 16, 16)   \
  X(270, 18, 16, 2, 15, 18)   \
  X(280, 10, 16, 3, 28, 10)   \
  X(336, 14, 16, 2, 28, 12)   \
  X(378, 14, 16, 2, 14, 27)   \
  X(400, 20, 16, 2, 20, 20)   \
  X(420, 21, 16, 1, 20, 21)   \
  X(432, 24, 16, 1, 24, 18)   \
  X(448, 32, 16, 1, 8, 14, 4) \
  X(486, 54, 16, 1, 9, 6, 9)  \
  X(490, 35, 16, 1, 14, 5, 7)

// Compiled convolution lengths.  Contiguous: M, threads per line, lines per
// CTA, CTAs per SM, radices; strided: M, threads per column, tile width, CTAs
// per SM, radices.  The passes are bound by instruction issue, so a length
// takes the smallest compiled M >= 2N - 1 rather than the next power of two;
// the set holds the lengths whose two FFTs cost least for their size (timed
// on 2^25 elements, us per pass at N = M / 2: 144 225, 180 276, 256 264, 360
// 330, 400 322, 512 387, 576 340, 800 411, 1024 478; e.g. N = 180 through
// 360 takes 0.6 of the time through 512).  A tighter M also spreads the
// rounding of the convolution over fewer unneeded outputs: against the power of
// two the relative error of one transform of such a line is 1.05 - 1.17 times
// as large in the mean over the lengths of an M (576 1.01, 800 1.06, 90, for
// 42 < N < 46, 1.19; 1.24 at most, N = 190: 1.35e-7 -> 1.67e-7), and 1.00 - 1.01
// where M stays a power of two.
#define TFFT_BLUE_CONTIG(X)            \
  X(32, 4, 64, 4, 8, 4)                \
  X(48, 4, 64, 4, 12, 4)               \
  X(64, 8, 32, 4, 8, 8)                \
  X(72, 9, 28, 4, 9, 8)                \
  X(80, 10, 25, 4, 10, 8)              \
  X(90, 10, 25, 4, 10, 9)              \
  X(128, 8, 32, 3, 16, 8)              \
  X(144, 12, 21, 3, 12, 12)            \
  X(180, 16, 16, 3, 12, 15)            \
  X(256, 16, 16, 3, 16, 16)            \
  X(288, 12, 21, 2, 24, 12)            \
  X(360, 20, 12, 2, 18, 20)            \
  X(400, 20, 12, 2, 20, 20)            \
  X(576, 32, 8, 2, 24, 24)             \
  X(800, 40, 6, 2, 4, 20, 10)          \
  X(1024, 64, 4, 3, 16, 16, 4)         \
  X(2048, 128, 2, 3, 16, 16, 8)        \
  X(4096, 256, 1, 3, 16, 16, 16)
#define TFFT_BLUE_STRIDED(X)           \
  X(32, 4, 32, 8, 8, 4)                \
  X(48, 4, 32, 8, 4, 12)               \
  X(64, 8, 16, 8, 8, 8)                \
  X(72, 6, 16, 8, 12, 6)               \
  X(80, 10, 16, 6, 10, 8)              \
  X(90, 10, 16, 6, 9, 10)              \
  X(128, 8, 16, 6, 16, 8)              \
  X(144, 12, 16, 4, 12, 12)            \
  X(180, 15, 16, 3, 12, 15)            \
  X(256, 16, 16, 3, 16, 16)            \
  X(288, 24, 16, 2, 4, 6, 12)          \
  X(360, 20, 16, 2, 18, 20)            \
  X(400, 20, 16, 2, 20, 20)            \
  X(576, 48, 8, 2, 12, 4, 12)          \
  X(800, 40, 8, 2, 4, 10, 20)          \
  X(1024, 64, 8, 1, 16, 16, 4)         \
  X(2048, 128, 4, 1, 16, 16, 8)        \
  X(4096, 256, 2, 1, 16, 16, 16)

// the kernel's shared-memory limit raised to 227 KB, once per device
#define TFFT_ALLOW_SMEM(kernel)                          \
  static PerDevice<cudaError_t> attr_cache;              \
  const cudaError_t attr = smem_attr_once(attr_cache, kernel, 227 * 1024)

template <int M, int T, int B, int MB, int... Rs>
cudaError_t run_blue_contig(const ContigArgs& a, const BlueArgs& b, cudaStream_t s) {
  constexpr int64_t kMaxGrid = 1 << 20;
  TFFT_ALLOW_SMEM((k_blue_contig_spec<M, T, B, MB, Rs...>));
  if (attr != cudaSuccess) return attr;
  if (a.lines_per_cta != B || 2 * b.N > M) return cudaErrorInvalidValue;
  const size_t smem = (size_t)B * blue_line_pitch<M, Rs...>() * sizeof(float2);
  int64_t grid = (a.nlines + B - 1) / B;
  if (grid > kMaxGrid) grid = kMaxGrid;
  if (grid < 1) return cudaSuccess;
  return launch_chained(k_blue_contig_spec<M, T, B, MB, Rs...>, dim3((unsigned)grid), dim3(T, B), smem, s, a.chained, a,
                        b);
}

template <int M, int T, int W, int MB, int... Rs>
cudaError_t run_blue_strided(const StridedArgs& a, const BlueArgs& b, cudaStream_t s) {
  TFFT_ALLOW_SMEM((k_blue_strided_spec<M, T, W, MB, Rs...>));
  if (attr != cudaSuccess) return attr;
  if (a.W != W || 2 * b.N > M) return cudaErrorInvalidValue;
  const size_t smem = blue_strided_smem<M, W>(b.N);
  // persistent: the per-CTA row table is computed once
  static PerDevice<int64_t> slots_cache;
  const int64_t slots = slots_cache.get(current_device(), [&] {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_blue_strided_spec<M, T, W, MB, Rs...>, W * T,
                                                  blue_strided_smem<M, W>(M / 2));
    return (int64_t)device_sm_count() * (per_sm > 0 ? per_sm : 1);
  });
  int64_t grid = a.nouter * a.ncolblocks;
  if (grid > slots) grid = slots;
  if (grid < 1) return cudaSuccess;
  return launch_chained(k_blue_strided_spec<M, T, W, MB, Rs...>, dim3((unsigned)grid), dim3(W, T), smem, s, a.chained, a,
                        b);
}

template <int M, int T, int W, int MB, int... Rs>
cudaError_t run_rader_strided(const StridedArgs& a, const BlueArgs& b, cudaStream_t s) {
  TFFT_ALLOW_SMEM((k_rader_strided<M, T, W, MB, Rs...>));
  if (attr != cudaSuccess) return attr;
  if (a.W != W || b.N != M + 1) return cudaErrorInvalidValue;
  constexpr size_t smem = rader_strided_smem<M, W>();
  static PerDevice<int64_t> slots_cache;
  const int64_t slots = slots_cache.get(current_device(), [&] {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_rader_strided<M, T, W, MB, Rs...>, W * T, smem);
    return (int64_t)device_sm_count() * (per_sm > 0 ? per_sm : 1);
  });
  int64_t grid = a.nouter * a.ncolblocks;
  if (grid > slots) grid = slots;
  if (grid < 1) return cudaSuccess;
  return launch_chained(k_rader_strided<M, T, W, MB, Rs...>, dim3((unsigned)grid), dim3(W, T), smem, s, a.chained, a, b);
}
#undef TFFT_ALLOW_SMEM

// compiled with the specialised passes' parts (tfft_spec_part.cu)
template <int P>
cudaError_t rader_strided_part(const StridedArgs& a, const BlueArgs& b, cudaStream_t s);
template <int P>
cudaError_t blue_contig_part(const ContigArgs& a, const BlueArgs& b, cudaStream_t s);
template <int P>
cudaError_t blue_strided_part(const StridedArgs& a, const BlueArgs& b, cudaStream_t s);

}  // namespace blue
}  // namespace tfft
