// Device-side building blocks of the compile-time specialised passes: the
// Stockham stage, register-held stage twiddles, shared-memory helpers and the
// per-tile bodies of the contiguous and strided passes.  Included by the pass
// kernels (tfft_spec.cu, tfft_tma.cu, tfft_tc.cu) and by the batched executor
// (tfft_batch.cu).
#pragma once

#include <type_traits>

#include "tfft_internal.h"

namespace tfft {
namespace tiles {

template <int S, int... Rs>
__host__ __device__ constexpr int radix_at() {
  constexpr int r[] = {Rs...};
  return r[S];
}

template <int S, int... Rs>
__host__ __device__ constexpr int span_at() {
  constexpr int r[] = {Rs...};
  int p = 1;
  for (int i = 0; i < S; ++i) p *= r[i];
  return p;
}

template <int I, int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

// A line of length L is worked by T threads.  A stage of radix R has L / R
// butterflies, nbf = ceil((L / R) / T) per thread: butterfly j = jt + q T,
// q < nbf, exists when j < L / R.  When every radix divides L / T this is
// L / (T R) butterflies each and no guard (the power-of-two plans); the
// others guard, their threads carry one butterfly fewer in some stages and
// hold up to emax() values.  T need not divide L.
template <int L, int T, int R>
__host__ __device__ constexpr int nbf() {
  return (L / R + T - 1) / T;
}

template <int L, int T, int R>
__host__ __device__ constexpr bool nbf_exact() {
  return (L / R) % T == 0;
}

template <int L, int T, int... Rs>
__host__ __device__ constexpr int emax() {
  constexpr int r[] = {Rs...};
  int m = 0;
  for (int i = 0; i < (int)sizeof...(Rs); ++i) {
    const int v = ((L / r[i] + T - 1) / T) * r[i];
    m = v > m ? v : m;
  }
  return m;
}

// Whether butterfly q of thread jt exists in a stage of radix R.
template <int L, int T, int R>
__device__ __forceinline__ bool bf_exists(int jt, int q) {
  if constexpr (nbf_exact<L, T, R>()) return true;
  else return jt + q * T < L / R;
}

// Offset of stage s in a plan's stage table (TwiddleTable): stages 1 .. s - 1
// hold (R - 1) Ns entries each.
template <int S, int... Rs>
__host__ __device__ constexpr int stage_table_at() {
  constexpr int r[] = {Rs...};
  int off = 0, ns = r[0];
  for (int i = 1; i < S; ++i) {
    off += (r[i] - 1) * ns;
    ns *= r[i];
  }
  return off;
}

// Where a contiguous pass reads stage s's twiddles (spec_stage's OFF): the
// stage table, or -1 for the roots (reads_stage_table).
template <int S, int... Rs>
__host__ __device__ constexpr int stage_table_off() {
  return reads_stage_table(sizeof...(Rs), radix_at<0, Rs...>()) ? stage_table_at<S, Rs...>() : -1;
}

// Twiddle (stage span Ns > 1) and size-R butterflies of a thread's work items.
// OFF < 0: tw is the table of the L roots; otherwise it is the plan's stage
// table, whose stage starts at OFF and holds twiddle r of butterflies k = 0 ..
// Ns - 1 consecutively.  In the contiguous passes a warp's lanes have
// consecutive k: one line of 16 twiddles per load instead of up to 16 lines
// (root r k L / (Ns R) lies r k apart), which kept the L1 busier than the data
// did.
template <int L, int T, int R, int Ns, int OFF = -1, int EM>
__device__ __forceinline__ void spec_stage(float2 (&v)[EM], int jt, const float2* __restrict__ tw) {
#pragma unroll
  for (int q = 0; q < nbf<L, T, R>(); ++q) {
    if (!bf_exists<L, T, R>(jt, q)) continue;
    if constexpr (Ns > 1) {
      const int j = jt + q * T;
      if constexpr (OFF >= 0) {
        const float2* row = tw + OFF + j % Ns;
#pragma unroll
        for (int r = 1; r < R; ++r) v[q * R + r] = cmul(v[q * R + r], __ldg(row + (r - 1) * Ns));
      } else {
        const int step = (j % Ns) * (L / (Ns * R));
#pragma unroll
        for (int r = 1; r < R; ++r) v[q * R + r] = cmul(v[q * R + r], __ldg(&tw[r * step]));
      }
    }
    Dft<R>::run(&v[q * R]);
  }
}

// Twiddles of every stage after the first for one thread.  They depend only
// on the thread's position in the line, so a persistent kernel loads them
// into registers once instead of once per tile where they fit beside its
// values: plans without guards and with at most 32 of them.  Others read
// them per tile.  Stage s (span Ns, radix R) multiplies item r of butterfly q
// by w_L^{r (j % Ns) L / (Ns R)} with j = jt + q T; the held values are
// stored from offset(s) on, (R - 1) per q.
template <int L, int T, int... Rs>
struct StageTwiddles {
  static constexpr int NST = sizeof...(Rs);
  __host__ __device__ static constexpr int offset(int s) {
    constexpr int r[] = {Rs...};
    int c = 0;
    for (int i = 1; i < s; ++i) c += (L / T / r[i]) * (r[i] - 1);
    return c;
  }
  static constexpr bool HELD = (nbf_exact<L, T, Rs>() && ...) && offset(NST) <= 32;
  static constexpr int COUNT = HELD ? offset(NST) : 0;
  float2 w[COUNT > 0 ? COUNT : 1];

  __device__ __forceinline__ void load(int jt, const float2* __restrict__ tw) {
    if constexpr (HELD)
      static_for<1, NST>([&](auto S) {
        constexpr int s = decltype(S)::value;
        constexpr int R = radix_at<s, Rs...>();
        constexpr int Ns = span_at<s, Rs...>();
        constexpr int off = offset(s);
#pragma unroll
        for (int q = 0; q < L / T / R; ++q) {
          const int step = ((jt + q * T) % Ns) * (L / (Ns * R));
#pragma unroll
          for (int r = 1; r < R; ++r) w[off + q * (R - 1) + r - 1] = __ldg(&tw[r * step]);
        }
      });
  }

  // Stage s on a thread's items.
  template <int s, int EM>
  __device__ __forceinline__ void stage(float2 (&v)[EM], int jt, const float2* __restrict__ tw) const {
    constexpr int R = radix_at<s, Rs...>();
    if constexpr (!HELD) {
      spec_stage<L, T, R, span_at<s, Rs...>()>(v, jt, tw);
    } else {
      constexpr int off = offset(s);
#pragma unroll
      for (int q = 0; q < L / T / R; ++q) {
        if constexpr (s > 0) {
#pragma unroll
          for (int r = 1; r < R; ++r) v[q * R + r] = cmul(v[q * R + r], w[off + q * (R - 1) + r - 1]);
        }
        Dft<R>::run(&v[q * R]);
      }
    }
  }
};

// threadIdx re-read inside a loop body, opaque to the compiler: it keeps the
// per-thread shared-memory addresses from being hoisted out of the tile loop
// (and held in registers across it).
__device__ __forceinline__ int opaque_tid_x() {
  int v;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(v));
  return v;
}
__device__ __forceinline__ int opaque_tid_y() {
  int v;
  asm volatile("mov.u32 %0, %%tid.y;" : "=r"(v));
  return v;
}

// Synchronises the threads of one line: a warp when the line's threads lie
// inside one (T divides 32), the whole CTA otherwise.
template <int T>
__device__ __forceinline__ void line_sync() {
  if constexpr (32 % T == 0) {
    __syncwarp();
  } else {
    __syncthreads();
  }
}

// Padded position inside a contiguous line: one spare slot every P elements.
// The first stage writes its outputs at stride R0 (its radix); with P = R0
// that stride becomes R0 + 1, odd, so 16 lanes of 8-byte stores hit 16
// distinct bank pairs.  P = 8 for a first radix below 8 or not a power of two.
template <int... Rs>
__host__ __device__ constexpr int pad_every() {
  constexpr int r[] = {Rs...};
  return (r[0] & (r[0] - 1)) == 0 && r[0] >= 8 ? r[0] : 8;
}

template <int P>
__device__ __forceinline__ int padp(int pos) {
  return pos + pos / P;
}

// Padded line pitch of the contiguous-line kernels (elements).
template <int L, int... Rs>
__host__ __device__ constexpr int line_pitch() {
  return L + L / pad_every<Rs...>();
}

// ------------------------------------------------------------ contiguous lines

// Global load, optionally L2-only (.cg): used where the data was written by
// other SMs earlier in the same launch (the batched executor).
template <bool CG>
__device__ __forceinline__ float2 ld(const float2* p) {
  if constexpr (CG) {
    return __ldcg(p);
  } else {
    return *p;
  }
}

// One group of B contiguous lines (group `tile`): thread jt of line ly.
template <int L, int T, int B, bool CG, int... Rs>
__device__ __forceinline__ void contig_tile(const ContigArgs& a, int64_t tile, float2* smem, int jt, int ly) {
  constexpr int NST = sizeof...(Rs);
  constexpr int LP = line_pitch<L, Rs...>();
  constexpr int P = pad_every<Rs...>();
  float2* sl = smem + ly * LP;
  const bool inv = a.sign > 0;
  const int64_t line = tile * B + ly;
  const bool act = line < a.nlines;
  const float2* src = a.in + line * L;
  float2* dst = a.out + line * L;
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
          float2 x = (act && bf_exists<L, T, R>(jt, q)) ? ld<CG>(src + jt + q * T + r * (L / R))
                                                        : make_float2(0.f, 0.f);
          if (inv) x.y = -x.y;
          v[q * R + r] = x;
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
    constexpr int OFF = CG ? -1 : stage_table_off<s, Rs...>();
    spec_stage<L, T, R, Ns, OFF>(v, jt, OFF < 0 ? a.tw : a.tws);
  });
  constexpr int RL = radix_at<NST - 1, Rs...>();
  const float oscale = contig_scale(a);
#pragma unroll
  for (int q = 0; q < nbf<L, T, RL>(); ++q)
#pragma unroll
    for (int r = 0; r < RL; ++r) {
      float2 x = cscale(v[q * RL + r], oscale);
      if (inv) x.y = -x.y;
      if (act && bf_exists<L, T, RL>(jt, q)) dst[jt + q * T + r * (L / RL)] = x;
    }
  line_sync<T>();  // the line's shared slots are free for the next group
}


// ------------------------------------------------------------ strided lines

// Per-tile scalars of a strided tile, computed by one thread per layout and
// shared through shared memory: the TileRows fold of the input (0) and output
// (1) layouts, the split of the FFT axis in each (part length q, and q + 1
// for the first r parts, Eq. decompose) and the column block.
struct TileShared {
  int64_t base[2], head[2], prod[2], tail[2];
  int q[2], r[2];
  int2 blk;
};

// Bytes of shared memory a strided tile of L x W takes: the tile, the two
// row tables, the shared scalars and, when `cached`, the per-CTA part/index
// table of the rows (two layouts).
template <int L, int W>
__host__ __device__ constexpr size_t strided_tile_smem(bool cached) {
  return (size_t)L * W * sizeof(float2) + 2 * (size_t)L * sizeof(int) + sizeof(TileShared) +
         (cached ? 2 * (size_t)L * sizeof(uint32_t) : 0);
}

template <int L, int W>
__device__ __forceinline__ uint32_t* strided_rowparts(float2* smem) {
  return reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(smem) + strided_tile_smem<L, W>(false));
}

// Part c and index l (packed c << 16 | l) of every row i < L along the FFT
// axis, input layout in [0, L), output layout in [L, 2L): they depend on the
// axis split only, so a persistent CTA computes them once.
template <int L>
__device__ __forceinline__ void strided_rowparts_init(const StridedArgs& a, uint32_t* rp, int tid, int nthreads) {
  for (int i = tid; i < 2 * L; i += nthreads) {
    const int row = i < L ? i : i - L;
    const int64_t N = i < L ? a.lin.N[a.axis] : a.lout.N[a.axis];
    const int64_t M = i < L ? a.lin.Mx[a.axis] : a.lout.Mx[a.axis];
    int64_t c = 0, l = row, n = N;
    if (M > 1) locate(N, M, row, c, l, n);
    rp[i] = ((uint32_t)c << 16) | (uint32_t)l;
  }
}

// The fold of one layout for tile position tp, written to ts slot `k`.
__device__ __forceinline__ void tile_fold(const StridedArgs& a, const DevLayout& lay, const StridedTilePos& tp,
                                          TileShared* ts, int k) {
  const TileRows tr(a, lay, tp);
  ts->base[k] = tr.base;
  ts->head[k] = tr.head;
  ts->prod[k] = tr.prod;
  ts->tail[k] = tr.tail;
  const uint32_t N = (uint32_t)tr.N, M = (uint32_t)tr.M;
  ts->q[k] = (int)(N / M);
  ts->r[k] = (int)(N - (N / M) * M);
}

// Element offset of row i of a layout from the shared fold (slot k): the
// part's offset plus the C-order index inside it.
__device__ __forceinline__ int row_offset(const DevLayout& lay, int axis, const TileShared* ts, int k, int64_t c,
                                          int64_t l) {
  const int64_t n = ts->q[k] + (c < ts->r[k] ? 1 : 0);
  return (int)(lay.offset[ts->base[k] + c * lay.rs[axis]] + (ts->head[k] * n + l) * ts->prod[k] + ts->tail[k]);
}

// One strided tile (outer index and column block `tile`): thread jt of
// column cx; tid = thread index in the CTA (W x T threads).  `rp` is the
// per-CTA part/index table of strided_rowparts_init, or null (then each row
// locates its part itself).
template <int L, int T, int W, bool CG, bool CHAIN, int... Rs>
__device__ __forceinline__ void strided_tile(const StridedArgs& a, int64_t tile, float2* smem, int cx, int jt,
                                             int tid, const uint32_t* rp = nullptr) {
  constexpr int NST = sizeof...(Rs);
  static_assert(W * T > 32, "the two layouts' folds are computed by threads 0 and 32");
  int* rin = reinterpret_cast<int*>(smem + L * W);
  int* rout = rin + L;
  TileShared* ts = reinterpret_cast<TileShared*>(rout + L);
  const bool inv = a.sign > 0;
  __syncthreads();  // the previous tile is done with the row tables and the scalars
  if (tid == 0) {
    const StridedTilePos tp(a, tile);
    tile_fold(a, a.lin, tp, ts, 0);
    ts->blk = tp.blk;
  } else if (tid == 32) {
    const StridedTilePos tp(a, tile);
    tile_fold(a, a.lout, tp, ts, 1);
  }
  __syncthreads();
  for (int i = tid; i < 2 * L; i += W * T) {
    const bool out = i >= L;
    const int row = out ? i - L : i;
    int64_t c = 0, l = row;
    if (rp != nullptr) {
      c = rp[i] >> 16;
      l = rp[i] & 0xFFFF;
    } else {
      int64_t n;
      const int64_t N = out ? a.lout.N[a.axis] : a.lin.N[a.axis];
      const int64_t M = out ? a.lout.Mx[a.axis] : a.lin.Mx[a.axis];
      if (M > 1) locate(N, M, row, c, l, n);
    }
    if (out)
      rout[row] = row_offset(a.lout, a.axis, ts, 1, c, l);
    else
      rin[row] = row_offset(a.lin, a.axis, ts, 0, c, l);
  }
  __syncthreads();
  const int2 blk = ts->blk;
  const bool act = cx < blk.y;
  // the tables of a chained pass's first tile are built while the previous
  // kernel drains
  if constexpr (CHAIN)
    if (tile == blockIdx.x) chain_wait();
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
          const int pos = jt + q * T + r * (L / R);
          float2 x = (act && bf_exists<L, T, R>(jt, q)) ? ld<CG>(a.in + rin[pos] + cx) : make_float2(0.f, 0.f);
          if (inv) x.y = -x.y;
          v[q * R + r] = x;
        }
    } else {
      constexpr int Rp = radix_at<s - 1, Rs...>();
      constexpr int Nsp = Ns / Rp;
      __syncthreads();
#pragma unroll
      for (int q = 0; q < nbf<L, T, Rp>(); ++q)
        if (bf_exists<L, T, Rp>(jt, q))
#pragma unroll
          for (int r = 0; r < Rp; ++r)
            smem[stockham_out_index(jt + q * T, Nsp, Rp, r) * W + cx] = v[q * Rp + r];
      __syncthreads();
#pragma unroll
      for (int q = 0; q < nbf<L, T, R>(); ++q)
        if (bf_exists<L, T, R>(jt, q))
#pragma unroll
          for (int r = 0; r < R; ++r) v[q * R + r] = smem[(jt + q * T + r * (L / R)) * W + cx];
    }
    spec_stage<L, T, R, Ns>(v, jt, a.tw);
  });
  constexpr int RL = radix_at<NST - 1, Rs...>();
#pragma unroll
  for (int q = 0; q < nbf<L, T, RL>(); ++q)
#pragma unroll
    for (int r = 0; r < RL; ++r) {
      float2 x = cscale(v[q * RL + r], a.scale);
      if (inv) x.y = -x.y;
      if (act && bf_exists<L, T, RL>(jt, q)) a.out[rout[jt + q * T + r * (L / RL)] + cx] = x;
    }
}

// One tile of an in-place pass along the leading axis of a layout that holds
// it whole (the last pass of every fused forward, the first of a backward).
// A rank's local array is then L rows of `inner` consecutive elements, all of
// them columns of independent lines, however many axes and odd extents they
// come from: the tile is up to W of them at column block `tile` mod
// a.merged_blocks of rank `tile` / a.merged_blocks, row i of it `inner`
// elements after row i - 1.  No column blocks, no row tables, no fold: every
// thread places the tile with one division and two loads, and only a rank's
// last tile is partial.
template <int L, int T, int W, bool CHAIN, int... Rs>
__device__ __forceinline__ void merged_tile(const StridedArgs& a, uint32_t tile, float2* smem, int cx, int jt) {
  constexpr int NST = sizeof...(Rs);
  const bool inv = a.sign > 0;
  const uint32_t rank = tile / (uint32_t)a.merged_blocks;
  const int c0 = (int)(tile - rank * (uint32_t)a.merged_blocks) * W;
  const int o0 = (int)__ldg(&a.lin.offset[rank]);
  const int inner = ((int)__ldg(&a.lin.offset[rank + 1]) - o0) / L;
  if constexpr (CHAIN)
    if (tile == blockIdx.x) chain_wait();
  if (c0 >= inner) return;  // a rank with fewer blocks than the widest (the whole CTA leaves)
  const bool act = c0 + cx < inner;
  // lanes past the last column load it again and store nothing
  const int at = o0 + (act ? c0 + cx : inner - 1);
  const float2* src = a.in + at;
  float2 v[emax<L, T, Rs...>()];
  static_for<0, NST>([&](auto S) {
    constexpr int s = decltype(S)::value;
    constexpr int R = radix_at<s, Rs...>();
    constexpr int Ns = span_at<s, Rs...>();
    if constexpr (s == 0) {
#pragma unroll
      for (int q = 0; q < nbf<L, T, R>(); ++q)
        if (bf_exists<L, T, R>(jt, q))
#pragma unroll
          for (int r = 0; r < R; ++r) {
            float2 x = src[(jt + q * T) * inner + r * (L / R) * inner];
            if (inv) x.y = -x.y;
            v[q * R + r] = x;
          }
    } else {
      constexpr int Rp = radix_at<s - 1, Rs...>();
      constexpr int Nsp = Ns / Rp;
      __syncthreads();
#pragma unroll
      for (int q = 0; q < nbf<L, T, Rp>(); ++q)
        if (bf_exists<L, T, Rp>(jt, q))
#pragma unroll
          for (int r = 0; r < Rp; ++r)
            smem[stockham_out_index(jt + q * T, Nsp, Rp, r) * W + cx] = v[q * Rp + r];
      __syncthreads();
#pragma unroll
      for (int q = 0; q < nbf<L, T, R>(); ++q)
        if (bf_exists<L, T, R>(jt, q))
#pragma unroll
          for (int r = 0; r < R; ++r) v[q * R + r] = smem[(jt + q * T + r * (L / R)) * W + cx];
    }
    spec_stage<L, T, R, Ns>(v, jt, a.tw);
  });
  constexpr int RL = radix_at<NST - 1, Rs...>();
  const float sc = a.scale, scy = inv ? -a.scale : a.scale;
  float2* dst = a.out + at;
#pragma unroll
  for (int q = 0; q < nbf<L, T, RL>(); ++q)
    if (act && bf_exists<L, T, RL>(jt, q))
#pragma unroll
      for (int r = 0; r < RL; ++r)
        dst[(jt + q * T) * inner + r * (L / RL) * inner] = make_float2(v[q * RL + r].x * sc, v[q * RL + r].y * scy);
}

// ------------------------------------------------------------ gathering passes
//
// Passes whose layouts cut the FFT axis (the axis d - 2 pass of a fused
// transform gathers its lines from one cut and scatters them to another): row
// i of a tile lies at part[c] + l prod for its part c and index l there.
// Where strided_tile folds a tile in two threads and builds both row tables
// behind three barriers before its first load, here the next tile is placed,
// one lane per part, and both its tables are built between the exchanges of
// the current one; one barrier per tile is left beside the exchanges'.

// Where a tile lies in one layout: the rank part and the index before (head)
// and after (tail, rows `prod` apart) the FFT axis, in 32 bits (every offset of
// a specialised pass fits).
struct TilePlace {
  uint32_t base, head, prod, tail;
  int2 blk;
  __device__ __forceinline__ TilePlace(const StridedArgs& a, const DevLayout& lay, uint32_t tile) {
    const uint32_t o = tile / (uint32_t)a.ncolblocks;
    blk = a.colblocks[tile - o * (uint32_t)a.ncolblocks];
    uint32_t go0 = o, go1 = 0;
    if (a.oax1 >= 0) {
      go0 = o / (uint32_t)a.on1;
      go1 = o - go0 * (uint32_t)a.on1;
    }
    base = head = tail = 0;
    prod = 1;
#pragma unroll
    for (int m = 0; m < MAXD; ++m) {
      if (m >= lay.d || m == a.axis) continue;
      const uint32_t g = (m == a.d - 1) ? (uint32_t)blk.x : (m == a.oax0) ? go0 : (m == a.oax1) ? go1 : 0;
      uint32_t local = g, n = (uint32_t)lay.q[m];
      if (lay.Mx[m] > 1) {  // inverse of Eq. decompose
        const uint32_t r = (uint32_t)lay.r[m], big = r * (n + 1);
        uint32_t c;
        if (g < big) {
          c = g / (n + 1);
          local = g - c * (n + 1);
          n += 1;
        } else {
          c = (g - big) / n;
          local = g - big - c * n;
          c += r;
        }
        base += c * (uint32_t)lay.rs[m];
      }
      if (m == lay.d - 1 && lay.pitch > 0) n = (uint32_t)lay.pitch;  // the innermost axis' storage extent
      if (m < a.axis) {
        head = head * n + local;
      } else {
        tail = tail * n + local;
        prod *= n;
      }
    }
  }
};

// Parts of each layout a CTA can hold (of each of two tiles).
constexpr int kGatherParts = 64;

struct GatherShared {
  int part[2][2][kGatherParts];  // offset of index 0 of every part: slot, side (input, output)
  int prod[2][2];
  int2 blk[2];
};

template <int L, int W>
__host__ __device__ constexpr size_t gather_smem() {
  return (size_t)L * W * sizeof(float2) + 4 * (size_t)L * sizeof(int) + sizeof(GatherShared);
}

// Places tile `tile` in slot p: threads 0 .. 31 the parts of the input layout
// (one each, in rounds), 32 .. 63 those of the output layout.
__device__ __forceinline__ void gather_place(const StridedArgs& a, uint32_t tile, GatherShared* gs, int p, int tid) {
  if (tid >= 64) return;
  const int side = tid >> 5;
  const DevLayout& lay = side ? a.lout : a.lin;
  const TilePlace t(a, lay, tile);
  const uint32_t q = (uint32_t)lay.q[a.axis], r = (uint32_t)lay.r[a.axis];
  for (uint32_t c = (uint32_t)tid & 31; c < (uint32_t)lay.Mx[a.axis]; c += 32)
    gs->part[p][side][c] = (int)((uint32_t)lay.offset[t.base + c * (uint32_t)lay.rs[a.axis]] +
                                 t.head * (q + (c < r ? 1 : 0)) * t.prod + t.tail);
  if ((tid & 31) == 0) gs->prod[p][side] = (int)t.prod;
  if (tid == 0) gs->blk[p] = t.blk;
}

// All tiles of a CTA.
template <int L, int T, int W, int... Rs>
__device__ __forceinline__ void gather_tiles(const StridedArgs& a, float2* smem) {
  constexpr int NST = sizeof...(Rs);
  static_assert(W * T >= 64 && NST >= 2, "two placing warps, one exchange at least");
  int* rin = reinterpret_cast<int*>(smem + L * W);
  int* rout = rin + L;
  uint32_t* rp = reinterpret_cast<uint32_t*>(rout + L);  // part and index of every row of both layouts, for the CTA's life
  GatherShared* gs = reinterpret_cast<GatherShared*>(rp + 2 * L);
  const int cx = threadIdx.x;
  const int tid = threadIdx.y * W + cx;
  const bool inv = a.sign > 0;
  const uint32_t ntiles = (uint32_t)(a.nouter * a.ncolblocks);
  if (a.chained) chain_next();
  for (uint32_t i = (uint32_t)tid; i < 2 * L; i += W * T) {
    const DevLayout& lay = i < L ? a.lin : a.lout;
    const uint32_t q = (uint32_t)lay.q[a.axis], r = (uint32_t)lay.r[a.axis], big = r * (q + 1);
    const uint32_t row = i < L ? i : i - L;
    const uint32_t c = row < big ? row / (q + 1) : r + (row - big) / q;
    rp[i] = (c << 16) | (row - c * q - (c < r ? c : r));
  }
  gather_place(a, blockIdx.x, gs, 0, tid);
  __syncthreads();
  auto build_rows = [&](int* rows, int side, int p) {
    const int prod = gs->prod[p][side];
    const int* part = gs->part[p][side];
    for (int i = tid; i < L; i += W * T) {
      const uint32_t cl = rp[side * L + i];
      rows[i] = part[cl >> 16] + (int)(cl & 0xFFFF) * prod;
    }
  };
  build_rows(rin, 0, 0);
  if (a.chained) chain_wait();
  int p = 0;
  for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, p ^= 1) {
    __syncthreads();  // the tile's input rows are complete
    const int jt = opaque_tid_y();
    const int2 blk = gs->blk[p];
    const bool act = cx < blk.y;
    const bool more = tile + gridDim.x < ntiles;
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
            const int pos = jt + q * T + r * (L / R);
            float2 x = (act && bf_exists<L, T, R>(jt, q)) ? a.in[rin[pos] + cx] : make_float2(0.f, 0.f);
            if (inv) x.y = -x.y;
            v[q * R + r] = x;
          }
      } else {
        constexpr int Rp = radix_at<s - 1, Rs...>();
        constexpr int Nsp = Ns / Rp;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < nbf<L, T, Rp>(); ++q)
          if (bf_exists<L, T, Rp>(jt, q))
#pragma unroll
            for (int r = 0; r < Rp; ++r) smem[stockham_out_index(jt + q * T, Nsp, Rp, r) * W + cx] = v[q * Rp + r];
        if constexpr (s == 1) {
          // every thread is past the previous tile's stores and this one's
          // loads: both tables and the other slot are free
          build_rows(rout, 1, p);
          if (more) gather_place(a, tile + gridDim.x, gs, p ^ 1, tid);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < nbf<L, T, R>(); ++q)
          if (bf_exists<L, T, R>(jt, q))
#pragma unroll
            for (int r = 0; r < R; ++r) v[q * R + r] = smem[(jt + q * T + r * (L / R)) * W + cx];
        if constexpr (s == 1)
          if (more) build_rows(rin, 0, p ^ 1);
      }
      spec_stage<L, T, R, Ns>(v, jt, a.tw);
    });
    constexpr int RL = radix_at<NST - 1, Rs...>();
#pragma unroll
    for (int q = 0; q < nbf<L, T, RL>(); ++q)
#pragma unroll
      for (int r = 0; r < RL; ++r) {
        float2 x = cscale(v[q * RL + r], a.scale);
        if (inv) x.y = -x.y;
        if (act && bf_exists<L, T, RL>(jt, q)) a.out[rout[jt + q * T + r * (L / RL)] + cx] = x;
      }
  }
}

// ------------------------------------------------------------ stages only

// The Stockham stages of a length-L FFT on the values a thread holds for
// column cx of an L x W tile in shared memory (the strided passes' layout:
// position i of the column at smem[i W + cx]): on entry v holds the first
// stage's inputs x[jt + q T + r L / R0], on exit the outputs at positions
// jt + q T + r L / RL (natural order, self-sorting); between stages the
// column goes through smem.  Starts and ends without a barrier: the caller
// orders smem use around it.
template <int L, int T, int W, int... Rs>
__device__ __forceinline__ void strided_stages(float2 (&v)[emax<L, T, Rs...>()], float2* smem, int cx, int jt,
                                               const float2* __restrict__ tw) {
  constexpr int NST = sizeof...(Rs);
  static_for<0, NST>([&](auto S) {
    constexpr int s = decltype(S)::value;
    constexpr int R = radix_at<s, Rs...>();
    constexpr int Ns = span_at<s, Rs...>();
    if constexpr (s > 0) {
      constexpr int Rp = radix_at<s - 1, Rs...>();
      constexpr int Nsp = Ns / Rp;
      __syncthreads();
#pragma unroll
      for (int q = 0; q < nbf<L, T, Rp>(); ++q)
        if (bf_exists<L, T, Rp>(jt, q))
#pragma unroll
          for (int r = 0; r < Rp; ++r) smem[stockham_out_index(jt + q * T, Nsp, Rp, r) * W + cx] = v[q * Rp + r];
      __syncthreads();
#pragma unroll
      for (int q = 0; q < nbf<L, T, R>(); ++q)
        if (bf_exists<L, T, R>(jt, q))
#pragma unroll
          for (int r = 0; r < R; ++r) v[q * R + r] = smem[(jt + q * T + r * (L / R)) * W + cx];
    }
    spec_stage<L, T, R, Ns>(v, jt, tw);
  });
}

// The same for one contiguous line in its padded line slot sl (the
// contiguous passes' layout), synchronising the line's threads; tws: the
// stage table of these radices.
template <int L, int T, int... Rs>
__device__ __forceinline__ void line_stages(float2 (&v)[emax<L, T, Rs...>()], float2* sl, int jt,
                                            const float2* __restrict__ tws) {
  constexpr int NST = sizeof...(Rs);
  constexpr int P = pad_every<Rs...>();
  static_for<0, NST>([&](auto S) {
    constexpr int s = decltype(S)::value;
    constexpr int R = radix_at<s, Rs...>();
    constexpr int Ns = span_at<s, Rs...>();
    if constexpr (s > 0) {
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
    spec_stage<L, T, R, Ns, stage_table_at<s, Rs...>()>(v, jt, tws);
  });
}

}  // namespace tiles
}  // namespace tfft
