// Compile-time specialised FFT passes (contiguous and strided): the kernels
// and launchers of the rows of tfft_spec_table.h.  Same Stockham schedule as
// the runtime-dispatched kernels (tfft_kernels.cu), but with the length, the
// radix sequence, the threads per line and the tile width fixed at compile
// time: every index, span and twiddle stride folds to a constant, the row
// tables hold 32-bit offsets, and the register budget is known to ptxas.
#pragma once

#include <type_traits>

#include "tfft_internal.h"
#include "tfft_spec_table.h"
#include "tfft_tiles.cuh"

namespace tfft {
namespace spec {

using namespace tiles;

// Registers sized for MB resident CTAs (1024 threads per SM for plans of up
// to 16 values per thread): more lines in flight per SM.  Against a
// 512-thread target: 256^3 pass 49.4 -> 46.7 us, 128^4 0.667 -> 0.603 ms.
template <int L, int T, int B, int MB, bool CHAIN, int... Rs>
__global__ void __launch_bounds__(T * B, MB) k_contig_spec(const ContigArgs a) {
  extern __shared__ float2 smem[];
  if constexpr (CHAIN) {
    chain_next();
    chain_wait();
  }
  for (int64_t tile = blockIdx.x; tile * B < a.nlines; tile += gridDim.x)
    contig_tile<L, T, B, false, Rs...>(a, tile, smem, opaque_tid_x(), threadIdx.y);
}

// Whether the plain strided kernel keeps the rows' part/index table for the
// CTA's lifetime (2L words): not at 4096, where it would halve the CTAs per SM.
__host__ __device__ constexpr bool strided_cache_rows(int L) { return L <= 2048; }

template <int L, int T, int W, int MB, bool CHAIN, int... Rs>
__global__ void __launch_bounds__(W * T, MB) k_strided_spec(const StridedArgs a) {
  extern __shared__ float2 smem[];
  const int64_t ntiles = a.nouter * a.ncolblocks;
  const int tid = threadIdx.y * W + threadIdx.x;
  uint32_t* rp = nullptr;
  if constexpr (CHAIN) chain_next();
  if constexpr (strided_cache_rows(L)) {
    rp = strided_rowparts<L, W>(smem);
    strided_rowparts_init<L>(a, rp, tid, W * T);  // published by the first tile's barriers
  }
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x)
    strided_tile<L, T, W, false, CHAIN, Rs...>(a, tile, smem, threadIdx.x, opaque_tid_y(), tid, rp);
}

template <int L, int T, int W, int MB, bool CHAIN, int... Rs>
__global__ void __launch_bounds__(W * T, MB) k_strided_merged(const StridedArgs a) {
  extern __shared__ float2 smem[];
  const uint32_t ntiles = (uint32_t)(a.nranks * a.merged_blocks);
  if constexpr (CHAIN) chain_next();
  for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x)
    merged_tile<L, T, W, CHAIN, Rs...>(a, tile, smem, threadIdx.x, opaque_tid_y());
}

template <int L, int T, int W, int MB, int... Rs>
__global__ void __launch_bounds__(W * T, MB) k_strided_gather(const StridedArgs a) {
  extern __shared__ float2 smem[];
  gather_tiles<L, T, W, Rs...>(a, smem);
}

// the kernel's shared-memory limit raised to 227 KB, once per device
#define TFFT_ALLOW_SMEM(kernel)                          \
  static PerDevice<cudaError_t> attr_cache;              \
  const cudaError_t attr = smem_attr_once(attr_cache, kernel, 227 * 1024)

constexpr int64_t kMaxGrid = 1 << 20;

template <int L, int T, int B, int MB, bool CHAIN, int... Rs>
cudaError_t run_contig(const ContigArgs& a, cudaStream_t s) {
  if constexpr (!CHAIN && chainable(L))
    if (a.chained) return run_contig<L, T, B, MB, true, Rs...>(a, s);
  TFFT_ALLOW_SMEM((k_contig_spec<L, T, B, MB, CHAIN, Rs...>));
  if (attr != cudaSuccess) return attr;
  const size_t smem = (size_t)B * line_pitch<L, Rs...>() * sizeof(float2);
  int64_t grid = (a.nlines + B - 1) / B;
  if (grid > kMaxGrid) grid = kMaxGrid;
  if (grid < 1) return cudaSuccess;
  return launch_chained(k_contig_spec<L, T, B, MB, CHAIN, Rs...>, dim3((unsigned)grid), dim3(T, B), smem, s, CHAIN ? a.chained : 0, a);
}

// Persistent launch: as many CTAs as fit at once, each taking every gridDim-th
// tile (in the plain pass, the row part table is then computed once per CTA).
// A merged pass over more than 512 MiB with four or more CTAs per SM runs one
// tile per CTA instead: it needs no set-up, and tiles that start in order keep
// the CTAs on neighbouring rows (128^4 0.703 -> 0.661 and 0.684 -> 0.640 ms;
// but 400^3, two CTAs per SM, 0.174 -> 0.188, and within the L2 100 x 320 x 320
// 26.6 -> 28.7 us).
template <int L, int T, int W, class K>
cudaError_t run_strided_tiles(K kern, const StridedArgs& a, size_t smem, int64_t ntiles, int chained, cudaStream_t s,
                              PerDevice<cudaError_t>& attr_cache, PerDevice<int64_t>& slots_cache) {
  const cudaError_t attr = smem_attr_once(attr_cache, kern, 227 * 1024);
  if (attr != cudaSuccess) return attr;
  if (a.W != W) return cudaErrorInvalidValue;
  const int64_t slots = slots_cache.get(current_device(), [&] {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, W * T, smem);
    return (int64_t)device_sm_count() * (per_sm > 0 ? per_sm : 1);
  });
  const bool in_order = a.merged_blocks > 0 && slots >= 4 * (int64_t)device_sm_count() &&
                        ntiles * L * W * (int64_t)sizeof(float2) > (int64_t(512) << 20);
  const int64_t grid = ntiles > slots && !in_order ? slots : ntiles;
  if (grid < 1) return cudaSuccess;
  return launch_chained(kern, dim3((unsigned)grid), dim3(W, T), smem, s, chained, a);
}

template <int L, int T, int W, int MB, bool CHAIN, int... Rs>
cudaError_t run_strided(const StridedArgs& a, cudaStream_t s) {
  // Gathering tiles: in chained calls from 96 rows on, where their set-up runs
  // before the wait (100 x 150 x 180 63.0 -> 60.3 us, 96 x 200 x 96 40.7 ->
  // 39.2; shorter lines gain nothing: 60 x 72 x 100 19.2 -> 19.5), otherwise
  // for the rows that gain from them (gather_blocks).
  constexpr int blocks = gather_blocks(L);
  if constexpr (!CHAIN && L <= 1024 && (L >= 96 || blocks != kGatherNone)) {
    const bool whole = a.ncolblocks * W == a.lin.N[a.d - 1];
    const bool gains = blocks == kGatherAny || (blocks == kGatherWhole && whole);
    if (a.merged_blocks == 0 && (gains || (a.chained && L >= 96)) &&
        a.lin.Mx[a.axis] <= kGatherParts && a.lout.Mx[a.axis] <= kGatherParts) {
      static PerDevice<cudaError_t> attr_cache;
      static PerDevice<int64_t> slots_cache;
      return run_strided_tiles<L, T, W>(k_strided_gather<L, T, W, MB, Rs...>, a, gather_smem<L, W>(),
                                        a.nouter * a.ncolblocks, a.chained, s, attr_cache, slots_cache);
    }
  }
  if constexpr (!CHAIN && chainable(L))
    if (a.chained) return run_strided<L, T, W, MB, true, Rs...>(a, s);
  const int chained = CHAIN ? a.chained : 0;
  // in-place leading-axis passes run merged columns (400^3 on 4 x 4 0.250 ->
  // 0.174 ms, 240^3 on 4 x 8 51 -> 41 us, 180 x 200 x 240 34.8 -> 24.6 us; over
  // every row at 2^24 elements 1.14 in the geometric mean).  The merged kernel
  // takes the launch bounds of the row-table kernel but forms every row's
  // address from the run-time `inner`: 57 of its 188 instantiations spill, 68
  // bytes at most at the powers of two up to 512, 96 132-140, 144 128-144, 288
  // and 576 124.  The worst lose to the row tables: 81 (180 bytes) 55 -> 60 us,
  // 243 (212) 65 -> 70, 392 (204) 64 -> 68; 864, 972 and 1000 lose 3-4 %.
  if (a.merged_blocks > 0) {
    static PerDevice<cudaError_t> attr_cache;
    static PerDevice<int64_t> slots_cache;
    return run_strided_tiles<L, T, W>(k_strided_merged<L, T, W, MB, CHAIN, Rs...>, a, (size_t)L * W * sizeof(float2),
                                      a.nranks * a.merged_blocks, chained, s, attr_cache, slots_cache);
  }
  static PerDevice<cudaError_t> attr_cache;
  static PerDevice<int64_t> slots_cache;
  return run_strided_tiles<L, T, W>(k_strided_spec<L, T, W, MB, CHAIN, Rs...>, a,
                                    strided_tile_smem<L, W>(strided_cache_rows(L)), a.nouter * a.ncolblocks, chained, s,
                                    attr_cache, slots_cache);
}

#undef TFFT_ALLOW_SMEM

// The rows are compiled in kSpecParts - 1 translation units (tfft_spec_part.cu),
// row L in part L mod kSpecParts.  With a prime above 7 the 2/3/5/7 lengths
// spread over the other remainders, and none is in part 0, which is not built.
constexpr int kSpecParts = 11;

// calls f(integral_constant<P>) for P == p
template <int P = 1, class F>
cudaError_t with_part(int p, F&& f) {
  if constexpr (P < kSpecParts)
    return p == P ? f(std::integral_constant<int, P>{}) : with_part<P + 1>(p, f);
  else
    return cudaErrorInvalidValue;
}

template <int P>
cudaError_t contig_part(const ContigArgs& a, cudaStream_t s);
template <int P>
cudaError_t strided_part(const StridedArgs& a, cudaStream_t s);

}  // namespace spec
}  // namespace tfft
