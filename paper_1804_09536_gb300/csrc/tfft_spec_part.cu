// One part of the specialised passes: the rows L of tfft_spec_table.h, and the
// convolution lengths M of tfft_blue.cuh, with L (M) mod kSpecParts ==
// TFFT_SPEC_PART (set by the build).
#include "tfft_blue.cuh"
#include "tfft_spec_pass.cuh"

namespace tfft {
namespace spec {

template <int P>
cudaError_t contig_part(const ContigArgs& a, cudaStream_t s) {
#define X(LL, T, B, MB, ...)                  \
  if constexpr (LL % kSpecParts == P)         \
    if (a.ap.L == LL) return run_contig<LL, T, B, MB, false, __VA_ARGS__>(a, s);
  TFFT_CONTIG_LINES(X)
#undef X
  return cudaErrorInvalidValue;
}

template <int P>
cudaError_t strided_part(const StridedArgs& a, cudaStream_t s) {
#define X(LL, T, W, MB, ...)                  \
  if constexpr (LL % kSpecParts == P)         \
    if (a.ap.L == LL) return run_strided<LL, T, W, MB, false, __VA_ARGS__>(a, s);
  TFFT_STRIDED_LINES(X)
#undef X
  return cudaErrorInvalidValue;
}

template cudaError_t contig_part<TFFT_SPEC_PART>(const ContigArgs& a, cudaStream_t s);
template cudaError_t strided_part<TFFT_SPEC_PART>(const StridedArgs& a, cudaStream_t s);

}  // namespace spec

namespace blue {

template <int P>
cudaError_t blue_contig_part(const ContigArgs& a, const BlueArgs& b, cudaStream_t s) {
#define X(MM, T, B, MB, ...)                  \
  if constexpr (MM % spec::kSpecParts == P)   \
    if (b.M == MM) return run_blue_contig<MM, T, B, MB, __VA_ARGS__>(a, b, s);
  TFFT_BLUE_CONTIG(X)
#undef X
  return cudaErrorInvalidValue;
}

template <int P>
cudaError_t blue_strided_part(const StridedArgs& a, const BlueArgs& b, cudaStream_t s) {
#define X(MM, T, W, MB, ...)                  \
  if constexpr (MM % spec::kSpecParts == P)   \
    if (b.M == MM) return run_blue_strided<MM, T, W, MB, __VA_ARGS__>(a, b, s);
  TFFT_BLUE_STRIDED(X)
#undef X
  return cudaErrorInvalidValue;
}

template <int P>
cudaError_t rader_strided_part(const StridedArgs& a, const BlueArgs& b, cudaStream_t s) {
#define X(MM, T, W, MB, ...)                  \
  if constexpr (MM % spec::kSpecParts == P)   \
    if (b.N == MM + 1) return run_rader_strided<MM, T, W, MB, __VA_ARGS__>(a, b, s);
  TFFT_RADER_STRIDED(X)
#undef X
  return cudaErrorInvalidValue;
}

template cudaError_t rader_strided_part<TFFT_SPEC_PART>(const StridedArgs& a, const BlueArgs& b, cudaStream_t s);
template cudaError_t blue_contig_part<TFFT_SPEC_PART>(const ContigArgs& a, const BlueArgs& b, cudaStream_t s);
template cudaError_t blue_strided_part<TFFT_SPEC_PART>(const StridedArgs& a, const BlueArgs& b, cudaStream_t s);

}  // namespace blue
}  // namespace tfft
