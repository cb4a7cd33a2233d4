// Convolution lengths and dispatch of the specialised Bluestein passes
// (tfft_blue.cuh; compiled in the parts of tfft_spec_part.cu).
#include "tfft_blue.cuh"
#include "tfft_spec_pass.cuh"

namespace tfft {

bool blue_spec_plan(int M, int& lines_per_cta, int& tile_width) {
  bool c = false, t = false;
#define X(MM, T, B, ...) \
  if (M == MM) {         \
    lines_per_cta = B;   \
    c = true;            \
  }
  TFFT_BLUE_CONTIG(X)
#undef X
#define X(MM, T, W, ...) \
  if (M == MM) {         \
    tile_width = W;      \
    t = true;            \
  }
  TFFT_BLUE_STRIDED(X)
#undef X
  return c && t;
}

void blue_spec_radices(int M, int& nst, int* radix) {
  nst = 0;
#define X(MM, T, B, MB, ...)                  \
  if (M == MM)                                \
    for (int r : {__VA_ARGS__}) radix[nst++] = r;
  TFFT_BLUE_CONTIG(X)
#undef X
}

int blue_spec_length(int N) {
  int best = 0;
#define X(MM, ...) \
  if (MM >= 2 * N - 1 && (best == 0 || MM < best)) best = MM;
  TFFT_BLUE_STRIDED(X)
#undef X
  return best;
}

bool rader_plan(int N, int& tile_width) {
#define X(MM, T, W, ...)  \
  if (N == MM + 1) {      \
    tile_width = W;       \
    return true;          \
  }
  TFFT_RADER_STRIDED(X)
#undef X
  return false;
}

cudaError_t launch_strided_rader(const StridedArgs& a, const BlueArgs& b, cudaStream_t s) {
  return spec::with_part((b.N - 1) % spec::kSpecParts,
                         [&](auto p) { return blue::rader_strided_part<decltype(p)::value>(a, b, s); });
}

cudaError_t launch_contig_blue_spec(const ContigArgs& a, const BlueArgs& b, cudaStream_t s) {
  return spec::with_part(b.M % spec::kSpecParts,
                         [&](auto p) { return blue::blue_contig_part<decltype(p)::value>(a, b, s); });
}

cudaError_t launch_strided_blue_spec(const StridedArgs& a, const BlueArgs& b, cudaStream_t s) {
  return spec::with_part(b.M % spec::kSpecParts,
                         [&](auto p) { return blue::blue_strided_part<decltype(p)::value>(a, b, s); });
}

}  // namespace tfft
