// Plans and dispatch of the compile-time specialised passes: the row of a
// length in tfft_spec_table.h and the translation unit that compiled it.
#include "tfft_blue.cuh"
#include "tfft_spec_pass.cuh"

namespace tfft {

namespace {

struct SpecRow {
  int L, T, width, nst, radix[6];
};

#define X(L, T, W, MB, ...) {L, T, W, (int)(sizeof((int[]){__VA_ARGS__}) / sizeof(int)), {__VA_ARGS__}},
const SpecRow kContigRows[] = {TFFT_CONTIG_LINES(X)};
const SpecRow kStridedRows[] = {TFFT_STRIDED_LINES(X)};
#undef X

// every row has a part that is built
#define X(L, ...) static_assert(L % spec::kSpecParts != 0);
TFFT_CONTIG_LINES(X)
TFFT_STRIDED_LINES(X)
TFFT_BLUE_CONTIG(X)
TFFT_BLUE_STRIDED(X)
TFFT_RADER_STRIDED(X)
#undef X

bool row_plan(const SpecRow& r, AxisPlan& ap, int& width) {
  ap.L = r.L;
  ap.E = (r.L + r.T - 1) / r.T;
  ap.T = r.T;
  ap.nst = r.nst;
  ap.code = 0;
  for (int s = 0; s < r.nst; ++s) {
    ap.radix[s] = r.radix[s];
    ap.code |= (uint64_t)r.radix[s] << (5 * s);
  }
  ap.spec = 1;
  width = r.width;
  return true;
}

}  // namespace

bool spec_plan(int L, bool strided, int64_t nelems, AxisPlan& ap, int& width) {
  if (nelems >= (int64_t(1) << 31)) return false;  // 32-bit row offsets
  if (strided) {
    for (const SpecRow& r : kStridedRows)
      if (r.L == L) return row_plan(r, ap, width);
  } else {
    for (const SpecRow& r : kContigRows)
      if (r.L == L) return row_plan(r, ap, width);
  }
  return false;
}

bool real_plan(int L, int64_t nelems, AxisPlan& ap, int& width) {
#define X(LL) \
  if (L == LL) return spec_plan(L, false, nelems, ap, width);
  TFFT_REAL_LENGTHS(X)
#undef X
  return false;
}

cudaError_t launch_contig_spec(const ContigArgs& a, cudaStream_t s) {
  return spec::with_part(a.ap.L % spec::kSpecParts,
                   [&](auto p) { return spec::contig_part<decltype(p)::value>(a, s); });
}

cudaError_t launch_strided_spec(const StridedArgs& a, cudaStream_t s) {
  return spec::with_part(a.ap.L % spec::kSpecParts,
                   [&](auto p) { return spec::strided_part<decltype(p)::value>(a, s); });
}

}  // namespace tfft
