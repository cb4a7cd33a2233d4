// Every butterfly of tfft_common.cuh on host memory (test infrastructure).
#include <type_traits>

#include "tfft_common.cuh"

using namespace tfft;

extern "C" int dft_radix(int R, float* v) {
  float2* x = reinterpret_cast<float2*>(v);
  switch (R) {
#define X(N) \
  case N:    \
    Dft<N>::run(x); \
    return 0;
    X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(12) X(14) X(15) X(16) X(18) X(20) X(21) X(24) X(25) X(27) X(28)
    X(30) X(32)
#undef X
  }
  return 1;
}
