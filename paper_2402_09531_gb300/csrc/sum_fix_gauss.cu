#include "sum_fix.cuh"

namespace dw {
namespace fx {

void launch_fix_gauss(int d, int RC, const FixArgs& a, int ctas, cudaStream_t s) {
  launch_fix_d<DWFMM_K_GAUSS>(d, RC, a, ctas, s);
}

void launch_fix_sym_gauss(int d, int RC, const FixSymArgs& a, int chunks, cudaStream_t s) {
  launch_sym_d<DWFMM_K_GAUSS>(d, RC, a, chunks, s);
}

}  // namespace fx
}  // namespace dw
