// FP32 instantiation of the hot-path passes (bulk of the mixed-precision iteration).
#include "gfp_kimpl.cuh"
namespace gfp {
template struct Passes<float>;
template bool cz_cols_ok<float>(int, int);
template bool cz_tma_ok<float>(int, int);
template int cy_cols_max<float>(int);
bool cz_swizzled(int n3, int cols) {
  if (cols != 8) return false;
  switch (n3) {
#define GFP_CASE(N) case N: return SPlanOk<N>::ok || N == ZL::LEN;
    GFP_FOR_CSIZES(GFP_CASE)
#undef GFP_CASE
    default: return false;
  }
}
}
