// Column passes on the interleaved intermediate: a share of the column lengths (compiled apart, so
// that the unrolled kernels build in parallel).
#include "k_col_il.cuh"

namespace t2sh {

cudaError_t launch_col_il_f(const Geom& g, IlPass pass, const float2* tw_y, const float* psi, const float2* in,
                            float2* t, cudaStream_t st) {
  switch (g.ny) {
#define X(n, ra, rb) case n: return il_go<n>(g, pass, tw_y, psi, in, t, st);
    T2SH_IL_LENGTHS_F(X)
#undef X
    default: return cudaErrorNotSupported;
  }
}

}  // namespace t2sh
