// Column passes on the interleaved intermediate: dispatch over the column lengths.
#include "k_col_il.cuh"

namespace t2sh {

#define X(p)                                                                                                        \
  cudaError_t launch_col_il_##p(const Geom& g, IlPass pass, const float2* tw_y, const float* psi, const float2* in, \
                                float2* t, cudaStream_t st);
X(a) X(b) X(c) X(d) X(e) X(f)
#undef X

// RB of the column length (0: none): the row passes need it for the slot rotation
int il_rb(int ny) {
  switch (ny) {
#define X(n, ra, rb) case n: return rb;
    T2SH_IL_LENGTHS(X)
#undef X
    default: return 0;
  }
}

cudaError_t launch_col_il(const Geom& g, IlPass pass, const float2* tw_y, const float* psi, const float2* in, float2* t,
                          cudaStream_t st) {
  if (g.K != 4 || g.nz % 4 != 0) return cudaErrorNotSupported;
  switch (g.ny) {
#define X(n, ra, rb) case n: return launch_col_il_a(g, pass, tw_y, psi, in, t, st);
    T2SH_IL_LENGTHS_A(X)
#undef X
#define X(n, ra, rb) case n: return launch_col_il_b(g, pass, tw_y, psi, in, t, st);
    T2SH_IL_LENGTHS_B(X)
#undef X
#define X(n, ra, rb) case n: return launch_col_il_c(g, pass, tw_y, psi, in, t, st);
    T2SH_IL_LENGTHS_C(X)
#undef X
#define X(n, ra, rb) case n: return launch_col_il_d(g, pass, tw_y, psi, in, t, st);
    T2SH_IL_LENGTHS_D(X)
#undef X
#define X(n, ra, rb) case n: return launch_col_il_e(g, pass, tw_y, psi, in, t, st);
    T2SH_IL_LENGTHS_E(X)
#undef X
#define X(n, ra, rb) case n: return launch_col_il_f(g, pass, tw_y, psi, in, t, st);
    T2SH_IL_LENGTHS_F(X)
#undef X
    default: return cudaErrorNotSupported;
  }
}

}  // namespace t2sh
