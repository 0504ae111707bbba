// Forward row passes on the interleaved intermediate.
#define T2SH_ROW_MODE ROW_FWD
#define T2SH_ROW_FIRST 1
#include "k_row_il.cuh"
