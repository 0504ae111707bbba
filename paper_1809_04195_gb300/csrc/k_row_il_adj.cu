// Adjoint row passes on the interleaved intermediate.
#define T2SH_ROW_MODE ROW_ADJ
#define T2SH_ROW_FIRST 0
#include "k_row_il.cuh"
