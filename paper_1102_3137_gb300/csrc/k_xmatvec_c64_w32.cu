// Mixed form, slices of width 16 < W <= 32 (the two-chain sweep of xmatvec_mixed.cuh).
#include "xmatvec_mixed.cuh"

DY_CHAIN_VARIANT(float, 32, k_xmatvec_m)
