// Mixed form, slices of width 32 < W <= 64 (the two-chain sweep of xmatvec_mixed.cuh).
#include "xmatvec_mixed.cuh"

DY_CHAIN_VARIANT(float, 64, k_xmatvec_m)
