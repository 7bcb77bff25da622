// FP64 form, slices of up to 32 sites (the two-chain sweep of xmatvec_mixed.cuh).
#include "xmatvec_mixed.cuh"

DY_CHAIN_VARIANT(double, 16, k_xmatvec_d)
DY_CHAIN_VARIANT(double, 32, k_xmatvec_d)
