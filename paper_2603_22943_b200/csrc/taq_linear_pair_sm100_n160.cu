// The dequant-GEMM's tiles of 256 rows x 160 columns, on pairs of CTAs.
#include "taq_prof.cuh"
TAQ_PROF_DEFINE(linear_pair_n160)
#include "taq_linear_pair_sm100.cuh"

template cudaError_t taq::linear::launch_pair<160>(const CUtensorMap&, const LinearArgs&, const LinearLayout&, const CUtensorMap&, int, size_t, cudaStream_t);
