// The dequant-GEMM's tiles of 256 rows x 128 columns, on pairs of CTAs.
#include "taq_prof.cuh"
TAQ_PROF_DEFINE(linear_pair_n128)
#include "taq_linear_pair_sm100.cuh"

template cudaError_t taq::linear::launch_pair<128>(const CUtensorMap&, const LinearArgs&, const LinearLayout&, const CUtensorMap&, int, size_t, cudaStream_t);
