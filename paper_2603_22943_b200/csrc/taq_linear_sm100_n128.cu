// The dequant-GEMM's tiles of 128 columns.
#include "taq_prof.cuh"
TAQ_PROF_DEFINE(linear_n128)
#include "taq_linear_sm100.cuh"

template cudaError_t taq::linear::launch_tile<128>(const CUtensorMap&, const LinearArgs&, const LinearLayout&, int, size_t, cudaStream_t);
