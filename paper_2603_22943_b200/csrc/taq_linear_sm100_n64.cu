// The dequant-GEMM's tiles of 64 columns.
#include "taq_prof.cuh"
TAQ_PROF_DEFINE(linear_n64)
#include "taq_linear_sm100.cuh"

template cudaError_t taq::linear::launch_tile<64>(const CUtensorMap&, const LinearArgs&, const LinearLayout&, int, size_t, cudaStream_t);
