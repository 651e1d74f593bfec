// Forward of BF16X2 models on warp tiles: interface.
#pragma once

#include "common.cuh"

namespace gna {

// GNA_ERR_UNSUPPORTED when the model or graph does not fit (the caller then takes tc.cu).
gna_status fx_workspace(const gna_graph* g, const Dims& m, int64_t B, size_t* bytes);
gna_status fx_run(const gna_graph* g, const Dims& m, const float* theta, const int8_t* spins, int64_t B, double* logpsi,
                  void* ws, size_t ws_bytes, cudaStream_t stream);

}  // namespace gna
