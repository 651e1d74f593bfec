// Sampler of BF16 models (plain moves), a warp per chain: interface.
#pragma once

#include "common.cuh"
#include "metro.cuh"

namespace gna {

// GNA_ERR_UNSUPPORTED when the model or graph does not fit (the caller then takes metro.cu).
gna_status mt_workspace(const gna_graph* g, const Dims& m, int64_t C, size_t* bytes);
gna_status mt_run(const MetroCall& c, void* ws, size_t ws_bytes, cudaStream_t stream);

}  // namespace gna
