// Float64 sampler (plain moves) and incremental local energy for tanh models: interface.
#pragma once

#include "common.cuh"
#include "metro.cuh"

namespace gna {

// All four return GNA_ERR_UNSUPPORTED when the model or graph does not fit (the caller then takes
// the kernels of metro.cu and simt.cu).
gna_status db_metro_workspace(const gna_graph* g, const Dims& m, int64_t C, size_t* bytes);
gna_status db_metro_run(const MetroCall& c, void* ws, size_t ws_bytes, cudaStream_t stream);
gna_status db_eloc_workspace(const gna_graph* g, const Dims& m, int64_t B, size_t* bytes);
gna_status db_eloc_run(const SimtCall& c, void* ws, size_t ws_bytes, cudaStream_t stream);

}  // namespace gna
