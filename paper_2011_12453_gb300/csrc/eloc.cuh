// Incremental local energy with split operands, one warp per tile of 16 rows: interface.
#pragma once

#include "tc.cuh"

namespace gna {

// GNA_ERR_UNSUPPORTED when the model or graph does not fit the kernel (the caller then takes
// the tensor-memory kernel of tc.cu).
gna_status el_workspace(const gna_graph* g, const Dims& m, int64_t B, size_t* bytes);
gna_status el_run(const TcCall& c, void* ws, size_t ws_bytes, cudaStream_t stream);

}  // namespace gna
