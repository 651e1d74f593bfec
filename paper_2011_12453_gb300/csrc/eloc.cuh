// Incremental local energy, one warp per tile of 16 rows: interface.  f32: an FP32 model (tanh, or
// ReLU + layer norm), without log Psi; else a BF16X2 model.
#pragma once

#include "tc.cuh"

namespace gna {

// GNA_ERR_UNSUPPORTED when the model or graph does not fit the kernel (the caller then takes
// kernel of tc.cu or simt.cu).
gna_status el_workspace(const gna_graph* g, const Dims& m, int64_t B, bool f32, size_t* bytes);
gna_status el_run(const TcCall& c, bool f32, void* ws, size_t ws_bytes, cudaStream_t stream);

}  // namespace gna
