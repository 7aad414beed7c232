// Connected-component labelling of a phase set, shared by the transport mask
// (kernels.cu) and the structure statistics (connect.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace cl {

// L[c] = smallest cell index of c's component (cells whose phase code's bit is
// in `set`), -1 elsewhere.  26 or 6 neighbours; y and z wrap when periodic, x
// never.  *err gets bit 2 when an iteration bound ran out.
cudaError_t launch_ccl(const uint8_t* phase, int nx, int ny, int nz, unsigned set, bool faces_only, bool periodic,
                       int* L, int* err, cudaStream_t s);

}  // namespace cl
