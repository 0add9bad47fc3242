// Records and launchers of the FP32 face and cell kernels (avs_step32.cu).
#pragma once

#include "avs_internal.h"

namespace avs {

// A cell's collision update out = k0 f + k1 g~ + kN N (k1 inside l2), and the
// reference velocity V of its raw moments.
struct alignas(16) Cell32Par {
    float U[3], k2;
    float al[3], l2;
    float k0, RTH, kN, pad;
    float V[3];
    float diag;              // implicit step: |V|/dt + |V|/tau~
};
static_assert(sizeof(Cell32Par) <= AVS_CELLPAR_BYTES, "cell parameter buffer");

cudaError_t launch_face32(avs_ctx* c, const double* Win, double dt);
cudaError_t launch_cell32(avs_ctx* c, const void* fin, void* fout, bool residual);
cudaError_t launch_raw32(avs_ctx* c, const void* fin, const double* W);

}  // namespace avs
