// Records and launchers of the FP32 face and cell kernels (avs_step32.cu).
#pragma once

#include "avs_internal.h"

namespace avs {

// A cell's update out = (u0 f + u1 g~ + un N) u3 with g~ the Shakhov equilibrium
// 2^(l2 + k2 |c|^2) (1 + (c . al)(|c|^2 / RT - D - 2)), c = xi - U, and the
// reference velocity V of its raw moments.
struct alignas(16) Cell32Par {
    float U[3], k2;
    float al[3], l2;
    float u0, u1, un, u3;
    float V[3], irt;
    float RTH, diag, pad[2];     // diag, implicit step: |V|/dt + |V|/tau~
};
static_assert(sizeof(Cell32Par) <= AVS_CELLPAR_BYTES, "cell parameter buffer");

// foot values of every face into c->flux, either gas; hd = dt / 2
void launch_foot32(avs_ctx* c, const void* fin, double hd);
// the monatomic gas
cudaError_t launch_face32(avs_ctx* c, const double* Win, double dt);
cudaError_t launch_cell32(avs_ctx* c, const void* fin, void* fout, bool residual);
cudaError_t launch_raw32(avs_ctx* c, const void* fin, const double* W);
// either gas; diag: per cell, or nullptr for the one in the cells' records (monatomic)
cudaError_t launch_micro32(avs_ctx* c, const void* fin, void* fout, const double* diag, int k_micro);

}  // namespace avs
