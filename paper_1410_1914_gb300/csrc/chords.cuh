// 13-direction pore lengths and diffusivities from bit masks (chords.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace cl {

// whether a box takes this path: its bit sets fit one double per cell, no run can exceed `most` cells, and the ratio of
// Knudsen to bulk diffusivity stays inside the f32 range
bool chord_bits_fit(int nx, int ny, int nz, int most, double dx, double vkn, double D_b);
// D (Eq. 7-9; 0 off the active set) of every cell; tot[0..2]: sums over the pore cells of their axis, face-diagonal
// and body-diagonal run lengths in cells, tot[3]: pore cells.  scratch: one double per cell.
cudaError_t launch_chord_bits(const uint8_t* phase, const uint8_t* active, int nx, int ny, int nz, double dx,
                              double vkn, double D_b, double D_ion, int knudsen, double* scratch, double* D,
                              unsigned long long* tot, cudaStream_t s);

}  // namespace cl
