// mra_sizes.h -- device memory of a problem's factors (host code only).
#pragma once
#include <cstdint>

namespace mra {

// Bytes of the factors that mra_build allocates: rc[m] regions' storage at every
// level m < M (V, L^{-1}, Ahat, omegahat, Lt^{-1}, G, g) and leaf stores for obs
// observations, ls entries of L_Sigma^{-1} and `leaves` leaves (H, z, L_Sigma^{-1}).
// gram: the Gram products run on the emulation engine, which takes the column
// scales of G and H (the emulated form, and the 3xTF32 form where gram_on_engine
// says so: on a complete tree with few observations a leaf the table of H is as
// large as H itself); emu: the row scales of V, L^{-1} and H as well.
inline double factor_bytes(int M, int r, bool emu, bool gram, const int64_t* rc, int64_t obs, int64_t ls, int64_t leaves) {
  double b = 0;
  for (int m = 0; m < M; ++m) {
    const double R = (double)rc[m], T = (m + 1) * (m + 2) / 2.0;
    b += 8.0 * R * ((double)r * m * r * 2 + r * r * 2 + T * r * r + (m + 1) * r + r);
    if (gram) b += 4.0 * R * m * r;
    if (emu) b += 4.0 * R * (((m * r + 127) / 128) * r + r);
  }
  b += 8.0 * ((double)obs * M * r + obs + ls);
  if (gram) b += 4.0 * (double)leaves * M * r;
  if (emu) b += 4.0 * (double)obs * ((M * r + 127) / 128);
  return b;
}

}  // namespace mra
