// Memory rule of the automatic factor choice (host only, no CUDA).
#pragma once
#include <cstddef>

namespace helm {

// BCR holds about 3 (and 5.3 while it factors; 6 counted) times the line factor's bytes.  On a short or
// odd line, where the line factor would do, it is taken automatically while that is a small part of
// the device: up to kBcrShortBytes, and above kBcrAlwaysBytes (0.4 % of 284 GB; not worth asking, one
// factor of 128^2 with three frequencies counts 0.3 GB) only if no more than an eighth of what is available.
constexpr size_t kBcrShortBytes = (size_t)16 << 30, kBcrAlwaysBytes = (size_t)1 << 30;
inline size_t short_bcr_bytes(size_t n_omega, size_t nx, size_t nz) { return 6 * 8 * n_omega * nx * nz * nz; }
// available(): bytes that a caller could still allocate
template <typename Available> bool short_bcr_fits(size_t bytes, Available available) {
    return bytes <= kBcrAlwaysBytes || (bytes <= kBcrShortBytes && bytes <= available() / 8);
}

}  // namespace helm
