// inst_w3.cu -- kernels and launchers for 512-bit keys of at most 192 spin
// orbitals, kept as three words on the device (hash annihilation): five of the
// eight words are zero, and every key read, written, compared or hashed was
// 64 bytes instead of 24.
#include "launch.cuh"

namespace hande {
Ops ops_w3(int kind) { return ops_for<3>(kind); }
}  // namespace hande
