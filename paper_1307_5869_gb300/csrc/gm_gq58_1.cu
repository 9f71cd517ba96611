// GQ58.1 instantiation of the torus-map ensemble kernels (see gm_host.cuh).
#include "gm_host.cuh"

namespace prand {
PRAND_GM_INSTANTIATE(PRAND_GQ58_1, gq58_1)
}  // namespace prand
