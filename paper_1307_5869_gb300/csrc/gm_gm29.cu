// GM29 instantiation of the torus-map ensemble kernels (see gm_host.cuh).
#include "gm_host.cuh"

namespace prand {
PRAND_GM_INSTANTIATE(PRAND_GM29, gm29)
}  // namespace prand
