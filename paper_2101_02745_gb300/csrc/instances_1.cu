// The heavy kernels of shape order 1.
#include "instances.cuh"

namespace emu_dev {
EMU_ORDER_INSTANCES(, 1)
EMU_RD_INSTANCES(, 1)
}  // namespace emu_dev
