// The heavy kernels of shape order 0.
#include "instances.cuh"

namespace emu_dev {
EMU_ORDER_INSTANCES(, 0)
EMU_RD_INSTANCES(, 0)
}  // namespace emu_dev
