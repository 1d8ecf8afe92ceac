// The heavy kernels of shape order 2.
#include "instances.cuh"

namespace emu_dev {
EMU_ORDER_INSTANCES(, 2)
EMU_RD_INSTANCES(, 2)
}  // namespace emu_dev
