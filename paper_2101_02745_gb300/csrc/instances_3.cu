// The heavy kernels of shape order 3.
#include "instances.cuh"

namespace emu_dev {
EMU_ORDER_INSTANCES(, 3)
}  // namespace emu_dev
