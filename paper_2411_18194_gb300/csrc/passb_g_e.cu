// passb_g_e.cu -- kernels of the general warp pass B (passb_g.cuh) of padded y
// lengths 1024 and 2048.
#define MMP_PASSB_G_KERNELS
#include "passb_g.cuh"

namespace mmp {
MMP_PASSB_G_ALL(32)
MMP_PASSB_G_LOW(32, 2)
}  // namespace mmp
