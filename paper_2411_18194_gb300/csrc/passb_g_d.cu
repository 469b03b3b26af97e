// passb_g_d.cu -- kernels of the general warp pass B (passb_g.cuh) of padded y
// lengths 768 and 1536.
#define MMP_PASSB_G_KERNELS
#include "passb_g.cuh"

namespace mmp {
MMP_PASSB_G_ALL(24)
MMP_PASSB_G_LOW(24, 2)
}  // namespace mmp
