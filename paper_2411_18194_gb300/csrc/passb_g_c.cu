// passb_g_c.cu -- kernels of the general warp pass B (passb_g.cuh) of padded y
// lengths 384 and 512.
#define MMP_PASSB_G_KERNELS
#include "passb_g.cuh"

namespace mmp {
MMP_PASSB_G_ALL(12)
MMP_PASSB_G_ALL(16)
}  // namespace mmp
