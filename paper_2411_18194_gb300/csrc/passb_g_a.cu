// passb_g_a.cu -- kernels of the general warp pass B (passb_g.cuh) of padded y
// lengths 64 .. 128.
#define MMP_PASSB_G_KERNELS
#include "passb_g.cuh"

namespace mmp {
MMP_PASSB_G_ALL(2)
MMP_PASSB_G_ALL(3)
MMP_PASSB_G_ALL(4)
}  // namespace mmp
