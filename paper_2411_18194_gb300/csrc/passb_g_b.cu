// passb_g_b.cu -- kernels of the general warp pass B (passb_g.cuh) of padded y
// lengths 192 and 256.
#define MMP_PASSB_G_KERNELS
#include "passb_g.cuh"

namespace mmp {
MMP_PASSB_G_ALL(6)
MMP_PASSB_G_ALL(8)
}  // namespace mmp
