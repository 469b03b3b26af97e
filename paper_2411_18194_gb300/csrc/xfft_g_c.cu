// xfft_g_c.cu -- general passes A and C (body in xfft_g.cuh): kernels of Px = 384, 512.
#define MMP_XFFT_G_KERNELS
#include "xfft_g.cuh"

namespace mmp {

MMP_XG(12, 1)
MMP_XG(16, 1)

}  // namespace mmp
