// xfft_g_a.cu -- general passes A and C (body in xfft_g.cuh): kernels of Px = 64, 96, 128.
#define MMP_XFFT_G_KERNELS
#include "xfft_g.cuh"

namespace mmp {

MMP_XG(2, 1)
MMP_XG(3, 1)
MMP_XG(4, 1)

}  // namespace mmp
