// xfft_g_b.cu -- general passes A and C (body in xfft_g.cuh): kernels of Px = 192, 256.
#define MMP_XFFT_G_KERNELS
#include "xfft_g.cuh"

namespace mmp {

MMP_XG(6, 1)
MMP_XG(8, 1)

}  // namespace mmp
