// xfft_g_g.cu -- general passes A and C (body in xfft_g.cuh): kernels of Px = 2048.
#define MMP_XFFT_G_KERNELS
#include "xfft_g.cuh"

namespace mmp {

MMP_XG(32, 2)

}  // namespace mmp
