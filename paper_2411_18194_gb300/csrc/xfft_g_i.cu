// xfft_g_i.cu -- general passes A and C (body in xfft_g.cuh): kernels of Px = 4096.
#define MMP_XFFT_G_KERNELS
#include "xfft_g.cuh"

namespace mmp {

MMP_XG(32, 4)

}  // namespace mmp
