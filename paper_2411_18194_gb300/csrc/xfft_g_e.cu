// xfft_g_e.cu -- general passes A and C (body in xfft_g.cuh): kernels of Px = 1024.
#define MMP_XFFT_G_KERNELS
#include "xfft_g.cuh"

namespace mmp {

MMP_XG(32, 1)

}  // namespace mmp
