// xfft_g_d.cu -- general passes A and C (body in xfft_g.cuh): kernels of Px = 768.
#define MMP_XFFT_G_KERNELS
#include "xfft_g.cuh"

namespace mmp {

MMP_XG(24, 1)

}  // namespace mmp
