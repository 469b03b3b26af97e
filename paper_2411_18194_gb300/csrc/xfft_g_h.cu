// xfft_g_h.cu -- general passes A and C (body in xfft_g.cuh): kernels of Px = 3072.
#define MMP_XFFT_G_KERNELS
#include "xfft_g.cuh"

namespace mmp {

MMP_XG(24, 4)

}  // namespace mmp
