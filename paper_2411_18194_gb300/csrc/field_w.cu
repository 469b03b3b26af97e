// field_w.cu -- pass C on the warp FFT engine (body in xfft_w.cuh): kernel
// instantiations and launcher.
#include "kernels.h"
#include "launch.cuh"
#include "xfft_w.cuh"

namespace mmp {

cudaError_t launch_field_w(const Grid& g, const DemagArgs& d, const Coefs& c, const FieldArgs& f, int nsub,
                           cudaStream_t s) {
  const int kind = (c.uniform ? 0 : 1) + (nsub == 2 ? 2 : 0);
  if (xg_split(g, kind)) return launch_xg(2, kind, g, nullptr, d, c, &f, s);   // every kind but 0
  const dim3 grid((g.ny + 1) / 2, g.nz);
  const size_t sm = field_w_smem();
  const cudaError_t e = set_smem(k_field_w<1, true>, sm, 1024);
  return e != cudaSuccess ? e : launch_chained(d.chain, k_field_w<1, true>, grid, kXwThreads, sm, s, g, d, c, f);
}

}  // namespace mmp
