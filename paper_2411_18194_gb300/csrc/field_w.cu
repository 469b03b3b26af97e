// field_w.cu -- pass C on the warp FFT engine (body in xfft_w.cuh): kernel
// and launcher.
#include "kernels.h"
#include "launch.cuh"
#include "xfft_w.cuh"

namespace mmp {

__global__ void __launch_bounds__(kXwThreads, 4) k_field_w(Grid g, DemagArgs d, Coefs co, FieldArgs f) {
  extern __shared__ __align__(16) unsigned char sraw[];
  after_predecessor();
  field_w_tile(sraw, g, d, co, f, blockIdx.y, 2 * blockIdx.x);
}

cudaError_t launch_field_w(const Grid& g, const DemagArgs& d, const Coefs& c, const FieldArgs& f, int nsub,
                           cudaStream_t s) {
  const int kind = (c.uniform ? 0 : 1) + (nsub == 2 ? 2 : 0);
  if (xg_split(g, kind)) return launch_xg(2, kind, g, nullptr, d, c, &f, s);   // every kind but 0
  const dim3 grid((g.ny + 1) / 2, g.nz);
  const size_t sm = field_w_smem();
  const cudaError_t e = set_smem(k_field_w, sm, 1024);
  return e != cudaSuccess ? e : launch_chained(d.chain, k_field_w, grid, kXwThreads, sm, s, g, d, c, f);
}

}  // namespace mmp
