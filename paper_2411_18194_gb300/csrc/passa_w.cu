// passa_w.cu -- pass A on the warp FFT engine (body in xfft_w.cuh): kernel
// and launcher.
#include "kernels.h"
#include "launch.cuh"
#include "xfft_w.cuh"

namespace mmp {

template <bool ASSEMBLE>
__global__ void __launch_bounds__(kXwThreads, 4) k_passA_w(Grid g, StageArgs a, DemagArgs d, Coefs co) {
  extern __shared__ __align__(16) unsigned char sraw[];
  after_predecessor();
  passA_w_tile<ASSEMBLE>(sraw, g, a, d, co, blockIdx.y, 2 * blockIdx.x);
}

cudaError_t launch_passA_w(const Grid& g, const StageArgs& a, const DemagArgs& d, const Coefs& c, cudaStream_t s) {
  // two sublattices: the general pass, whose loads of a stage's vectors are in
  // flight together and whose elastic parts have blocks of their own
  // (antiferromagnet 1024x256x1, four steps: 2902 -> 2665 us)
  if (a.nsub == 2) return launch_xg(0, 0, g, &a, d, c, nullptr, s);
  const dim3 grid((g.ny + 1) / 2, g.nz);
  const size_t sm = passa_w_smem();
  auto go = [&](auto kernel) {
    const cudaError_t e = set_smem(kernel, sm, 64);
    return e != cudaSuccess ? e : launch_chained(d.chain, kernel, grid, kXwThreads, sm, s, g, a, d, c);
  };
  return a.stage != nullptr && a.y != nullptr ? go(k_passA_w<true>) : go(k_passA_w<false>);
}

}  // namespace mmp
