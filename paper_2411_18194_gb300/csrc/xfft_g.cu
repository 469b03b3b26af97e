// xfft_g.cu -- launcher of the general passes A and C (body in xfft_g.cuh;
// kernels instantiated per padded x length in xfft_g_*.cu).
#include "xfft_g.cuh"

#include <string.h>

#include <algorithm>

namespace mmp {

bool xg_shape(const Grid& g, int* M, int* Q) {
  switch (g.Px) {
    case 64: case 96: case 128: case 192: case 256: case 384: case 512: case 768: case 1024:
      *M = g.Px / 32; *Q = 1; return true;
    case 1536: case 2048: *M = g.Px / 64; *Q = 2; return true;
    case 3072: case 4096: *M = g.Px / 128; *Q = 4; return true;
    default: return false;
  }
}

// Threads: the transforms' warps; more where the assembly (nx / 2 items of pass
// A) or the cells (nx / 2 items of four cells, or 2 nx cells) fill them.
XgPlan xg_plan(const Grid& g, int pass, bool cells) {
  XgPlan l{};
  int M = 0, Q = 0;
  xg_shape(g, &M, &Q);
  const int warps = M <= 8 ? 1 : 3 * Q;
  const int items = pass == 2 && cells ? 2 * g.nx : (g.nx + 1) / 2;
  l.threads = std::min(xg_maxthr(Q), std::max(32 * warps, (items + 31) / 32 * 32));
  const size_t W = (size_t)3 * Q * xg_pitch(M, Q) * sizeof(float2), HX = g.Px / 2;
  l.smem = pass == 0 ? 3 * HX * sizeof(float2) + W
                     : xg_gather_bytes(M, Q) + (Q == 1 ? 1 : 2) * 6 * HX * sizeof(float);
  return l;
}

static cudaError_t launch_xg_list(int pass, int kind, const Grid& g, const XgArgs& p, const BatchInst* insts,
                           const BatchItem* items, int nitems, int stage, cudaStream_t st) {
  int M = 0, Q = 0;
  if (!xg_shape(g, &M, &Q)) return cudaErrorInvalidValue;
  const XgPlan pl = xg_plan(g, pass, pass == 2 && (kind != 0 || (g.nx & 3)));
  XgLaunch l;
  l.grid = insts ? dim3(nitems) : dim3((g.ny + 1) / 2, g.nz);
  l.threads = pl.threads;
  l.smem = pl.smem;
  if (Q == 1) {
    switch (M) {
      case 2: return launch_xg_t<2, 1>(pass, kind, p, l, insts, items, stage, st);
      case 3: return launch_xg_t<3, 1>(pass, kind, p, l, insts, items, stage, st);
      case 4: return launch_xg_t<4, 1>(pass, kind, p, l, insts, items, stage, st);
      case 6: return launch_xg_t<6, 1>(pass, kind, p, l, insts, items, stage, st);
      case 8: return launch_xg_t<8, 1>(pass, kind, p, l, insts, items, stage, st);
      case 12: return launch_xg_t<12, 1>(pass, kind, p, l, insts, items, stage, st);
      case 16: return launch_xg_t<16, 1>(pass, kind, p, l, insts, items, stage, st);
      case 24: return launch_xg_t<24, 1>(pass, kind, p, l, insts, items, stage, st);
      default: return launch_xg_t<32, 1>(pass, kind, p, l, insts, items, stage, st);
    }
  }
  if (Q == 2)
    return M == 24 ? launch_xg_t<24, 2>(pass, kind, p, l, insts, items, stage, st)
                   : launch_xg_t<32, 2>(pass, kind, p, l, insts, items, stage, st);
  return M == 24 ? launch_xg_t<24, 4>(pass, kind, p, l, insts, items, stage, st)
                 : launch_xg_t<32, 4>(pass, kind, p, l, insts, items, stage, st);
}

cudaError_t launch_xg(int pass, int kind, const Grid& g, const StageArgs* a, const DemagArgs& d, const Coefs& c,
                      const FieldArgs* f, cudaStream_t st) {
  XgArgs p;
  memset(&p, 0, sizeof p);
  p.g = g;
  p.d = d;
  p.co = c;
  if (a) p.a = *a;
  if (f) p.f = *f;
  return launch_xg_list(pass, kind, g, p, nullptr, nullptr, 0, 0, st);
}

cudaError_t launch_xg_batch(int pass, const Grid& g, const BatchInst* insts, const BatchItem* items, int nitems,
                            int stage, cudaStream_t st) {
  static const XgArgs none{};
  return launch_xg_list(pass, 0, g, none, insts, items, nitems, stage, st);
}

}  // namespace mmp
