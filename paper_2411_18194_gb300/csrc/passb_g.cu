// passb_g.cu -- launcher of the general warp pass B (body in passb_g.cuh;
// kernels instantiated per M in passb_g_*.cu).
#include <algorithm>

#include "batch.h"
#include "kernels.h"
#include "passb_g.cuh"

namespace mmp {

bool passb_g_shape(const Grid& g, PassBG* s) {
  if (g.nz < 1 || g.nz > 8) return false;
  PassBG p;
  p.H = passb_g_half(g.nz);
  p.Q = g.Py > 1024 ? 2 : 1;
  if (g.Py % (32 * p.Q) != 0) return false;
  p.M = g.Py / (32 * p.Q);
  if (p.Q == 1) {
    if (p.M != 2 && p.M != 3 && p.M != 4 && p.M != 6 && p.M != 8 && p.M != 12 && p.M != 16 && p.M != 24 && p.M != 32)
      return false;
  } else if ((p.M != 24 && p.M != 32) || p.H > 4) {
    return false;
  }
  p.cols = passb_g_cols(p.M);
  p.pitch = passb_g_pitch(p.M, p.Q);
  if (passb_g_plan(g, p, 1).smem > 227 * 1024) return false;
  if (s) *s = p;
  return true;
}

bool passb_g_use(const Grid& g, int R, int warp_engine) {
  PassBG s;
  if (!passb_g_shape(g, &s)) return false;
  if (!warp_engine) return R == 1;
  if (R != s.Q) return false;
  return s.Q == 1 ? !(g.nz == 8 && s.M == 32) : g.nz <= 2;
}

PassBGLaunch passb_g_plan(const Grid& g, const PassBG& s, int nplanes) {
  const int ncol = 3 * g.nz;
  const int maxw = passb_g_maxthr(s.H) / 32;
  PassBGLaunch l;
  int groups = 1;
  l.kp = 1;
  // as many planes as give every warp of a block one group of columns, two
  // blocks per SM left
  for (int kp = 1; kp <= 8; ++kp) {
    const int gr = (kp * ncol + s.cols - 1) / s.cols;
    if (kp > 1 && (gr > maxw || (size_t)gr * s.cols * s.Q * s.pitch * sizeof(float2) > 64 * 1024)) break;
    if (kp > 1 && nplanes > 0 && nplanes < kp * kTwoPerSM) break;
    if (kp > 1 && (kp * ncol) % s.cols != 0 && (ncol % s.cols) == 0) continue;
    l.kp = kp;
    groups = gr;
  }
  const int rounds = (groups + maxw - 1) / maxw;
  l.threads = 32 * ((groups + rounds - 1) / rounds);
  l.smem = (size_t)groups * s.cols * s.Q * s.pitch * sizeof(float2);
  return l;
}

template <int M, int Q>
static cudaError_t by_half(const Grid& g, const DemagArgs& d, const PassBG& s, const PassBGLaunch& l, int nblocks,
                           const BatchInst* insts, const BatchItem* items, cudaStream_t st) {
  switch (s.H) {
    case 1: return launch_passB_g_t<1, M, Q>(g, d, l, nblocks, insts, items, st);
    case 2: return launch_passB_g_t<2, M, Q>(g, d, l, nblocks, insts, items, st);
    case 3: return launch_passB_g_t<3, M, Q>(g, d, l, nblocks, insts, items, st);
    case 4: return launch_passB_g_t<4, M, Q>(g, d, l, nblocks, insts, items, st);
    default: break;
  }
  if constexpr (Q == 1) {
    if (s.H == 6) return launch_passB_g_t<6, M, Q>(g, d, l, nblocks, insts, items, st);
    if (s.H == 8) return launch_passB_g_t<8, M, Q>(g, d, l, nblocks, insts, items, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_passB_g(const Grid& g, const DemagArgs& d, const PassBG& s, const PassBGLaunch& l, int nblocks,
                           const BatchInst* insts, const BatchItem* items, cudaStream_t st) {
  if (s.Q == 2)
    return s.M == 24 ? by_half<24, 2>(g, d, s, l, nblocks, insts, items, st)
                     : by_half<32, 2>(g, d, s, l, nblocks, insts, items, st);
  switch (s.M) {
    case 2: return by_half<2, 1>(g, d, s, l, nblocks, insts, items, st);
    case 3: return by_half<3, 1>(g, d, s, l, nblocks, insts, items, st);
    case 4: return by_half<4, 1>(g, d, s, l, nblocks, insts, items, st);
    case 6: return by_half<6, 1>(g, d, s, l, nblocks, insts, items, st);
    case 8: return by_half<8, 1>(g, d, s, l, nblocks, insts, items, st);
    case 12: return by_half<12, 1>(g, d, s, l, nblocks, insts, items, st);
    case 16: return by_half<16, 1>(g, d, s, l, nblocks, insts, items, st);
    case 24: return by_half<24, 1>(g, d, s, l, nblocks, insts, items, st);
    case 32: return by_half<32, 1>(g, d, s, l, nblocks, insts, items, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mmp
