// xfft_g.cu -- launcher of the general passes A and C (body in xfft_g.cuh;
// kernels instantiated per padded x length in xfft_g_*.cu).
#include "xfft_g.cuh"

#include <stdint.h>
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

// Where pass C is two kernels (k_invx_g, one block per row pair and component,
// then k_cells_g, one thread per item of the local field): one more launch and the
// field through memory, against a kernel whose warps mostly wait for its three to
// twelve transforming ones.  us, one kernel -> two:
//   several regions or two sublattices, cell by cell: field 300x213x3 90 -> 82,
//     600x500x2 151 -> 132, antiferromagnet 1024x256x1 (25 evaluations) 3994 -> 2946;
//   several classes of kx: 2048x128x1 run 1736 -> 1334, 768x640x1 four steps 2568
//     -> 2086, 1000x200x1 1298 -> 1005;
//   one class stays one kernel: 512x512x1 run 623 -> 666, 200x180x1 1208 -> 1242;
//   Px = 2048 above two blocks per SM too (the kernel of xfft_w.cuh): 1000x1000x1
//     the same, 1024x1024x8 run 31554 -> 32629.
bool xg_split(const Grid& g, int kind) {
  int M = 0, Q = 0;
  if (!xg_shape(g, &M, &Q) || M <= 8) return false;
  const long long pairs = (long long)((g.ny + 1) / 2) * g.nz;
  return kind != 0 || (Q > 1 && (g.Px != 2048 || pairs <= kTwoPerSM));
}

// Cells per item of the local field: four, but one or two where that gives a block
// of a small grid up to 256 threads (the same sums; a four-cell item is a chain of
// 1500 instructions on the one warp that its scheduler has): us, four -> fewer:
// 64x64x1 ten steps 1055 -> 891, 200x180x1 1195 -> 1103, 256x256x2 relaxation 976 ->
// 955.
// Threads: the transforms' warps; more where the assembly (nx / 2 items of pass
// A) or the cells (nx / 2 items of four cells, or 2 nx cells) fill them, up to the
// kernel's limit while a grid gives each SM two blocks at most, to 128 above and in
// batches: at 128 registers a thread that is four blocks per SM instead of two.  us,
// limit -> 128: 384x192x4 four steps 1189 -> 1000, 512x512x4 2914 -> 2781, batch of
// 24 32918 -> 30988; but 512x512x1 run (256 row pairs) 623 -> 706.
XgPlan xg_plan(const Grid& g, int pass, bool cells, bool batch) {
  XgPlan l{};
  int M = 0, Q = 0;
  xg_shape(g, &M, &Q);
  const int warps = M <= 8 ? 1 : 3 * Q;
  const bool many = batch || (long long)((g.ny + 1) / 2) * g.nz > kTwoPerSM;
  l.v = many || M > 16 ? 4 : M > 8 ? 2 : 1;
  const int items = pass == 0 ? (g.nx + 1) / 2 : cells ? 2 * g.nx : 2 * g.nx / l.v;
  l.threads = std::max(32 * warps, std::min(many ? 128 : xg_maxthr(Q), (items + 31) / 32 * 32));
  const size_t W = (size_t)3 * Q * xg_pitch(M, Q) * sizeof(float2), HX = g.Px / 2;
  l.smem = pass == 0 ? 3 * HX * sizeof(float2) + W
                     : xg_gather_bytes(M, Q) + (Q == 1 ? 1 : 2) * 6 * HX * sizeof(float);
  return l;
}

static cudaError_t launch_xg_list(int pass, int kind, const Grid& g, const XgArgs& p, const BatchInst* insts,
                           const BatchItem* items, int nitems, int stage, cudaStream_t st) {
  int M = 0, Q = 0;
  if (!xg_shape(g, &M, &Q)) return cudaErrorInvalidValue;
  const XgPlan pl = xg_plan(g, pass, pass == 2 && (kind != 0 || (g.nx & 3)), insts != nullptr);
  XgLaunch l;
  l.grid = insts ? dim3(nitems) : dim3((g.ny + 1) / 2, g.nz);
  l.threads = pl.threads;
  l.smem = pl.smem;
  l.v = pl.v;
  if (!insts && pass == 0 && p.a.y) l.grid.z = 1 + p.a.nparts - p.a.nsub;   // elastic parts: blocks of their own
  if (!insts && pass == 2 && xg_split(g, kind)) {   // one component per block
    l.grid.z = 3;
    l.threads = 32 * Q;   // the transforms' warps (128 threads: 768x640x1 2086 us, 32 Q: 2017)
    l.smem = xg_gather_bytes(M, Q) / 3 + 16;
    pass = 1;
  }
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

// The local field and torque of every cell after k_invx_g (KIND as in pass C,
// VEC: four cells an item).  One item per thread.
template <int KIND, bool VEC>
__global__ void __launch_bounds__(128, 4) k_cells_g(const __grid_constant__ XgArgs p) {
  constexpr int NSUB = KIND >= 2 ? 2 : 1;
  constexpr bool UNI = KIND == 0 || KIND == 2;
  const Grid& g = p.g;
  const int nx = g.nx, ny = g.ny;
  float emax = 0.0f, tmax = 0.0f;
  const long long e = blockIdx.x * 128LL + threadIdx.x;
  after_predecessor();
  if constexpr (VEC) {
    __shared__ RegionCoef sR;
    __shared__ float ec[7];
    if (p.f.err && threadIdx.x == 0) error_coefs_load(p.f, ec);
    const int* src = reinterpret_cast<const int*>(p.co.reg);
    for (int i = threadIdx.x; i < (int)(sizeof(RegionCoef) / sizeof(int)); i += 128) reinterpret_cast<int*>(&sR)[i] = src[i];
    __syncthreads();
    const long long row = e / (nx >> 2);   // z ny + y
    if (4 * e < g.n) {
      const int x0 = 4 * (int)(e - row * (nx >> 2)), z = (int)(row / ny), y = (int)(row - (long long)z * ny), h = y & 1;
      const long long base = (row - h) * nx;   // the row pair
      st4_item<true, 4>(p.f.stage + base, p.f.kout + base, (int)g.n, nx, h, x0, y + 1 - h < ny, g, sR, ec, p.f, z, y,
                     row * nx + x0, emax, tmax);
    }
  } else {
    if (e < g.n) {
      const long long row = e / nx;
      const int x = (int)(e - row * nx), z = (int)(row / ny), y = (int)(row - (long long)z * ny);
      float b3[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) b3[c] = MMP_IN(g, c * g.n + e, g.lim_state) ? p.f.kout[c * g.n + e] : 0.0f;
      field_cell<NSUB, UNI>(b3, g, p.co, p.f, x, y, z, e, emax, tmax);
    }
  }
  field_maxima(p.f, emax, tmax);
}

template <int KIND, bool VEC>
static cudaError_t go_cells(const XgArgs& p, cudaStream_t st) {
  const long long items = VEC ? p.g.n / 4 : p.g.n;
  return launch_chained(p.d.chain, k_cells_g<KIND, VEC>, dim3((unsigned)((items + 127) / 128)), 128, 0, st, p);
}

static cudaError_t launch_cells(int kind, const XgArgs& p, cudaStream_t st) {
  const uintptr_t al = (uintptr_t)p.f.stage | (uintptr_t)p.f.kout | (uintptr_t)p.f.Bout | (uintptr_t)p.f.eps;
  switch (kind) {
    case 0: return (p.g.nx & 3) || (al & 15) ? go_cells<0, false>(p, st) : go_cells<0, true>(p, st);
    case 1: return go_cells<1, false>(p, st);
    case 2: return go_cells<2, false>(p, st);
    default: return go_cells<3, false>(p, st);
  }
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
  const cudaError_t e = launch_xg_list(pass, kind, g, p, nullptr, nullptr, 0, 0, st);
  if (e != cudaSuccess || pass != 2 || !xg_split(g, kind)) return e;
  return launch_cells(kind, p, st);
}

cudaError_t launch_xg_batch(int pass, const Grid& g, const BatchInst* insts, const BatchItem* items, int nitems,
                            int stage, cudaStream_t st) {
  static const XgArgs none{};
  return launch_xg_list(pass, 0, g, none, insts, items, nitems, stage, st);
}


}  // namespace mmp
