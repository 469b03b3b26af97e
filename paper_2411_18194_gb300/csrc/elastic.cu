// elastic.cu -- strain/stress and elastic force (4th-order stencils in the
// bulk, divergence = -G^T of the gradient G) plus the magnetoelastic force.
#include <cooperative_groups.h>
#include "kernels.h"
#include "launch.cuh"
#include "stage.cuh"

namespace cg = cooperative_groups;

namespace mmp {

// ---------------------------------------------------------- elastic -------
// Gradient operator G along an axis of n cells (rows: one-sided 2nd order at
// an edge, central 2nd order one cell in, central 4th order in the bulk;
// (f1 - f0)/h for n = 2); the divergence is -G^T.
__device__ __forceinline__ float gcoef(int i, int j, int n, float ih) {
  if (n == 1) return 0.0f;
  if (n == 2) return j == 0 ? -ih : (j == 1 ? ih : 0.0f);
  int dj = j - i;
  if (i == 0) return dj == 0 ? -1.5f * ih : dj == 1 ? 2.0f * ih : dj == 2 ? -0.5f * ih : 0.0f;
  if (i == n - 1) return dj == -2 ? 0.5f * ih : dj == -1 ? -2.0f * ih : dj == 0 ? 1.5f * ih : 0.0f;
  if (i == 1 || i == n - 2) return dj == -1 ? -0.5f * ih : dj == 1 ? 0.5f * ih : 0.0f;
  const float c = ih * (1.0f / 12.0f);
  return dj == -2 ? c : dj == -1 ? -8.0f * c : dj == 1 ? 8.0f * c : dj == 2 ? -c : 0.0f;
}

// (G f)(cell) along an axis: row `i` of G applied to f.
__device__ __forceinline__ float grad_at(const float* __restrict__ f, long long cell, int i, int n,
                                         long long stride, float ih) {
  float acc = 0.0f;
  int lo = i - 2 < 0 ? 0 : i - 2, hi = i + 2 > n - 1 ? n - 1 : i + 2;
  for (int j = lo; j <= hi; ++j) {
    float c = gcoef(i, j, n, ih);
    if (c != 0.0f) acc = fmaf(c, f[cell + (long long)(j - i) * stride], acc);
  }
  return acc;
}

// (G^T s)(cell) along an axis: sum_i G[i][j] s_i, j the cell's index.
__device__ __forceinline__ float gradT_at(const float* __restrict__ s, long long cell, int j, int n,
                                          long long stride, float ih) {
  float acc = 0.0f;
  int lo = j - 2 < 0 ? 0 : j - 2, hi = j + 2 > n - 1 ? n - 1 : j + 2;
  for (int i = lo; i <= hi; ++i) {
    float c = gcoef(i, j, n, ih);
    if (c != 0.0f) acc = fmaf(c, s[cell + (long long)(i - j) * stride], acc);
  }
  return acc;
}

// Bulk rows of G (4th-order central) and of G^T, with the coefficients and
// the order of the multiply-adds of grad_at / gradT_at, so a bulk cell gets
// bitwise the same value without the per-term coefficient selection.
__device__ __forceinline__ float grad_bulk(const float* __restrict__ f, long long cell, long long st, float ih) {
  const float c = ih * (1.0f / 12.0f);
  float acc = fmaf(c, f[cell - 2 * st], 0.0f);
  acc = fmaf(-8.0f * c, f[cell - st], acc);
  acc = fmaf(8.0f * c, f[cell + st], acc);
  return fmaf(-c, f[cell + 2 * st], acc);
}
__device__ __forceinline__ float gradT_bulk(const float* __restrict__ s, long long cell, long long st, float ih) {
  const float c = ih * (1.0f / 12.0f);
  float acc = fmaf(-c, s[cell - 2 * st], 0.0f);
  acc = fmaf(8.0f * c, s[cell - st], acc);
  acc = fmaf(-8.0f * c, s[cell + st], acc);
  return fmaf(c, s[cell + 2 * st], acc);
}
// Whether every axis of more than one cell has index i with all the rows the
// operator needs in the 4th-order bulk: G: 2 <= i <= n - 3; G^T: 4 <= i <= n - 5.
__device__ __forceinline__ bool in_bulk(const int (&idx)[3], const int (&ext)[3], int margin) {
  bool b = true;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if (ext[a] > 1) b = b && idx[a] >= margin && idx[a] <= ext[a] - 1 - margin;
  return b;
}

// Whether row idx of one axis of n cells is in the bulk of G (margin 2) or G^T (4).
__device__ __forceinline__ bool axis_bulk(int idx, int n, int margin) { return idx >= margin && idx <= n - 1 - margin; }

// One thread a cell, cells packed into blocks whatever the extents: a row of its own
// blocks left most threads of a narrow grid idle, and a cell at one edge took the slow
// rows along every axis (antiferromagnet without demag, us an evaluation, before ->
// packed and by axis: 8x4096x1 151 -> 53, 129x8000x1 787 -> 298, 65x65x65 367 -> 150;
// with demag 1024x1024x1 351 -> 293).  The coordinates come from exact divisions by
// multiplication: 64-bit divisions cost the kernels a third of their time.
constexpr int kElThreads = 128;
// q = c / d for 0 <= c < 2^31: m = ceil(2^(31 + l) / d), l = ceil(log2 d), so m < 2^32 and the
// excess c (m d - 2^(31 + l)) / 2^(31 + l) stays below 1.
struct FastDiv {
  unsigned m, s, d;
};
static FastDiv fast_div(unsigned d) {
  unsigned l = 0;
  while ((1u << l) < d) ++l;
  return {(unsigned)(((1ull << (31 + l)) + d - 1) / d), 31 + l, d};
}
__device__ __forceinline__ unsigned div_by(unsigned c, const FastDiv& f) {
  return (unsigned)(((unsigned long long)c * f.m) >> f.s);
}
struct CellDiv {
  FastDiv x, y;
};
static CellDiv cell_div(const Grid& g) { return {fast_div(g.nx), fast_div(g.ny)}; }
template <bool HZ>
__device__ __forceinline__ void cell_index(const CellDiv& f, unsigned cell, int (&idx)[3]) {
  const unsigned row = div_by(cell, f.x), z = HZ ? div_by(row, f.y) : 0;
  idx[0] = (int)(cell - row * f.x.d);
  idx[1] = (int)(row - z * f.y.d);
  idx[2] = (int)z;
}

// The three components' gradients along one axis (zero for one cell).
__device__ __forceinline__ void grad3(const float* __restrict__ f, long long n, long long cell, int i, int ext,
                                      long long st, float ih, float (&G)[3]) {
  if (ext == 1) return;
  if (axis_bulk(i, ext, 2)) {
#pragma unroll
    for (int j = 0; j < 3; ++j) G[j] = grad_bulk(f + j * n, cell, st, ih);
  } else {
#pragma unroll
    for (int j = 0; j < 3; ++j) G[j] = grad_at(f + j * n, cell, i, ext, st, ih);
  }
}

// Both elastic kernels are bound by the latency of their neighbour loads (24 and
// about 80 a cell): a cell whose rows are all in the 4th-order bulk takes a path
// with no selection between them, so that they are in flight together; the
// selection per term and the 64-bit divisions of the index took most of the time
// before.  1024x256x1 with two sublattices, cold L2, us a launch, general form -> bulk
// path in rows -> packed and by axis: strain 25, 20, 12.5; force 59, 38, 30.5.
// Antiferromagnet 1024x256x1, four steps (25 launches of each): 2678 -> 2253 us by the
// last of these.
// HZ: nz > 1.
template <bool HZ>
__global__ void __launch_bounds__(kElThreads) k_strain(Grid g, ElasticArgs e, CellDiv fd, int nsub) {
  const long long n = g.n;
  const float* u = e.stage + (long long)3 * nsub * n;
  const float* v = u + 3 * n;
  constexpr int NA = HZ ? 3 : 2;
  const long long cell = (long long)blockIdx.x * kElThreads + threadIdx.x;
  if (cell < n) {
    int idx[3];
    cell_index<HZ>(fd, (unsigned)cell, idx);
    const int ext[3] = {g.nx, g.ny, g.nz};
    const long long st[3] = {1, g.nx, (long long)g.nx * g.ny};
    float G[3][3] = {}, Gv[3][3] = {};
    if (in_bulk(idx, ext, 2)) {
#pragma unroll
      for (int a = 0; a < NA; ++a)
        if (ext[a] > 1) {
#pragma unroll
          for (int j = 0; j < 3; ++j) G[a][j] = grad_bulk(u + j * n, cell, st[a], g.ih[a]);
          if (e.eta != 0.0f)
#pragma unroll
            for (int j = 0; j < 3; ++j) Gv[a][j] = grad_bulk(v + j * n, cell, st[a], g.ih[a]);
        }
    } else {   // by axis: most of these cells are at the edge of one axis only
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        grad3(u, n, cell, idx[a], ext[a], st[a], g.ih[a], G[a]);
        if (e.eta != 0.0f) grad3(v, n, cell, idx[a], ext[a], st[a], g.ih[a], Gv[a]);
      }
    }
    float eps[6] = {G[0][0], G[1][1], G[2][2], 0.5f * (G[0][1] + G[1][0]), 0.5f * (G[0][2] + G[2][0]),
                    0.5f * (G[1][2] + G[2][1])};
    float epv[6] = {Gv[0][0], Gv[1][1], Gv[2][2], 0.5f * (Gv[0][1] + Gv[1][0]), 0.5f * (Gv[0][2] + Gv[2][0]),
                    0.5f * (Gv[1][2] + Gv[2][1])};
#pragma unroll
    for (int c = 0; c < 6; ++c) e.eps[c * n + cell] = eps[c];
    float sig[6];
    sig[0] = e.c11 * eps[0] + e.c12 * (eps[1] + eps[2]);
    sig[1] = e.c11 * eps[1] + e.c12 * (eps[0] + eps[2]);
    sig[2] = e.c11 * eps[2] + e.c12 * (eps[0] + eps[1]);
    sig[3] = 2.0f * e.c44 * eps[3];
    sig[4] = 2.0f * e.c44 * eps[4];
    sig[5] = 2.0f * e.c44 * eps[5];
    if (e.eta != 0.0f) {
      sig[0] += e.eta * (e.c11 * epv[0] + e.c12 * (epv[1] + epv[2]));
      sig[1] += e.eta * (e.c11 * epv[1] + e.c12 * (epv[0] + epv[2]));
      sig[2] += e.eta * (e.c11 * epv[2] + e.c12 * (epv[0] + epv[1]));
      sig[3] += e.eta * 2.0f * e.c44 * epv[3];
      sig[4] += e.eta * 2.0f * e.c44 * epv[4];
      sig[5] += e.eta * 2.0f * e.c44 * epv[5];
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) e.sig[c * n + cell] = sig[c];
  }
}

// Force of one cell.  BULK: every row of G and G^T it needs is in the bulk; else each
// axis is looked at by itself.
template <bool UNI, bool HZ, bool BULK>
__device__ __forceinline__ void elastic_force(const Grid& g, const ElasticArgs& e, const Coefs& co, int nsub,
                                              long long cell, const int (&idx)[3], float (&f)[3]) {
  const long long n = g.n;
  constexpr int NA = HZ ? 3 : 2;
  constexpr int sidx[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};   // sigma_ab as component of sig[6]
  const int ext[3] = {g.nx, g.ny, g.nz};
  const long long st[3] = {1, g.nx, (long long)g.nx * g.ny};
#pragma unroll
  for (int a = 0; a < NA; ++a)
    if (ext[a] > 1) {
      if (BULK || axis_bulk(idx[a], ext[a], 4)) {
#pragma unroll
        for (int b = 0; b < 3; ++b) f[b] -= gradT_bulk(e.sig + sidx[a][b] * n, cell, st[a], g.ih[a]);
      } else {
#pragma unroll
        for (int b = 0; b < 3; ++b) f[b] -= gradT_at(e.sig + sidx[a][b] * n, cell, idx[a], ext[a], st[a], g.ih[a]);
      }
    }
  if (!(e.terms & 64u)) return;
  const int reg = UNI ? 0 : co.regions[cell];
  for (int s = 0; s < nsub; ++s) {
    const float* m = e.stage + (long long)3 * s * n;
    const RegionCoef& R = co.reg[s * MMP_MAX_REGIONS + reg];
    float G[3][3] = {};
#pragma unroll
    for (int a = 0; a < NA; ++a) {
      if (BULK) {
        if (ext[a] > 1)
#pragma unroll
          for (int j = 0; j < 3; ++j) G[a][j] = grad_bulk(m + j * n, cell, st[a], g.ih[a]);
      } else {
        grad3(m, n, cell, idx[a], ext[a], st[a], g.ih[a], G[a]);
      }
    }
    const float mx = m[cell], my = m[n + cell], mz = m[2 * n + cell];
    const float B1 = R.b1, B2 = R.b2;
    f[0] += 2.0f * B1 * mx * G[0][0] + B2 * (mx * (G[1][1] + G[2][2]) + my * G[1][0] + mz * G[2][0]);
    f[1] += 2.0f * B1 * my * G[1][1] + B2 * (my * (G[0][0] + G[2][2]) + mx * G[0][1] + mz * G[2][1]);
    f[2] += 2.0f * B1 * mz * G[2][2] + B2 * (mz * (G[0][0] + G[1][1]) + mx * G[0][2] + my * G[1][2]);
  }
}

// Six blocks an SM (72 registers): without the bound it takes 128 to 160 and the
// 65x65x65 magnet 233 us an evaluation instead of 150, 1024x1024x1 320 instead of 293.
template <bool UNI, bool HZ>
__global__ void __launch_bounds__(kElThreads, 6) k_elastic_rhs(Grid g, ElasticArgs e, Coefs co, CellDiv fd,
                                                            int nsub) {
  const long long n = g.n;
  const float* v = e.stage + (long long)3 * (nsub + 1) * n;
  float* ku = e.kout + (long long)3 * nsub * n;
  float* kv = ku + 3 * n;
  const long long cell = (long long)blockIdx.x * kElThreads + threadIdx.x;
  if (cell < n) {
    int idx[3];
    cell_index<HZ>(fd, (unsigned)cell, idx);
    const int ext[3] = {g.nx, g.ny, g.nz};
    const float vc[3] = {v[cell], v[n + cell], v[2 * n + cell]};
    float f[3] = {0.0f, 0.0f, 0.0f};
    if (in_bulk(idx, ext, 4)) elastic_force<UNI, HZ, true>(g, e, co, nsub, cell, idx, f);
    else elastic_force<UNI, HZ, false>(g, e, co, nsub, cell, idx, f);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ku[c * n + cell] = vc[c];
      kv[c * n + cell] = f[c] * e.inv_rho;
    }
  }
}

static unsigned elastic_blocks(const Grid& g) { return (unsigned)((g.n + kElThreads - 1) / kElThreads); }

cudaError_t launch_strain(const Grid& g, const ElasticArgs& e, int nsub, cudaStream_t s) {
  const CellDiv fd = cell_div(g);
  if (g.nz > 1) k_strain<true><<<elastic_blocks(g), kElThreads, 0, s>>>(g, e, fd, nsub);
  else k_strain<false><<<elastic_blocks(g), kElThreads, 0, s>>>(g, e, fd, nsub);
  return cudaGetLastError();
}

cudaError_t launch_elastic_rhs(const Grid& g, const ElasticArgs& e, const Coefs& c, int nsub, cudaStream_t s) {
  const unsigned grid = elastic_blocks(g);
  const CellDiv fd = cell_div(g);
  if (c.uniform) {
    if (g.nz > 1) k_elastic_rhs<true, true><<<grid, kElThreads, 0, s>>>(g, e, c, fd, nsub);
    else k_elastic_rhs<true, false><<<grid, kElThreads, 0, s>>>(g, e, c, fd, nsub);
  } else {
    if (g.nz > 1) k_elastic_rhs<false, true><<<grid, kElThreads, 0, s>>>(g, e, c, fd, nsub);
    else k_elastic_rhs<false, false><<<grid, kElThreads, 0, s>>>(g, e, c, fd, nsub);
  }
  return cudaGetLastError();
}

}  // namespace mmp
