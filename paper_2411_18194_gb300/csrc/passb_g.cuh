// passb_g.cuh -- the general pass B of the demag convolution on the warp
// transforms of gfft.cuh: every padded y length Py = Q * 32 M (Q = 1 or 2 ky
// classes, all of them in one CTA) and every nz <= 8, for planes that fit in
// one CTA's shared memory.  A CTA takes `kp` consecutive kx planes of the
// spectrum T[kx][c][z][y]:
//   1. forward y transform of every column (3 nz per plane), NB columns per
//      warp, read from T straight into registers (y < ny <= Py / 2: the zero
//      half is not held), the result into the warp's columns of W;
//   2. per kx and |ky|, one thread: ky and its mirror Py - ky with one row of
//      the kernel octant: z transform (padded length 2 H, as its even and odd
//      halves), the 3x3 symmetric kernel multiply, inverse z transform;
//   3. inverse y transform of every column, the y < ny outputs to T.
//
// What bounds it and why this layout: the block Stockham pass this replaces
// for these planes spent its time in barriers and run-time index arithmetic
// with 19 % of the warps active, and the warp pass B of passb_w.cuh gives one
// CTA per SM with all but one of its warps idle when a plane has few columns.
// Here a plane takes only the warps its columns fill, several CTAs share an SM
// (their loads of T cover one another's transforms, so no staging copy), and
// with three columns per plane and per warp (nz = 1, M <= 8) a warp does a
// plane alone and no block barrier remains.  What bounds it now is the latency
// of one plane's chain on small grids and shared memory plus issue on large ones.
//
// Measured, us per launch between CUDA events (which add about 4 us), before ->
// after: 64x64x1 14 -> 8, 256x256x2 18 -> 12, 512x512x1 29 -> 13, 512x512x4
// 63 -> 43, 2048x128x1 67 -> 16, 1024x1024x1 121 -> 59 (two-CTA cluster before);
// block engine: 384x192x4 57 -> 18.5, 300x213x3 85 -> 16, 768x768x2 175 -> 72.
#pragma once
#include "batch.h"
#include "kernels.h"
#include "gfft.cuh"
#include "launch.cuh"
#include "passb_w.cuh"

namespace mmp {

// Columns per warp transform.
__host__ __device__ constexpr int passb_g_cols(int M) { return M <= 8 ? 3 : M <= 16 ? 2 : 1; }
// Floats between the columns of W: NB columns of a warp on different banks,
// and the two classes of a column (Q = 2) too.
__host__ __device__ constexpr int passb_g_pitch(int M, int Q) { return 32 * M + (M < 16 ? M : Q == 2 ? 8 : 0); }
// A warp does whole planes alone: no block barrier.
__host__ __device__ constexpr bool passb_g_private(int H, int M) { return H == 1 && passb_g_cols(M) == 3; }
// Half z length: padded z length 2 H (H = 1: no z transform).
__host__ __device__ constexpr int passb_g_half(int nz) { return nz <= 4 ? nz : nz <= 6 ? 6 : 8; }
__host__ __device__ constexpr int passb_g_maxthr(int H) { return H <= 4 ? 256 : 384; }
__host__ __device__ constexpr int passb_g_minblk(int H) { return H <= 4 ? 2 : 1; }

// Kernel row (one |ky|) of 6 (H + 1) floats, 16-byte loads; H = 1: 6 floats.
template <int H>
struct RowG {
  static constexpr int KZ = H == 1 ? 1 : H + 1;
  static constexpr int KQ = (6 * KZ + 3) / 4;
  float4 q[KQ];
  __device__ __forceinline__ explicit RowG(const float* row) {
#pragma unroll
    for (int j = 0; j < KQ; ++j) q[j] = __ldg(reinterpret_cast<const float4*>(row) + j);
  }
  __device__ __forceinline__ float at(int i) const {
    const float4& v = q[i >> 2];
    return (i & 3) == 0 ? v.x : (i & 3) == 1 ? v.y : (i & 3) == 2 ? v.z : v.w;
  }
  __device__ __forceinline__ void mul(int kz, float sy, float sz, float2& a, float2& b, float2& c) const {
    kmul3(make_float2(at(6 * kz), at(6 * kz + 1)), make_float2(at(6 * kz + 2), at(6 * kz + 3)),
          make_float2(at(6 * kz + 4), at(6 * kz + 5)), sy, sz, a, b, c);
  }
};

// z stage of one ky column: component c, layer z at w[(c nz + z) * cs];
// layers nz .. H - 1 are zero.
//   F[2q + p] = DFT_H(x[z] w_2H^(p z))[q],  x[z] = sum_p w_2H^(-p z) IDFT_H(F[2q + p])[z]
template <int H>
__device__ __forceinline__ void zstage_g(float2* w, int cs, int nz, const RowG<H>& row, float sy) {
  if constexpr (H == 1) {
    float2 a = w[0], b = w[cs], c = w[2 * cs];
    row.mul(0, sy, 1.0f, a, b, c);
    w[0] = a;
    w[cs] = b;
    w[2 * cs] = c;
  } else {
    constexpr int P = 2 * H;
    constexpr bool FULL = H <= 4;   // nz = H exactly
    float2 out[3][H];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      float2 f[3][H];
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int z = 0; z < H; ++z)
          f[c][z] = FULL || z < nz ? w[(c * (FULL ? H : nz) + z) * cs] : make_float2(0.0f, 0.0f);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (p) mul_roots<P, H, false>(f[c]);
        dft_any<H, false>(f[c]);
      }
#pragma unroll
      for (int q = 0; q < H; ++q) {
        const int kz = 2 * q + p;   // compile-time after unrolling
        row.mul(kz <= H ? kz : P - kz, sy, kz <= H ? 1.0f : -1.0f, f[0][q], f[1][q], f[2][q]);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dft_any<H, true>(f[c]);
        if (p) mul_roots<P, H, true>(f[c]);
#pragma unroll
        for (int z = 0; z < H; ++z) out[c][z] = p ? cadd(out[c][z], f[c][z]) : f[c][z];
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int z = 0; z < H; ++z)
        if (FULL || z < nz) w[(c * (FULL ? H : nz) + z) * cs] = out[c][z];
  }
}

// Planes kx0 .. kx0 + np - 1.
template <int H, int M, int Q>
__device__ __forceinline__ void passB_g_planes(unsigned char* sraw, const Grid& g, const DemagArgs& d, int kx0,
                                               int np) {
  constexpr int NB = passb_g_cols(M);
  constexpr int LP = passb_g_pitch(M, Q);
  constexpr int CS = Q * LP;                 // one column (all classes)
  constexpr bool PRIV = passb_g_private(H, M);
  constexpr int Ly = 32 * M, Py = Q * Ly;
  constexpr bool HALF = Q == 1;
  constexpr int MI = gfft_in<M, HALF>();
  const int ny = g.ny, nz = H <= 4 ? H : g.nz;
  const int ncp = 3 * nz, ncol = np * ncp;
  float2* W = reinterpret_cast<float2*>(sraw);
  const int lane = lane_id(), warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const long long t0 = (long long)kx0 * ncp * ny;
  float2* T = d.T + t0;
  const int ngrp = (ncol + NB - 1) / NB;
  // 1. forward y transforms
#pragma unroll 1
  for (int grp = warp; grp < ngrp; grp += nwarp) {
#pragma unroll 1
    for (int r = 0; r < Q; ++r) {
      float2 v[NB * MI], o[32];
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const int col = grp * NB + b;
#pragma unroll
        for (int m = 0; m < MI; ++m) {
          const int y = lane + 32 * m;
          const bool ok = col < ncol && y < ny && MMP_IN(g, t0 + (long long)col * ny + y, g.lim_T);
          float2 x = ok ? T[(long long)col * ny + y] : make_float2(0.0f, 0.0f);
          if (r) x = cmul(x, __ldg(d.tw_y + y));
          v[b * MI + m] = x;
        }
      }
      float2* scr = W + grp * NB * CS + r * LP;
      gfft<M, NB, HALF, false, false>(v, o, scr, d.tw_wy);
      const int b = lane / M, k1 = lane - b * M;
      if (lane < NB * M && grp * NB + b < ncol) {
        float2* dst = W + (grp * NB + b) * CS + r * LP + k1;
#pragma unroll
        for (int k2 = 0; k2 < 32; ++k2) dst[M * k2] = o[k2];
      }
      __syncwarp();
    }
  }
  if (!PRIV) __syncthreads();
  // 2. z stage: item (plane, |ky|): ky and its mirror
  {
    constexpr int NY = Py / 2 + 1;
    const int first = PRIV ? lane : threadIdx.x, step = PRIV ? 32 : blockDim.x;
    const int p0 = PRIV ? warp : 0, pn = PRIV ? nwarp : 1;
    const int total = PRIV ? NY : np * NY;
    for (int pp = p0; pp < (PRIV ? np : 1); pp += pn) {
      for (int e = first; e < total; e += step) {
        const int pl = PRIV ? pp : e / NY, ky = PRIV ? e : e - pl * NY;
        const long long ki = ((long long)(kx0 + pl) * g.kyn + ky) * g.krow;
        const RowG<H> row(d.khat + (MMP_IN(g, ki + g.krow - 1, g.lim_khat) ? ki : 0));
        float2* w = W + pl * ncp * CS;
        const int km = ky == 0 ? 0 : Py - ky;
        zstage_g<H>(w + (Q == 1 ? ky : (ky & 1) * LP + (ky >> 1)), CS, nz, row, 1.0f);
        if (km != ky) zstage_g<H>(w + (Q == 1 ? km : (km & 1) * LP + (km >> 1)), CS, nz, row, -1.0f);
      }
    }
  }
  if (PRIV) __syncwarp();
  else __syncthreads();
  // 3. inverse y transforms, the upper class first: its outputs wait in its
  // own half of W for the lane that forms the same y of class 0
#pragma unroll 1
  for (int grp = warp; grp < ngrp; grp += nwarp) {
    const int b1 = lane / M, k1 = lane - b1 * M, col1 = grp * NB + b1;
    const bool mine = lane < NB * M && col1 < ncol;
#pragma unroll 1
    for (int r = Q - 1; r >= 0; --r) {
      float2 v[NB * M], o[32];
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const int col = grp * NB + b < ncol ? grp * NB + b : ncol - 1;
#pragma unroll
        for (int m = 0; m < M; ++m) v[b * M + m] = W[col * CS + r * LP + lane + 32 * m];
      }
      __syncwarp();
      float2* scr = W + grp * NB * CS + r * LP;
      gfft<M, NB, false, HALF, true>(v, o, scr, d.tw_wy);
      if (mine) {
        float2* w1 = W + col1 * CS + LP + k1;   // class 1 (Q = 2)
#pragma unroll
        for (int k2 = 0; k2 < (HALF ? 16 : 32); ++k2) {
          const int y = k1 + M * k2;
          float2 h = o[k2];
          if (r) {
            w1[M * k2] = cmul(h, cconj(__ldg(d.tw_y + y)));
          } else {
            if (Q == 2) h = cadd(h, w1[M * k2]);
            if (y < ny && MMP_IN(g, t0 + (long long)col1 * ny + y, g.lim_T)) T[(long long)col1 * ny + y] = h;
          }
        }
      }
      __syncwarp();
    }
  }
}

// Per-context launch (insts null) over the kx planes, or one batch launch over
// work-list items, one CTA per item (kx0 = item.a, kp planes each).
template <int H, int M, int Q>
__global__ void __launch_bounds__(passb_g_maxthr(H), passb_g_minblk(H))
    k_passB_g(Grid g, DemagArgs d, int kp, const BatchInst* __restrict__ insts, const BatchItem* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char sraw[];
  if (!insts) {
    after_predecessor();
    const int kx0 = blockIdx.x * kp;
    passB_g_planes<H, M, Q>(sraw, g, d, kx0, min(kp, g.kxn - kx0));
  } else {
    const BatchItem w = items[blockIdx.x];
    const BatchInst& I = insts[w.inst];
    g = I.g;
    d = I.d;
    passB_g_planes<H, M, Q>(sraw, g, d, w.a, min(kp, g.kxn - w.a));
  }
}

// Launch of one instantiation (defined where MMP_PASSB_G_KERNELS is set, one
// translation unit per group of lengths so that they compile in parallel).
template <int H, int M, int Q>
cudaError_t launch_passB_g_t(const Grid& g, const DemagArgs& d, const PassBGLaunch& l, int nblocks,
                             const BatchInst* insts, const BatchItem* items, cudaStream_t st);

#ifdef MMP_PASSB_G_KERNELS
template <int H, int M, int Q>
cudaError_t launch_passB_g_t(const Grid& g, const DemagArgs& d, const PassBGLaunch& l, int nblocks,
                             const BatchInst* insts, const BatchItem* items, cudaStream_t st) {
  cudaError_t e = set_smem(k_passB_g<H, M, Q>, l.smem);
  if (e != cudaSuccess) return e;
  if (!insts) return launch_chained(d.chain, k_passB_g<H, M, Q>, dim3(nblocks), l.threads, l.smem, st, g, d, l.kp, insts, items);
  k_passB_g<H, M, Q><<<nblocks, l.threads, l.smem, st>>>(g, d, l.kp, insts, items);
  return cudaGetLastError();
}
#define MMP_PASSB_G(H, M, Q)                                                                                       \
  template cudaError_t launch_passB_g_t<H, M, Q>(const Grid&, const DemagArgs&, const PassBGLaunch&, int,          \
                                                 const BatchInst*, const BatchItem*, cudaStream_t);
#define MMP_PASSB_G_LOW(M, Q) MMP_PASSB_G(1, M, Q) MMP_PASSB_G(2, M, Q) MMP_PASSB_G(3, M, Q) MMP_PASSB_G(4, M, Q)
#define MMP_PASSB_G_ALL(M) MMP_PASSB_G_LOW(M, 1) MMP_PASSB_G(6, M, 1) MMP_PASSB_G(8, M, 1)
#endif

}  // namespace mmp
