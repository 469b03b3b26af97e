// xfft_g.cuh -- the general passes A and C of the demag convolution on the
// warp transforms of gfft.cuh: padded x lengths Px = Q * 32 M of 64 .. 4096
// (Q = 1, 2 or 4 classes of kx, k = Q k' + r).  A CTA takes one row pair (rows
// y0, y0 + 1 of plane z), packed as one complex row z[x] = M_a[x] + i M_b[x]:
//   pass A: stage assembly of both rows, M = sum_s Ms m_s into shared memory,
//     forward transforms, the two rows' half spectra to T[kx][c][z][y];
//   pass C: both rows' half spectra gathered by asynchronous copies, inverse
//     transforms, then the local field and torque of every cell (four cells an
//     item, stencil4.cuh, or one cell, field.cuh).
// With Q = 1 a transform holds only the nonzero half of its input (pass A) and
// forms only the needed half of its output (pass C).  With Q > 1, N = Px / Q:
//   Z[Q k' + r] = DFT_N( sum_j (-i)^(r j) z[x + j N] w_Px^(r x) )[k'],  j < Q / 2
//   z[x + j N] = sum_r i^(r j) w_Px^(-r x) IDFT_N(Z[Q k' + r])[x],
// (-i)^(r j) exact.
//
// What bounds it and why this layout: the block Stockham passes this replaces
// need a block barrier around every radix pass and run-time index arithmetic;
// at these sizes they waited on barriers and on the chain load -> transform ->
// store with few blocks in flight.  Here three warps (one for M <= 8, all three
// components in its lanes) do a row pair's transforms with warp barriers only,
// and the smallest tile, one row pair, gives the most blocks.
// Cold L2, us per launch now, A and C: 64x64x1 6.6 and 7.7, 512x512x1 11 and 16.5,
// 2048x128x1 31 and 10 + 10 (two kernels; 47 as one), 1024x256x1 of two sublattices
// 23 and 8 + 21 (A 45 and C 100 on the kernels of xfft_w.cuh).  Before, whole passes:
// 512x512x1 run 1577 -> 726 us, 2048x128x1 run 4094 -> 1865, with what follows 630 and
// 1337.
#pragma once
#include "batch.h"
#include "copy.cuh"
#include "field.cuh"
#include "gfft.cuh"
#include "kernels.h"
#include "launch.cuh"
#include "stencil4.cuh"

namespace mmp {

template <int M, int Q>
struct Xg {
  static constexpr int NB = M <= 8 ? 3 : 1;        // transforms per warp (components)
  static constexpr int N = 32 * M, Px = Q * N, HX = Px / 2;
  static constexpr int GRP = NB == 3 ? 1 : 3 * Q;  // warps that transform
  static constexpr int LP = (xg_pitch(M, Q));      // complex values of one transform's region
  static constexpr int W = 3 * Q * LP;             // complex values of all regions
};

template <int V>
struct VecF { float v[V]; };
// V floats at p, or zeros where !ok, without a branch: the loads of one item
// are issued back to back.
template <int V>
__device__ __forceinline__ VecF<V> ld_if(const float* p, bool ok) {
  VecF<V> r;
  if constexpr (V == 2) {
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %3, 0; mov.f32 %0, 0f00000000; mov.f32 %1, 0f00000000; @q ld.global.v2.f32 {%0, %1}, [%2]; }"
                 : "=f"(r.v[0]), "=f"(r.v[1]) : "l"(p), "r"((unsigned)ok) : "memory");
  } else {
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %2, 0; mov.f32 %0, 0f00000000; @q ld.global.f32 %0, [%1]; }"
                 : "=f"(r.v[0]) : "l"(p), "r"((unsigned)ok) : "memory");
  }
  return r;
}

// Stage value of part p at V cells of both rows, three components: v[c][h].
// All vectors of a group (y and k_1 .. k_3, then the rest) are in flight at once.
template <int V>
__device__ __forceinline__ void xg_stage(const Grid& g, const StageArgs& a, bool assemble, long long idx0, bool two,
                                         VecF<V> (&v)[3][2]) {
  const long long n = g.n;
  const int nx = g.nx;
  const float* src = assemble ? a.y : a.stage;
  const int nk = assemble ? a.nk : 0;
  bool ok[3][2];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      ok[c][h] = (h == 0 || two) && MMP_IN(g, idx0 + c * n + h * nx + V - 1, g.lim_state);
  VecF<V> w[3][3][2];
  auto load = [&](int j0, int j) {
    const bool have = j0 + j < nk;
    const float* k = have ? a.k[j0 + j] : src;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int h = 0; h < 2; ++h) w[j][c][h] = ld_if<V>(k + idx0 + c * n + h * nx, have && ok[c][h]);
  };
  auto add = [&](int j0, int j) {
    if (j0 + j < nk) {
      const float cj = a.coef[j0 + j];
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int i = 0; i < V; ++i) v[c][h].v[i] = fmaf(cj, w[j][c][h].v[i], v[c][h].v[i]);
    }
  };
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int h = 0; h < 2; ++h) v[c][h] = ld_if<V>(src + idx0 + c * n + h * nx, ok[c][h]);
#pragma unroll
  for (int j = 0; j < 3; ++j) load(0, j);
#pragma unroll
  for (int j = 0; j < 3; ++j) add(0, j);
  if (nk > 3) {
#pragma unroll
    for (int j = 0; j < 3; ++j) load(3, j);
#pragma unroll
    for (int j = 0; j < 3; ++j) add(3, j);
  }
  if (nk > 6) {   // no method here has more than six previous stages
    load(6, 0);
    add(6, 0);
  }
}

template <int V>
__device__ __forceinline__ void xg_store(const Grid& g, float* p, long long idx, const VecF<V>& v) {
  if (!MMP_IN(g, idx + V - 1, g.lim_state)) return;
  if constexpr (V == 2) *reinterpret_cast<float2*>(p + idx) = make_float2(v.v[0], v.v[1]);
  else p[idx] = v.v[0];
}

// Assembly of both rows of the parts p0 .. p1 - 1: items of V cells in each row;
// M of the sublattices into Z[c][x] = (row a, row b).
template <int V>
__device__ __forceinline__ void xg_assemble(const Grid& g, const StageArgs& a, const Coefs& co, float2* Z, int hx,
                                            int p0, int p1, int z, int y0) {
  const int nx = g.nx;
  const long long n = g.n, row0 = (long long)nx * (y0 + (long long)g.ny * z);
  const bool two = y0 + 1 < g.ny, assemble = a.y != nullptr, uni = co.uniform != 0;
  const int nsub = a.nsub;
  for (int x0 = V * threadIdx.x; x0 < nx; x0 += V * blockDim.x) {
    for (int p = p0; p < p1; ++p) {
      const long long idx0 = 3LL * p * n + row0 + x0;
      VecF<V> v[3][2];
      xg_stage<V>(g, a, assemble, idx0, two, v);
      if (assemble && a.normalize && p < nsub) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int i = 0; i < V; ++i) {
            const float m0 = v[0][h].v[i], m1 = v[1][h].v[i], m2 = v[2][h].v[i];
            const float nn = m0 * m0 + m1 * m1 + m2 * m2;
            const float r = nn > 0.0f ? rnorm3df(m0, m1, m2) : 1.0f;
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c][h].v[i] *= r;
          }
      }
      if (assemble) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          xg_store<V>(g, a.stage, idx0 + c * n, v[c][0]);
          if (two) xg_store<V>(g, a.stage, idx0 + c * n + nx, v[c][1]);
        }
      }
      if (p >= nsub) continue;   // elastic parts: assembled, not transformed
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const long long cell = row0 + x0 + i;
        float ms[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int reg = uni || (h && !two) || !MMP_IN(g, cell + h * nx, n) ? 0 : co.regions[cell + h * nx];
          ms[h] = co.reg[p * MMP_MAX_REGIONS + reg].ms;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float2 acc = p ? Z[c * hx + x0 + i] : make_float2(0.0f, 0.0f);
          acc.x = fmaf(ms[0], v[c][0].v[i], acc.x);
          acc.y = fmaf(ms[1], v[c][1].v[i], acc.y);
          Z[c * hx + x0 + i] = acc;
        }
      }
    }
  }
}

// part 0: the sublattices and the transforms; part q > 0: elastic part q - 1,
// assembled and not transformed, in a block of its own.
template <int M, int Q>
__device__ __forceinline__ void passA_g_tile(unsigned char* sraw, const XgArgs& s, int part, int z, int y0) {
  using X = Xg<M, Q>;
  constexpr int NB = X::NB, N = X::N, LP = X::LP, HX = X::HX;
  constexpr bool HALF = Q == 1;
  constexpr int MI = gfft_in<M, HALF>();
  const Grid& g = s.g;
  const int nx = g.nx, ny = g.ny;
  float2* Z = reinterpret_cast<float2*>(sraw);   // [3][HX] input rows
  float2* W = Z + 3 * HX;                        // [3][Q][LP] transforms
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  const unsigned long long al = reinterpret_cast<unsigned long long>(s.a.stage) |
                                reinterpret_cast<unsigned long long>(s.a.y);
  unsigned long long alk = 0;
#pragma unroll
  for (int j = 0; j < 7; ++j) alk |= j < s.a.nk ? reinterpret_cast<unsigned long long>(s.a.k[j]) : 0ull;
  const int p0 = part ? s.a.nsub + part - 1 : 0, p1 = part ? p0 + 1 : s.a.nsub;
  if (!(nx & 1) && !((al | alk) & 7)) xg_assemble<2>(g, s.a, s.co, Z, HX, p0, p1, z, y0);
  else xg_assemble<1>(g, s.a, s.co, Z, HX, p0, p1, z, y0);
  if (part) return;
  __syncthreads();
  if (warp < X::GRP) {
    const int c0 = NB == 3 ? 0 : warp / Q, r = NB == 3 ? 0 : warp - c0 * Q;
    float2 v[NB * MI], o[32];
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int m = 0; m < MI; ++m) {
        const int x = lane + 32 * m;
        const float2* Zc = Z + (c0 + b) * HX;
        float2 q = x < nx && x < HX ? Zc[x] : make_float2(0.0f, 0.0f);
        if constexpr (Q == 4) {
          const float2 u = x + N < nx ? Zc[x + N] : make_float2(0.0f, 0.0f);
          const float2 t = (r & 1) ? make_float2(u.y, -u.x) : u;   // (-i)^r up to the sign
          q = r < 2 ? cadd(q, t) : csub(q, t);
        }
        if (Q > 1 && r) q = cmul(q, __ldg(s.d.tw_wx2 + r * x));
        v[b * MI + m] = q;
      }
    float2* scr = W + (c0 * Q + r) * LP;
    gfft<M, NB, HALF, false, false>(v, o, scr, s.d.tw_wx);
    const int b = lane / M, k1 = lane - b * M;
    if (lane < NB * M) {
      float2* dst = scr + b * LP + k1;
#pragma unroll
      for (int k2 = 0; k2 < 32; ++k2) dst[M * k2] = o[k2];
    }
  }
  __syncthreads();
  // the two rows' half spectra
  const bool two = y0 + 1 < ny;
  float2* T = s.d.T;
  const bool wide = two && !(ny & 1) && !(reinterpret_cast<unsigned long long>(T) & 15);
  const long long kst = (long long)3 * g.nz * ny, cst = (long long)g.nz * ny, t0 = (long long)z * ny + y0;
  for (int e = threadIdx.x; e < 3 * (HX + 1); e += blockDim.x) {
    const int c = e / (HX + 1), k = e - c * (HX + 1), km = k == 0 ? 0 : X::Px - k;
    const float2* Wc = W + c * Q * LP;
    const float2 Zk = Wc[(k % Q) * LP + k / Q], Zm = Wc[(km % Q) * LP + km / Q];
    const float2 A = make_float2(0.5f * (Zk.x + Zm.x), 0.5f * (Zk.y - Zm.y));
    const float2 B = make_float2(0.5f * (Zk.y + Zm.y), -0.5f * (Zk.x - Zm.x));
    const long long ti = t0 + k * kst + c * cst;
    if (!MMP_IN(g, ti + (two ? 1 : 0), g.lim_T)) continue;
    if (wide) {
      *reinterpret_cast<float4*>(T + ti) = make_float4(A.x, A.y, B.x, B.y);
    } else {
      T[ti] = A;
      if (two) T[ti + 1] = B;
    }
  }
}

// KIND 0: one sublattice, uniform material; 1: one sublattice, regions; 2: two
// sublattices, uniform; 3: two sublattices, regions.  V: cells per item (KIND 0).
template <int M, int Q, int KIND, int V>
__device__ __forceinline__ void passC_g_tile(unsigned char* sraw, const XgArgs& s, int z, int y0) {
  using X = Xg<M, Q>;
  constexpr int NB = X::NB, N = X::N, LP = X::LP, HX = X::HX;
  constexpr bool HALF = Q == 1;
  const Grid& g = s.g;
  const int nx = g.nx, ny = g.ny;
  float4* G = reinterpret_cast<float4*>(sraw);   // [3][HX + 1]: (X_a, X_b); then the transforms' regions
  float2* W = reinterpret_cast<float2*>(sraw);   // [3][Q][LP]
  float* bd = reinterpret_cast<float*>(sraw + (Q == 1 ? 0 : xg_gather_bytes(M, Q)));   // [3][2][HX]
  float* ms = reinterpret_cast<float*>(sraw + xg_gather_bytes(M, Q)) + (Q == 1 ? 0 : 6 * HX);
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  const bool two = y0 + 1 < ny;
  const long long kst = (long long)3 * g.nz * ny, cst = (long long)g.nz * ny, t0 = (long long)z * ny + y0;
  const float2* T = s.d.T;
  // 1. gather T[k][c][z][y0 .. y0 + 1], k <= HX; the tile rows of m
  if (two && !(ny & 1) && !(reinterpret_cast<unsigned long long>(T) & 15)) {
    for (int e = threadIdx.x; e < 3 * (HX + 1); e += blockDim.x) {
      const int c = e / (HX + 1), k = e - c * (HX + 1);
      const long long ti = t0 + k * kst + c * cst;
      if (MMP_IN(g, ti + 1, g.lim_T)) cp_async16(G + e, T + ti);
    }
  } else {
    for (int e = threadIdx.x; e < 3 * (HX + 1); e += blockDim.x) {
      const int c = e / (HX + 1), k = e - c * (HX + 1);
      const long long ti = t0 + k * kst + c * cst;
      if (!MMP_IN(g, ti + (two ? 1 : 0), g.lim_T)) continue;
      cp_async8(reinterpret_cast<float2*>(G + e), T + ti);
      if (two) cp_async8(reinterpret_cast<float2*>(G + e) + 1, T + ti + 1);
      else reinterpret_cast<float2*>(G + e)[1] = make_float2(0.0f, 0.0f);
    }
  }
  cp_async_commit();
  bool vec = false;
  if constexpr (KIND == 0) {
    const unsigned long long al = reinterpret_cast<unsigned long long>(s.f.stage) |
                                  reinterpret_cast<unsigned long long>(s.f.kout) |
                                  reinterpret_cast<unsigned long long>(s.f.Bout) |
                                  reinterpret_cast<unsigned long long>(s.f.eps);
    vec = !(nx & 3) && !(al & 15);
    if (vec) {
      const int q = nx >> 2, nrows = two ? 2 : 1;
      const long long row0 = (long long)nx * (y0 + (long long)ny * z);
      for (int e = threadIdx.x; e < 3 * nrows * q; e += blockDim.x) {
        const int ch = e / q, j = e - ch * q, c = ch / nrows, h = ch - c * nrows;
        const long long si = c * g.n + row0 + (long long)h * nx + 4 * j;
        if (MMP_IN(g, si + 3, g.lim_state)) cp_async16(ms + (2 * c + h) * HX + 4 * j, s.f.stage + si);
      }
    }
  }
  cp_async_commit();
  cp_async_wait_one();
  __syncthreads();
  // 2. inverse transforms: Z[k] = X_a[k] + i X_b[k] (k <= HX), conj X_a[Px - k] + i conj X_b[Px - k] above
  float2 o[32];
  const int c0 = NB == 3 ? 0 : warp / Q, r = NB == 3 ? 0 : warp - c0 * Q;
  float2* scr = W + (c0 * Q + r) * LP;
  const int b1 = lane / M, k1 = lane - b1 * M;
  {
    float2 v[NB * M];
    if (warp < X::GRP) {
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int m = 0; m < M; ++m) {
          const int k = Q * (lane + 32 * m) + r;
          const bool lo = k <= HX;
          const float4 q = G[(c0 + b) * (HX + 1) + (lo ? k : X::Px - k)];
          v[b * M + m] = lo ? make_float2(q.x - q.w, q.y + q.z) : make_float2(q.x + q.w, q.z - q.y);
        }
    }
    __syncthreads();   // every warp holds its input: G becomes the transforms' regions
    if (warp < X::GRP) {
      gfft<M, NB, false, HALF, true>(v, o, scr, s.d.tw_wx);
      if (Q > 1 && lane < M) {
#pragma unroll
        for (int k2 = 0; k2 < 32; ++k2) {
          const int x = k1 + M * k2;
          scr[x] = r ? cmul(o[k2], cconj(__ldg(s.d.tw_wx2 + r * x))) : o[k2];
        }
      }
    }
  }
  cp_async_wait_all();
  if (NB == 1) __syncthreads();
  if constexpr (Q == 1) {
    if (warp < X::GRP && lane < NB * M) {
      float* dst = bd + (c0 + b1) * 2 * HX + k1;
#pragma unroll
      for (int k2 = 0; k2 < 16; ++k2) {
        dst[M * k2] = o[k2].x;
        dst[HX + M * k2] = o[k2].y;
      }
    }
  } else {
    for (int e = threadIdx.x; e < 3 * N; e += blockDim.x) {
      const int c = e / N, x = e - c * N;
      const float2* t = W + c * Q * LP + x;
      float* dst = bd + c * 2 * HX + x;
      if constexpr (Q == 2) {
        const float2 u = cadd(t[0], t[LP]);
        dst[0] = u.x;
        dst[HX] = u.y;
      } else {
        const float2 p = cadd(t[0], t[2 * LP]), q = cadd(t[LP], t[3 * LP]);
        const float2 pm = csub(t[0], t[2 * LP]), qm = csub(t[LP], t[3 * LP]);
        dst[0] = p.x + q.x;
        dst[HX] = p.y + q.y;
        dst[N] = pm.x - qm.y;        // + i (t1 - t3)
        dst[HX + N] = pm.y + qm.x;
      }
    }
  }
  __syncthreads();
  // 3. local field and torque
  constexpr int NSUB = KIND >= 2 ? 2 : 1;
  constexpr bool UNI = KIND == 0 || KIND == 2;
  if (KIND == 0 && vec) field_cells4<true, V>(ms, bd, 2 * HX, HX, two ? 2 : 1, g, s.co, s.f, z, y0);
  else field_cells<NSUB, true, UNI>(bd, 2 * HX, HX, two ? 2 : 1, g, s.co, s.f, z, y0);
}

// Word copy into shared memory (16-byte-free: the structs are multiples of 4).
template <typename S>
__device__ __forceinline__ void xg_copy(S& dst, const S& src) {
  const int* p = reinterpret_cast<const int*>(&src);
  int* q = reinterpret_cast<int*>(&dst);
  for (int i = threadIdx.x; i < (int)(sizeof(S) / sizeof(int)); i += blockDim.x) q[i] = p[i];
}

// The tile of this block: of the launch's grid (insts null; p holds the
// arguments) or of a batch work list.
__device__ __forceinline__ BatchItem xg_tile(XgArgs& s, const XgArgs& p, const BatchInst* insts,
                                             const BatchItem* items, int stage) {
  if (!insts) {
    xg_copy(s, p);
    after_predecessor();
    __syncthreads();
    if (p.a.cdev) {   // a captured attempt: this step's coefficients
      if (threadIdx.x < 7) s.a.coef[threadIdx.x] = __ldg(p.a.cdev + threadIdx.x);
      __syncthreads();
    }
    return BatchItem{0, (int)blockIdx.x, (int)blockIdx.y};
  }
  const BatchItem w = items[blockIdx.x];
  const BatchInst& I = insts[w.inst];
  xg_copy(s.g, I.g);
  xg_copy(s.d, I.d);
  xg_copy(s.co, I.co);
  // as batch_args, one entry a lane: by one thread this chain of loads from the
  // descriptor lasted longer than a small tile's transforms
  if (threadIdx.x < 32) {
    const int j = threadIdx.x, p = I.par;
    float* const k1 = I.kbuf[p];
    float* const k7 = I.kbuf[p ^ 1];
    float* kj = j == 0 ? k1 : j < 6 ? I.kmid[j - 1] : k7;
    const bool last = stage == 6;
    if (j < 7) {
      s.a.k[j] = j < stage ? kj : nullptr;
      s.a.coef[j] = j < stage ? I.coef[stage][j] : 0.0f;
      s.f.ecoef[j] = last ? I.ecoef[j] : 0.0f;
      if (j < 6) s.f.ek[j] = last ? kj : nullptr;
      if (j == stage) s.f.kout = kj;
    } else if (j == 7) {
      float* st = I.ybuf[stage == 0 ? p : p ^ 1];
      s.a.y = stage == 0 ? nullptr : I.ybuf[p];
      s.a.stage = st;
      s.f.stage = st;
    } else if (j == 8) {
      s.a.nk = stage;
      s.a.cdev = nullptr;
      s.f.cdev = nullptr;
      s.a.normalize = last;
      s.a.nparts = 1;
      s.a.nsub = 1;
      s.f.Bout = nullptr;
      s.f.eps = nullptr;
      s.f.terms = I.terms;
      s.f.relax = I.relax;
      s.f.err = last ? I.red : nullptr;
      s.f.torque_max = last ? I.red + 1 : nullptr;
    }
  }
  __syncthreads();
  return w;
}

template <int M, int Q>
__global__ void __launch_bounds__(xg_maxthr(Q), xg_minblk(Q))
    k_passA_g(const __grid_constant__ XgArgs p, const BatchInst* __restrict__ insts,
              const BatchItem* __restrict__ items, int stage) {
  extern __shared__ __align__(16) unsigned char sraw[];
  __shared__ __align__(16) XgArgs s;
  const BatchItem w = xg_tile(s, p, insts, items, stage);
  passA_g_tile<M, Q>(sraw, s, blockIdx.z, w.b, 2 * w.a);
}

// The inverse x transforms of one component (blockIdx.z) of a row pair; the
// demag field waits where the cell's stage derivative will be written.
template <int M, int Q>
__global__ void __launch_bounds__(xg_maxthr(Q), xg_minblk(Q)) k_invx_g(const __grid_constant__ XgArgs p) {
  using X = Xg<M, Q>;
  constexpr int N = X::N, LP = X::LP, HX = X::HX;
  constexpr bool HALF = Q == 1;
  static_assert(X::NB == 1, "one component per warp");
  extern __shared__ __align__(16) unsigned char sraw[];
  float4* G = reinterpret_cast<float4*>(sraw);   // [HX + 1]: (X_a, X_b); then the transforms' regions
  float2* W = reinterpret_cast<float2*>(sraw);   // [Q][LP]
  const Grid& g = p.g;
  const int nx = g.nx, ny = g.ny, y0 = 2 * blockIdx.x, z = blockIdx.y, c = blockIdx.z;
  const int lane = lane_id(), r = threadIdx.x >> 5;
  const bool two = y0 + 1 < ny;
  const long long kst = (long long)3 * g.nz * ny, t0 = ((long long)c * g.nz + z) * ny + y0;
  const float2* T = p.d.T;
  after_predecessor();
  if (two && !(ny & 1) && !(reinterpret_cast<unsigned long long>(T) & 15)) {
    for (int k = threadIdx.x; k <= HX; k += blockDim.x)
      if (MMP_IN(g, t0 + k * kst + 1, g.lim_T)) cp_async16(G + k, T + t0 + k * kst);
  } else {
    for (int k = threadIdx.x; k <= HX; k += blockDim.x) {
      if (!MMP_IN(g, t0 + k * kst + (two ? 1 : 0), g.lim_T)) continue;
      cp_async8(reinterpret_cast<float2*>(G + k), T + t0 + k * kst);
      if (two) cp_async8(reinterpret_cast<float2*>(G + k) + 1, T + t0 + k * kst + 1);
      else reinterpret_cast<float2*>(G + k)[1] = make_float2(0.0f, 0.0f);
    }
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();
  float2 v[M], o[32];
  if (r < Q) {
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const int k = Q * (lane + 32 * m) + r;
      const bool lo = k <= HX;
      const float4 q = G[lo ? k : X::Px - k];
      v[m] = lo ? make_float2(q.x - q.w, q.y + q.z) : make_float2(q.x + q.w, q.z - q.y);
    }
  }
  __syncthreads();
  float* out = p.f.kout + c * g.n + (long long)nx * (y0 + (long long)ny * z);
  if (r < Q) {
    float2* scr = W + r * LP;
    gfft<M, 1, false, HALF, true>(v, o, scr, p.d.tw_wx);
    if (lane < M) {
#pragma unroll
      for (int k2 = 0; k2 < (HALF ? 16 : 32); ++k2) {
        const int x = lane + M * k2;
        if (Q > 1) {
          scr[x] = r ? cmul(o[k2], cconj(__ldg(p.d.tw_wx2 + r * x))) : o[k2];
        } else if (x < nx && MMP_IN(g, (out - p.f.kout) + x, g.lim_state)) {
          out[x] = o[k2].x;
          if (two) out[nx + x] = o[k2].y;
        }
      }
    }
  }
  if constexpr (Q > 1) {
    __syncthreads();
    auto put = [&](int x, float2 u) {
      if (x >= nx || !MMP_IN(g, (out - p.f.kout) + x, g.lim_state)) return;
      out[x] = u.x;
      if (two) out[nx + x] = u.y;
    };
    for (int x = threadIdx.x; x < N; x += blockDim.x) {
      const float2* t = W + x;
      if constexpr (Q == 2) {
        put(x, cadd(t[0], t[LP]));
      } else {
        const float2 e = cadd(t[0], t[2 * LP]), q = cadd(t[LP], t[3 * LP]);
        const float2 em = csub(t[0], t[2 * LP]), qm = csub(t[LP], t[3 * LP]);
        put(x, make_float2(e.x + q.x, e.y + q.y));
        put(x + N, make_float2(em.x - qm.y, em.y + qm.x));   // + i (t1 - t3)
      }
    }
  }
}

template <int M, int Q, int KIND, int V>
__global__ void __launch_bounds__(xg_maxthr(Q), xg_minblk(Q))
    k_passC_g(const __grid_constant__ XgArgs p, const BatchInst* __restrict__ insts,
              const BatchItem* __restrict__ items, int stage) {
  extern __shared__ __align__(16) unsigned char sraw[];
  __shared__ __align__(16) XgArgs s;
  const BatchItem w = xg_tile(s, p, insts, items, stage);
  passC_g_tile<M, Q, KIND, V>(sraw, s, w.b, 2 * w.a);
}

struct XgLaunch {
  dim3 grid;
  int threads;
  size_t smem;
  int v;       // cells per item of pass C's local field
};

template <int M, int Q>
cudaError_t launch_xg_t(int pass, int kind, const XgArgs& p, const XgLaunch& l, const BatchInst* insts,
                        const BatchItem* items, int stage, cudaStream_t st);

#ifdef MMP_XFFT_G_KERNELS
template <typename K>
static cudaError_t xg_go(K kernel, const XgArgs& p, const XgLaunch& l, const BatchInst* insts, const BatchItem* items,
                         int stage, cudaStream_t st) {
  cudaError_t e = set_smem(kernel, l.smem, sizeof(XgArgs) + sizeof(RegionCoef) + 256);
  if (e != cudaSuccess) return e;
  if (!insts) return launch_chained(p.d.chain, kernel, l.grid, l.threads, l.smem, st, p, insts, items, stage);
  kernel<<<l.grid, l.threads, l.smem, st>>>(p, insts, items, stage);
  return cudaGetLastError();
}
template <int M, int Q>
cudaError_t launch_xg_t(int pass, int kind, const XgArgs& p, const XgLaunch& l, const BatchInst* insts,
                        const BatchItem* items, int stage, cudaStream_t st) {
  if (pass == 0) return xg_go(k_passA_g<M, Q>, p, l, insts, items, stage, st);
  if constexpr (M > 8) {
    if (pass == 1) {
      const cudaError_t e = set_smem(k_invx_g<M, Q>, l.smem);
      return e != cudaSuccess ? e : launch_chained(p.d.chain, k_invx_g<M, Q>, l.grid, l.threads, l.smem, st, p);
    }
  }
  if (kind == 0 && M <= 16 && l.v != 4) return xg_go(k_passC_g<M, Q, 0, M <= 8 ? 1 : M <= 16 ? 2 : 4>, p, l, insts, items, stage, st);
  if (kind == 0) return xg_go(k_passC_g<M, Q, 0, 4>, p, l, insts, items, stage, st);
  if constexpr (M <= 8) {   // above, several regions or sublattices take k_invx_g and k_cells_g (xg_split)
    if (kind == 1) return xg_go(k_passC_g<M, Q, 1, 4>, p, l, insts, items, stage, st);
    if (kind == 2) return xg_go(k_passC_g<M, Q, 2, 4>, p, l, insts, items, stage, st);
    return xg_go(k_passC_g<M, Q, 3, 4>, p, l, insts, items, stage, st);
  }
  return cudaErrorInvalidValue;
}
#define MMP_XG(M, Q)                                                                                              \
  template cudaError_t launch_xg_t<M, Q>(int, int, const XgArgs&, const XgLaunch&, const BatchInst*,              \
                                         const BatchItem*, int, cudaStream_t);
#endif

}  // namespace mmp
