// gfft.cuh -- warp-level FFTs of every length N = 32 M of the zero-padded
// axes (M in {1, 2, 3, 4, 6, 8, 12, 16, 24, 32}: N = 32 .. 1024 with at most
// one factor 3), the transform engine of the general passes (passb_g.cuh,
// xfft_g.cuh).
//
// The factorisation is that of wfft.cuh (n = l + 32 m, k = k1 + M k2: a DFT of
// length M in the registers of lane l, one twiddle per value, one transpose
// through the warp's own shared memory, a DFT32 in the registers of lane
// (b, k1)), generalised in three ways:
//   - lengths 3 * 2^k: the DFT of length 3 Q (Q = 1, 2, 4, 8) by the prime
//     factor map n = Q n1 + 3 n2, k = k1 (mod 3), k2 (mod Q): a DFT3 and a
//     DFTQ without twiddles between them, every index a compile-time constant;
//   - NB transforms per warp with NB M <= 32: few transforms (small grids) take
//     few registers each and more warps, instead of always 32 values a lane;
//   - zero padding: a transform of length N whose inputs beyond N / 2 are zero
//     (HIN) takes only its first M / 2 registers, split exactly into the even
//     and odd outputs of its DFT_M (two DFT_(M/2)); a transform of which only
//     the outputs below N / 2 are used (HOUT) leaves out the last butterfly's
//     second half.  So a padded axis of length N costs one transform of
//     half-filled registers, without separate even and odd twiddle passes.
#pragma once
#include "wfft.cuh"

namespace mmp {

// cos(2 pi k / 96), k = 0 .. 24 (a quarter wave); other k by symmetry.
__host__ __device__ constexpr float kCos96q(int k) {
  constexpr float t[25] = {
      1.0f,
      0.99785892323860347908f,
      0.99144486137381038215f,
      0.98078528040323044913f,
      0.96592582628906828675f,
      0.94693012949510566414f,
      0.92387953251128675613f,
      0.89687274153268830392f,
      0.86602540378443864676f,
      0.83146961230254523708f,
      0.79335334029123516458f,
      0.75183980747897739641f,
      0.70710678118654752440f,
      0.65934581510006886430f,
      0.60876142900872066437f,
      0.55557023301960222474f,
      0.5f,
      0.44228869021900126280f,
      0.38268343236508977173f,
      0.32143946530316154250f,
      0.25881904510252076235f,
      0.19509032201612826785f,
      0.13052619222005159155f,
      0.06540312923014306819f,
      0.0f};
  return t[k];
}
__host__ __device__ constexpr float cos96(int k) {
  k = ((k % 96) + 96) % 96;
  return k <= 24 ? kCos96q(k) : k <= 48 ? -kCos96q(48 - k) : k <= 72 ? -kCos96q(k - 48) : kCos96q(96 - k);
}
__host__ __device__ constexpr float sin96(int k) { return cos96(k - 24); }

// a * w_N^K (forward, exp(-2 pi i K / N)) or its conjugate (inverse); N | 96.
template <int N, int K, bool INV>
__device__ __forceinline__ float2 mul_root(float2 a) {
  static_assert(96 % N == 0, "roots of unity of orders dividing 96");
  constexpr int k = (96 / N * K) % 96;
  if constexpr (k == 0) return a;
  else if constexpr (k == 24) return mul_mi<INV>(a);
  else if constexpr (k == 48) return make_float2(-a.x, -a.y);
  else if constexpr (k == 72) return mul_mi<!INV>(a);
  else {
    constexpr float c = cos96(k), s = sin96(k);
    return INV ? make_float2(fmaf(c, a.x, -s * a.y), fmaf(c, a.y, s * a.x))
               : make_float2(fmaf(c, a.x, s * a.y), fmaf(c, a.y, -s * a.x));
  }
}

template <int M, bool INV>
__device__ __forceinline__ void dft_any(float2 (&t)[M]);

// DFT of length 3 Q (Q = 2, 4, 8) by the prime factor map.
template <int Q, bool INV>
__device__ __forceinline__ void dft_3q(float2 (&t)[3 * Q]) {
  constexpr int N = 3 * Q;
  float2 u[3][Q];
#pragma unroll
  for (int n1 = 0; n1 < 3; ++n1) {
#pragma unroll
    for (int n2 = 0; n2 < Q; ++n2) u[n1][n2] = t[(Q * n1 + 3 * n2) % N];
    dft_m<Q, INV>(u[n1]);
  }
#pragma unroll
  for (int k2 = 0; k2 < Q; ++k2) {
    // n = Q n1 + 3 n2 gives w_N^(n k) = w_3^(n1 k) w_Q^(n2 k)
    dft3<INV>(u[0][k2], u[1][k2], u[2][k2]);
  }
#pragma unroll
  for (int k = 0; k < N; ++k) t[k] = u[k % 3][k % Q];
}

// In-register DFT of length M in {1, 2, 3, 4, 6, 8, 12, 16, 24, 32}.
template <int M, bool INV>
__device__ __forceinline__ void dft_any(float2 (&t)[M]) {
  if constexpr (M == 3) dft3<INV>(t[0], t[1], t[2]);
  else if constexpr (M % 3 == 0) dft_3q<M / 3, INV>(t);
  else dft_m<M, INV>(t);
}

// t[m] *= w_N^m for m = 1 .. M - 1 (compile-time factors)
template <int N, int M, bool INV, int m = 1>
__device__ __forceinline__ void mul_roots(float2 (&t)[M]) {
  if constexpr (m < M) {
    t[m] = mul_root<N, m, INV>(t[m]);
    mul_roots<N, M, INV, m + 1>(t);
  }
}

// Registers of one transform's input: with HIN the inputs l + 32 m of m >= M / 2
// are zero and not held (odd M: none are left out, M = 3 keeps two of three).
template <int M, bool HIN>
__host__ __device__ constexpr int gfft_in() {
  return !HIN ? M : M == 1 ? 1 : (M + 1) / 2;
}

// The transpose scratch of NB transforms: NB M rows of 32 complex values.
template <int M, int NB>
__host__ __device__ constexpr int gfft_scratch() { return NB * M * 32; }

// Forward DFT of NB transforms of length N = 32 M up to the transpose: v holds
// x_b[l + 32 m] at v[b * gfft_in + m]; on return lane j < NB M holds in o the
// 32 inputs of its final DFT32 (transform b = j / M, outputs k1 + M k2,
// k1 = j mod M); other lanes hold a copy of lane 0's.  scr: the warp's scratch
// (free on entry and on exit).  tw: w_N^(l k1) at [k1 * 32 + l], global memory.
template <int M, int NB, bool HIN>
__device__ __forceinline__ void gfft_head(const float2 (&v)[NB * gfft_in<M, HIN>()], float2 (&o)[32], float2* scr,
                                          const float2* __restrict__ tw) {
  constexpr int MI = gfft_in<M, HIN>();
  const int l = lane_id();
  float2 t[NB][M];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if constexpr (HIN && M % 2 == 0) {
      // X[2q] = DFT_(M/2)(x)[q], X[2q + 1] = DFT_(M/2)(x w_M^m)[q]
      constexpr int Hm = M / 2;
      float2 e[Hm], d[Hm];
#pragma unroll
      for (int m = 0; m < Hm; ++m) { e[m] = v[b * MI + m]; d[m] = e[m]; }
      mul_roots<M, Hm, false>(d);
      if constexpr (Hm > 1) {
        dft_any<Hm, false>(e);
        dft_any<Hm, false>(d);
      }
#pragma unroll
      for (int q = 0; q < Hm; ++q) { t[b][2 * q] = e[q]; t[b][2 * q + 1] = d[q]; }
    } else {
#pragma unroll
      for (int m = 0; m < M; ++m) t[b][m] = m < MI ? v[b * MI + m] : make_float2(0.0f, 0.0f);
      if constexpr (M > 1) dft_any<M, false>(t[b]);
    }
  }
#pragma unroll
  for (int k1 = 0; k1 < M; ++k1) {
    const float2 w = k1 == 0 ? make_float2(1.0f, 0.0f) : __ldg(tw + k1 * 32 + l);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int r = b * M + k1;
      scr[r * 32 + (l ^ r)] = k1 == 0 ? t[b][0] : cmul(t[b][k1], w);
    }
  }
  __syncwarp();
  // lanes without a row read row 0 again (a guard around the loads would keep
  // both sides of 64 registers alive and spill)
  const int lr = NB * M == 32 || l < NB * M ? l : 0;
#pragma unroll
  for (int c = 0; c < 32; ++c) o[c] = scr[lr * 32 + (c ^ lr)];
  __syncwarp();
}

// The final DFT32 (forward); HOUT: only outputs k2 < 16 are formed.
template <bool HOUT>
__device__ __forceinline__ void gfft_tail(float2 (&v)[32]) {
  if constexpr (!HOUT) {
    dft32<false>(v);
  } else {
    float2 e[16], o[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      e[i] = v[2 * i];
      o[i] = v[2 * i + 1];
    }
    dft16<false>(e);
    dft16<false>(o);
#define MMP_R2H(K) v[K] = cadd(e[K], mul_w32<K, false>(o[K]));
    MMP_R2H(0) MMP_R2H(1) MMP_R2H(2) MMP_R2H(3) MMP_R2H(4) MMP_R2H(5) MMP_R2H(6) MMP_R2H(7)
    MMP_R2H(8) MMP_R2H(9) MMP_R2H(10) MMP_R2H(11) MMP_R2H(12) MMP_R2H(13) MMP_R2H(14) MMP_R2H(15)
#undef MMP_R2H
  }
}

// NB transforms of length 32 M by one warp (INV: exp(+2 pi i k n / N), no 1/N,
// as the conjugate of the forward transform of the conjugate).  v as in
// gfft_head; on return lane j < NB M holds o[k2] = X_b[k1 + M k2].
template <int M, int NB, bool HIN, bool HOUT, bool INV>
__device__ __forceinline__ void gfft(float2 (&v)[NB * gfft_in<M, HIN>()], float2 (&o)[32], float2* scr,
                                     const float2* __restrict__ tw) {
  if (INV) {
#pragma unroll
    for (int i = 0; i < NB * gfft_in<M, HIN>(); ++i) v[i].y = -v[i].y;
  }
  gfft_head<M, NB, HIN>(v, o, scr, tw);
  gfft_tail<HOUT>(o);
  if (INV) {
#pragma unroll
    for (int i = 0; i < (HOUT ? 16 : 32); ++i) o[i].y = -o[i].y;
  }
}

}  // namespace mmp
