// tensor.cu -- FP64 construction of the demag kernel spectrum on the device.
//
// Methods, "Magnetostatic field": the cell-to-cell demag tensor N is the
// analytical result of Newell, Williams and Dunlop below a cutoff radius and
// an asymptotic result above it.  Built here in FP64 (the Newell second
// differences cancel catastrophically) and transformed in FP64; only the
// final spectrum is rounded to FP32.
//
//  * Newell: N_xx is the 27-point second difference (weights 2, -1, -1 per
//    axis) of f(x, y, z), N_xy that of g(x, y, z), divided by 4 pi V.
//  * Far field: N_ab(r) = -V/(4 pi) sum_{alpha even, |alpha| <= 2P}
//    E[s^alpha]/alpha! d^(alpha + e_a + e_b)(1/r), the expansion of the
//    cell-pair average over the difference s of two uniform points of a
//    cell (triangular per axis, E[s^2k] = 2 D^2k / ((2k+1)(2k+2))).  The
//    derivatives of 1/r = F(r^2), F(q) = q^(-1/2), use the Hermite-type
//    chain rule  d^t_x F(x^2 + ...) = sum_i t!/(i!(t-2i)!) (2x)^(t-2i) F^(t-i)
//    applied per axis, with F^(n)(r^2) = (-1)^n (2n-1)!!/2^n r^(-2n-1).
//    The far-field terms are evaluated in FP32 (no cancellation there that
//    FP32 cannot carry: the kernel is smooth and ~1/r^3 above the cutoff).
//  * Spectrum: the kernel of the zero-padded convolution is even or odd in
//    each axis, so its DFT is real: along an axis with padded length P the
//    transform is N(0) + 2 sum_i N(i) cos(2 pi k i / P) (even) or
//    -2i sum_i N(i) sin(2 pi k i / P) (odd); two odd axes give the factor
//    (-i)^2 = -1.  Only the octant 0 <= k <= P/2 is stored.  Axes with
//    P >= 64 are transformed by an FP64 FFT of the evenly or oddly extended
//    line, shorter ones by the direct sums.
#include <math.h>
#include "kernels.h"
#include "launch.cuh"

namespace mmp {

namespace {

constexpr double kPi = 3.14159265358979323846;
constexpr int kOrder = 4;                  // expansion through E[s^8]
constexpr int kNmax = 2 * kOrder + 2;      // highest derivative order of 1/r

__device__ __noinline__ double newell_f(double x, double y, double z) {
  x = fabs(x); y = fabs(y); z = fabs(z);
  double x2 = x * x, y2 = y * y, z2 = z * z;
  double R = sqrt(x2 + y2 + z2);
  double out = (2.0 * x2 - y2 - z2) * R / 6.0;
  double rxz = sqrt(x2 + z2), rxy = sqrt(x2 + y2);
  if (rxz > 0) out += 0.5 * y * (z2 - x2) * asinh(y / rxz);
  if (rxy > 0) out += 0.5 * z * (y2 - x2) * asinh(z / rxy);
  if (x > 0) out -= x * y * z * atan(y * z / (x * R));
  return out;
}

__device__ __noinline__ double newell_g(double x, double y, double z) {
  double sgn = ((x < 0) != (y < 0)) ? -1.0 : 1.0;
  if (x == 0 || y == 0) sgn = 0.0;
  x = fabs(x); y = fabs(y); z = fabs(z);
  double x2 = x * x, y2 = y * y, z2 = z * z;
  double R = sqrt(x2 + y2 + z2);
  double out = -x * y * R / 3.0;
  double rxy = sqrt(x2 + y2), ryz = sqrt(y2 + z2), rxz = sqrt(x2 + z2);
  if (rxy > 0) out += x * y * z * asinh(z / rxy);
  if (ryz > 0) out += y / 6.0 * (3.0 * z2 - y2) * asinh(x / ryz);
  if (rxz > 0) out += x / 6.0 * (3.0 * z2 - x2) * asinh(y / rxz);
  if (z > 0) out -= z * z2 / 6.0 * atan(x * y / (z * R));
  if (y > 0) out -= z * y2 / 2.0 * atan(x * z / (y * R));
  if (x > 0) out -= z * x2 / 2.0 * atan(y * z / (x * R));
  return sgn * out;
}

template <bool G>
__device__ double second_difference(double X, double Y, double Z, double a, double b, double c) {
  const double w[3] = {-1.0, 2.0, -1.0};
  double acc = 0.0;
#pragma unroll 1
  for (int i = 0; i < 3; ++i)
#pragma unroll 1
    for (int j = 0; j < 3; ++j)
#pragma unroll 1
      for (int k = 0; k < 3; ++k) {
        double f = G ? newell_g(X + (i - 1) * a, Y + (j - 1) * b, Z + (k - 1) * c)
                     : newell_f(X + (i - 1) * a, Y + (j - 1) * b, Z + (k - 1) * c);
        acc += w[i] * w[j] * w[k] * f;
      }
  return acc / (4.0 * kPi * a * b * c);
}

// Far field in FP32.  Above the cutoff the kernel is smooth and of size
// ~1/r^3; its terms are evaluated in single precision (relative rounding
// ~1e-7 of the kernel's scale there, against the 1e-5 Ms field bar), with
// every index a compile-time constant after unrolling.
// c(t, i) = t! / (i! (t - 2i)!), the coefficients of the chain rule
// d^t_x F(x^2 + ..) = sum_i c(t, i) (2x)^(t - 2i) F^(t - i).
__host__ __device__ constexpr float chain_coef(int t, int i) {
  float v = 1.0f;
  for (int m = t - 2 * i + 1; m <= t; ++m) v *= (float)m;   // t! / (t - 2i)!
  for (int m = 2; m <= i; ++m) v /= (float)m;               // / i!
  return v;
}
// d^T_x d^U_y d^V_z (1/r) from px[e] = (2X)^e (etc.) and Fn[n] = F^(n)(r^2)
template <int T, int U, int V>
__device__ __forceinline__ float inv_r_derivative(const float (&px)[kNmax + 1], const float (&py)[kNmax + 1],
                                                  const float (&pz)[kNmax + 1], const float (&Fn)[kNmax + 1]) {
  float acc = 0.0f;
#pragma unroll
  for (int i = 0; i <= T / 2; ++i)
#pragma unroll
    for (int j = 0; j <= U / 2; ++j)
#pragma unroll
      for (int k = 0; k <= V / 2; ++k) {
        const float c = chain_coef(T, i) * chain_coef(U, j) * chain_coef(V, k);
        acc = fmaf(c * px[T - 2 * i] * py[U - 2 * j], pz[V - 2 * k] * Fn[T + U + V - i - j - k], acc);
      }
  return acc;
}

// N octant: out[comp][k][j][i] for offsets (i dx, j dy, k dz); cell sizes
// scaled by the largest one (N is scale invariant).
// Moment weights of the far-field expansion, w[a][b][e] =
// E[s_x^2a] E[s_y^2b] E[s_z^2e] / ((2a)! (2b)! (2e)!) (a + b + e <= kOrder),
// E[s^2k] = 2 d^2k / ((2k+1)(2k+2)) for the difference s of two uniform
// points of a cell of width d (1 for k = 0); built on the host in FP64.
struct FarWeights {
  float w[kOrder + 1][kOrder + 1][kOrder + 1];
};

// Far-field sums of the orders 2 (A + B + E), E, then B, then A ascending.  The
// diagonal components share their derivatives: d^(2A, 2B, 2E)(1/r) is the term
// (A - 1, B, E) of xx, (A, B - 1, E) of yy and (A, B, E - 1) of zz, so it is
// formed once for the three.
template <int A, int B, int E>
__device__ __forceinline__ void far_terms(const FarWeights& fw, const float (&px)[kNmax + 1],
                                          const float (&py)[kNmax + 1], const float (&pz)[kNmax + 1],
                                          const float (&Fn)[kNmax + 1], float (&acc)[6]) {
  if constexpr (A + B + E >= 1) {
    const float D = inv_r_derivative<2 * A, 2 * B, 2 * E>(px, py, pz, Fn);
    if constexpr (A > 0) acc[0] = fmaf(fw.w[A - 1][B][E], D, acc[0]);
    if constexpr (B > 0) acc[1] = fmaf(fw.w[A][B - 1][E], D, acc[1]);
    if constexpr (E > 0) acc[2] = fmaf(fw.w[A][B][E - 1], D, acc[2]);
  }
  if constexpr (A + B + E <= kOrder) {
    const float w = fw.w[A][B][E];
    acc[3] = fmaf(w, inv_r_derivative<2 * A + 1, 2 * B + 1, 2 * E>(px, py, pz, Fn), acc[3]);
    acc[4] = fmaf(w, inv_r_derivative<2 * A + 1, 2 * B, 2 * E + 1>(px, py, pz, Fn), acc[4]);
    acc[5] = fmaf(w, inv_r_derivative<2 * A, 2 * B + 1, 2 * E + 1>(px, py, pz, Fn), acc[5]);
  }
  if constexpr (A + B + E < kOrder + 1) far_terms<A, B, E + 1>(fw, px, py, pz, Fn, acc);
  else if constexpr (A + B < kOrder + 1) far_terms<A, B + 1, 0>(fw, px, py, pz, Fn, acc);
  else if constexpr (A < kOrder + 1) far_terms<A + 1, 0, 0>(fw, px, py, pz, Fn, acc);
}

// Newell's f and g on the lattice of offsets that the second differences of the
// near octant touch: point (i, j, k) of m[0] x m[1] x m[2], function c (f for
// xx, yy, zz with the axes in turn, g for xy, xz, yz) at lat[c][k][j][i].  A
// point is shared by up to 27 differences of each component; formed anew for
// each, one thread's chain of 162 evaluations (FP64 asinh, atan and square
// roots) took longer than the rest of the octant (256x256x4
// geometry with its first field 5476 -> 3417 us; the lattice takes 38).
__global__ void k_newell_lattice(double* __restrict__ lat, int mx, int my, int mz, double dx, double dy, double dz) {
  const int per = mx * my * mz;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 6 * per) return;
  const int c = idx / per, r = idx - c * per;
  const double X = (r % mx) * dx, Y = (r / mx % my) * dy, Z = (r / (mx * my)) * dz;
  lat[idx] = c == 0   ? newell_f(X, Y, Z)
             : c == 1 ? newell_f(Y, X, Z)
             : c == 2 ? newell_f(Z, Y, X)
             : c == 3 ? newell_g(X, Y, Z)
             : c == 4 ? newell_g(X, Z, Y)
                      : newell_g(Y, Z, X);
}

// The second difference of component c at (i, j, k) from the lattice: f is even
// in every axis, g odd in its two axes.
__device__ __forceinline__ double lattice_difference(const double* __restrict__ lat, int c, int i, int j, int k,
                                                     int mx, int my, int mz) {
  const double w[3] = {-1.0, 2.0, -1.0};
  const bool ox = c == 3 || c == 4, oy = c == 3 || c == 5, oz = c == 4 || c == 5;
  double acc = 0.0;
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b)
      for (int e = 0; e < 3; ++e) {
        const int x = i + a - 1, y = j + b - 1, z = k + e - 1;
        double s = w[a] * w[b] * w[e];
        if (x < 0 && ox) s = -s;
        if (y < 0 && oy) s = -s;
        if (z < 0 && oz) s = -s;
        acc += s * lat[(long long)c * mx * my * mz + abs(x) + (long long)mx * (abs(y) + (long long)my * abs(z))];
      }
  return acc;
}

// lat: the lattice of extents mx, my, mz (null: the differences are formed
// point by point).
__global__ void k_tensor_octant(double* __restrict__ out, int nx, int ny, int nz, double dx,
                                double dy, double dz, double rc, FarWeights fw, const double* __restrict__ lat,
                                int mx, int my, int mz) {
  long long n = (long long)nx * ny * nz;
  long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= n) return;
  int i = idx % nx, j = (idx / nx) % ny, k = idx / ((long long)nx * ny);
  double X = i * dx, Y = j * dy, Z = k * dz;
  const bool near = sqrt(X * X + Y * Y + Z * Z) < rc;
  if (near && lat) {
    for (int c = 0; c < 6; ++c)
      out[c * n + idx] = lattice_difference(lat, c, i, j, k, mx, my, mz) / (4.0 * kPi * dx * dy * dz);
  } else if (near) {
    out[idx] = second_difference<false>(X, Y, Z, dx, dy, dz);
    out[n + idx] = second_difference<false>(Y, X, Z, dy, dx, dz);
    out[2 * n + idx] = second_difference<false>(Z, Y, X, dz, dy, dx);
    out[3 * n + idx] = second_difference<true>(X, Y, Z, dx, dy, dz);
    out[4 * n + idx] = second_difference<true>(X, Z, Y, dx, dz, dy);
    out[5 * n + idx] = second_difference<true>(Y, Z, X, dy, dz, dx);
  } else {
    const float x = (float)X, y = (float)Y, z = (float)Z;
    float px[kNmax + 1], py[kNmax + 1], pz[kNmax + 1], Fn[kNmax + 1];
    px[0] = py[0] = pz[0] = 1.0f;
#pragma unroll
    for (int e = 1; e <= kNmax; ++e) {
      px[e] = px[e - 1] * 2.0f * x;
      py[e] = py[e - 1] * 2.0f * y;
      pz[e] = pz[e - 1] * 2.0f * z;
    }
    const float r2 = x * x + y * y + z * z, ir2 = 1.0f / r2;
    Fn[0] = 1.0f / sqrtf(r2);   // F^(n) = (-1)^n (2n-1)!!/2^n r^(-2n-1)
#pragma unroll
    for (int m = 1; m <= kNmax; ++m) Fn[m] = Fn[m - 1] * (-(2.0f * m - 1.0f) / 2.0f) * ir2;
    float acc[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    far_terms<0, 0, 0>(fw, px, py, pz, Fn, acc);
    const double V = dx * dy * dz;
#pragma unroll
    for (int c = 0; c < 6; ++c) out[c * n + idx] = -V / (4.0 * kPi) * (double)acc[c];
  }
}

// One axis of the real cos/sin transform.  in: [6][e2][e1][e0] with the
// transformed axis of extent nin; out: same with extent nout = P/2+1.
// trig[t] = (cos, sin)(2 pi t / P), t in [0, P).
__global__ void k_tensor_axis(const double* __restrict__ in, double* __restrict__ out, int e0, int e1,
                              int e2, int axis, int nin, int nout, int P, const double2* __restrict__ trig,
                              int odd_mask) {
  int o0 = axis == 0 ? nout : e0, o1 = axis == 1 ? nout : e1, o2 = axis == 2 ? nout : e2;
  long long per = (long long)o0 * o1 * o2;
  long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= 6 * per) return;
  int comp = idx / per;
  long long r = idx - comp * per;
  int i0 = r % o0, i1 = (r / o0) % o1, i2 = r / ((long long)o0 * o1);
  int kk = axis == 0 ? i0 : (axis == 1 ? i1 : i2);
  long long stride = axis == 0 ? 1 : (axis == 1 ? (long long)e0 : (long long)e0 * e1);
  long long base = (long long)comp * e0 * e1 * e2 + (long long)(axis == 0 ? 0 : i0) +
                   (long long)(axis == 1 ? 0 : i1) * e0 + (long long)(axis == 2 ? 0 : i2) * e0 * e1;
  bool odd = (odd_mask >> comp) & 1;
  double acc = odd ? 0.0 : in[base];
  for (int i = 1; i < nin; ++i) {
    int t = (int)(((long long)kk * i) % P);
    double w = odd ? trig[t].y : trig[t].x;
    acc += 2.0 * w * in[base + i * stride];
  }
  out[comp * per + r] = acc;
}

// One axis of the real cos/sin transform by an FP64 FFT, for padded lengths
// P >= 64 (P = 2^a or 3 * 2^a): two lines of one component per complex
// transform.  A line is extended to length P evenly (N(P - i) = N(i)) or oddly
// (N(P - i) = -N(i)); its DFT is then real (even: N(0) + 2 sum N(i) cos) or
// imaginary (odd: -i times 2 sum N(i) sin), so the DFT of line a + i line b holds
// both: even Re and Im, odd -Im and Re, the same values as k_tensor_axis.
// Stockham passes in shared memory: radix 8, one of 4 or 2, then 3 where it
// divides P (pass of radix R with Ns outputs per sub-transform: inputs j + r P/R,
// twiddle w_(Ns R)^(r (j mod Ns)), outputs at (j / Ns) Ns R + j mod Ns + r Ns);
// Ns is a power of two in every pass.
// What bounds it is the FP64 rate (2 lanes a clock and SM): two lines a transform
// and radix 8 take 0.4 of the operations of one line by radix 2.  A block takes
// NL neighbouring lines, so that along y and z its loads and stores are whole
// sectors.  256x256x4, x and y axis each: 225 us (one line, radix 2) -> 104.
template <int R>
__device__ __forceinline__ void dft64(double2 (&v)[R]) {
  auto two = [](double2& a, double2& b) {
    const double2 t = a;
    a = make_double2(t.x + b.x, t.y + b.y);
    b = make_double2(t.x - b.x, t.y - b.y);
  };
  auto mi = [](double2 a) { return make_double2(a.y, -a.x); };   // -i a
  if constexpr (R == 2) {
    two(v[0], v[1]);
  } else if constexpr (R == 3) {
    // w3 = exp(-2 pi i / 3) = (-1/2, -s3)
    const double s3 = 0.86602540378443864676;
    const double2 t = make_double2(v[1].x + v[2].x, v[1].y + v[2].y);
    const double2 d = make_double2(v[1].x - v[2].x, v[1].y - v[2].y);
    const double2 m = make_double2(v[0].x - 0.5 * t.x, v[0].y - 0.5 * t.y);
    v[0] = make_double2(v[0].x + t.x, v[0].y + t.y);
    v[1] = make_double2(m.x + s3 * d.y, m.y - s3 * d.x);
    v[2] = make_double2(m.x - s3 * d.y, m.y + s3 * d.x);
  } else if constexpr (R == 4) {
    two(v[0], v[2]);
    two(v[1], v[3]);
    v[3] = mi(v[3]);
    two(v[0], v[1]);
    two(v[2], v[3]);
    const double2 t = v[1];   // outputs 0, 2, 1, 3
    v[1] = v[2];
    v[2] = t;
  } else {
    const double h = 0.70710678118654752440;
    double2 e[4], o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      e[i] = v[i];
      o[i] = v[i + 4];
      two(e[i], o[i]);
    }
    // odd outputs: DFT4 of o[i] w8^i
    o[1] = make_double2(h * (o[1].x + o[1].y), h * (o[1].y - o[1].x));
    o[2] = mi(o[2]);
    o[3] = make_double2(h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y));
    dft64<4>(e);
    dft64<4>(o);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[2 * i] = e[i];
      v[2 * i + 1] = o[i];
    }
  }
}

template <int R>
__device__ __forceinline__ void fft64_pass(const double2* __restrict__ x, double2* __restrict__ y, int P, int npair,
                                           int lns, const double2* __restrict__ trig) {
  const int NR = P / R, Ns = 1 << lns, step = NR >> lns;
  for (int e = threadIdx.x; e < npair * NR; e += blockDim.x) {
    const int t = e / NR, j = e - t * NR, k = j & (Ns - 1);
    const double2* xt = x + t * P;
    double2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = xt[j + r * NR];
    if (k)
#pragma unroll
      for (int r = 1; r < R; ++r) {
        const double2 w = trig[r * k * step];   // (cos, sin), r k step < P: the forward twiddle is its conjugate
        v[r] = make_double2(v[r].x * w.x + v[r].y * w.y, v[r].y * w.x - v[r].x * w.y);
      }
    dft64<R>(v);
    double2* yt = y + t * P + (j >> lns) * Ns * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) yt[r * Ns] = v[r];
  }
  __syncthreads();
}

constexpr int kFft64Threads = 128;
// Pairs of lines per block: about 1024 values.
__host__ __device__ __forceinline__ int fft64_pairs(int P) { return P >= 1024 ? 1 : P >= 512 ? 2 : P >= 256 ? 4 : 8; }

__global__ void __launch_bounds__(kFft64Threads) k_tensor_axis_fft(const double* __restrict__ in,
                                                                   double* __restrict__ out, int e0, int e1, int e2,
                                                                   int axis, int nin, int nout, int P, int npair,
                                                                   const double2* __restrict__ trig, int odd_mask) {
  extern __shared__ double2 fbuf[];
  double2* x = fbuf;
  double2* y = fbuf + npair * P;
  // lines of one component: their coordinates (i0, i1, i2) with 0 on the transformed axis
  const int l0 = axis == 0 ? 1 : e0, l1 = axis == 1 ? 1 : e1, l2 = axis == 2 ? 1 : e2;
  const int lines = l0 * l1 * l2, nl = 2 * npair, per = (lines + nl - 1) / nl;
  const int comp = blockIdx.x / per, line0 = (blockIdx.x - comp * per) * nl, have = min(nl, lines - line0);
  const bool odd = (odd_mask >> comp) & 1;
  const long long istride = axis == 0 ? 1 : (axis == 1 ? (long long)e0 : (long long)e0 * e1);
  const int q0 = axis == 0 ? nout : e0, q1 = axis == 1 ? nout : e1, q2 = axis == 2 ? nout : e2;
  const long long ostride = axis == 0 ? 1 : (axis == 1 ? (long long)q0 : (long long)q0 * q1);
  auto base = [&](int line, int f0, int f1, int f2) {
    const int i0 = line % l0, i1 = (line / l0) % l1, i2 = line / (l0 * l1);
    return (long long)comp * f0 * f1 * f2 + i0 + (long long)i1 * f0 + (long long)i2 * f0 * f1;
  };
  double* xf = reinterpret_cast<double*>(x);
  for (int i = threadIdx.x; i < 2 * npair * P; i += blockDim.x) xf[i] = 0.0;
  __syncthreads();
  for (int e = threadIdx.x; e < have * nin; e += blockDim.x) {   // nin <= P / 2: no overlap of i and P - i
    const int l = axis == 0 ? e / nin : e % have, i = axis == 0 ? e - l * nin : e / have;
    const double v = in[base(line0 + l, e0, e1, e2) + i * istride];
    double* xl = xf + 2 * (l >> 1) * P + (l & 1);
    if (i == 0) {
      xl[0] = odd ? 0.0 : v;
    } else {
      xl[2 * i] = v;
      xl[2 * (P - i)] = odd ? -v : v;
    }
  }
  __syncthreads();
  auto swap = [&]() { double2* t = x; x = y; y = t; };
  int lns = 0, rest = P % 3 == 0 ? P / 3 : P;
  while (rest >= 8) {
    fft64_pass<8>(x, y, P, npair, lns, trig);
    swap();
    lns += 3;
    rest >>= 3;
  }
  if (rest == 4) {
    fft64_pass<4>(x, y, P, npair, lns, trig);
    swap();
    lns += 2;
  } else if (rest == 2) {
    fft64_pass<2>(x, y, P, npair, lns, trig);
    swap();
    lns += 1;
  }
  if (P % 3 == 0) {
    fft64_pass<3>(x, y, P, npair, lns, trig);
    swap();
  }
  const double* of = reinterpret_cast<const double*>(x);
  for (int e = threadIdx.x; e < have * nout; e += blockDim.x) {
    const int l = axis == 0 ? e / nout : e % have, k = axis == 0 ? e - l * nout : e / have;
    const double* z = of + 2 * ((l >> 1) * P + k);
    out[base(line0 + l, q0, q1, q2) + k * ostride] = !odd ? z[l & 1] : (l & 1) ? z[0] : -z[1];
  }
}

// Final scaling and layout change to float [kx][ky][krow], row = 6 floats
// per kz (xx, yy, zz, xy, xz, yz) and zero padding to krow.
__global__ void k_tensor_store(const double* __restrict__ in, float* __restrict__ out, int mx, int my,
                               int mz, int krow, double scale_even, double scale_odd2) {
  long long per = (long long)mx * my * mz;
  long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= per) return;
  int ix = idx % mx, iy = (idx / mx) % my, iz = idx / ((long long)mx * my);
  long long row = ((long long)ix * my + iy) * krow;
  if (iz == 0)
    for (int c = 6 * mz; c < krow; ++c) out[row + c] = 0.0f;
  long long o = row + iz * 6;
  for (int c = 0; c < 6; ++c) out[o + c] = (float)(in[c * per + idx] * (c < 3 ? scale_even : scale_odd2));
}

}  // namespace

cudaError_t build_kernel_spectrum(const KernelBuild& kb, cudaStream_t s) {
  const int nx = kb.n[0], ny = kb.n[1], nz = kb.n[2];
  double L = fmax(kb.cell[0], fmax(kb.cell[1], kb.cell[2]));
  long long n = (long long)nx * ny * nz;
  FarWeights fw;
  {
    const double d[3] = {kb.cell[0] / L, kb.cell[1] / L, kb.cell[2] / L};
    double m[3][kOrder + 1];
    double f2[kOrder + 1];
    for (int k = 0; k <= kOrder; ++k) {
      double f = 1.0;
      for (int q = 2; q <= 2 * k; ++q) f *= q;
      f2[k] = f;                                   // (2k)!
      for (int ax = 0; ax < 3; ++ax)
        m[ax][k] = k == 0 ? 1.0 : 2.0 * pow(d[ax], 2 * k) / ((2.0 * k + 1.0) * (2.0 * k + 2.0));
    }
    for (int a = 0; a <= kOrder; ++a)
      for (int b = 0; b <= kOrder; ++b)
        for (int e = 0; e <= kOrder; ++e)
          fw.w[a][b][e] = a + b + e > kOrder ? 0.0f
                                             : (float)(m[0][a] * m[1][b] * m[2][e] / (f2[a] * f2[b] * f2[e]));
  }
  // the lattice of the near octant: offsets below the cutoff and one beyond, in
  // the buffer that the first transform overwrites
  const double dl[3] = {kb.cell[0] / L, kb.cell[1] / L, kb.cell[2] / L};
  int m[3];
  for (int ax = 0; ax < 3; ++ax) m[ax] = (int)fmin((double)kb.n[ax], floor(kb.rc / dl[ax]) + 1.0) + 1;
  const bool lattice = (long long)m[0] * m[1] * m[2] <= n;
  if (lattice) {
    const int total = 6 * m[0] * m[1] * m[2];
    k_newell_lattice<<<(total + 63) / 64, 64, 0, s>>>(kb.buf1, m[0], m[1], m[2], dl[0], dl[1], dl[2]);
  }
  k_tensor_octant<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(kb.buf0, nx, ny, nz, dl[0], dl[1], dl[2], kb.rc, fw,
                                                              lattice ? kb.buf1 : nullptr, m[0], m[1], m[2]);
  // odd masks per axis: x odd for xy, xz; y odd for xy, yz; z odd for xz, yz
  const int odd[3] = {(1 << 3) | (1 << 4), (1 << 3) | (1 << 5), (1 << 4) | (1 << 5)};
  int e[3] = {nx, ny, nz};
  double* src = kb.buf0;
  double* dst = kb.buf1;
  for (int a = 0; a < 3; ++a) {
    if (kb.P[a] == 1) continue;
    int nout = kb.P[a] / 2 + 1;
    const long long lines = 6LL * (a == 0 ? 1 : e[0]) * (a == 1 ? 1 : e[1]) * (a == 2 ? 1 : e[2]);
    if (kb.P[a] >= 64) {   // FP64 FFT of line pairs
      const int np = fft64_pairs(kb.P[a]);
      const size_t sm = (size_t)2 * np * kb.P[a] * sizeof(double2);
      const cudaError_t err = set_smem(k_tensor_axis_fft, sm);
      if (err != cudaSuccess) return err;
      const long long blocks = 6 * ((lines / 6 + 2 * np - 1) / (2 * np));
      k_tensor_axis_fft<<<(unsigned)blocks, kFft64Threads, sm, s>>>(src, dst, e[0], e[1], e[2], a, e[a], nout,
                                                                    kb.P[a], np, kb.trig[a], odd[a]);
    } else {               // short axes: the direct sums
      const long long total = lines * nout;
      k_tensor_axis<<<(unsigned)((total + 127) / 128), 128, 0, s>>>(src, dst, e[0], e[1], e[2], a, e[a], nout,
                                                                    kb.P[a], kb.trig[a], odd[a]);
    }
    e[a] = nout;
    double* t = src; src = dst; dst = t;
  }
  double scale = -kMu0 / ((double)kb.P[0] * kb.P[1] * kb.P[2]);
  long long per = (long long)e[0] * e[1] * e[2];
  k_tensor_store<<<(unsigned)((per + 127) / 128), 128, 0, s>>>(src, kb.out, e[0], e[1], e[2], kb.krow, scale,
                                                                -scale);
  return cudaGetLastError();
}

}  // namespace mmp
