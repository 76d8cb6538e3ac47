// The contraction over the FFTLog frequencies as a chirp transform (a3 and its transpose), for k
// grids that are uniform in ln k:  ln k_q = x0 + q d.
//
// With eta_n = 2 pi n/L and beta = 2 pi d/L the phase of Eq. 3.4-3.5 is e^{-i eta_n ln k_q} =
// e^{-i eta_n x0} e^{-i beta n q}, and with n = n0 + m, m q = (m^2 + q^2 - (m - q)^2)/2 (Bluestein):
//   sum_{n >= n0} F_n G_n e^{-i eta_n ln k_q} = b_q sum_m [F_n G_n a_n] h_{q - m},
//   a_n = e^{-i eta_n x0 - i beta m^2/2},  b_q = e^{-i beta (n0 q + q^2/2)},  h_t = e^{+i beta t^2/2},
// a linear convolution with one fixed filter: two FFTs of M >= (frequencies) + N_k - 1 points per
// row (walker, tracer, multipole) instead of 4 n_h N_k operations.  The transpose is the same
// convolution with the roles of m and q exchanged:
//   sum_q d_q e^{-i eta_n ln k_q} = a_n sum_q [d_q b_q] h_{n - q}                  (n0 = 0),
// multiplied by G[l][n] and summed over the multipoles before the factor a_n.
//
// One CTA of M/E threads (E = 16 or 32 points each) runs one row at a time: a forward FFT of passes
// E x E x M/E^2 with the frequencies left in digit-reversed order, the product with the
// filter's spectrum (stored in that order), and the inverse passes in reverse.  Each pass works in
// registers; passes exchange through shared memory in place (a thread writes back the places it has
// read), so the second and third pass, which stay within 16 neighbouring threads, need a warp
// barrier only (or shuffles) and a row needs two CTA barriers.  The window of the frequencies and of the k points
// is at most M/2 in the HALF form: half of the first pass's inputs are then zero and half of the
// last pass's outputs unused.
//
// FP64: bound by the FP64 pipe (two FMA per clock and SM): about 1080 FP64 instructions per thread and
// row of 2048 points, so the largest radix whose points fit the registers (fewest twiddle products)
// and eight resident warps are enough.  15 tracers x 103 multipoles, N = 2048, N_k = 1024: 459 us
// forward and 440 us transposed (75 % of the pipe's rate; the last of six turns of two CTAs per SM is
// nearly empty), against 5.9 ms each for the direct sums.
//
// FP32: bound by shared-memory and table accesses (1750 wavefronts of the load/store pipe per row of
// 2048 points) and, close behind, by instruction issue: about 2070 clocks per row and SM with four
// resident CTAs (16 warps).  1545 such rows 19 us forward and 20 us transposed; 287 100 rows (256 walkers
// with ragged lists) 1.89 and 1.80 ms; 89 970 rows of 8192 points 3.74 and 3.21 ms.  The GEMMs over all
// frequencies took 56 and 58 us, 7.9 and 12.3 ms, 14.6 and 11.9 ms, with another 23 us, 1.7 ms and
// 1.5 ms for their operand images.  Errors against 64 bits (N5K shape): Delta 1.3e-7 (GEMMs 1.9e-7),
// normalised C 2.7e-5 (3.1e-5), W_bar 4.2e-7 (9.7e-7); white-noise windows 1.6e-7 (1.4e-7), 5.9e-5
// (6.0e-5), 4.8e-7 (7.4e-7).
#pragma once
#include <algorithm>
#include <type_traits>

#include "f32x2.cuh"
#include "swcl_internal.h"

namespace swcl {
namespace chirp {

template <class T> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };
template <class T> using V2 = typename Vec2<T>::type;

template <class T> __device__ __forceinline__ V2<T> mk(T x, T y) { V2<T> v; v.x = x; v.y = y; return v; }
template <class V> __device__ __forceinline__ V add(V a, V b) { a.x += b.x; a.y += b.y; return a; }
template <class V> __device__ __forceinline__ V sub(V a, V b) { a.x -= b.x; a.y -= b.y; return a; }
// FP32: both components in one instruction (the same two roundings); 2.12 -> 1.96 ms forward and 2.22 ->
// 1.89 ms transposed for 287 100 rows of 2048 points, together with the constant offsets below
template <> __device__ __forceinline__ float2 add<float2>(float2 a, float2 b) { return f2_add(a, b); }
template <> __device__ __forceinline__ float2 sub<float2>(float2 a, float2 b) { return f2_sub(a, b); }
// a + c b and a - c b with a real constant c
template <class V, class T> __device__ __forceinline__ V axpy(T c, V b, V a) {
  a.x = fma(c, b.x, a.x);
  a.y = fma(c, b.y, a.y);
  return a;
}
template <> __device__ __forceinline__ float2 axpy<float2, float>(float c, float2 b, float2 a) {
  return f2_fma(make_float2(c, c), b, a);
}
// a b, and a conj(b)
template <class V> __device__ __forceinline__ V mul(V a, V b) {
  V r;
  r.x = fma(a.x, b.x, -a.y * b.y);
  r.y = fma(a.x, b.y, a.y * b.x);
  return r;
}
template <class V> __device__ __forceinline__ V mulc(V a, V b) {
  V r;
  r.x = fma(a.x, b.x, a.y * b.y);
  r.y = fma(a.y, b.x, -a.x * b.y);
  return r;
}
// a times i S (S = +1 or -1)
template <int S, class V> __device__ __forceinline__ V rot(V a) {
  V r;
  if constexpr (S > 0) { r.x = -a.y; r.y = a.x; } else { r.x = a.y; r.y = -a.x; }
  return r;
}

// A table value that every row reads again (L1).  volatile keeps the load in the loop over rows: hoisted
// out of it, the tables would take more registers than the data.
__device__ __forceinline__ float2 ld_tab(const float2* p) {
  float2 v;
  asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ double2 ld_tab(const double2* p) {
  double2 v;
  asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}

// ---- DFTs in registers, X_k = sum_n v_n e^{2 pi i S n k / R}, natural order in and out ----

template <int S, class V> __device__ __forceinline__ void dft4(V& a, V& b, V& c, V& d) {
  const V s0 = add(a, c), d0 = sub(a, c), s1 = add(b, d), d1 = rot<S>(sub(b, d));
  a = add(s0, s1);
  b = add(d0, d1);
  c = sub(s0, s1);
  d = sub(d0, d1);
}
// c = d = 0
template <int S, class V> __device__ __forceinline__ void dft4_half(V& a, V& b, V& c, V& d) {
  const V a0 = a, b0 = b, r = rot<S>(b);
  a = add(a0, b0);
  b = add(a0, r);
  c = sub(a0, b0);
  d = sub(a0, r);
}

// cos and sin of 2 pi j/32 (j mod 32; the quadrant's nine values, the rest by symmetry)
__host__ __device__ constexpr double cos32(int j) {
  constexpr double c[9] = {1.0, 0.98078528040323044913, 0.92387953251128675613,
                           0.83146961230254523708, 0.70710678118654752440,
                           0.55557023301960222474, 0.38268343236508977173,
                           0.19509032201612826785, 0.0};
  j &= 31;
  if (j > 16) j = 32 - j;
  return j <= 8 ? c[j] : -c[16 - j];
}
__host__ __device__ constexpr double sin32(int j) { return cos32(j + 24); }   // cos(x - pi/2)

// e^{2 pi i S J / 32} = tw_scale(J) i^(S k) (1 + i S t), k the nearest quarter turn and t the tangent of the
// rest, |t| <= 1: tw_tan is the product without the scale, one FMA per component, and the scale goes
// into the FMAs of the additions that follow.  A 4-point DFT with three constant factors so takes 22
// operations instead of 28: 16-point passes 144 and not 160, 8-point ones 52 and not 56.  (A published way
// to fit FFTs to multiply-add units: Linzer and Feig, IEEE Trans. Signal Process. 41, 1993; Goedecker, SIAM J.
// Sci. Comput. 18, 1997.)
__host__ __device__ constexpr int tw_quarter(int J) { return ((J & 31) + 4) >> 3; }
__host__ __device__ constexpr int tw_rest(int J) { return (J & 31) - 8 * tw_quarter(J); }   // -4 .. 3
__host__ __device__ constexpr double tw_scale(int J) { return cos32(tw_rest(J)); }

template <int S, int J, class V> __device__ __forceinline__ V tw_tan(V v) {
  using T = decltype(v.x);
  constexpr int r = tw_rest(J), k = tw_quarter(J) & 3;
  V u = v;
  if constexpr (r == -4) {
    u.x = S > 0 ? v.x + v.y : v.x - v.y;
    u.y = S > 0 ? v.y - v.x : v.y + v.x;
  } else if constexpr (r != 0) {
    constexpr T t = (T)(S * sin32(r) / cos32(r));
    u.x = fma(-t, v.y, v.x);
    u.y = fma(t, v.x, v.y);
  }
  if constexpr (k == 1) return rot<S>(u);
  if constexpr (k == 3) return rot<-S>(u);
  if constexpr (k == 2) {
    u.x = -u.x;
    u.y = -u.y;
  }
  return u;
}
// a + c b with c = 1 as an addition
template <int NUM, int DEN, class V> __device__ __forceinline__ V add_scaled(V a, V b, bool minus) {
  using T = decltype(a.x);
  constexpr double c = tw_scale(NUM) / tw_scale(DEN);
  if constexpr (c == 1.0) return minus ? sub(a, b) : add(a, b);
  else return axpy((T)(minus ? -c : c), b, a);
}
// the 4-point DFT of a, b w^JB, c w^JC, d w^JD (w = e^{2 pi i S / 32})
template <int S, int JB, int JC, int JD, class V> __device__ __forceinline__ void dft4_tw(V& a, V& b, V& c, V& d) {
  const V bp = tw_tan<S, JB>(b), cp = tw_tan<S, JC>(c), dp = tw_tan<S, JD>(d);
  const V s0 = add_scaled<JC, 0>(a, cp, false), d0 = add_scaled<JC, 0>(a, cp, true);
  const V s1 = add_scaled<JD, JB>(bp, dp, false), d1 = rot<S>(add_scaled<JD, JB>(bp, dp, true));
  a = add_scaled<JB, 0>(s0, s1, false);
  b = add_scaled<JB, 0>(d0, d1, false);
  c = add_scaled<JB, 0>(s0, s1, true);
  d = add_scaled<JB, 0>(d0, d1, true);
}

template <int S, class V> __device__ __forceinline__ void dft2(V* v) {
  const V a = v[0];
  v[0] = add(a, v[1]);
  v[1] = sub(a, v[1]);
}
template <int S, class V> __device__ __forceinline__ void dft8(V* v) {
  V u[4], w[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    u[j] = add(v[j], v[j + 4]);
    w[j] = sub(v[j], v[j + 4]);
  }
  dft4<S>(u[0], u[1], u[2], u[3]);
  dft4_tw<S, 4, 8, 12>(w[0], w[1], w[2], w[3]);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    v[2 * j] = u[j];
    v[2 * j + 1] = w[j];
  }
}
// the same with v[4..7] = 0
template <int S, class V> __device__ __forceinline__ void dft8_half(V* v) {
  V u[4] = {v[0], v[1], v[2], v[3]};
  V w[4] = {v[0], v[1], v[2], v[3]};
  dft4<S>(u[0], u[1], u[2], u[3]);
  dft4_tw<S, 4, 8, 12>(w[0], w[1], w[2], w[3]);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    v[2 * j] = u[j];
    v[2 * j + 1] = w[j];
  }
}
// n = 4 n1 + n2, k = k1 + 4 k2
template <int S, bool HALF, class V> __device__ __forceinline__ void dft16(V* v) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if constexpr (HALF) dft4_half<S>(v[j], v[j + 4], v[j + 8], v[j + 12]);
    else dft4<S>(v[j], v[j + 4], v[j + 8], v[j + 12]);
  }
  // now v[4 k1 + n2]; times w16^{n2 k1}
  dft4<S>(v[0], v[1], v[2], v[3]);
  dft4_tw<S, 2, 4, 6>(v[4], v[5], v[6], v[7]);
  dft4_tw<S, 4, 8, 12>(v[8], v[9], v[10], v[11]);
  dft4_tw<S, 6, 12, 18>(v[12], v[13], v[14], v[15]);
  // v[4 k1 + k2] -> X[k1 + 4 k2]
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = a + 1; b < 4; ++b) {
      const V t = v[4 * a + b];
      v[4 * a + b] = v[4 * b + a];
      v[4 * b + a] = t;
    }
}
template <int S, int K1, class V> __device__ __forceinline__ void dft_row32(V* r) {   // times w32^{n2 k1}
  if constexpr (K1 == 0) dft4<S>(r[0], r[1], r[2], r[3]);
  else dft4_tw<S, K1, 2 * K1, 3 * K1>(r[0], r[1], r[2], r[3]);
}
// n = 4 n1 + n2, n1 < 8, k = k1 + 8 k2
template <int S, bool HALF, class V> __device__ __forceinline__ void dft32(V* v) {
  V y[8][4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    V c[8];
#pragma unroll
    for (int a = 0; a < 8; ++a) c[a] = v[4 * a + j];
    if constexpr (HALF) dft8_half<S>(c); else dft8<S>(c);
#pragma unroll
    for (int a = 0; a < 8; ++a) y[a][j] = c[a];
  }
  dft_row32<S, 0>(y[0]);
  dft_row32<S, 1>(y[1]);
  dft_row32<S, 2>(y[2]);
  dft_row32<S, 3>(y[3]);
  dft_row32<S, 4>(y[4]);
  dft_row32<S, 5>(y[5]);
  dft_row32<S, 6>(y[6]);
  dft_row32<S, 7>(y[7]);
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) v[a + 8 * b] = y[a][b];
}
// R points; HALF: v[R/2 .. R-1] = 0 on input
template <int R, int S, bool HALF = false, class V> __device__ __forceinline__ void dft(V* v) {
  if constexpr (R == 2) dft2<S>(v);
  else if constexpr (R == 4) dft4<S>(v[0], v[1], v[2], v[3]);
  else if constexpr (R == 8) dft8<S>(v);
  else if constexpr (R == 16) dft16<S, HALF>(v);
  else dft32<S, HALF>(v);
}

// ---- the plan of one size ----

// M = E x E x M/E^2 points, E per thread: passes of radix E at strides S1 and S2, then of radix R3 at
// stride 1.  E = 16, and 32 at M = 8192.  In FP32 E = 32 at M = 2048, with the last pass by shuffles, has
// a third fewer shared-memory and table accesses, but with 168 registers fewer warps to hide them:
// 2.3 ms against 2.0 ms for 287 100 rows.
template <int LOGM, class T> struct Plan {
  static constexpr int M = 1 << LOGM;
  static constexpr int E = LOGM == 13 ? 32 : 16;
  static constexpr int S1 = M / E, S2 = S1 / E, R3 = S2;
  static constexpr int kT = S1;                        // threads per CTA
  static constexpr int KP = E / S2;                    // third-pass columns per thread
  static constexpr int kSmem = M + M / E;              // elements, padded by one in E
  static_assert(S2 >= 1 && S2 <= 16, "the exchange of passes 2 and 3 stays within a warp");
};
// Element i sits at i + i/E.  The three access patterns split into a thread's base and a constant:
// k S1 + t, g S1 + n3 + j S2 and g S1 + (n3 KP + e) S2 + j (t < S1; n3 < S2, S2 divides E).
template <class P> __device__ __forceinline__ int base1(int t) { return t + t / P::E; }
template <class P> __device__ __forceinline__ constexpr int off1(int k) { return k * (P::S1 + P::S1 / P::E); }
template <class P> __device__ __forceinline__ int base2(int g, int n3) { return g * (P::S1 + P::S1 / P::E) + n3; }
template <class P> __device__ __forceinline__ constexpr int off2(int j) { return j * P::S2 + j * P::S2 / P::E; }
template <class P> __device__ __forceinline__ int base3(int g, int n3) {
  return g * (P::S1 + P::S1 / P::E) + n3 * (P::E + 1);
}
template <class P> __device__ __forceinline__ constexpr int off3(int e, int j) { return e * P::S2 + j; }

template <class P> __device__ __forceinline__ void cta_sync() {
  if constexpr (P::kT <= 32) __syncwarp();
  else __syncthreads();
}

// Tables of one size in global memory: tw1[(k1 - 1) S1 + t] = e^{-2 pi i t k1 / M}, k1 = 1..E-1;
// tw2[(k2 - 1) S2 + j] = e^{-2 pi i j k2 / S1}, k2 = 1..E-1.

// v[j] = x[t + j S1] -> the spectrum in this thread's registers (digit-reversed order)
template <class P, bool HALF, class V>
__device__ __forceinline__ void fft_fwd(V* v, V* sm, const V* __restrict__ tw1, const V* __restrict__ tw2) {
  const int t = threadIdx.x;
  dft<P::E, -1, HALF>(v);
  V* s1 = sm + base1<P>(t);
  s1[0] = v[0];
#pragma unroll
  for (int k = 1; k < P::E; ++k) s1[off1<P>(k)] = mul(v[k], ld_tab(tw1 + (k - 1) * P::S1 + t));
  cta_sync<P>();
  const int g = t / P::S2, n3 = t % P::S2;
  V *s2 = sm + base2<P>(g, n3), *s3 = sm + base3<P>(g, n3);
#pragma unroll
  for (int j = 0; j < P::E; ++j) v[j] = s2[off2<P>(j)];
  dft<P::E, -1>(v);
  s2[0] = v[0];
#pragma unroll
  for (int k = 1; k < P::E; ++k) s2[off2<P>(k)] = mul(v[k], ld_tab(tw2 + (k - 1) * P::S2 + n3));
  __syncwarp();
#pragma unroll
  for (int e = 0; e < P::KP; ++e) {
    V* u = v + e * P::R3;
#pragma unroll
    for (int j = 0; j < P::R3; ++j) u[j] = s3[off3<P>(e, j)];
    dft<P::R3, -1>(u);
  }
}

// the spectrum as fft_fwd leaves it -> v[j] = x[t + j S1] (unscaled inverse); the caller's next
// fft_fwd may follow without a barrier (its first writes go to the places this thread read last)
template <class P, class V>
__device__ __forceinline__ void fft_inv(V* v, V* sm, const V* __restrict__ tw1, const V* __restrict__ tw2) {
  const int t = threadIdx.x;
  const int g = t / P::S2, n3 = t % P::S2;
  V *s1 = sm + base1<P>(t), *s2 = sm + base2<P>(g, n3), *s3 = sm + base3<P>(g, n3);
#pragma unroll
  for (int e = 0; e < P::KP; ++e) {
    V* u = v + e * P::R3;
    dft<P::R3, 1>(u);
#pragma unroll
    for (int j = 0; j < P::R3; ++j) s3[off3<P>(e, j)] = u[j];
  }
  __syncwarp();
  v[0] = s2[0];
#pragma unroll
  for (int k = 1; k < P::E; ++k) v[k] = mulc(s2[off2<P>(k)], ld_tab(tw2 + (k - 1) * P::S2 + n3));
  dft<P::E, 1>(v);
#pragma unroll
  for (int j = 0; j < P::E; ++j) s2[off2<P>(j)] = v[j];
  cta_sync<P>();
  v[0] = s1[0];
#pragma unroll
  for (int k = 1; k < P::E; ++k) v[k] = mulc(s1[off1<P>(k)], ld_tab(tw1 + (k - 1) * P::S1 + t));
  dft<P::E, 1>(v);
}

// x -> x * h (cyclic), filt[e T + t] = spectrum of h over M in the order of fft_fwd's registers
template <class P, bool HALF, class V>
__device__ __forceinline__ void convolve(V* v, V* sm, const V* __restrict__ tw1,
                                         const V* __restrict__ tw2, const V* __restrict__ filt) {
  fft_fwd<P, HALF>(v, sm, tw1, tw2);
#pragma unroll
  for (int e = 0; e < P::E; ++e) v[e] = mul(v[e], ld_tab(filt + e * P::kT + threadIdx.x));
  fft_inv<P>(v, sm, tw1, tw2);
}

// ---- kernels ----

template <class T> struct ChirpArgs {
  const V2<T>* tw1;
  const V2<T>* tw2;
  const V2<T>* filt;     // spectrum of h over M
  const V2<T>* a;        // [n_in] a_{n0 + m} (forward)
  const V2<T>* b;        // [N_k] b_q
  const V2<T>* g;        // Gamma table [n_cls][N_ell][n_h]
  const int* cls_of;
  const T* kw;           // FP64: stencil weights [tracer stride lw_ts][N_k][4]; FP32: kpow mu [N_tr][4][N_k]
  long lw_ts;
  const double* kpow;    // FP64: [N_tr][N_k]
  const int* head;       // FP32 forward: [walker N_tr + tracer] the frequencies below this are in Delta already
  const int* off;        // ragged lists (null: multipoles l_lo .. l_lo + n_l - 1)
  const int* idx;
  int N_tr, NI, n_h, N_k, N_ell, l_lo, n_l, r, n0;
  int n_chunk, n_total, chunk0;   // CTAs of a row: shares chunk0 .. chunk0 + n_chunk - 1 of n_total
};

// FP64: kpow lw; FP32: the product is tabulated
__device__ __forceinline__ double k_weight(const ChirpArgs<double>& A, int i, int s, int q) {
  return A.kpow[(size_t)i * A.N_k + q] * A.kw[(size_t)i * A.lw_ts + (size_t)q * 4 + s];
}
__device__ __forceinline__ float k_weight(const ChirpArgs<float>& A, int i, int s, int q) {
  return __ldg(A.kw + ((size_t)i * 4 + s) * A.N_k + q);
}
__device__ __forceinline__ double2 coef_at(const cplx* p) { return make_double2(p->x, p->y); }
__device__ __forceinline__ float2 coef_at(const float4* p) {
  return *reinterpret_cast<const float2*>(p);   // the high parts of a double-float pair
}

// the multipoles of walker w that this chunk of a row works on: positions [u0, u1) of its list
__device__ __forceinline__ void chunk_range(int n, int n_chunk, int chunk, int& u0, int& u1) {
  u0 = (int)((long)n * chunk / n_chunk);
  u1 = (int)((long)n * (chunk + 1) / n_chunk);
}

// resident threads the registers are cut for: 255 registers in FP64 (one pipe of the SM is the bound)
// and with 32 points per thread, 128 in FP32 with 16 (at 2048 points and many rows 2.0 ms; 2.1 ms with
// 102 registers, 2.3 ms with 168)
template <class T, int LOGM> constexpr int resident_threads() {
  return sizeof(T) == 8 || Plan<LOGM, T>::E == 32 ? 256 : 512;
}
template <class T, int LOGM> constexpr int min_blocks() {
  constexpr int n = resident_threads<T, LOGM>() / Plan<LOGM, T>::kT;
  return n > 32 ? 32 : n > 0 ? n : 1;
}

// Delta[w][l - l_lo][i][q] (+)= sum_s kw_is[q] Re sum_{n >= n0} F_wisn G[l][n] e^{-i eta_n ln k_q}
// FP64 (n0 = 1): the term n = 0, whose phase is 1, is added and Delta is written; FP32 (n0 > 0):
// the terms below head >= n0 are in Delta already.  CT: cplx (FP64) or float4 (double-float pairs, FP32).
template <int LOGM, class T, class CT, bool HALF>
__global__ void __launch_bounds__(Plan<LOGM, T>::kT, min_blocks<T, LOGM>())
k_chirp_fwd(T* __restrict__ delta, const CT* __restrict__ coef, ChirpArgs<T> A) {
  using P = Plan<LOGM, T>;
  using V = V2<T>;
  constexpr bool kDc = sizeof(T) == 8;
  constexpr int NI = HALF ? P::E / 2 : P::E;     // inputs and outputs of a thread
  extern __shared__ __align__(16) unsigned char chirp_sm[];
  V* sm = reinterpret_cast<V*>(chirp_sm);
  const int t = threadIdx.x;
  const int chunk = blockIdx.x % A.n_chunk, wi = blockIdx.x / A.n_chunk;
  const int i = wi % A.N_tr, w = wi / A.N_tr;
  const int lo = A.off ? A.off[w] : 0;
  int u0, u1;
  chunk_range(A.off ? A.off[w + 1] - lo : A.n_l, A.n_total, A.chunk0 + chunk, u0, u1);
  const V* G0 = A.g + (size_t)A.cls_of[i] * A.N_ell * A.n_h;
  const int n_in = A.n_h - A.n0;
  for (int s = 0; s < A.r; ++s) {
    const CT* F = coef + ((size_t)wi * A.NI + s) * A.n_h;
    V f[HALF ? NI : 1], cs[HALF ? NI : 1];
    T km[kDc && HALF ? NI : 1];
    const int m0 = kDc ? 0 : A.head[wi] - A.n0;   // first frequency here, from n0
    if constexpr (HALF) {
#pragma unroll
      for (int e = 0; e < NI; ++e) {
        const int m = t + e * P::S1;
        // (a row's tensor-core rounds end below frequency 256)
        f[e] = m < n_in && (e * P::S1 >= 192 || m >= m0) ? mul(coef_at(F + A.n0 + m), A.a[m]) : mk<T>(0, 0);
        const T k = m < A.N_k ? k_weight(A, i, s, m) : T(0);
        const V b = m < A.N_k ? A.b[m] : mk<T>(0, 0);
        cs[e] = mk<T>(k * b.x, k * b.y);
        if constexpr (kDc) km[e] = k;
      }
    }
    // A row of zeros, as the tangents of all tracers that a perturbation does not touch are, transforms
    // to zeros.  (A NaN compares unequal.)  Forward mode along 8 tangents, two of which move one window
    // each, 15 tracers, 103 multipoles, N = 2048, N_k = 1024: 3935 -> 871 us, and the same 480 us as
    // before where no row is zero.  In FP32 the test costs 3 to 9 % where no row is zero.
    if constexpr (kDc) {
      bool live = false;
      for (int m = t - 1; m < n_in; m += P::kT) {
        const V x = coef_at(F + A.n0 + m);
        live = live || x.x != T(0) || x.y != T(0);
      }
      if (!__syncthreads_or(live)) {
        if (s == 0) {
          for (int u = u0; u < u1; ++u) {
            const int l = A.off ? A.idx[lo + u] : A.l_lo + u;
            T* out = delta + (((size_t)w * A.n_l + (l - A.l_lo)) * A.N_tr + i) * A.N_k;
            for (int q = t; q < A.N_k; q += P::kT) out[q] = T(0);
          }
        }
        continue;
      }
    }
    for (int u = u0; u < u1; ++u) {
      const int l = A.off ? A.idx[lo + u] : A.l_lo + u;
      const V* G = G0 + (size_t)l * A.n_h + A.n0;
      V v[P::E];
#pragma unroll
      for (int e = 0; e < NI; ++e) {
        const int m = t + e * P::S1;
        if constexpr (HALF) {
          v[e] = m < n_in ? mul(f[e], __ldg(G + m)) : mk<T>(0, 0);
        } else {
          v[e] = m >= m0 && m < n_in ? mul(mul(coef_at(F + A.n0 + m), A.a[m]), __ldg(G + m)) : mk<T>(0, 0);
        }
      }
#pragma unroll
      for (int e = NI; e < P::E; ++e) v[e] = mk<T>(0, 0);
      T dc = 0;
      if constexpr (kDc) {
        const V f0 = coef_at(F), g0 = __ldg(G - 1);
        dc = fma(f0.x, g0.x, -f0.y * g0.y);
      }
      convolve<P, HALF>(v, sm, A.tw1, A.tw2, A.filt);
      T* out = delta + (((size_t)w * A.n_l + (l - A.l_lo)) * A.N_tr + i) * A.N_k;
#pragma unroll
      for (int e = 0; e < NI; ++e) {
        const int q = t + e * P::S1;
        if (q < A.N_k) {
          T x;
          if constexpr (HALF) {
            x = fma(v[e].x, cs[e].x, -v[e].y * cs[e].y);
            if constexpr (kDc) x = fma(km[e], dc, x);
          } else {
            const V b = A.b[q];
            x = fma(v[e].x, b.x, -v[e].y * b.y);
            if constexpr (kDc) x += dc;
            x *= k_weight(A, i, s, q);
          }
          if (kDc && s == 0) out[q] = x;
          else out[q] += x;
        }
      }
    }
  }
}

// The transpose: part[chunk][(w, i, s)][n] = sum over the multipoles of share chunk0 + chunk of
// G[l][n] sum_q [kw_is[q] Dbar_i(l, q) b_q] h_{n - q}  (n0 = 0); the chunks are added in FP64 by
// k_chirp_sum.
template <int LOGM, class T, bool HALF>
__global__ void __launch_bounds__(Plan<LOGM, T>::kT, min_blocks<T, LOGM>())
k_chirp_adj(V2<T>* __restrict__ part, const T* __restrict__ dbar, ChirpArgs<T> A) {
  using P = Plan<LOGM, T>;
  using V = V2<T>;
  constexpr int NI = HALF ? P::E / 2 : P::E;         // inputs of a thread
  constexpr int NO = HALF ? P::E / 2 + 1 : P::E;     // outputs (n_h <= M/2 + 1)
  extern __shared__ __align__(16) unsigned char chirp_sm[];
  V* sm = reinterpret_cast<V*>(chirp_sm);
  const int t = threadIdx.x;
  const int chunk = blockIdx.x % A.n_chunk, wi = blockIdx.x / A.n_chunk;
  const int i = wi % A.N_tr, w = wi / A.N_tr;
  const int lo = A.off ? A.off[w] : 0;
  int u0, u1;
  chunk_range(A.off ? A.off[w + 1] - lo : A.n_l, A.n_total, A.chunk0 + chunk, u0, u1);
  const V* G0 = A.g + (size_t)A.cls_of[i] * A.N_ell * A.n_h;
  const size_t rows = (size_t)(gridDim.x / A.n_chunk) * A.r;
  for (int s = 0; s < A.r; ++s) {
    V cs[HALF ? NI : 1];
    if constexpr (HALF) {
#pragma unroll
      for (int e = 0; e < NI; ++e) {
        const int q = t + e * P::S1;
        const T k = q < A.N_k ? k_weight(A, i, s, q) : T(0);
        const V b = q < A.N_k ? A.b[q] : mk<T>(0, 0);
        cs[e] = mk<T>(k * b.x, k * b.y);
      }
    }
    V acc[NO];
#pragma unroll
    for (int e = 0; e < NO; ++e) acc[e] = mk<T>(0, 0);
    for (int u = u0; u < u1; ++u) {
      const int l = A.off ? A.idx[lo + u] : A.l_lo + u;
      const T* d = dbar + (((size_t)w * A.n_l + (l - A.l_lo)) * A.N_tr + i) * A.N_k;
      V v[P::E];
#pragma unroll
      for (int e = 0; e < NI; ++e) {
        const int q = t + e * P::S1;
        const T x = q < A.N_k ? d[q] : T(0);
        if constexpr (HALF) {
          v[e] = mk<T>(x * cs[e].x, x * cs[e].y);
        } else {
          const V b = q < A.N_k ? A.b[q] : mk<T>(0, 0);
          const T k = q < A.N_k ? x * k_weight(A, i, s, q) : T(0);
          v[e] = mk<T>(k * b.x, k * b.y);
        }
      }
#pragma unroll
      for (int e = NI; e < P::E; ++e) v[e] = mk<T>(0, 0);
      convolve<P, HALF>(v, sm, A.tw1, A.tw2, A.filt);
      const V* G = G0 + (size_t)l * A.n_h;
#pragma unroll
      for (int e = 0; e < NO; ++e) {
        const int n = t + e * P::S1;
        if (n < A.n_h) {
          const V g = __ldg(G + n);
          acc[e].x = fma(v[e].x, g.x, fma(-v[e].y, g.y, acc[e].x));
          acc[e].y = fma(v[e].x, g.y, fma(v[e].y, g.x, acc[e].y));
        }
      }
    }
    V* out = part + ((size_t)chunk * rows + (size_t)wi * A.r + s) * A.n_h;
#pragma unroll
    for (int e = 0; e < NO; ++e) {
      const int n = t + e * P::S1;
      if (n < A.n_h) out[n] = acc[e];
    }
  }
}

// cbar[(w, i, s)][n] (+)= conj(a_n sum_chunk part[chunk][(w, i, s)][n]); rows s >= r
// (padding of the profile rows) are zeros.  Grid: rows x (n_h / 32); thread (n, group) adds the
// chunks group, group + 8, ... in order, then the eight groups are added in order, so that a row's
// hundred or so chunks are not one serial chain of loads.
//
// FP64 parts are added in FP64.  FP32 parts are added in pairs of FP32 values (TwoSum: the rounding of
// every addition is carried in the second one), which hold 48 bits of the sum; widening each part
// to FP64 first was bound by the FP64 pipe: 256 walkers of 15 rows 452 -> 186 us, 30 rows of 2049 values
// 166 -> 42 us, 15 rows 7.8 -> 3.9 us.  Where a pair leaves the range of FP32, the sum is
// repeated in FP64.
constexpr int kSumN = 32, kSumG = 8;
template <class T> struct SumAcc;
template <> struct SumAcc<double> {
  double2 s;
  __device__ __forceinline__ void zero() { s = make_double2(0.0, 0.0); }
  __device__ __forceinline__ void add(double2 v) { s.x += v.x; s.y += v.y; }
  __device__ __forceinline__ void join(const SumAcc& o) { add(o.s); }
  __device__ __forceinline__ double2 value() const { return s; }
};
template <> struct SumAcc<float> {
  float2 s, c;
  __device__ __forceinline__ void zero() { s = c = make_float2(0.f, 0.f); }
  __device__ __forceinline__ void add(float2 v) {
    const float2 sn = chirp::add(s, v), bp = sub(sn, s);
    c = chirp::add(c, chirp::add(sub(s, sub(sn, bp)), sub(v, bp)));
    s = sn;
  }
  __device__ __forceinline__ void join(const SumAcc& o) { add(o.s); c = chirp::add(c, o.c); }
  __device__ __forceinline__ double2 value() const {
    return make_double2((double)s.x + (double)c.x, (double)s.y + (double)c.y);
  }
};
template <class T>
__global__ void __launch_bounds__(kSumN * kSumG)
k_chirp_sum(cplx* __restrict__ cbar, const V2<T>* __restrict__ part, const double2* __restrict__ a,
            int n_rows, int NI, int r, int n_h, int n_chunk, bool accumulate) {
  __shared__ SumAcc<T> red[kSumG][kSumN];
  const int nb = (n_h + kSumN - 1) / kSumN;
  const int nl = threadIdx.x % kSumN, grp = threadIdx.x / kSumN;
  const int n = (blockIdx.x % nb) * kSumN + nl;
  const int row = blockIdx.x / nb, wi = row / NI, s = row % NI;
  const size_t per = (size_t)n_rows * r * n_h;
  const V2<T>* p = part + ((size_t)wi * r + s) * n_h + n;
  SumAcc<T> x;
  x.zero();
  if (n < n_h && s < r) {
#pragma unroll 4
    for (int c = grp; c < n_chunk; c += kSumG) x.add(p[(size_t)c * per]);
  }
  red[grp][nl] = x;
  __syncthreads();
  if (grp || n >= n_h) return;
  const int ng = min(kSumG, n_chunk);
#pragma unroll
  for (int g = 1; g < kSumG; ++g)
    if (g < ng) x.join(red[g][nl]);
  cplx* out = cbar + (size_t)row * n_h + n;
  if (s >= r) {
    if (!accumulate) *out = {0.0, 0.0};
    return;
  }
  double2 v = x.value();
  if constexpr (sizeof(T) == 4) {
    if (!(isfinite(x.s.x) && isfinite(x.s.y) && isfinite(x.c.x) && isfinite(x.c.y))) {
      v = make_double2(0.0, 0.0);
      for (int c = 0; c < n_chunk; ++c) {
        const V2<T> u = p[(size_t)c * per];
        v.x += (double)u.x;
        v.y += (double)u.y;
      }
    }
  }
  const double2 f = a[n];
  cplx o = {fma(v.x, f.x, -v.y * f.y), -fma(v.x, f.y, v.y * f.x)};
  if (accumulate) { o.x += out->x; o.y += out->y; }
  *out = o;
}

// ---- tables ----

// e^{2 pi i S f}, f = frac(n (ch + cl)) with the product's rounding error kept
__device__ __forceinline__ double dd_cycles(double n, double ch, double cl) {
  const double p = n * ch;
  return (p - rint(p)) + fma(n, ch, -p) + n * cl;
}
__device__ __forceinline__ double2 unit(double cycles) {
  double s, c;
  sincospi(2.0 * cycles, &s, &c);
  return make_double2(c, s);
}
template <class T> __device__ __forceinline__ V2<T> cast2(double2 v) { return mk<T>((T)v.x, (T)v.y); }

// tw1, tw2 of the plan, a_{n0 + m} (m < n_in, type TA) and b_q (q < N_k).  cc = d/(2 L) and
// xx = x0/L in double-double: beta m^2/2 = 2 pi cc m^2 and eta_n x0 = 2 pi n xx.
template <int LOGM, class T, class TA>
__global__ void k_chirp_tables(V2<T>* __restrict__ tw1, V2<T>* __restrict__ tw2, V2<TA>* __restrict__ a,
                               V2<T>* __restrict__ b, int n0, int n_in, int N_k, double2 cc, double2 xx) {
  using P = Plan<LOGM, T>;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < (P::E - 1) * P::S1) {
    const long k1 = e / P::S1 + 1, t = e % P::S1;
    tw1[e] = cast2<T>(unit(-(double)((k1 * t) & (P::M - 1)) / P::M));
  }
  if (e < (P::E - 1) * P::S2) {
    const int k2 = e / P::S2 + 1, j = e % P::S2;
    tw2[e] = cast2<T>(unit(-(double)((k2 * j) & (P::S1 - 1)) / P::S1));
  }
  if (e < n_in) {
    const double m = e, n = n0 + e;
    a[e] = cast2<TA>(unit(-(dd_cycles(n, xx.x, xx.y) + dd_cycles(m * m, cc.x, cc.y))));
  }
  if (e < N_k) {
    const double q = e;
    b[e] = cast2<T>(unit(-dd_cycles(q * q + 2.0 * n0 * q, cc.x, cc.y)));
  }
}

// spectrum of h_t/M, t = -t_lo .. t_hi (t_lo + t_hi < M, the rest zero), in FP64, one CTA
template <int LOGM, class T>
__global__ void __launch_bounds__(Plan<LOGM, T>::kT)
k_chirp_filter(V2<T>* __restrict__ filt, int t_lo, int t_hi, double2 cc, const double2* __restrict__ tw1,
               const double2* __restrict__ tw2) {
  using P = Plan<LOGM, T>;   // T's order of the spectrum
  extern __shared__ __align__(16) unsigned char chirp_sm[];
  double2 v[P::E];
#pragma unroll
  for (int e = 0; e < P::E; ++e) {
    const int p = threadIdx.x + e * P::S1;
    const int x = p <= t_hi ? p : p - P::M;
    v[e] = make_double2(0.0, 0.0);
    if (x >= -t_lo) {
      v[e] = unit(dd_cycles((double)x * x, cc.x, cc.y));
      v[e].x *= 1.0 / P::M;
      v[e].y *= 1.0 / P::M;
    }
  }
  fft_fwd<P, false>(v, reinterpret_cast<double2*>(chirp_sm), tw1, tw2);
#pragma unroll
  for (int e = 0; e < P::E; ++e) filt[e * P::kT + threadIdx.x] = cast2<T>(v[e]);
}

// tw1 and tw2 of T's plan in FP64, for the filter
template <int LOGM, class T>
__global__ void k_chirp_twiddles64(double2* __restrict__ tw1, double2* __restrict__ tw2) {
  using P = Plan<LOGM, T>;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < (P::E - 1) * P::S1) tw1[e] = unit(-(double)(((long)(e / P::S1 + 1) * (e % P::S1)) & (P::M - 1)) / P::M);
  if (e < (P::E - 1) * P::S2) tw2[e] = unit(-(double)((e / P::S2 + 1) * (e % P::S2) & (P::S1 - 1)) / P::S1);
}

// ---- host side of one precision (instantiated in chirp_f64.cu and chirp_f32.cu) ----

template <int LOGM, class T> constexpr size_t smem_bytes(size_t elem = sizeof(V2<T>)) {
  return elem * Plan<LOGM, T>::kSmem;
}

template <class F> cudaError_t with_smem(F kern, size_t smem) {
  return smem > 48 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                          : cudaSuccess;
}

// Elements of a direction's tables: tw1 and tw2 (FP64 ones first, for the filter), filt, b, a
struct TabLayout {
  size_t tw1d, tw2d, tw1, tw2, filt, b, a, bytes;
};
template <class T> TabLayout tab_layout(int logm, int n_in, int N_k, size_t a_elem) {
  const size_t M = (size_t)1 << logm;   // tw1 and tw2 hold fewer than M values each
  TabLayout L;
  size_t o = 0;
  auto put = [&](size_t bytes) { const size_t at = o; o += (bytes + 255) & ~size_t(255); return at; };
  L.tw1d = put(16 * M);
  L.tw2d = put(16 * M / 16);
  L.tw1 = sizeof(T) == 8 ? L.tw1d : put(8 * M);
  L.tw2 = sizeof(T) == 8 ? L.tw2d : put(8 * M / 16);
  L.filt = put(sizeof(V2<T>) * M);
  L.b = put(sizeof(V2<T>) * N_k);
  L.a = put(a_elem * n_in);
  L.bytes = o;
  return L;
}

template <int LOGM, class T, class TA>
cudaError_t build_tables(uint8_t* p, const TabLayout& L, int n0, int n_in, int N_k, int t_lo, int t_hi,
                         double2 cc, double2 xx, cudaStream_t s) {
  using P = Plan<LOGM, T>;
  const int n = std::max({P::M, n_in, N_k});
  const unsigned grid = (unsigned)((n + 255) / 256);
  double2 *tw1d = (double2*)(p + L.tw1d), *tw2d = (double2*)(p + L.tw2d);
  k_chirp_tables<LOGM, T, TA><<<grid, 256, 0, s>>>((V2<T>*)(p + L.tw1), (V2<T>*)(p + L.tw2), (V2<TA>*)(p + L.a),
                                                   (V2<T>*)(p + L.b), n0, n_in, N_k, cc, xx);
  if (sizeof(T) == 4) k_chirp_twiddles64<LOGM, T><<<grid, 256, 0, s>>>(tw1d, tw2d);
  const size_t smem = smem_bytes<LOGM, T>(sizeof(double2));
  cudaError_t e = with_smem(k_chirp_filter<LOGM, T>, smem);
  if (e != cudaSuccess) return e;
  k_chirp_filter<LOGM, T><<<1, P::kT, smem, s>>>((V2<T>*)(p + L.filt), t_lo, t_hi, cc, tw1d, tw2d);
  return cudaGetLastError();
}

template <class T, class F> cudaError_t by_size(int logm, F f) {
  switch (logm) {
    case 9: return f(std::integral_constant<int, 9>());
    case 10: return f(std::integral_constant<int, 10>());
    case 11: return f(std::integral_constant<int, 11>());
    case 12: return f(std::integral_constant<int, 12>());
    case 13: return f(std::integral_constant<int, 13>());
    default: return cudaErrorInvalidValue;
  }
}

template <class T, class CT>
cudaError_t launch_fwd(int logm, bool half, T* delta, const CT* coef, const ChirpArgs<T>& A, int n_rows,
                       cudaStream_t s) {
  return by_size<T>(logm, [&](auto lm) {
    constexpr int LM = decltype(lm)::value;
    auto kern = half ? k_chirp_fwd<LM, T, CT, true> : k_chirp_fwd<LM, T, CT, false>;
    constexpr size_t smem = smem_bytes<LM, T>();
    cudaError_t e = with_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((long)n_rows * A.n_chunk), Plan<LM, T>::kT, smem, s>>>(delta, coef, A);
    return cudaGetLastError();
  });
}
template <class T>
cudaError_t launch_adj(int logm, bool half, V2<T>* part, const T* dbar, const ChirpArgs<T>& A, int n_rows,
                       cudaStream_t s) {
  return by_size<T>(logm, [&](auto lm) {
    constexpr int LM = decltype(lm)::value;
    auto kern = half ? k_chirp_adj<LM, T, true> : k_chirp_adj<LM, T, false>;
    constexpr size_t smem = smem_bytes<LM, T>();
    cudaError_t e = with_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((long)n_rows * A.n_chunk), Plan<LM, T>::kT, smem, s>>>(part, dbar, A);
    return cudaGetLastError();
  });
}

}  // namespace chirp
}  // namespace swcl
