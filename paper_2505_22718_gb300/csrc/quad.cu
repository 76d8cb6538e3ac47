// a4: the k-quadrature of Eq. 2.1, C_l^{ij} = A_i A_j sum_q u_q Delta_i(l,q) Delta_j(l,q),
// u_q = wk2[q] P(k_q), and the reductions of its reverse mode (a5):
//   Pbar_q   = wk2[q] sum_l sum_i A_i Delta_i T_i,   T_i = sum_j S_ij A_j Delta_j,
//   Dbar_i   = 2 A_i u_q T_i,
//   Abar_i   = 2 sum_l sum_j S_ij A_j U_ij            (U = C at unit amplitudes),
// with S = (Cbar + Cbar^T)/2 (zero for multipoles outside a walker's list).
//
// The unit-amplitude spectra U of the FP64 form are formed in two passes: partial sums of each
// unordered pair (i <= j) over chunks of 256 k points (one CTA per multipole and chunk), then the
// chunks added in a fixed order and written to both (i,j) and (j,i), so C is symmetric bit for
// bit and the same from run to run.  Delta in FP32 (mixed paths) goes through k_quad_blocks or
// k_quad_stream below: FP32 products, compensated FP32 sums (TwoSum; the rounding of each addition carried in
// a second float), FP64 above them.
#include <algorithm>

#include "f32x2.cuh"
#include "tc_common.cuh"
#include "swcl_internal.h"

namespace swcl {
namespace {

constexpr int QT = 256;    // threads
constexpr int KC = 256;    // k points per CTA (one partial sum per pair and chunk)
constexpr int KS = KC + 1; // shared row stride: lanes reading rows j at the same k point fall in
                           // different banks
static_assert(QT == KC, "k_quad_part stages one k point per thread");

// Partial pair sums over one chunk of KC k points: part[w][l - l_lo][kc][p] for unordered pairs
// p = (i <= j).  Grid (multipole, k chunk, walker).  Thread t handles pair p = t % npair for the
// k points t / npair, t / npair + G, ... of the chunk (G = QT / npair groups); groups are combined
// in shared memory in a fixed order.
//
// Bound by the FP64 pipe (two FMA per clock and SM): Delta_i u is formed once per row and k point and staged
// beside Delta (SCALED), which leaves one FMA per pair instead of a product and an FMA.  103 multipoles, 15
// tracers, 1024 k points, alone on the GPU: 60 -> 33 us.  Above 55 tracers both do not fit
// the shared memory and the product is formed per pair.
template <bool SCALED>
__global__ void __launch_bounds__(QT)
k_quad_part(double* __restrict__ part, const double* __restrict__ delta, const double* __restrict__ P,
            const double* __restrict__ wk2, int N_tr, int N_k, int n_l, int n_kc) {
  extern __shared__ double qsm[];
  double* Ds = qsm;                               // [N_tr][KS]
  double* Es = qsm + (SCALED ? N_tr * KS : 0);    // [N_tr][KS] Delta u
  __shared__ double us[KC];
  __shared__ double red[QT];
  const int ll = blockIdx.x, kc = blockIdx.y, w = blockIdx.z;
  const int q0 = kc * KC;
  const int npair = N_tr * (N_tr + 1) / 2;
  const double* dl = delta + ((size_t)w * n_l + ll) * N_tr * N_k;
  {
    // one k point per thread (QT == KC); the rows' loads are unrolled so that several are in
    // flight at once
    const int qq = threadIdx.x, q = q0 + qq;
    const double u = q < N_k ? wk2[q] * P[(size_t)w * N_k + q] : 0.0;
    if constexpr (!SCALED) us[qq] = u;
#pragma unroll 8
    for (int t = 0; t < N_tr; ++t) {
      const double d = q < N_k ? dl[(size_t)t * N_k + q] : 0.0;
      Ds[t * KS + qq] = d;
      if constexpr (SCALED) Es[t * KS + qq] = d * u;
    }
  }
  __syncthreads();
  const int ngroups = max(1, QT / npair);
  double* out = part + (((size_t)w * n_l + ll) * n_kc + kc) * npair;
  for (int p0 = 0; p0 < npair; p0 += QT) {
    const int p = p0 + (ngroups > 1 ? threadIdx.x % npair : threadIdx.x);
    const int group = ngroups > 1 ? threadIdx.x / npair : 0;
    const bool active = p < npair && group < ngroups;
    double acc = 0.0;
    if (active) {
      int r = p, i = 0;                           // unordered pair index -> (i <= j)
      while (r >= N_tr - i) { r -= N_tr - i; ++i; }
      const int j = i + r;
      const double* di = Es + i * KS;
      const double* dj = Ds + j * KS;
#pragma unroll 4
      for (int qq = group; qq < KC; qq += ngroups)
        acc = fma(SCALED ? di[qq] : di[qq] * us[qq], dj[qq], acc);
    }
    if (ngroups > 1) {
      red[threadIdx.x] = acc;
      __syncthreads();
      if (active && group == 0) {
        double s2 = acc;
        for (int g = 1; g < ngroups; ++g) s2 += red[g * npair + threadIdx.x];
        out[p] = s2;
      }
      __syncthreads();
    } else if (active) {
      out[p] = acc;
    }
  }
}

// U[w][l][i][j] = U[w][l][j][i] = sum over the k chunks of the pair's partial sums (in order)
__global__ void k_quad_reduce(double* __restrict__ U, const double* __restrict__ part, int N_tr,
                              int N_ell, int l_lo, int n_l, int n_kc, int n_walk) {
  const int npair = N_tr * (N_tr + 1) / 2;
  const long total = (long)n_walk * n_l * npair;
  for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
    const int p = (int)(e % npair);
    const long wl = e / npair;                       // w * n_l + ll
    const int ll = (int)(wl % n_l), w = (int)(wl / n_l);
    const double* src = part + (size_t)wl * n_kc * npair + p;
    double s = 0.0;
    for (int kc = 0; kc < n_kc; ++kc) s += src[(size_t)kc * npair];
    int r = p, i = 0;
    while (r >= N_tr - i) { r -= N_tr - i; ++i; }
    const int j = i + r;
    double* u = U + ((size_t)w * N_ell + l_lo + ll) * N_tr * N_tr;
    u[i * N_tr + j] = s;
    u[j * N_tr + i] = s;
  }
}

// ---- FP32 form: register blocks of 4 x 4 tracer pairs ----
//
// Delta rows lie in shared memory as in global memory ([tracer][k], rows padded to a multiple of four
// tracers with zeros), brought by asynchronous 16-byte copies, and u = wk2 P in FP32.  A warp takes
// the block of pairs (4 ib .. 4 ib + 3) x (4 jb .. 4 jb + 3), ib <= jb; lane l takes the k points
// l, l + 32, ... (consecutive lanes read consecutive words: no bank conflicts).  Per k point a lane
// forms a_i = Delta_i u (four products, rounded as in the two-pass form) and sixteen products a_i Delta_j;
// after every four points the block sums go into compensated (TwoSum) accumulators.  The 32 lanes are
// then combined by a butterfly that halves the pairs each lane holds at every step (each combination a
// TwoSum), so lane pair (2p, 2p + 1) ends with pair p of the block.  The order of every addition is
// fixed: the result is the same from run to run.
//
// Two kernels.  k_quad_blocks: one CTA per (multipole, k chunk, walker) with all its copies in flight at
// once; with one chunk the sum, widened to FP64, is U itself (both triangles); with several, the
// per-chunk sums go through the chunk reduction of the FP64 form.  k_quad_stream, where many rows of more
// than ten blocks need several chunks each: resident CTAs that stream the rows through a ring of stages,
// so that the next rows arrive while a block is summed, combined and written, and the lanes are combined
// once per row instead of once per chunk.  30 tracers, 2999 multipoles, 4096 k: 1842 us and 80 us for the
// chunk reduction with one CTA per row and chunk, 1494 us so.  Packed FP32 (two points per instruction)
// took as long and spilled; 30 warps with 64 registers instead of 20 with 96 took 2460 us.
constexpr int QB_MAX_WARPS = 20;             // per SM, 96 registers each
constexpr int QB_SMEM = 100 * 1024;          // staged rows per CTA at most (2 CTAs per SM)

__device__ __forceinline__ void qb_two_sum(float& s, float& c, float b) {
  const float sn = s + b;
  const float bp = sn - s;
  c += (s - (sn - bp)) + (b - bp);
  s = sn;
}

// (s, c) += (rs, rc): the sums' rounding error from TwoSum, the compensations added
__device__ __forceinline__ void qb_combine(float& s, float& c, float rs, float rc) {
  const float sn = s + rs;
  const float bp = sn - s;
  const float e = (s - (sn - bp)) + (rs - bp);
  c = (c + rc) + e;
  s = sn;
}

// one butterfly step: lanes with (lane & OFF) keep the upper half of their H pairs
template <int H, int OFF>
__device__ __forceinline__ void qb_scatter_step(float* s, float* c, int lane) {
  const bool up = lane & OFF;
#pragma unroll
  for (int p = 0; p < H; ++p) {
    const float keep_s = up ? s[p + H] : s[p], keep_c = up ? c[p + H] : c[p];
    const float ss = up ? s[p] : s[p + H], sc = up ? c[p] : c[p + H];
    const float rs = __shfl_xor_sync(0xffffffffu, ss, OFF);
    const float rc = __shfl_xor_sync(0xffffffffu, sc, OFF);
    s[p] = keep_s;
    c[p] = keep_c;
    qb_combine(s[p], c[p], rs, rc);
  }
}

// One group of up to 128 k points of a block: n = 64 or 128; ra, rb and ru are at this lane's first point
__device__ __forceinline__ void qb_group(float* s, float* c, const float* ra, const float* rb, const float* ru,
                                         int pitch, int n) {
  float bs[16];
#pragma unroll
  for (int k = 0; k < 128; k += 32) {
    if (k == 64 && n <= 64) break;
    const float u = ru[k];
    float ai[4], dj[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      ai[x] = ra[x * pitch + k] * u;
      dj[x] = rb[x * pitch + k];
    }
#pragma unroll
    for (int p = 0; p < 16; ++p) bs[p] = k == 0 ? ai[p >> 2] * dj[p & 3] : fmaf(ai[p >> 2], dj[p & 3], bs[p]);
  }
#pragma unroll
  for (int p = 0; p < 16; ++p) qb_two_sum(s[p], c[p], bs[p]);
}

// The 32 lanes' sums of a block's sixteen pairs -> pair lane / 2
__device__ __forceinline__ float2 qb_lanes(float* s, float* c, int lane) {
  qb_scatter_step<8, 16>(s, c, lane);
  qb_scatter_step<4, 8>(s, c, lane);
  qb_scatter_step<2, 4>(s, c, lane);
  qb_scatter_step<1, 2>(s, c, lane);
  const float os = __shfl_xor_sync(0xffffffffu, s[0], 1), oc = __shfl_xor_sync(0xffffffffu, c[0], 1);
  qb_combine(s[0], c[0], os, oc);
  return make_float2(s[0], c[0]);
}

// block b -> (ib <= jb)
__device__ __forceinline__ void qb_block(int b, int n_ib, int& ib, int& jb) {
  ib = 0;
  while (b >= n_ib - ib) { b -= n_ib - ib; ++ib; }
  jb = ib + b;
}

__global__ void __launch_bounds__(QB_MAX_WARPS * 32, 1)
k_quad_blocks(double* __restrict__ U, double* __restrict__ part, const float* __restrict__ delta,
              const double* __restrict__ P, const double* __restrict__ wk2, int N_tr, int N_k,
              int N_ell, int l_lo, int n_l, int kcap, int n_kc, int ks, bool vec4,
              const int* __restrict__ listed) {
  extern __shared__ float4 qb_smv[];
  float* qb_sm = reinterpret_cast<float*>(qb_smv);
  const int ll = blockIdx.x, kc = blockIdx.y, w = blockIdx.z;
  const int n_ib = (N_tr + 3) / 4, nb = n_ib * (n_ib + 1) / 2;
  const int npair = N_tr * (N_tr + 1) / 2;
  const int q0 = kc * kcap;
  const int nk = min(kcap, N_k - q0);
  const int nk64 = (nk + 63) & ~63;
  double* Uw = U + ((size_t)w * N_ell + l_lo + ll) * N_tr * N_tr;
  double* pw = part + (((size_t)w * n_l + ll) * n_kc + kc) * npair;
  if (listed && listed[w * n_l + ll] < 0) {
    // a multipole the walker does not list: zero sums (its Delta rows are not read)
    if (n_kc == 1)
      for (int e = threadIdx.x; e < N_tr * N_tr; e += blockDim.x) Uw[e] = 0.0;
    else
      for (int e = threadIdx.x; e < npair; e += blockDim.x) pw[e] = 0.0;
    return;
  }
  const int rows = 4 * n_ib;
  float* Ds = qb_sm;                                            // [rows][kcap]
  float* us = qb_sm + (size_t)rows * kcap;                      // [kcap]
  const float* dl = delta + ((size_t)w * n_l + ll) * N_tr * N_k + q0;
  if (vec4) {
    // rows start on 16-byte boundaries (N_k and q0 multiples of 4): 16-byte copies, the part of
    // a group past the chunk's end (and every padding row) filled with zeros by the copy itself
    const int ng = nk64 >> 2;
    for (int e = threadIdx.x; e < rows * ng; e += blockDim.x) {
      const int t = e / ng, gq = e - t * ng;
      const int left = nk - 4 * gq;
      const int bytes = t < N_tr ? (left >= 4 ? 16 : left > 0 ? 4 * left : 0) : 0;
      const float* src = bytes ? dl + (size_t)t * N_k + 4 * gq : dl;
      const unsigned dst = (unsigned)__cvta_generic_to_shared(Ds + (size_t)t * kcap + 4 * gq);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
                   "r"(bytes) : "memory");
    }
  } else {
    for (int e = threadIdx.x; e < rows * nk64; e += blockDim.x) {
      const int t = e / nk64, kk = e - t * nk64;
      const int bytes = t < N_tr && kk < nk ? 4 : 0;
      const float* src = bytes ? dl + (size_t)t * N_k + kk : dl;
      const unsigned dst = (unsigned)__cvta_generic_to_shared(Ds + (size_t)t * kcap + kk);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src),
                   "r"(bytes) : "memory");
    }
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  for (int kk = threadIdx.x; kk < nk64; kk += blockDim.x)
    us[kk] = kk < nk ? (float)(wk2[q0 + kk] * P[(size_t)w * N_k + q0 + kk]) : 0.0f;
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  // warp wi: k part h = wi / wb of ks, blocks bw, bw + wb, ... (bw = wi % wb); part h takes the
  // 64-point groups [h n64 / ks, (h + 1) n64 / ks) of the chunk
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int wb = (blockDim.x >> 5) / ks, h = wi / wb, bw = wi - h * wb;
  const int n64 = nk64 >> 6;
  const int k_lo = 64 * (h * n64 / ks), k_hi = 64 * ((h + 1) * n64 / ks);
  float2* red = reinterpret_cast<float2*>(us + kcap);         // [ks][nb][16] (sum, compensation)
  for (int b = bw; b < nb && h < ks; b += wb) {
    int ib, jb;
    qb_block(b, n_ib, ib, jb);
    const float* ra = Ds + (size_t)(4 * ib) * kcap + lane;
    const float* rb = Ds + (size_t)(4 * jb) * kcap + lane;
    const float* ru = us + lane;
    float s2[16], c2[16];
#pragma unroll
    for (int p = 0; p < 16; ++p) s2[p] = c2[p] = 0.0f;
    for (int g0 = k_lo; g0 < k_hi; g0 += 128) qb_group(s2, c2, ra + g0, rb + g0, ru + g0, kcap, k_hi - g0);
    const float2 t = qb_lanes(s2, c2, lane);
    if (!(lane & 1)) red[((size_t)h * nb + b) * 16 + (lane >> 1)] = t;
  }
  __syncthreads();
  // the k parts of each pair, added in order; pair p of block b is (4 ib + p / 4, 4 jb + p % 4)
  for (int e = threadIdx.x; e < nb * 16; e += blockDim.x) {
    const int b = e >> 4, p = e & 15;
    int ib, jb;
    qb_block(b, n_ib, ib, jb);
    const int i = 4 * ib + (p >> 2), j = 4 * jb + (p & 3);
    if (i >= N_tr || j >= N_tr || i > j) continue;
    float2 t = red[e];
    for (int hh = 1; hh < ks; ++hh) {
      const float2 o = red[(size_t)hh * nb * 16 + e];
      qb_combine(t.x, t.y, o.x, o.y);
    }
    const double v = (double)t.x + (double)t.y;
    if (n_kc == 1) {
      Uw[i * N_tr + j] = v;
      Uw[j * N_tr + i] = v;
    } else {
      pw[i * N_tr - i * (i - 1) / 2 + (j - i)] = v;
    }
  }
}

// Items (walker, multipole, part of the blocks), an equal share of consecutive ones per CTA.  A part's
// blocks have a warp each; their accumulators live over all the k points of a row.
constexpr int QS_RING = 4;                   // stages; three are in flight while one is summed
constexpr int QS_MAX_K = 8192;               // u of all k points stays in shared memory
__global__ void __launch_bounds__(QB_MAX_WARPS * 32, 1)
k_quad_stream(double* __restrict__ U, const float* __restrict__ delta, const double* __restrict__ P,
              const double* __restrict__ wk2, int N_tr, int N_k, int N_ell, int l_lo, int n_l, int n_walk,
              int n_part, int nbp, int lg_sk, bool vec4) {
  extern __shared__ float4 qb_smv[];
  const int n_ib = (N_tr + 3) / 4, nb = n_ib * (n_ib + 1) / 2, rows = 4 * n_ib;
  const int sk = 1 << lg_sk, n_st = (N_k + sk - 1) >> lg_sk, nk64 = (N_k + 63) & ~63;
  float* ring = reinterpret_cast<float*>(qb_smv);               // [QS_RING][rows][sk]
  float* us = ring + (size_t)QS_RING * rows * sk;               // [nk64]
  const int lane = threadIdx.x & 31, bw = threadIdx.x >> 5;
  const long n_item = (long)n_walk * n_l * n_part;
  const int it0 = (int)(n_item * blockIdx.x / gridDim.x), it1 = (int)(n_item * (blockIdx.x + 1) / gridDim.x);
  // the producer's place: stage pst of item pit
  int pit = it0, pst = 0, slot = 0;
  auto issue = [&](int to) {
    if (pit < it1) {
      const int k0 = pst << lg_sk, ns = min(sk, nk64 - k0);
      const float* dl = delta + (size_t)(pit / n_part) * N_tr * N_k;
      float* st = ring + (size_t)to * rows * sk;
      if (vec4) {
        for (int e = threadIdx.x; e < rows << (lg_sk - 2); e += blockDim.x) {
          const int t = e >> (lg_sk - 2), kk = (e & ((sk >> 2) - 1)) << 2, left = N_k - k0 - kk;
          if (kk >= ns) continue;
          const int bytes = t < N_tr && left > 0 ? 16 : 0;      // N_k is a multiple of 4
          const float* src = bytes ? dl + (size_t)t * N_k + k0 + kk : dl;
          const unsigned dst = (unsigned)__cvta_generic_to_shared(st + (t << lg_sk) + kk);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
                       "r"(bytes) : "memory");
        }
      } else {
        for (int e = threadIdx.x; e < rows << lg_sk; e += blockDim.x) {
          const int t = e >> lg_sk, kk = e & (sk - 1);
          if (kk >= ns) continue;
          const int bytes = t < N_tr && k0 + kk < N_k ? 4 : 0;
          const float* src = bytes ? dl + (size_t)t * N_k + k0 + kk : dl;
          const unsigned dst = (unsigned)__cvta_generic_to_shared(st + (t << lg_sk) + kk);
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src),
                       "r"(bytes) : "memory");
        }
      }
      if (++pst == n_st) {
        pst = 0;
        ++pit;
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");   // empty past the end: the count goes on
  };
#pragma unroll
  for (int x = 0; x < QS_RING - 1; ++x) issue(x);
  int cur_w = -1;
  for (int it = it0; it < it1; ++it) {
    const int wl = it / n_part, part = it - wl * n_part, w = wl / n_l, ll = wl - w * n_l;
    double* Uw = U + ((size_t)w * N_ell + l_lo + ll) * N_tr * N_tr;
    if (w != cur_w) {
      __syncthreads();   // the sums of the walker before have read us
      for (int q = threadIdx.x; q < nk64; q += blockDim.x)
        us[q] = q < N_k ? (float)(wk2[q] * P[(size_t)w * N_k + q]) : 0.0f;
      cur_w = w;
    }
    const int b = part * nbp + bw;
    const bool work = b < nb;
    int ib, jb;
    qb_block(work ? b : 0, n_ib, ib, jb);
    const int oa = ((4 * ib) << lg_sk) + lane, ob = ((4 * jb) << lg_sk) + lane;
    float s2[16], c2[16];
#pragma unroll
    for (int p = 0; p < 16; ++p) s2[p] = c2[p] = 0.0f;
    for (int st = 0; st < n_st; ++st) {
      // this stage has arrived, and every warp is done with the one before, whose place is free
      asm volatile("cp.async.wait_group %0;\n" ::"n"(QS_RING - 2) : "memory");
      __syncthreads();
      issue(slot == 0 ? QS_RING - 1 : slot - 1);
      const float* d = ring + (size_t)slot * rows * sk;
      slot = slot + 1 == QS_RING ? 0 : slot + 1;
      if (!work) continue;
      const int k0 = st << lg_sk, ns = min(sk, nk64 - k0);
      const float* ru = us + k0 + lane;
      for (int g0 = 0; g0 < ns; g0 += 128) qb_group(s2, c2, d + oa + g0, d + ob + g0, ru + g0, sk, ns - g0);
    }
    if (!work) continue;
    const float2 t = qb_lanes(s2, c2, lane);
    if (!(lane & 1)) {
      const int p = lane >> 1, i = 4 * ib + (p >> 2), j = 4 * jb + (p & 3);
      if (i <= j && j < N_tr) {
        const double v = (double)t.x + (double)t.y;
        Uw[i * N_tr + j] = v;
        Uw[j * N_tr + i] = v;
      }
    }
  }
}

// C[o][i][j] = A_i A_j U[w][l][i][j] for the packed (walker, listed multipole) outputs.
__global__ void k_scale_pack(double* __restrict__ C, const double* __restrict__ U,
                             const double* __restrict__ amp, const int* __restrict__ off,
                             const int* __restrict__ idx, int n_walk, int N_tr, int N_ell,
                             long n_out, int* __restrict__ status) {
  long o = blockIdx.x;
  if (o >= n_out) return;
  int w, l;
  if (off) {
    // walker of output o: largest w with off[w] <= o
    int lo = 0, hi = n_walk;
    while (hi - lo > 1) { int mid = (lo + hi) >> 1; if (off[mid] <= o) lo = mid; else hi = mid; }
    w = lo;
    l = idx[o];
  } else {
    w = (int)(o / N_ell);
    l = (int)(o % N_ell);
  }
  const double* u = U + ((size_t)w * N_ell + l) * N_tr * N_tr;
  const double* A = amp + (size_t)w * N_tr;
  for (int e = threadIdx.x; e < N_tr * N_tr; e += blockDim.x) {
    int i = e / N_tr, j = e - i * N_tr;
    double ai = A[i], aj = A[j];
    double s = (i <= j) ? ai * aj : aj * ai;
    const double v = s * u[e];
    flag_nonfinite(status, v);
    C[o * N_tr * N_tr + e] = v;
  }
}

// Cbar_full[w][l] = (Cbar + Cbar^T)/2 on listed multipoles, 0 elsewhere.
__global__ void k_unpack_sym(double* __restrict__ Cf, const double* __restrict__ Cb,
                             const int* __restrict__ off, const int* __restrict__ idx,
                             int n_walk, int N_tr, int N_ell, long n_out) {
  long o = blockIdx.x;
  if (o >= n_out) return;
  int w, l;
  if (off) {
    int lo = 0, hi = n_walk;
    while (hi - lo > 1) { int mid = (lo + hi) >> 1; if (off[mid] <= o) lo = mid; else hi = mid; }
    w = lo;
    l = idx[o];
  } else {
    w = (int)(o / N_ell);
    l = (int)(o % N_ell);
  }
  const double* s = Cb + o * N_tr * N_tr;
  double* d = Cf + ((size_t)w * N_ell + l) * N_tr * N_tr;
  for (int e = threadIdx.x; e < N_tr * N_tr; e += blockDim.x) {
    int i = e / N_tr, j = e - i * N_tr;
    d[e] = 0.5 * (s[i * N_tr + j] + s[j * N_tr + i]);
  }
}

// amp_bar[w][i] = 2 sum_l sum_j S_ij A_j U_ij
// One CTA per tracer and walker; 1024 threads where a tracer has more than 4096 terms (30 tracers, 2999
// multipoles: 218 us with 256 threads, 122 us beside the FFTLog adjoint).
template <int AT>
__global__ void __launch_bounds__(AT) k_amp_bar(double* __restrict__ abar, const double* __restrict__ Cf,
                          const double* __restrict__ U, const double* __restrict__ amp,
                          int N_tr, int N_ell, int* __restrict__ status) {
  const int w = blockIdx.y;
  const int i = blockIdx.x;
  __shared__ double red[AT];
  double s = 0.0;
  const double* A = amp + (size_t)w * N_tr;
#pragma unroll 4
  for (int e = threadIdx.x; e < N_ell * N_tr; e += blockDim.x) {
    int l = e / N_tr, j = e - l * N_tr;
    size_t base = (((size_t)w * N_ell + l) * N_tr + i) * N_tr + j;
    s = fma(Cf[base] * A[j], U[base], s);
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    flag_nonfinite(status, red[0]);
    abar[(size_t)w * N_tr + i] = 2.0 * red[0];
  }
}

// Delta_bar and the P_bar partial sums.  Grid: (k tile of DT QT points, one multipole, walker);
// QT consecutive k points per thread.  S_ij A_j is staged per multipole chunk in shared memory,
// transposed (St[j][i], rows padded to a multiple of DG with zeros) so that DG consecutive rows i
// load as one vector, in the arithmetic type T (FP32 for the mixed paths, FP64 for the FP64 path);
// Delta_j(l, q) sits in a per-thread shared column.  Each thread forms T_i for DG rows i at a time,
// DG independent FMA chains over j in ascending order.  The P_bar partial of each multipole chunk
// is a compensated sum (TwoSum) written as FP64 to pbar_part[chunk][w][q]; k_pbar_reduce adds the
// chunks.  A launch covers the multipoles [l_lo, l_lo + n_l) of the Delta buffer it is given (a
// multipole chunk when Delta is recomputed chunk by chunk); the reduction runs once after the last
// chunk.
constexpr int DT = 256;   // threads per CTA
constexpr int LC = 1;   // multipoles per CTA: one, for enough CTAs to hide the load latency
constexpr int DG = 4;   // rows i per pass

__host__ __device__ inline int delta_bar_pitch(int N_tr) { return (N_tr + DG - 1) / DG * DG; }

__device__ __forceinline__ void lds4(const float* p, float (&v)[4]) {
  const float4 x = *reinterpret_cast<const float4*>(p);
  v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void lds4(const double* p, double (&v)[4]) {
  const double2 x = reinterpret_cast<const double2*>(p)[0];
  const double2 y = reinterpret_cast<const double2*>(p)[1];
  v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
}

template <typename T>
__device__ __forceinline__ void two_sum_acc(T& s, T& c, T x) {
  const T sn = s + x;
  const T bp = sn - s;
  c += (s - (sn - bp)) + (x - bp);
  s = sn;
}

// QT consecutive k points per thread: with QT = 2 every shared load of S feeds 2 DG FMAs and
// Delta and Dbar move as 8-byte pairs, but one point per thread at 256 threads per CTA measured
// faster (more warps to hide the load latency), so both types use QT = 1; the sums of each k
// point are the same in either form.
template <typename T> struct DbarQ { static constexpr int QT = 1; };
template <> struct DbarQ<float> { static constexpr int QT = 1; };

template <typename T>
__global__ void __launch_bounds__(DT)
k_delta_bar(T* __restrict__ dbar, double* __restrict__ pbar_part, const T* __restrict__ delta,
            const double* __restrict__ Cf, const double* __restrict__ amp,
            const double* __restrict__ P, const double* __restrict__ wk2, int N_tr, int N_k,
            int N_ell, int n_walk, int l_lo, int n_l, const int* __restrict__ listed) {
  constexpr int QT = DbarQ<T>::QT, DQ = DT * QT;
  pdl_trigger();   // the next kernel of the step may be scheduled
  pdl_wait();      // Delta and the cotangent come from the kernels before
  extern __shared__ __align__(16) unsigned char dsm_raw[];
  const int NP = delta_bar_pitch(N_tr);
  T* St = reinterpret_cast<T*>(dsm_raw);           // [N_tr][NP]  St[j][i] = S_ij A_j
  T* Dl = St + N_tr * NP;                          // [N_tr][DQ]
  T* As = Dl + N_tr * DQ;                          // [N_tr] A_i
  const int w = blockIdx.z;
  // Delta and Dbar hold multipoles [l_lo, l_lo + n_l); Cf all N_ell (LC = 1 multipole per CTA)
  const int l0 = l_lo + blockIdx.y;
  const int qt = threadIdx.x * QT;                 // this thread's first column of Dl
  const int q0 = blockIdx.x * DQ + qt;
  if (listed && listed[w * n_l + (l0 - l_lo)] < 0) {
    // a multipole the walker does not list: S = 0, so Dbar = 0 and the P_bar partial is 0; its
    // Delta rows are not read and its Dbar rows are not used
#pragma unroll
    for (int u = 0; u < QT; ++u)
      if (q0 + u < N_k) pbar_part[((size_t)l0 * n_walk + w) * N_k + q0 + u] = 0.0;
    return;
  }
  const double* A = amp + (size_t)w * N_tr;
  const double* Cl = Cf + ((size_t)w * N_ell + l0) * N_tr * N_tr;
  for (int e = threadIdx.x; e < N_tr * NP; e += DT) {
    const int j = e / NP, i = e - j * NP;
    St[e] = i < N_tr ? (T)(Cl[i * N_tr + j] * A[j]) : T(0);
  }
  for (int e = threadIdx.x; e < N_tr; e += DT) As[e] = (T)A[e];
  T two_u[QT];
#pragma unroll
  for (int u = 0; u < QT; ++u)
    two_u[u] = (q0 + u < N_k) ? (T)(2.0 * wk2[q0 + u] * P[(size_t)w * N_k + q0 + u]) : T(0);
  const T* dl = delta + ((size_t)w * n_l + l0 - l_lo) * N_tr * N_k;
  const bool pair = QT == 2 && (N_k & 1) == 0 && q0 + 1 < N_k;   // 8-byte aligned pair
#pragma unroll 5
  for (int t = 0; t < N_tr; ++t) {
    if (pair) {
      *reinterpret_cast<float2*>(Dl + t * DQ + qt) = *reinterpret_cast<const float2*>(dl + (size_t)t * N_k + q0);
    } else {
#pragma unroll
      for (int u = 0; u < QT; ++u) Dl[t * DQ + qt + u] = (q0 + u < N_k) ? dl[(size_t)t * N_k + q0 + u] : T(0);
    }
  }
  __syncthreads();
  if (q0 >= N_k) return;
  T ps[QT], pc[QT];
#pragma unroll
  for (int u = 0; u < QT; ++u) ps[u] = pc[u] = T(0);
  const T* dq = Dl + qt;
  T* db = dbar + ((size_t)w * n_l + l0 - l_lo) * N_tr * N_k + q0;
  for (int i0 = 0; i0 < N_tr; i0 += DG) {
    T t[DG][QT];
#pragma unroll
    for (int g = 0; g < DG; ++g)
#pragma unroll
      for (int u = 0; u < QT; ++u) t[g][u] = 0;
#pragma unroll 5
    for (int j = 0; j < N_tr; ++j) {
      T sv[DG];
      lds4(St + j * NP + i0, sv);
      T d[QT];
#pragma unroll
      for (int u = 0; u < QT; ++u) d[u] = dq[j * DQ + u];
#pragma unroll
      for (int g = 0; g < DG; ++g)
#pragma unroll
        for (int u = 0; u < QT; ++u) t[g][u] = fma(sv[g], d[u], t[g][u]);
    }
#pragma unroll
    for (int g = 0; g < DG; ++g) {
      const int ii = i0 + g;
      if (ii < N_tr) {
        const T ai = As[ii];
        T o[QT];
#pragma unroll
        for (int u = 0; u < QT; ++u) {
          two_sum_acc(ps[u], pc[u], ai * dq[ii * DQ + u] * t[g][u]);
          o[u] = two_u[u] * ai * t[g][u];
        }
        if (pair) {
          *reinterpret_cast<float2*>(db + (size_t)ii * N_k) = make_float2((float)o[0], (float)o[QT - 1]);
        } else {
#pragma unroll
          for (int u = 0; u < QT; ++u)
            if (q0 + u < N_k) db[(size_t)ii * N_k + u] = o[u];
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < QT; ++u)
    if (q0 + u < N_k) pbar_part[((size_t)l0 * n_walk + w) * N_k + q0 + u] = (double)ps[u] + (double)pc[u];
}

// FP32 form for up to 32 tracers: two neighbouring k points per thread in packed arithmetic, Delta_j of
// both in registers (NJ rows, those past N_tr zero), S_ij A_j from shared memory as doubled values
// {x, x} by broadcast 16-byte loads.  Per point the sums are those of k_delta_bar in the same order.
// What bounds it: with many multipoles and walkers the traffic of Delta, Dbar and the P_bar partials;
// k_delta_bar, which re-read Delta_j from shared memory for every group of rows, was bound by issue.
// 256 points of 15 tracers, ragged lists: 827 us with k_delta_bar, 530 us here; 30 tracers, 2999 multipoles,
// 4096 k 1267 and 1129 us; one point, 103 multipoles 12.2 and 10.1 us.
template <int NJ>
__global__ void __launch_bounds__(128)
k_delta_bar2(float* __restrict__ dbar, double* __restrict__ pbar_part, const float* __restrict__ delta,
             const double* __restrict__ Cf, const double* __restrict__ amp,
             const double* __restrict__ P, const double* __restrict__ wk2, int N_tr, int N_k,
             int N_ell, int n_walk, int l_lo, int n_l, const int* __restrict__ listed) {
  pdl_trigger();   // the next kernel of the step may be scheduled
  pdl_wait();      // Delta and the cotangent come from the kernels before
  __shared__ __align__(16) float2 St[NJ * NJ];   // St[j][i] = S_ij A_j, twice
  __shared__ float As[NJ];
  const int w = blockIdx.z, l0 = l_lo + blockIdx.y;
  const int q0 = (blockIdx.x * 128 + threadIdx.x) * 2;
  const bool in0 = q0 < N_k, in1 = q0 + 1 < N_k;
  double* pb = pbar_part + ((size_t)l0 * n_walk + w) * N_k + q0;
  if (listed && listed[w * n_l + (l0 - l_lo)] < 0) {
    // a multipole the walker does not list: S = 0, so Dbar = 0 and the P_bar partial is 0; its
    // Delta rows are not read and its Dbar rows are not used
    if (in0) pb[0] = 0.0;
    if (in1) pb[1] = 0.0;
    return;
  }
  const size_t row0 = ((size_t)w * n_l + l0 - l_lo) * N_tr * N_k + q0;
  const bool pair = in1 && (N_k & 1) == 0;   // 8-byte aligned
  float2 d[NJ];
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    d[j] = make_float2(0.f, 0.f);
    if (j < N_tr) {
      const float* p = delta + row0 + (size_t)j * N_k;
      if (pair) {
        d[j] = *reinterpret_cast<const float2*>(p);
      } else {
        if (in0) d[j].x = p[0];
        if (in1) d[j].y = p[1];
      }
    }
  }
  const double* A = amp + (size_t)w * N_tr;
  const double* Cl = Cf + ((size_t)w * N_ell + l0) * N_tr * N_tr;
  for (int e = threadIdx.x; e < NJ * NJ; e += 128) {
    const int j = e / NJ, i = e % NJ;
    const float v = i < N_tr && j < N_tr ? (float)(Cl[i * N_tr + j] * A[j]) : 0.0f;
    St[e] = make_float2(v, v);
  }
  if (threadIdx.x < NJ) As[threadIdx.x] = threadIdx.x < N_tr ? (float)A[threadIdx.x] : 0.0f;
  float2 two_u;
  two_u.x = in0 ? (float)(2.0 * wk2[q0] * P[(size_t)w * N_k + q0]) : 0.0f;
  two_u.y = in1 ? (float)(2.0 * wk2[q0 + 1] * P[(size_t)w * N_k + q0 + 1]) : 0.0f;
  __syncthreads();
  if (!in0) return;
  float2 ps = make_float2(0.f, 0.f), pc = ps;
#pragma unroll
  for (int i0 = 0; i0 < NJ; i0 += 4) {
    if (i0 >= N_tr) break;
    float2 t[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) t[g] = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const float4 s01 = *reinterpret_cast<const float4*>(St + j * NJ + i0);
      const float4 s23 = *reinterpret_cast<const float4*>(St + j * NJ + i0 + 2);
      t[0] = f2_fma(make_float2(s01.x, s01.y), d[j], t[0]);
      t[1] = f2_fma(make_float2(s01.z, s01.w), d[j], t[1]);
      t[2] = f2_fma(make_float2(s23.x, s23.y), d[j], t[2]);
      t[3] = f2_fma(make_float2(s23.z, s23.w), d[j], t[3]);
    }
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int ii = i0 + g;
      if (ii < N_tr) {
        const float2 ai = make_float2(As[ii], As[ii]);
        // TwoSum of A_i Delta_i T_i
        const float2 x = f2_mul(f2_mul(ai, d[ii]), t[g]);
        const float2 sn = f2_add(ps, x), bp = f2_sub(sn, ps);
        pc = f2_add(pc, f2_add(f2_sub(ps, f2_sub(sn, bp)), f2_sub(x, bp)));
        ps = sn;
        const float2 o = f2_mul(f2_mul(two_u, ai), t[g]);
        float* out = dbar + row0 + (size_t)ii * N_k;
        if (pair) {
          *reinterpret_cast<float2*>(out) = o;
        } else {
          out[0] = o.x;
          if (in1) out[1] = o.y;
        }
      }
    }
  }
  if (pair) {
    *reinterpret_cast<double2*>(pb) = make_double2((double)ps.x + (double)pc.x, (double)ps.y + (double)pc.y);
  } else {
    pb[0] = (double)ps.x + (double)pc.x;
    if (in1) pb[1] = (double)ps.y + (double)pc.y;
  }
}

// P_bar = wk2 x the sum over the chunks (multipoles).  One thread per k point and walker took the chunks
// one after the other: 16 CTAs and 2999 dependent loads at the large shape, 520 us.  Here eight threads
// share a point (chunks g, g + 8, ..., then the eight sums in order): 66 us; one
// point, 103 multipoles 16.8 and 8.0 us.
constexpr int PQ = 32, PG = 8;
__global__ void __launch_bounds__(PQ * PG)
k_pbar_reduce(double* __restrict__ Pbar, const double* __restrict__ part,
              const double* __restrict__ wk2, int n_chunk, int n_walk, int N_k,
              int* __restrict__ status) {
  __shared__ double red[PG][PQ];
  const int tl = threadIdx.x % PQ, g = threadIdx.x / PQ;
  const long t = (long)blockIdx.x * PQ + tl, n = (long)n_walk * N_k;
  double s = 0.0;
  if (t < n) {
#pragma unroll 8
    for (int c = g; c < n_chunk; c += PG) s += part[(size_t)c * n + t];
  }
  red[g][tl] = s;
  __syncthreads();
  if (g || t >= n) return;
#pragma unroll
  for (int u = 1; u < PG; ++u) s += red[u][tl];
  const double v = wk2[t % N_k] * s;
  flag_nonfinite(status, v);
  Pbar[t] = v;
}

}  // namespace

size_t quad_scratch_bytes(int n_walk, int N_tr, int N_k, int n_l) {
  return sizeof(double) * (size_t)n_walk * n_l * ((N_k + KC - 1) / KC) * (N_tr * (N_tr + 1) / 2);
}

cudaError_t launch_pair_reduce(double* U, const double* part, int n_walk, int N_tr, int N_ell,
                               int l_lo, int n_l, int n_chunk, cudaStream_t s) {
  const long total = (long)n_walk * n_l * (N_tr * (N_tr + 1) / 2);
  const int grid = (int)std::min<long>((total + 255) / 256, 152L * 8);
  k_quad_reduce<<<grid, 256, 0, s>>>(U, part, N_tr, N_ell, l_lo, n_l, n_chunk, n_walk);
  return cudaGetLastError();
}

cudaError_t launch_quad_fp64(double* U, const double* delta, const double* P, const double* wk2,
                             int n_walk, int N_tr, int N_k, int N_ell, int l_lo, int n_l,
                             double* scratch, cudaStream_t s) {
  const size_t row = (size_t)KS * sizeof(double);
  const bool scaled = N_tr <= 55;
  const size_t smem = N_tr * row * (scaled ? 2 : 1);
  auto kern = scaled ? k_quad_part<true> : k_quad_part<false>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  const int n_kc = (N_k + KC - 1) / KC;
  kern<<<dim3(n_l, n_kc, n_walk), QT, smem, s>>>(scratch, delta, P, wk2, N_tr, N_k, n_l, n_kc);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const long total = (long)n_walk * n_l * N_tr * (N_tr + 1) / 2;
  const unsigned grid = (unsigned)std::min<long>((total + 255) / 256, 152L * 16);
  k_quad_reduce<<<grid, 256, 0, s>>>(U, scratch, N_tr, N_ell, l_lo, n_l, n_kc, n_walk);
  return cudaGetLastError();
}

cudaError_t launch_quad_f32(double* U, const float* delta, const double* P, const double* wk2,
                            int n_walk, int N_tr, int N_k, int N_ell, int l_lo, int n_l,
                            double* scratch, cudaStream_t s, const int* listed) {
  if (n_walk <= 0 || n_l <= 0) return cudaSuccess;
  const int n_ib = (N_tr + 3) / 4, nb = n_ib * (n_ib + 1) / 2;
  const bool vec4 = N_k % 4 == 0 && ((uintptr_t)delta & 15) == 0;
  const long n_row = (long)n_walk * n_l;
  // k parts per block: with few CTAs (one walker), enough warps per CTA to hide the shared-load
  // and FMA latencies; with many, one part (each further part repeats the lane combination)
  const long n_cta0 = (long)n_walk * N_ell * ((N_k + 1023) / 1024);
  const int ks = n_cta0 >= 2 * 152 ? 1 : std::max(1, std::min(4, QB_MAX_WARPS / nb));
  const int warps = ks * std::min(nb, QB_MAX_WARPS / ks);
  const size_t red_bytes = sizeof(float2) * (size_t)ks * nb * 16;
  // k points per CTA: the largest power of two up to 1024 whose rows fit QB_SMEM
  int kcap = 1024;
  while (kcap > 64 && (size_t)kcap * (16 * n_ib + 4) + red_bytes > (size_t)QB_SMEM) kcap >>= 1;
  const int n_kc = (N_k + kcap - 1) / kcap;
  const size_t smem = (size_t)kcap * (16 * n_ib + 4) + red_bytes;
  // A stream of rows: from two rows per SM on (by all the multipoles, so that a launch over a part of them
  // sums in the same order), where the other form needs several chunks per row and more blocks than half
  // the warps.  Its equal shares want equal rows: ragged lists stay with the CTAs per row, which the
  // hardware hands out.  More than twenty blocks go in parts (each reads the rows again, from L2); stages
  // of up to 32 KB keep 100 KB in flight per SM.
  if ((long)n_walk * N_ell >= 2 * 152 && !listed && n_kc > 1 && nb > QB_MAX_WARPS / 2 && N_k <= QS_MAX_K &&
      n_row * nb < (1L << 31)) {
    const int n_part = (nb + QB_MAX_WARPS - 1) / QB_MAX_WARPS, nbp = (nb + n_part - 1) / n_part;
    int lg_sk = 7;
    while (lg_sk < 10 && (size_t)(4 * n_ib) * (8 << lg_sk) <= 32 * 1024) ++lg_sk;
    const size_t ring = sizeof(float) * ((size_t)QS_RING * (4 * n_ib) * (1 << lg_sk) + ((N_k + 63) & ~63));
    cudaError_t e = cudaFuncSetAttribute(k_quad_stream, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ring);
    if (e != cudaSuccess) return e;
    k_quad_stream<<<(unsigned)std::min<long>(n_row * n_part, 152), nbp * 32, ring, s>>>(
        U, delta, P, wk2, N_tr, N_k, N_ell, l_lo, n_l, n_walk, n_part, nbp, lg_sk, vec4);
    return cudaGetLastError();
  }
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_quad_blocks, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
  }
  dim3 g(n_l, n_kc, n_walk);
  k_quad_blocks<<<g, warps * 32, smem, s>>>(U, scratch, delta, P, wk2, N_tr, N_k, N_ell, l_lo,
                                            n_l, kcap, n_kc, ks, vec4, listed);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || n_kc == 1) return e;
  const long total = (long)n_walk * n_l * N_tr * (N_tr + 1) / 2;
  const unsigned grid = (unsigned)std::min<long>((total + 255) / 256, 152L * 16);
  k_quad_reduce<<<grid, 256, 0, s>>>(U, scratch, N_tr, N_ell, l_lo, n_l, n_kc, n_walk);
  return cudaGetLastError();
}

cudaError_t launch_scale_pack(double* C, const double* U, const double* amp, const int* off,
                              const int* idx, int n_walk, int N_tr, int N_ell, int64_t n_out,
                              cudaStream_t s, int* status) {
  if (n_out == 0) return cudaSuccess;
  k_scale_pack<<<(unsigned)n_out, 128, 0, s>>>(C, U, amp, off, idx, n_walk, N_tr, N_ell, n_out,
                                               status);
  return cudaGetLastError();
}

cudaError_t launch_unpack_sym(double* Cf, const double* Cb, const int* off, const int* idx,
                              int n_walk, int N_tr, int N_ell, int64_t n_out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(Cf, 0, (size_t)n_walk * N_ell * N_tr * N_tr * sizeof(double), s);
  if (e != cudaSuccess || n_out == 0) return e;
  k_unpack_sym<<<(unsigned)n_out, 128, 0, s>>>(Cf, Cb, off, idx, n_walk, N_tr, N_ell, n_out);
  return cudaGetLastError();
}

cudaError_t launch_amp_bar(double* amp_bar, const double* Cf, const double* U, const double* amp,
                           int n_walk, int N_tr, int N_ell, cudaStream_t s, int* status) {
  dim3 g(N_tr, n_walk);
  if ((long)N_ell * N_tr > 4096) k_amp_bar<1024><<<g, 1024, 0, s>>>(amp_bar, Cf, U, amp, N_tr, N_ell, status);
  else k_amp_bar<256><<<g, 256, 0, s>>>(amp_bar, Cf, U, amp, N_tr, N_ell, status);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_delta_bar(T* dbar, const T* delta, const double* Cf, const double* amp,
                             const double* P, const double* wk2, int n_walk, int N_tr, int N_k,
                             int N_ell, int l_lo, int n_l, double* scratch, cudaStream_t s,
                             const int* listed, bool pdl) {
  if constexpr (sizeof(T) == 4) {
    // up to 32 tracers, whose rows fit the registers
    if (N_tr <= 32) {
      auto kern = N_tr <= 4 ? k_delta_bar2<4> : N_tr <= 8 ? k_delta_bar2<8> : N_tr <= 16 ? k_delta_bar2<16>
                                                                                         : k_delta_bar2<32>;
      return launch_k(pdl, kern, dim3((N_k + 255) / 256, n_l, n_walk), dim3(128), 0, s, dbar, scratch, delta, Cf,
                      amp, P, wk2, N_tr, N_k, N_ell, n_walk, l_lo, n_l, listed);
    }
  }
  constexpr int DQ = DT * DbarQ<T>::QT;
  const size_t smem = (size_t)(N_tr * delta_bar_pitch(N_tr) + N_tr * DQ + N_tr) * sizeof(T);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_delta_bar<T>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  dim3 g((N_k + DQ - 1) / DQ, n_l, n_walk);
  return launch_k(pdl, k_delta_bar<T>, g, dim3(DT), smem, s, dbar, scratch, delta, Cf, amp, P, wk2,
                  N_tr, N_k, N_ell, n_walk, l_lo, n_l, listed);
}

cudaError_t launch_pbar_reduce(double* P_bar, const double* scratch, const double* wk2,
                               int n_walk, int N_k, int N_ell, cudaStream_t s, int* status) {
  const int n_chunk = (N_ell + LC - 1) / LC;
  const long n = (long)n_walk * N_k;
  k_pbar_reduce<<<(unsigned)((n + PQ - 1) / PQ), PQ * PG, 0, s>>>(P_bar, scratch, wk2, n_chunk, n_walk, N_k,
                                                           status);
  return cudaGetLastError();
}

size_t delta_bar_scratch_bytes(int n_walk, int N_k, int N_ell) {
  return sizeof(double) * (size_t)((N_ell + LC - 1) / LC) * n_walk * N_k;
}

template cudaError_t launch_delta_bar<double>(double*, const double*, const double*,
                                              const double*, const double*, const double*, int,
                                              int, int, int, int, int, double*, cudaStream_t,
                                              const int*, bool);
template cudaError_t launch_delta_bar<float>(float*, const float*, const double*, const double*,
                                             const double*, const double*, int, int, int, int,
                                             int, int, double*, cudaStream_t, const int*, bool);

}  // namespace swcl
