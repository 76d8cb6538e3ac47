// FP32 instances (the mixed form in basis mode) of the chirp transforms (chirp.cuh).
#include "chirp.cuh"

namespace swcl {

using namespace chirp;

namespace {

constexpr size_t kA = sizeof(double2);   // room for either type

// a_n is FP32 forward (it multiplies FP32 coefficients) and FP64 in the transpose (it multiplies the
// FP64 sums over multipoles)
ChirpArgs<float> args(const ChirpDir& d, const ChirpRun& r, const float2* g, const int* cls_of, const float* kmu) {
  const TabLayout L = tab_layout<float>(d.logm, r.n_h - d.n0, r.N_k, kA);
  const uint8_t* p = (const uint8_t*)d.tab.p;
  ChirpArgs<float> A;
  A.tw1 = (const float2*)(p + L.tw1);
  A.tw2 = (const float2*)(p + L.tw2);
  A.filt = (const float2*)(p + L.filt);
  A.a = (const float2*)(p + L.a);
  A.b = (const float2*)(p + L.b);
  A.g = g;
  A.cls_of = cls_of;
  A.kw = kmu;
  A.lw_ts = 0;
  A.kpow = nullptr;
  A.head = nullptr;
  A.off = r.off;
  A.idx = r.idx;
  A.N_tr = r.N_tr; A.NI = r.NI; A.n_h = r.n_h; A.N_k = r.N_k; A.N_ell = r.N_ell;
  A.l_lo = r.l_lo; A.n_l = r.n_l; A.r = r.rank; A.n0 = d.n0; A.n_chunk = r.n_chunk;
  A.n_total = r.n_total; A.chunk0 = r.chunk0;
  return A;
}

}  // namespace

int chirp32_ctas_per_sm(int logm) {
  int n = 1;
  by_size<float>(logm, [&](auto lm) {
    n = min_blocks<float, decltype(lm)::value>();
    return cudaSuccess;
  });
  return n;
}

size_t chirp32_table_bytes(int logm, int n_in, int N_k) {
  return tab_layout<float>(logm, n_in, N_k, kA).bytes;
}

cudaError_t chirp32_build(void* tab, int logm, int n0, int n_in, int N_k, int t_lo, int t_hi, const double* cc,
                          const double* xx, bool forward, cudaStream_t s) {
  const TabLayout L = tab_layout<float>(logm, n_in, N_k, kA);
  const double2 c2 = make_double2(cc[0], cc[1]), x2 = make_double2(xx[0], xx[1]);
  return by_size<float>(logm, [&](auto lm) {
    constexpr int LM = decltype(lm)::value;
    return forward ? build_tables<LM, float, float>((uint8_t*)tab, L, n0, n_in, N_k, t_lo, t_hi, c2, x2, s)
                   : build_tables<LM, float, double>((uint8_t*)tab, L, n0, n_in, N_k, t_lo, t_hi, c2, x2, s);
  });
}

cudaError_t chirp32_forward(const ChirpDir& d, float* delta, const float4* coef, const float2* g, const int* cls_of,
                            const float* kmu, const int* head, const ChirpRun& r, cudaStream_t s) {
  ChirpArgs<float> A = args(d, r, g, cls_of, kmu);
  A.head = head;
  return launch_fwd<float>(d.logm, d.half, delta, coef, A, r.n_walk * r.N_tr, s);
}

cudaError_t chirp32_adjoint(const ChirpDir& d, void* part, const float* dbar, const float2* g, const int* cls_of,
                            const float* kmu, const ChirpRun& r, cudaStream_t s) {
  return launch_adj<float>(d.logm, d.half, (float2*)part, dbar, args(d, r, g, cls_of, kmu), r.n_walk * r.N_tr, s);
}

cudaError_t chirp32_sum(cplx* cbar, const void* part, const ChirpDir& d, const ChirpRun& r, bool accumulate,
                        cudaStream_t s) {
  const TabLayout L = tab_layout<float>(d.logm, r.n_h, r.N_k, kA);
  const int rows = r.n_walk * r.N_tr;
  const long grid = (long)rows * r.NI * ((r.n_h + kSumN - 1) / kSumN);
  k_chirp_sum<float><<<(unsigned)grid, kSumN * kSumG, 0, s>>>(cbar, (const float2*)part,
                                                              (const double2*)((const uint8_t*)d.tab.p + L.a), rows,
                                                              r.NI, r.rank, r.n_h, r.n_chunk, accumulate);
  return cudaGetLastError();
}

}  // namespace swcl
