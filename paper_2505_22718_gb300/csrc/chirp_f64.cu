// FP64 instances of the chirp transforms (chirp.cuh).
#include "chirp.cuh"

namespace swcl {

using namespace chirp;

namespace {

ChirpArgs<double> args(const ChirpDir& d, const ChirpRun& r, const cplx* g, const int* cls_of, const double* w,
                       long w_ts, const double* kpow) {
  const TabLayout L = tab_layout<double>(d.logm, r.n_h - d.n0, r.N_k, sizeof(double2));
  const uint8_t* p = (const uint8_t*)d.tab.p;
  ChirpArgs<double> A;
  A.tw1 = (const double2*)(p + L.tw1);
  A.tw2 = (const double2*)(p + L.tw2);
  A.filt = (const double2*)(p + L.filt);
  A.a = (const double2*)(p + L.a);
  A.b = (const double2*)(p + L.b);
  A.g = (const double2*)g;
  A.cls_of = cls_of;
  A.kw = w;
  A.lw_ts = w_ts;
  A.kpow = kpow;
  A.head = nullptr;
  A.off = r.off;
  A.idx = r.idx;
  A.N_tr = r.N_tr; A.NI = r.NI; A.n_h = r.n_h; A.N_k = r.N_k; A.N_ell = r.N_ell;
  A.l_lo = r.l_lo; A.n_l = r.n_l; A.r = r.rank; A.n0 = d.n0; A.n_chunk = r.n_chunk;
  A.n_total = r.n_total; A.chunk0 = r.chunk0;
  return A;
}

}  // namespace

int chirp64_ctas_per_sm(int logm) {
  int n = 1;
  by_size<double>(logm, [&](auto lm) {
    n = min_blocks<double, decltype(lm)::value>();
    return cudaSuccess;
  });
  return n;
}

size_t chirp64_table_bytes(int logm, int n_in, int N_k) {
  return tab_layout<double>(logm, n_in, N_k, sizeof(double2)).bytes;
}

cudaError_t chirp64_build(void* tab, int logm, int n0, int n_in, int N_k, int t_lo, int t_hi, const double* cc,
                          const double* xx, cudaStream_t s) {
  const TabLayout L = tab_layout<double>(logm, n_in, N_k, sizeof(double2));
  return by_size<double>(logm, [&](auto lm) {
    return build_tables<decltype(lm)::value, double, double>((uint8_t*)tab, L, n0, n_in, N_k, t_lo, t_hi,
                                                             make_double2(cc[0], cc[1]),
                                                             make_double2(xx[0], xx[1]), s);
  });
}

cudaError_t chirp64_forward(const ChirpDir& d, double* delta, const cplx* coef, const cplx* g, const int* cls_of,
                            const double* w, long w_ts, const double* kpow, const ChirpRun& r, cudaStream_t s) {
  return launch_fwd<double>(d.logm, d.half, delta, coef, args(d, r, g, cls_of, w, w_ts, kpow), r.n_walk * r.N_tr, s);
}

cudaError_t chirp64_adjoint(const ChirpDir& d, void* part, const double* dbar, const cplx* g, const int* cls_of,
                            const double* w, long w_ts, const double* kpow, const ChirpRun& r, cudaStream_t s) {
  return launch_adj<double>(d.logm, d.half, (double2*)part, dbar, args(d, r, g, cls_of, w, w_ts, kpow),
                            r.n_walk * r.N_tr, s);
}

cudaError_t chirp64_sum(cplx* cbar, const void* part, const ChirpDir& d, const ChirpRun& r, bool accumulate,
                        cudaStream_t s) {
  const TabLayout L = tab_layout<double>(d.logm, r.n_h, r.N_k, sizeof(double2));
  const int rows = r.n_walk * r.N_tr;
  const long grid = (long)rows * r.NI * ((r.n_h + kSumN - 1) / kSumN);
  k_chirp_sum<double><<<(unsigned)grid, kSumN * kSumG, 0, s>>>(cbar, (const double2*)part,
                                                     (const double2*)((const uint8_t*)d.tab.p + L.a), rows, r.NI,
                                                     r.rank, r.n_h, r.n_chunk, accumulate);
  return cudaGetLastError();
}

}  // namespace swcl
