// Nucleon two-point function (eq. Nop and the P+- projections of Sec. 2.3)
// on an FP64 propagator; the kernels and the
// contraction formulas are in nucleon_kernels.cuh.
#include "nucleon_kernels.cuh"

int contract_sites_per_cta(const qcd_ctx* c) {
  return nucleon::sites_per_cta((long long)c->g.L[1] * c->g.L[2] * c->g.L[3]);
}

template <typename R, bool CANONICAL>
static qcd_status launch_sites(qcd_ctx* c, const void* prop, int ns, double2* partials) {
  const size_t smem = nucleon::cta_smem<R>(ns);
  QCD_CUDA_OK(allow_smem(nucleon::k_sites<R, CANONICAL>, nucleon::cta_smem<R>(nucleon::MAX_SITES)));
  nucleon::k_sites<R, CANONICAL><<<c->g.V / ns, nucleon::cta_threads(ns), smem, c->stream>>>((const double2*)prop,
                                                                                             c->g.V, ns, partials);
  QCD_CUDA_OK(cudaGetLastError());
  return QCD_OK;
}

// corr_dev: [2][T] double2.  prop: 12 FP64 spinors (rhs = 3 spin + colour), internal layout
// or, with canonical, that of the C-ABI.  partials: at least 2 V / ns double2.
qcd_status contract_nucleon(qcd_ctx* c, const void* prop, int t0, double* corr_dev, int precision,
                            double2* partials, int canonical) {
  const int ns = contract_sites_per_cta(c);
  const int nb = c->g.V / ns;
  const int T = c->g.L[0];
  const int per_t = nb / T;
  const int bc3 = c->g.bc_t * c->g.bc_t * c->g.bc_t;
  // algorithmic cost per site: the 144 complex propagator entries read once;
  // 9 colour pairs x (96 + 12 + 2) complex multiply-adds
  ProfScope ps(c, FAM_CONTRACT, (double)c->g.V * 144 * 16, (double)c->g.V * 9 * 110 * 8, 2);
  if (precision == QCD_PREC_F64)
    QCD_TRY((canonical ? launch_sites<double, true> : launch_sites<double, false>)(c, prop, ns, partials));
  else
    QCD_TRY((canonical ? launch_sites<float, true> : launch_sites<float, false>)(c, prop, ns, partials));
  nucleon::k_timeslices<<<T, 256, 0, c->stream>>>(partials, per_t, T, t0, bc3, (double2*)corr_dev);
  QCD_CUDA_OK(cudaGetLastError());
  return QCD_OK;
}
