// The FP64 SpMV kernels and the outer operator.
#include "spmv_inst.cuh"

namespace fsi {

namespace {

RowClass row_class(const Bsr& A1, const Bsr& A2, int* ctas) {
  const auto [blocks, rows] = cta_split(A1, A1.tpr64);
  *ctas = blocks;
  return {A1.nbr,  A1.tpr64, rows,       pair_order(A1, A2), A1.rowptr.p,   A1.colind.p,   A1.v64.p,
          A1.nnzb, A2.rowptr.p, A2.colind.p, A2.v64.p,          A2.nnzb};
}

template <int D, template <class, int> class Epi>
void launch_operator(const Bsr& AVV, const Bsr& AVP, const Bsr& APV, const Bsr& APP, const double* x,
                     const Epi<double, D>& ev, const Epi<double, 1>& ep, cudaStream_t s) {
  const SpmvTuning& tu = spmv_tuning();
  int cv = 0, cp = 0;
  const RowClass V = row_class(AVV, AVP, &cv), P = row_class(APV, APP, &cp);
  const bool built = tu.setup_depth == 0;
  const bool early = built && loads_early(cv + cp, V.rows_per_cta, V.tpr, kEarlyCtas64);
  launch_k(early ? k_operator_rows<D, Epi, true> : k_operator_rows<D, Epi, false>, cv + cp, 256, 0, s, V, P, cp,
           tu.prefetch > 0 ? kPrefetchCap : 0, built ? kDepBuilt : 0, x, x + AVV.rows(), ev, ep);
}

}  // namespace

void spmv_operator(const Bsr& AVV, const Bsr& AVP, const Bsr& APV, const Bsr& APP, const double* x, const double* b,
                   double* y, cudaStream_t s) {
  const int64_t nv = AVV.rows();
  if (AVV.nbr == 0 || APP.nbr == 0) {   // (AVP has the velocity rows, APV the pressure rows)
    const Bsr& A = AVV.nbr ? AVV : APP;   // no pressures, or no velocities: then nv = 0
    if (b) spmv2_resid<double>(A, x, nullptr, nullptr, b, y, s);
    else spmv2_axpby<double>(A, x, nullptr, nullptr, 1.0, 0.0, y, s);
    return;
  }
  auto run = [&]<int D>() {
    if (b)
      launch_operator<D, EpiResid>(AVV, AVP, APV, APP, x, {b, y}, {b + nv, y + nv}, s);
    else
      launch_operator<D, EpiAxpby>(AVV, AVP, APV, APP, x, {y, 1.0, 0.0}, {y + nv, 1.0, 0.0}, s);
  };
  require(AVV.br == AVV.bc && APV.br == 1 && APV.bc == AVV.br && AVP.br == AVV.br, "outer operator: block shapes");
  if (AVV.br == 2) run.operator()<2>();
  else if (AVV.br == 3) run.operator()<3>();
  else throw Error(EINVAL_, "outer operator: unsupported block size " + std::to_string(AVV.br));
}

FSI_INST(double)

}  // namespace fsi
