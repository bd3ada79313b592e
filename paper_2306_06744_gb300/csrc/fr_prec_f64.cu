// fr_prec_f64.cu -- the FP64 form: interface kernel in double, element and trace kernels with
// fixed-point contractions (fr_stage_fx.cuh).
#include "fr_stage_fx.cuh"

namespace frg {

int launch_traces_f64(int dim, int p, const double* u, int64_t M, const DevOps& o, void* tr, const int8_t* mask,
                      cudaStream_t s, Err* err, const int64_t* d_M) {
  if (M <= 0) return 0;
  const TraceFx ops = make_trace_fx(p, o);
  FR_NP_DISPATCH(dim, p, ({
                   using SS = Sz<DD, NN>;
                   const unsigned nb = unsigned((M + SS::EPB - 1) / SS::EPB);
                   launch_dependent(k_traces_fx<DD, NN>, nb, SS::BT, s, u, M, ops, static_cast<double*>(tr), mask, d_M);
                 }));
  FR_LAUNCH_CHECK(err);
  return 0;
}
int launch_faces_f64(int dim, int p, FaceArgs A, const DevOps& ops, cudaStream_t s, Err* err) {
  return launch_faces_impl<double>(dim, p, A, ops, s, err);
}
int launch_stage_f64(int dim, int p, const StageArgs& A, const DevOps& o, cudaStream_t s, Err* err) {
  if (A.M <= 0) return 0;
  const OpsFx ops = make_ops_fx(dim, p, o, A.gamma);
  FR_NP_DISPATCH(dim, p, ({
                   using SS = Sz<DD, NN>;
                   const unsigned nb = unsigned((A.M + SS::EPB - 1) / SS::EPB);
                   if (launch_dependent(k_stage_fx<DD, NN>, nb, SS::BT, s, A, ops) != cudaSuccess)
                     return set_error(err, FR_ECUDA, "element kernel launch");
                 }));
  FR_LAUNCH_CHECK(err);
  return 0;
}

}  // namespace frg
