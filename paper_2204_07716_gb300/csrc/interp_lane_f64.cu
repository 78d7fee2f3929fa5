// The lane-per-sample interpolation of interp_lane.cuh in FP64.
#include "interp_lane.cuh"

namespace fk {

// Launched when the plan's window width is one of the instantiated ones
// (*launched says so); other widths go through interp.cu's runtime kernel.
cudaError_t run_interp_lane_f64(fkreg_plan_s* P, int b, int n_rhs_real, int n_probes,
                                void* mhat_at_x, cudaStream_t st, int nacc, int F2, void* vout,
                                bool* launched) {
  LaneLaunch<double> L{P, {}, static_cast<double*>(mhat_at_x), static_cast<double*>(vout), st, {P->poly}};
  L.a.b = b;
  L.a.order = P->order;
  L.a.rec = t2_record_stride(F2, sizeof(double));
  L.a.F2 = F2;
  L.a.n_rhs_real = n_rhs_real;
  L.a.n_probes = n_probes;
  L.a.cplx = P->o.y_complex;
  L.a.n_rhs_out = P->nrhs;
  L.a.nacc = nacc;
  L.a.nbw = P->nbw;
  *launched = true;
  const int w = P->geo.w, d = P->d;
#define FK_W(DD, WW) \
  if (d == DD && w == WW) return lane_dispatch<double, DD, WW>(L)
  FK_W(1, 7);
  FK_W(2, 7);
  FK_W(3, 7);
  FK_W(1, 10);
  FK_W(2, 10);
  FK_W(1, 13);
  FK_W(2, 13);
#undef FK_W
  *launched = false;
  return cudaSuccess;
}

}  // namespace fk
