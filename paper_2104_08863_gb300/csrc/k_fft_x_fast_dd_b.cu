// x-transform kernels, group 1 of the half-lengths: FP64 field, FP64 half spectrum.
#include "k_fft_x_fast.cuh"

namespace pp {
cudaError_t launch_fwd_x_fast_dd_b(const Geometry& g, const DevTables& tb, FwdMode mode, const FwdArgs& args,
                                   cplx<double>* spec, cudaStream_t st) {
  return launch_fwd_x_fast_impl<double, double, 1>(g, tb, tb.d, mode, args, spec, st);
}
cudaError_t launch_inv_x_fast_dd_b(const Geometry& g, const DevTables& tb, InvMode mode, const cplx<double>* spec,
                                   double* out, double scale, bool accumulate, cudaStream_t st, PairArgs pair) {
  return launch_inv_x_fast_impl<double, double, 1>(g, tb, tb.d, mode, spec, out, scale, accumulate, st, pair);
}
}  // namespace pp
