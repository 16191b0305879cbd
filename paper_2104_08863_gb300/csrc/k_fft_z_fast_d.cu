// FP64 instantiations of the specialised z-transform.
#include "k_fft_z_fast.cuh"

namespace pp {
template cudaError_t launch_fft_z_fast<double>(const Geometry&, const Tables<double>&, int, cplx<double>*, cudaStream_t, int, int);
template int fft_z_fast_tile<double>(const Geometry&);
}  // namespace pp
