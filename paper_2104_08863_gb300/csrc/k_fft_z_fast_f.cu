// FP32 instantiations of the specialised z-transform.
#include "k_fft_z_fast.cuh"

namespace pp {
template cudaError_t launch_fft_z_fast<float>(const Geometry&, const Tables<float>&, int, cplx<float>*, cudaStream_t, int, int);
template int fft_z_fast_tile<float>(const Geometry&);
}  // namespace pp
