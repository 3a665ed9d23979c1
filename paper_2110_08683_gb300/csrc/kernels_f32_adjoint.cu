// kernels_f32_adjoint.cu -- the reverse-mode kernels, FP32: reconstruction, Riemann solver and detection in float;
// state, candidate and RK sums in double.
#include "kernels_impl.cuh"
template struct gpm::LaunchA<float>;
