// kernels_f32.cu -- the stage kernels, FP32: reconstruction, Riemann solver and detection in float;
// state, candidate and RK sums in double.
#include "kernels_impl.cuh"
template struct gpm::Launch<float>;
