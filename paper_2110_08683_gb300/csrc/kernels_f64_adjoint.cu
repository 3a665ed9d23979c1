// kernels_f64_adjoint.cu -- the reverse-mode kernels, FP64.
#include "kernels_impl.cuh"
template struct gpm::LaunchA<double>;
