// kernels_f64.cu -- the stage kernels, FP64.
#include "kernels_impl.cuh"
template struct gpm::Launch<double>;
