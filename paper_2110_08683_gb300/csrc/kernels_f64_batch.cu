// kernels_f64_batch.cu -- the batched kernels, FP64.
#include "kernels_impl.cuh"
template struct gpm::LaunchB<double>;
