// The persistent coarse GMRES in FP64 (coarse_gmres.cuh).
#include "coarse_gmres.cuh"

namespace mgeig {

const void *coarse_gmres_kernel_f64() { return (const void *)coarse_gmres_kernel<double, 0>; }

}  // namespace mgeig
