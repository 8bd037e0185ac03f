// The persistent coarse GMRES with IEEE half links (coarse_gmres.cuh).
#include "coarse_gmres.cuh"

namespace mgeig {

const void *coarse_gmres_kernel_f16() { return (const void *)coarse_gmres_kernel<float, 2>; }

}  // namespace mgeig
