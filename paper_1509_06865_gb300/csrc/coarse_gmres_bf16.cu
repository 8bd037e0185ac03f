// The persistent coarse GMRES with bfloat16 links (coarse_gmres.cuh).
#include "coarse_gmres.cuh"

namespace mgeig {

const void *coarse_gmres_kernel_bf16() { return (const void *)coarse_gmres_kernel<float, 1>; }

}  // namespace mgeig
