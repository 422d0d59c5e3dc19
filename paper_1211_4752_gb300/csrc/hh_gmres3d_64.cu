// complex128 instantiations of the 3-D GMRES step kernels (hh_gmres3d.cuh).
#include "hh_gmres3d.cuh"

namespace hh {
HH_GM3D_INST(double)
}  // namespace hh
