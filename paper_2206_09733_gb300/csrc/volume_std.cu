// Element kernels of the standard form (Sec. 3.5): all degrees, both
// precisions, Euler and Navier-Stokes.
#include "volume_dev.cuh"
#include "volume_kernel.cuh"
#include "volume_row.cuh"

namespace hs3d {
HS3D_VOLUME_FORM_TU(HS3D_VOL_STANDARD)
HS3D_VOLUME_DEV_FORM_TU(HS3D_VOL_STANDARD)
}  // namespace hs3d
