// Instantiation of the FP64 kernels of the DG levels, 3D, p = 5.
#include "dg_fx.cuh"

namespace dgmg {
template struct FxRun<3, 6>;
}  // namespace dgmg
