// Instantiation of the FP64 kernels of the DG levels, 3D, p = 4.
#include "dg_fx.cuh"

namespace dgmg {
template struct FxRun<3, 5>;
}  // namespace dgmg
