// Instantiation of the FP64 kernels of the DG levels, 3D, p = 1 .. 3.
#include "dg_fx.cuh"

namespace dgmg {
template struct FxRun<3, 2>;
template struct FxRun<3, 3>;
template struct FxRun<3, 4>;
}  // namespace dgmg
