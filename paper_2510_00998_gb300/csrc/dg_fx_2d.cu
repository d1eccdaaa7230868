// Instantiation of the FP64 kernels of the DG levels, 2D.
#include "dg_fx.cuh"

namespace dgmg {
template struct FxRun<2, 2>;
template struct FxRun<2, 3>;
template struct FxRun<2, 4>;
template struct FxRun<2, 5>;
template struct FxRun<2, 6>;
template struct FxRun<2, 7>;
}  // namespace dgmg
