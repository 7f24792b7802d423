// Kernels of the marching form for 7 channels (a unit of its own, so that the units
// compile in parallel).
#include "march2d.cuh"

namespace vomt {
namespace march {

Kernels pick_k7(int, int un, int wn, bool reg, bool res) { return pick_norms<7>(un, wn, reg, res); }

}  // namespace march
}  // namespace vomt
