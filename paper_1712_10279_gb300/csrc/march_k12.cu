// Kernels of the marching form for one and two channels (a unit of its own, so that the
// units compile in parallel).
#include "march2d.cuh"

namespace vomt {
namespace march {

Kernels pick_k12(int k, int un, int wn, bool reg, bool res)
{
    return k == 1 ? pick_norms<1>(un, wn, reg, res) : pick_norms<2>(un, wn, reg, res);
}

}  // namespace march
}  // namespace vomt
