// Instances of the cluster-resident kernel (gx_crs.cuh): adjoint, 1 hour per thread item.
#include "gx_crs.cuh"

namespace gx {
CrsFn crs_pick_adj1(int kw, int hpl, int reg) { return crs_pick_impl<1, 1>(kw, hpl, reg); }
}  // namespace gx
