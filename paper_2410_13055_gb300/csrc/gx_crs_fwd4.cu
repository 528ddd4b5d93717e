// Instances of the cluster-resident kernel (gx_crs.cuh): forward, 4 hours per thread item.
#include "gx_crs.cuh"

namespace gx {
CrsFn crs_pick_fwd4(int kw, int hpl, int reg) { return crs_pick_impl<0, 4>(kw, hpl, reg); }
}  // namespace gx
