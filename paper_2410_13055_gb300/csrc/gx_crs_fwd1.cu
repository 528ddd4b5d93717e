// Instances of the cluster-resident kernel (gx_crs.cuh): forward, 1 hour per thread item.
#include "gx_crs.cuh"

namespace gx {
CrsFn crs_pick_fwd1(int kw, int hpl, int reg) { return crs_pick_impl<0, 1>(kw, hpl, reg); }
}  // namespace gx
