// Instances of the fixed-point 2D passes (fx2d.cuh): node grids, isotropic stencil, red-black sweeps.
#include "fx2d.cuh"

namespace mg {
namespace fx2 {
FX2_RUN(node_rbgs_quarter) { return dispatch<false, false, kQuarter>(a, rows, nu, zero, corr, out, nparts, s); }
FX2_RUN(node_rbgs_iso) { return dispatch<false, false, kIso>(a, rows, nu, zero, corr, out, nparts, s); }
}  // namespace fx2
}  // namespace mg
