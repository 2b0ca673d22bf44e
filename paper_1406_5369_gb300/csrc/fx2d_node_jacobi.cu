// Instances of the fixed-point 2D passes (fx2d.cuh): node grids, isotropic stencil, omega-Jacobi.
#include "fx2d.cuh"

namespace mg {
namespace fx2 {
FX2_RUN(node_jacobi_iso) { return dispatch<false, true, kIso>(a, rows, nu, zero, corr, out, nparts, s); }
}  // namespace fx2
}  // namespace mg
