// Instances of the fixed-point 2D passes (fx2d.cuh): node grids, anisotropic stencil.
#include "fx2d.cuh"

namespace mg {
namespace fx2 {
FX2_RUN(node_rbgs_gen) { return dispatch<false, false, kGen>(a, rows, nu, zero, corr, out, nparts, s); }
FX2_RUN(node_jacobi_gen) { return dispatch<false, true, kGen>(a, rows, nu, zero, corr, out, nparts, s); }
}  // namespace fx2
}  // namespace mg
