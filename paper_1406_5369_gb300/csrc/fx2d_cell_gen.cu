// Instances of the fixed-point 2D passes (fx2d.cuh): cell grids, anisotropic stencil.
#include "fx2d.cuh"

namespace mg {
namespace fx2 {
FX2_RUN(cell_rbgs_gen) { return dispatch<true, false, kGen>(a, rows, nu, zero, corr, out, nparts, s); }
FX2_RUN(cell_jacobi_gen) { return dispatch<true, true, kGen>(a, rows, nu, zero, corr, out, nparts, s); }
}  // namespace fx2
}  // namespace mg
