// Instances of the fixed-point 2D passes (fx2d.cuh): cell grids, isotropic stencil.
#include "fx2d.cuh"

namespace mg {
namespace fx2 {
FX2_RUN(cell_rbgs_iso) { return dispatch<true, false, kIso>(a, rows, nu, zero, corr, out, nparts, s); }
FX2_RUN(cell_jacobi_iso) { return dispatch<true, true, kIso>(a, rows, nu, zero, corr, out, nparts, s); }
}  // namespace fx2
}  // namespace mg
