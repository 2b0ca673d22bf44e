// Instances of the fixed-point 3D passes (fx3d.cuh): omega-Jacobi.
#include "fx3d.cuh"

namespace mg {
namespace fx3 {
FX3_RUN(jacobi_iso) { return dispatch<true, kIso>(a, zero, corr, out, nparts, s); }
FX3_RUN(jacobi_gen) { return dispatch<true, kGen>(a, zero, corr, out, nparts, s); }
}  // namespace fx3
}  // namespace mg
