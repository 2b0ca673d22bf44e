// Instances of the fixed-point 3D passes (fx3d.cuh): red-black sweeps.
#include "fx3d.cuh"

namespace mg {
namespace fx3 {
FX3_RUN(rbgs_iso) { return dispatch<false, kIso>(a, zero, corr, out, nparts, s); }
FX3_RUN(rbgs_gen) { return dispatch<false, kGen>(a, zero, corr, out, nparts, s); }
}  // namespace fx3
}  // namespace mg
