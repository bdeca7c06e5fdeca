// Instantiations of the stage paths for dim = 2, 4 variable(s), F32.
#include "launch.cuh"

namespace dol {

void register_paths_d2e_f32(PathFns *t) { register_paths<2, 4, PREC_F32>(t); }

}  // namespace dol
