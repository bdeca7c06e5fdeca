// Instantiations of the stage paths for dim = 3, 5 variable(s), F32.
#include "launch.cuh"

namespace dol {

void register_paths_d3e_f32(PathFns *t) { register_paths<3, 5, PREC_F32>(t); }

}  // namespace dol
