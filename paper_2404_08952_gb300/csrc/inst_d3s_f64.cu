// Instantiations of the stage paths for dim = 3, 1 variable(s), F64.
#include "launch.cuh"

namespace dol {

void register_paths_d3s_f64(PathFns *t) { register_paths<3, 1, PREC_F64>(t); }

}  // namespace dol
