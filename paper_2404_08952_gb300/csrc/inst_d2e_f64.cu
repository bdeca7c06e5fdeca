// Instantiations of the stage paths for dim = 2, 4 variable(s), F64.
#include "launch.cuh"

namespace dol {

void register_paths_d2e_f64(PathFns *t) { register_paths<2, 4, PREC_F64>(t); }

}  // namespace dol
