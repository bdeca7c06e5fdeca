// Instantiations of the stage paths for dim = 3, 1 variable(s), BF16.
#include "launch.cuh"

namespace dol {

void register_paths_d3s_bf16(PathFns *t) { register_paths<3, 1, PREC_BF16>(t); }

}  // namespace dol
