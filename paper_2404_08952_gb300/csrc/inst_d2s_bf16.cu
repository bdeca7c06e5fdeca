// Instantiations of the stage paths for dim = 2, 1 variable(s), BF16.
#include "launch.cuh"

namespace dol {

void register_paths_d2s_bf16(PathFns *t) { register_paths<2, 1, PREC_BF16>(t); }

}  // namespace dol
