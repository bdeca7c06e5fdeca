// Instantiations of the persistent batched stage (first- and second-order DOLINC stencils).
#include "launch.cuh"

namespace dol {

void register_batch_f32(BatchFns *t) { register_batch<PREC_F32>(t); }

}  // namespace dol
