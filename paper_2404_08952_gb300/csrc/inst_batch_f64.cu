// Instantiations of the persistent batched stage (first- and second-order DOLINC stencils).
#include "launch.cuh"

namespace dol {

void register_batch_f64(BatchFns *t) { register_batch<PREC_F64>(t); }

}  // namespace dol
