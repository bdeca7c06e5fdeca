// Instantiations of the persistent batched stage (first- and second-order DOLINC stencils).
#include "launch.cuh"

namespace dol {

void register_batch_bf16(BatchFns *t) { register_batch<PREC_BF16>(t); }

}  // namespace dol
