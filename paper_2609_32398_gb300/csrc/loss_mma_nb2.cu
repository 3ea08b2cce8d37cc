// The tensor-core loss kernel at 2 boxes of 32 experts.
#include "loss_mma.cuh"

namespace dol {

DOL_LOSS_MMA_INSTANCE(2)

}  // namespace dol
