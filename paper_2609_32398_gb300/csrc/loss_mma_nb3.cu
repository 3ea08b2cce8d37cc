// The tensor-core loss kernel at 3 boxes of 32 experts.
#include "loss_mma.cuh"

namespace dol {

DOL_LOSS_MMA_INSTANCE(3)

}  // namespace dol
