// The tensor-core loss kernel at 1 box of 32 experts.
#include "loss_mma.cuh"

namespace dol {

DOL_LOSS_MMA_INSTANCE(1)

}  // namespace dol
