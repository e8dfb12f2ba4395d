// Training of the learned decoder: the two-shots-per-block kernels of nms_train.cuh.
#include "nms_train.cuh"

namespace qldpc {

const void *train_kernel_x2(const TrainChoice &tc, int loss_kind, bool backward)
{
    return backward ? train_kernel<2, true>(tc, loss_kind) : train_kernel<2, false>(tc, loss_kind);
}

}  // namespace qldpc
