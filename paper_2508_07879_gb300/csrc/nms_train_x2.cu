// Training of the learned decoder: the two-shots-per-block forward kernels of nms_train.cuh.
#include "nms_train.cuh"

namespace qldpc {

const void *train_forward_x2(const TrainChoice &tc, int loss_kind) { return forward_kernel<2>(tc, loss_kind); }

}  // namespace qldpc
