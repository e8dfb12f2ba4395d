// Training of the learned decoder: the one-shot-per-block kernels of nms_train.cuh, the weights' edge groups,
// and the Adam step.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include <cuda_runtime.h>

#include "nms_train.cuh"

namespace qldpc {
namespace kern {

// CSR edge order to edge groups (padding is 0: it only ever scales zeros).
__global__ void permute_weights_kernel(const float *__restrict__ w_csr, const int32_t *__restrict__ slot_edge, int32_t T,
                                       int32_t m, int32_t dc_max, int32_t wstride, int32_t group, int32_t nnz,
                                       float *__restrict__ w_groups)
{
    const int64_t S = int64_t(m) * wstride, total = int64_t(T) * S;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
        const int64_t t = i / S;
        const int32_t x = int32_t(i - t * S), g = x / (m * group), c = (x - g * m * group) / group;
        const int32_t j = g * group + x % group;
        const int32_t e = j < dc_max ? __ldg(slot_edge + size_t(j) * m + c) : -1;
        w_groups[i] = e >= 0 ? w_csr[t * nnz + e] : 0.0f;
    }
}

// The gradient's edge groups in CSR edge order.
__global__ void gather_grad_kernel(const float *__restrict__ grad_groups, const uint32_t *__restrict__ eslot, int32_t T,
                                   int32_t m, int32_t wstride, int32_t group, int32_t nnz, float *__restrict__ grad)
{
    const int64_t total = int64_t(T) * nnz;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
        const int64_t t = i / nnz, e = i - t * nnz;
        const uint32_t sl = __ldg(eslot + e), j = sl / uint32_t(m), c = sl - j * uint32_t(m);
        grad[i] = grad_groups[t * m * wstride + train_edge_at(group, int(c), int(j), m)];
    }
}

// One Adam step (Kingma and Ba, 2015) in the form of PyTorch's single-tensor implementation:
//   m = m + (1 - b1) (g - m);  v = b2 v + (1 - b2) g^2;
//   p = p - (lr / (1 - b1^t)) * m / (sqrt(v) / sqrt(1 - b2^t) + eps)
__global__ void adam_kernel(float *__restrict__ param, const float *__restrict__ grad, float *__restrict__ m1,
                            float *__restrict__ m2, int64_t count, float beta1, float beta2, float eps,
                            float step_size, float bc2_sqrt)
{
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x) {
        const float g = grad[i];
        const float a = m1[i] + (1.0f - beta1) * (g - m1[i]);
        const float v = beta2 * m2[i] + (1.0f - beta2) * g * g;
        m1[i] = a;
        m2[i] = v;
        param[i] = param[i] - step_size * (a / (sqrtf(v) / bc2_sqrt + eps));
    }
}

}  // namespace kern

const void *train_forward_x1(const TrainChoice &tc, int loss_kind) { return forward_kernel<1>(tc, loss_kind); }

const void *train_backward(const TrainChoice &tc, int loss_kind)
{
    const bool syn = loss_kind == kLossSyndrome;
#define QLDPC_K(DCV, UNI, DVV)                                                                  \
    if (tc.dc == DCV && tc.uniform == UNI && tc.dvb == DVV)                                     \
        return syn ? reinterpret_cast<const void *>(&kern::nms_backward_kernel<DCV, UNI, DVV, true>) \
                   : reinterpret_cast<const void *>(&kern::nms_backward_kernel<DCV, UNI, DVV, false>);
    QLDPC_TRAIN_SHORT(QLDPC_K)
    QLDPC_TRAIN_LONG(QLDPC_K)
#undef QLDPC_K
    return nullptr;
}

cudaError_t launch_training(const void *kernel, const TrainParams &p, int grid, int threads, size_t smem,
                            cudaStream_t stream)
{
    void *args[] = {const_cast<TrainParams *>(&p)};
    const cudaError_t e = cudaLaunchKernel(kernel, dim3(unsigned(grid)), dim3(unsigned(threads)), args, smem, stream);
    return e != cudaSuccess ? e : cudaGetLastError();
}

namespace {
int elementwise_grid(int64_t count)
{
    return int(std::max<int64_t>(1, std::min<int64_t>((count + 255) / 256, 4096)));
}
}  // namespace

cudaError_t launch_permute_weights(const float *w_csr, const DeviceGraph &g, int32_t T, int32_t wstride, int group,
                                   float *w_groups, cudaStream_t stream)
{
    kern::permute_weights_kernel<<<elementwise_grid(int64_t(T) * g.m * wstride), 256, 0, stream>>>(
        w_csr, g.slot_edge, T, g.m, g.dc_max, wstride, group, g.nnz, w_groups);
    return cudaGetLastError();
}

cudaError_t launch_gather_grad(const float *grad_groups, const DeviceGraph &g, int32_t T, int32_t wstride, int group,
                               float *grad, cudaStream_t stream)
{
    kern::gather_grad_kernel<<<elementwise_grid(int64_t(T) * g.nnz), 256, 0, stream>>>(grad_groups, g.eslot, T, g.m, wstride,
                                                                                       group, g.nnz, grad);
    return cudaGetLastError();
}

cudaError_t launch_adam(float *param, const float *grad, float *m1, float *m2, int64_t count, int32_t step,
                        float lr, float beta1, float beta2, float eps, cudaStream_t stream)
{
    const double bc1 = 1.0 - std::pow(double(beta1), double(step));
    const double bc2 = 1.0 - std::pow(double(beta2), double(step));
    kern::adam_kernel<<<elementwise_grid(count), 256, 0, stream>>>(param, grad, m1, m2, count, beta1, beta2, eps,
                                                                   float(double(lr) / bc1), float(std::sqrt(bc2)));
    return cudaGetLastError();
}

}  // namespace qldpc
