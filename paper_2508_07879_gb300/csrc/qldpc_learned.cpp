// Host side of the learned-decoder entry points of include/qldpc.h: weight upload for learned
// decoding, workspace sizing, argument validation and launches of the training kernels
// (nms_train.cuh), the Adam step, the device error sampler and the logical-failure test.  No
// arithmetic of the method runs here.
#include "qldpc.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include <cuda_runtime.h>

#include "graph.h"
#include "msa_launch.h"

using namespace qldpc;
using namespace qldpc::detail;

namespace {

constexpr int32_t kMaxLearnedIters = 4096;
constexpr size_t kAlign = 256;

size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

// Compiled training variant for a graph (see nms_train.cuh), or dc = -1 if none.
TrainChoice train_choice(const qldpc_graph *g)
{
    const int dvb = dv_bucket(g->dv_max);
    if (g->uniform_rows && g->dc_max >= 6 && g->dc_max <= 8 && dvb <= 8) return TrainChoice{g->dc_max, true, dvb};
    const int dcb = dc_bucket(g->dc_max);
    if (dcb < 0 || dvb < 0) return TrainChoice{-1, false, 0};
    return TrainChoice{dcb, false, std::max(8, dvb)};
}

struct TrainPlan {
    TrainChoice tc{};
    int threads[2] = {};                             // [backward]
    int grid[2][2] = {};                             // [loss kind][backward]
    const void *kernel[2][2] = {};
    size_t smem[2][2] = {};
    int32_t wstride = 0, group = 4;
    size_t w_off = 0, state_off = 0, part_off = 0, total = 0;
};

int plan_training_uncached(const qldpc_graph *g, int32_t batch, int32_t T, TrainPlan &tp);

// The plan of the graph's last (batch, T), else a new one (occupancy queries cost host time on
// every training step otherwise).
int plan_training(const qldpc_graph *g, int32_t batch, int32_t T, TrainPlan &tp)
{
    static_assert(sizeof(TrainPlan) <= sizeof(g->train_plan), "plan cache too small");
    qldpc_graph *mg = const_cast<qldpc_graph *>(g);
    std::lock_guard<std::mutex> lk(mg->train_mu);
    if (mg->train_batch == batch && mg->train_T == T) {
        std::memcpy(&tp, mg->train_plan, sizeof(TrainPlan));
        return QLDPC_OK;
    }
    if (int rc = plan_training_uncached(g, batch, T, tp)) return rc;
    std::memcpy(mg->train_plan, &tp, sizeof(TrainPlan));
    mg->train_batch = batch;
    mg->train_T = T;
    return QLDPC_OK;
}

// Forward.  Two shots per block share weights and edge lists, where they fit and every SM still gets
// several blocks; below that the batch is spread one shot per block (LP-1054, T = 20, syndrome loss, one
// against two shots per block, us: 456 shots 112 | 133, 608 shots 139 | 135, 4096 shots 725 | 669; 72 checks on 144
// variables, 608 shots 47 | 51, 1216 shots 62 | 59, 4096 shots 149 | 133).
constexpr int kPairShotsPerSm = 3;

int plan_forward(const qldpc_graph *g, int32_t batch, int shots, TrainPlan &tp)
{
    for (int kind = 0; kind < 2; ++kind) {
        tp.kernel[kind][0] = shots == 2 ? train_forward_x2(tp.tc, kind) : train_forward_x1(tp.tc, kind);
        if (!tp.kernel[kind][0]) return QLDPC_ERR_UNSUPPORTED;
        tp.smem[kind][0] = train_layout(g->m, g->nv, g->dc_max, shots, false, kind == kLossSyndrome).total;
        if (int rc = ensure_kernel_attrs(tp.kernel[kind][0], tp.smem[kind][0], g->smem_optin)) return rc;
        tp.grid[kind][0] = int((int64_t(batch) + shots - 1) / shots);
    }
    // threads: one pass over the checks of a small code
    tp.threads[0] = std::min(kTrainThreads, std::max(64, (g->m + 31) / 32 * 32));
    return QLDPC_OK;
}

// Backward.  One shot per block of 128 threads, four blocks an SM that take the shots in waves (up to two shots per SM, where
// no order is left to keep, each its own block of the forward's size: LP-1054, 304 shots 149 us).  The blocks add into one
// buffer, small shares into sums that have grown large, so the order in which shots arrive shows.  LP-1054, 4096 shots,
// T = 20, syndrome loss: a gradient is off an exactly rounded sum by 7e-6 of its norm, two runs of these waves differ by
// 5e-7, and other schedules lie further from them than that: two shots per block 7.7e-7 (1153 us, where the waves take
// 1572), blocks of 192 threads 1.5e-6, the two halves of the batch in turn 5e-6.  What the next step can make of such
// distances (nms_train.cuh) decides for the order that training has always had.
constexpr int kBackwardThreads = 128, kBackwardBlocksPerSm = 4, kBackwardWideShotsPerSm = 2;

int plan_backward(const qldpc_graph *g, int32_t batch, TrainPlan &tp)
{
    const bool wide = int64_t(batch) <= int64_t(kBackwardWideShotsPerSm) * g->sm_count;
    tp.threads[1] = wide ? tp.threads[0] : kBackwardThreads;
    for (int kind = 0; kind < 2; ++kind) {
        tp.kernel[kind][1] = train_backward(tp.tc, kind);
        if (!tp.kernel[kind][1]) return QLDPC_ERR_UNSUPPORTED;
        tp.smem[kind][1] = train_layout(g->m, g->nv, g->dc_max, 1, true, kind == kLossSyndrome).total;
        if (int rc = ensure_kernel_attrs(tp.kernel[kind][1], tp.smem[kind][1], g->smem_optin)) return rc;
        int per_sm = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, tp.kernel[kind][1], tp.threads[1], tp.smem[kind][1]);
        if (e != cudaSuccess) return cuda_status(e);
        if (per_sm < 1) return QLDPC_ERR_UNSUPPORTED;
        tp.grid[kind][1] = wide ? batch : int(std::min<int64_t>(batch, int64_t(std::min(per_sm, kBackwardBlocksPerSm)) * g->sm_count));
    }
    return QLDPC_OK;
}

int plan_training_uncached(const qldpc_graph *g, int32_t batch, int32_t T, TrainPlan &tp)
{
    tp.tc = train_choice(g);
    if (tp.tc.dc < 0) return QLDPC_ERR_UNSUPPORTED;
    if (!g->dg.vslot16) return QLDPC_ERR_UNSUPPORTED;   // (more edge slots than any training block holds)
    int rc = QLDPC_ERR_UNSUPPORTED;
    if (int64_t(batch) > int64_t(kPairShotsPerSm) * g->sm_count) rc = plan_forward(g, batch, 2, tp);
    if (rc == QLDPC_ERR_UNSUPPORTED) rc = plan_forward(g, batch, 1, tp);
    if (!rc) rc = plan_backward(g, batch, tp);
    if (rc) return rc;
    tp.group = train_group(tp.tc.dc, tp.tc.uniform);
    tp.wstride = (g->dc_max + tp.group - 1) / tp.group * tp.group;
    const size_t rows = size_t(T) * size_t(g->m) * size_t(tp.wstride) * sizeof(float);
    tp.w_off = 0;
    tp.state_off = align_up(rows);
    tp.part_off = tp.state_off + align_up(size_t(batch) * size_t(T) * size_t(g->m) * sizeof(uint4));
    tp.total = tp.part_off + align_up(rows);
    return QLDPC_OK;
}

int check_workspace(const TrainPlan &tp, const void *ws, size_t bytes)
{
    if (!ws || bytes < tp.total || (reinterpret_cast<uintptr_t>(ws) % kAlign) != 0) return QLDPC_ERR_INVALID_ARG;
    return QLDPC_OK;
}

TrainParams train_params(const qldpc_graph *g, const TrainPlan &tp, const uint8_t *syn, const uint8_t *target,
                         int32_t batch, const float *prior, int32_t T, void *ws)
{
    TrainParams p{};
    char *b = static_cast<char *>(ws);
    p.g = g->dg;
    p.syn = syn;
    p.target = target;
    p.prior = prior;
    p.w = reinterpret_cast<const float *>(b + tp.w_off);
    p.wstride = tp.wstride;
    p.state = reinterpret_cast<uint4 *>(b + tp.state_off);
    p.partial = reinterpret_cast<float *>(b + tp.part_off);
    p.T = T;
    p.batch = batch;
    return p;
}

}  // namespace

extern "C" {

int qldpc_graph_set_weights(qldpc_graph *g, const float *weights, int32_t T)
{
    if (!g || T < 0 || T > kMaxLearnedIters || (T > 0 && !weights)) return QLDPC_ERR_INVALID_ARG;
    if (int rc = check_device(g)) return rc;
    if (T == 0) {
        if (g->d_weights) cudaFree(g->d_weights);
        g->d_weights = nullptr;
        g->learned_T = 0;
        return QLDPC_OK;
    }
    const size_t count = size_t(T) * size_t(g->nnz);
    std::vector<float> host(count);
    cudaError_t e = cudaMemcpy(host.data(), weights, count * sizeof(float), cudaMemcpyDefault);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return QLDPC_ERR_INVALID_ARG;   // not a readable host or device range
    }
    for (float x : host)
        if (!std::isfinite(x)) return QLDPC_ERR_INVALID_ARG;
    // edge groups: the weight of CSR edge e at position j of row i sits at train_edge_at(4, i, j, m)
    const size_t S = learned_stride(g->dc_max, g->m);
    std::vector<uint32_t> eslot(size_t(g->nnz));
    e = cudaMemcpy(eslot.data(), g->dg.eslot, eslot.size() * sizeof(uint32_t), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_status(e);
    for (uint32_t &x : eslot) x = uint32_t(train_edge_at(4, int(x % uint32_t(g->m)), int(x / uint32_t(g->m)), g->m));
    std::vector<float> slot(size_t(T) * S, 0.0f);
    for (int32_t t = 0; t < T; ++t)
        for (int32_t i = 0; i < g->nnz; ++i) slot[size_t(t) * S + eslot[size_t(i)]] = host[size_t(t) * g->nnz + i];
    float *d = nullptr;
    e = cudaMalloc(&d, slot.size() * sizeof(float));
    if (e != cudaSuccess) return cuda_status(e);
    e = cudaMemcpy(d, slot.data(), slot.size() * sizeof(float), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(d);
        return cuda_status(e);
    }
    if (g->d_weights) cudaFree(g->d_weights);
    g->d_weights = d;
    g->learned_T = T;
    return QLDPC_OK;
}

int qldpc_nms_workspace_bytes(const qldpc_graph *g, int32_t batch, int32_t T, size_t *bytes)
{
    if (!g || !bytes || batch < 1 || T < 1 || T > kMaxLearnedIters) return QLDPC_ERR_INVALID_ARG;
    if (int rc = check_device(g)) return rc;
    TrainPlan tp;
    if (int rc = plan_training(g, batch, T, tp)) return rc;
    *bytes = tp.total;
    return QLDPC_OK;
}

int qldpc_nms_forward(const qldpc_graph *g, const uint8_t *syndromes, const uint8_t *targets, int32_t batch,
                      const float *prior, const float *weights, int32_t T, const float *loss_weights,
                      int32_t loss, float *out_loss, float *out_post, void *workspace, size_t workspace_bytes,
                      void *stream)
{
    if (loss != QLDPC_LOSS_ERROR && loss != QLDPC_LOSS_SYNDROME) return QLDPC_ERR_INVALID_ARG;
    if (!g || !syndromes || (!targets && loss == QLDPC_LOSS_ERROR) || !prior || !weights || !out_loss || batch < 1 ||
        T < 1 || T > kMaxLearnedIters)
        return QLDPC_ERR_INVALID_ARG;
    if (int rc = check_device(g)) return rc;
    TrainPlan tp;
    if (int rc = plan_training(g, batch, T, tp)) return rc;
    if (int rc = check_workspace(tp, workspace, workspace_bytes)) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    TrainParams p = train_params(g, tp, syndromes, targets, batch, prior, T, workspace);
    p.loss = out_loss;
    p.post = out_post;
    p.loss_w = loss_weights;
    p.loss_kind = loss;
    cudaError_t e = launch_permute_weights(weights, g->dg, T, tp.wstride, tp.group, const_cast<float *>(p.w), st);
    if (e == cudaSuccess) e = launch_training(tp.kernel[loss][0], p, tp.grid[loss][0], tp.threads[0], tp.smem[loss][0], st);
    return cuda_status(e);
}

int qldpc_nms_backward(const qldpc_graph *g, const uint8_t *syndromes, const uint8_t *targets, int32_t batch,
                       const float *prior, int32_t T, const float *loss_weights, int32_t loss,
                       const float *grad_loss, float *out_grad, void *workspace, size_t workspace_bytes,
                       void *stream)
{
    if (loss != QLDPC_LOSS_ERROR && loss != QLDPC_LOSS_SYNDROME) return QLDPC_ERR_INVALID_ARG;
    if (!g || !syndromes || (!targets && loss == QLDPC_LOSS_ERROR) || !prior || !grad_loss || !out_grad ||
        batch < 1 || T < 1 || T > kMaxLearnedIters)
        return QLDPC_ERR_INVALID_ARG;
    if (int rc = check_device(g)) return rc;
    TrainPlan tp;
    if (int rc = plan_training(g, batch, T, tp)) return rc;
    if (int rc = check_workspace(tp, workspace, workspace_bytes)) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    TrainParams p = train_params(g, tp, syndromes, targets, batch, prior, T, workspace);
    p.grad_loss = grad_loss;
    p.loss_w = loss_weights;
    p.loss_kind = loss;
    cudaError_t e = cudaMemsetAsync(p.partial, 0, tp.total - tp.part_off, st);
    if (e == cudaSuccess) e = launch_training(tp.kernel[loss][1], p, tp.grid[loss][1], tp.threads[1], tp.smem[loss][1], st);
    if (e == cudaSuccess) e = launch_gather_grad(p.partial, g->dg, T, tp.wstride, tp.group, out_grad, st);
    return cuda_status(e);
}

int qldpc_adam_step(float *params, const float *grads, float *exp_avg, float *exp_avg_sq, int64_t count,
                    int32_t step, float lr, float beta1, float beta2, float eps, void *stream)
{
    if (count < 0 || step < 1 || !std::isfinite(lr) || !(beta1 >= 0.0f && beta1 < 1.0f) ||
        !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps >= 0.0f) || !std::isfinite(eps))
        return QLDPC_ERR_INVALID_ARG;
    if (count == 0) return QLDPC_OK;
    if (!params || !grads || !exp_avg || !exp_avg_sq) return QLDPC_ERR_INVALID_ARG;
    return cuda_status(launch_adam(params, grads, exp_avg, exp_avg_sq, count, step, lr, beta1, beta2, eps,
                                   static_cast<cudaStream_t>(stream)));
}

int qldpc_sample_errors(const qldpc_graph *g, uint64_t seed, int64_t first_shot, int32_t batch, double p_lo,
                        double p_hi, uint8_t *out_err, uint8_t *out_syn, void *stream)
{
    if (!g || batch < 0 || first_shot < 0) return QLDPC_ERR_INVALID_ARG;
    if (!(p_lo >= 0.0 && p_hi <= 1.0 && p_lo <= p_hi)) return QLDPC_ERR_INVALID_ARG;
    if (batch == 0) return QLDPC_OK;
    if (!out_err || !out_syn) return QLDPC_ERR_INVALID_ARG;
    if (int rc = check_device(g)) return rc;
    if (int rc = ensure_kernel_attrs(sample_kernel_ptr(), sample_smem(g->m, g->n), g->smem_optin)) return rc;
    return cuda_status(launch_sample(g->dg, seed, first_shot, batch, p_lo, p_hi, out_err, out_syn, g->sm_count,
                                     static_cast<cudaStream_t>(stream)));
}

int qldpc_logical_failures(const uint8_t *logicals, int32_t k, int32_t n, const uint8_t *errors,
                           const uint8_t *decisions, const uint8_t *ok, int32_t batch, uint8_t *out_fail,
                           void *stream)
{
    if (k < 1 || n < 1 || batch < 0) return QLDPC_ERR_INVALID_ARG;
    if (batch == 0) return QLDPC_OK;
    if (!logicals || !errors || !decisions || !ok || !out_fail) return QLDPC_ERR_INVALID_ARG;
    if ((size_t(k) + 1) * size_t((n + 31) / 32) * 4 > 48 * 1024) return QLDPC_ERR_UNSUPPORTED;
    int dev = 0, sms = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return QLDPC_ERR_CUDA;
    const LogicalPlan pl = plan_logical(k, n);
    if (int rc = ensure_kernel_attrs(pl.kernel, pl.smem, size_t(optin))) return rc;
    return cuda_status(launch_logical(pl, logicals, k, n, errors, decisions, ok, batch, out_fail, sms,
                                      static_cast<cudaStream_t>(stream)));
}

}  // extern "C"
