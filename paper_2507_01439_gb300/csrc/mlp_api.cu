// C ABI of the proposal-MLP trainer (include/turboreg_internal.h): FP32
// master weights, Adam moments and gradient on the device; the forward,
// backward and update run in the kernels of mlp.cu.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <random>
#include <vector>

#include "tr_common.cuh"
#include "tr_mlp.h"
#include "turboreg_internal.h"

using namespace tr;

struct turboreg_mlp {
    int device = 0;
    int32_t max_samples = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int32_t step = 0;
    float* w = nullptr;      // FP32 master [P]
    float* wbf = nullptr;    // BF16-rounded copy used by the forward [P]
    float* mom = nullptr;    // Adam first moment [P]
    float* vel = nullptr;    // Adam second moment [P]
    // gradient [P], loss, error bits: cleared by one kernel, read by one copy
    float* grad = nullptr;
    float* loss = nullptr;   // grad + P
    uint32_t* err = nullptr; // grad + P + 1
    int32_t stalls = 0;      // failure injection: training passes left that stall
    // page-locked [P + 4]: a parameter vector or gradient, loss, error bits on their
    // way out; then a step's loss, and the steps left out that no call has reported yet
    float* host = nullptr;
    std::mutex host_mu;            // one call at a time between its copy into `host` and its reading of it
    float* step_loss = nullptr;    // host + P + 2
    uint32_t* skipped = nullptr;   // host + P + 3
};

namespace {

#define TM_CHECK(expr)                                                                           \
    do {                                                                                         \
        cudaError_t e_ = (expr);                                                                 \
        if (e_ != cudaSuccess) {                                                                 \
            std::fprintf(stderr, "turboreg mlp: %s failed: %s\n", #expr, cudaGetErrorString(e_)); \
            return TURBOREG_ERR_CUDA;                                                            \
        }                                                                                        \
    } while (0)

void free_all(turboreg_mlp* t)
{
    void* ptrs[] = {t->w, t->wbf, t->mom, t->vel, t->grad};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    if (t->host) cudaFreeHost(t->host);
}

// grad, loss (device) = those of the mean BCE over m samples.
int backward(turboreg_mlp* t, const float* feat, const float* label, int32_t m)
{
    const uint32_t dbg = t->stalls > 0 ? TR_DBG_STALL_TRAIN : 0u;
    if (t->stalls > 0) --t->stalls;
    launch_mlp_train(feat, label, m, t->wbf, t->grad, t->loss, t->err, dbg, t->stream);
    TM_CHECK(cudaGetLastError());
    return TURBOREG_OK;
}

// With the stream idle and host_mu held: TIMEOUT if steps were left out since the last report
// (once; they do not count as steps).
int report_skipped(turboreg_mlp* t)
{
    const uint32_t k = *t->skipped;
    *t->skipped = 0u;
    t->step -= static_cast<int32_t>(k);
    return k != 0u ? TURBOREG_ERR_TIMEOUT : TURBOREG_OK;
}

// `count` values at `src` (device) through the page-locked buffer; the stream
// is then idle; the caller holds host_mu until it has read the buffer, so that
// several threads may read one trainer.  (A copy to pageable memory would be staged by the driver.)
int fetch(turboreg_mlp* t, const float* src, size_t count)
{
    TM_CHECK(cudaMemcpyAsync(t->host, src, sizeof(float) * count, cudaMemcpyDeviceToHost, t->stream));
    TM_CHECK(cudaStreamSynchronize(t->stream));
    return TURBOREG_OK;
}

}  // namespace

extern "C" {

int turboreg_mlp_create(int device, int32_t max_samples, uint64_t seed, void* cuda_stream, turboreg_mlp** out)
{
    if (!out || max_samples < 1) return TURBOREG_ERR_INVALID_ARG;
    *out = nullptr;
    TM_CHECK(cudaSetDevice(device));
    turboreg_mlp* t = new (std::nothrow) turboreg_mlp();
    if (!t) return TURBOREG_ERR_OOM;
    t->device = device;
    t->max_samples = max_samples;
    cudaError_t e = cudaSuccess;
    auto al = [&](void** p, size_t b) {
        if (e == cudaSuccess) e = cudaMalloc(p, b);
    };
    al(reinterpret_cast<void**>(&t->w), sizeof(float) * kMlpParams);
    al(reinterpret_cast<void**>(&t->wbf), sizeof(float) * kMlpParams);
    al(reinterpret_cast<void**>(&t->mom), sizeof(float) * kMlpParams);
    al(reinterpret_cast<void**>(&t->vel), sizeof(float) * kMlpParams);
    al(reinterpret_cast<void**>(&t->grad), sizeof(float) * (kMlpParams + 2));
    if (e == cudaSuccess) e = cudaMallocHost(reinterpret_cast<void**>(&t->host), sizeof(float) * (kMlpParams + 4));
    if (e == cudaSuccess) {
        t->step_loss = t->host + kMlpParams + 2;
        t->skipped = reinterpret_cast<uint32_t*>(t->host + kMlpParams + 3);
        *t->skipped = 0u;
    }
    t->loss = t->grad + kMlpParams;
    t->err = reinterpret_cast<uint32_t*>(t->grad + kMlpParams + 1);
    if (e == cudaSuccess) e = mlp_setup();
    if (e == cudaSuccess) {
        if (cuda_stream) t->stream = static_cast<cudaStream_t>(cuda_stream);
        else {
            e = cudaStreamCreateWithFlags(&t->stream, cudaStreamNonBlocking);
            t->own_stream = true;
        }
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        free_all(t);
        delete t;
        return e == cudaErrorMemoryAllocation ? TURBOREG_ERR_OOM : TURBOREG_ERR_CUDA;
    }
    // He-normal initialisation (std = sqrt(2 / fan_in)), zero biases
    std::vector<float> w(kMlpParams, 0.f);
    std::mt19937_64 rng(seed);
    auto fill = [&](int off, int out_dim, int in_dim) {
        std::normal_distribution<float> nd(0.f, std::sqrt(2.f / static_cast<float>(in_dim)));
        for (int k = 0; k < out_dim * in_dim; ++k) w[off + k] = nd(rng);
    };
    fill(kW1, 64, 8);
    fill(kW2, 128, 64);
    fill(kW3, 64, 128);
    fill(kW4, 1, 64);
    int rc = turboreg_mlp_set_params(t, w.data());
    if (rc == TURBOREG_OK) {
        std::vector<float> z(kMlpParams, 0.f);
        rc = turboreg_mlp_set_state(t, z.data(), z.data(), 0);
    }
    if (rc != TURBOREG_OK) {
        turboreg_mlp_destroy(t);
        return rc;
    }
    *out = t;
    return TURBOREG_OK;
}

void turboreg_mlp_destroy(turboreg_mlp* t)
{
    if (!t) return;
    cudaSetDevice(t->device);
    if (t->stream) cudaStreamSynchronize(t->stream);
    free_all(t);
    if (t->own_stream && t->stream) cudaStreamDestroy(t->stream);
    delete t;
}

int turboreg_mlp_debug_stall(turboreg_mlp* t, int32_t calls)
{
    if (!t || calls < 0) return TURBOREG_ERR_INVALID_ARG;
    t->stalls = calls;
    return TURBOREG_OK;
}

int turboreg_mlp_debug_blocks(turboreg_mlp* t, int32_t m)
{
    if (!t || m < 1 || m > t->max_samples) return -TURBOREG_ERR_INVALID_ARG;
    if (cudaSetDevice(t->device) != cudaSuccess) return -TURBOREG_ERR_CUDA;
    return mlp_train_blocks(m);
}

int turboreg_mlp_get_params(turboreg_mlp* t, float* params)
{
    if (!t || !params) return TURBOREG_ERR_INVALID_ARG;
    TM_CHECK(cudaSetDevice(t->device));
    std::lock_guard<std::mutex> lk(t->host_mu);
    const int rc = fetch(t, t->w, kMlpParams);
    if (rc != TURBOREG_OK) return rc;
    std::memcpy(params, t->host, sizeof(float) * kMlpParams);
    return report_skipped(t);
}

int turboreg_mlp_set_params(turboreg_mlp* t, const float* params)
{
    if (!t || !params) return TURBOREG_ERR_INVALID_ARG;
    for (int k = 0; k < kMlpParams; ++k)
        if (!std::isfinite(params[k])) return TURBOREG_ERR_NONFINITE;
    TM_CHECK(cudaSetDevice(t->device));
    TM_CHECK(cudaMemcpyAsync(t->w, params, sizeof(float) * kMlpParams, cudaMemcpyHostToDevice, t->stream));
    launch_mlp_round(t->w, t->wbf, t->stream);
    TM_CHECK(cudaGetLastError());
    TM_CHECK(cudaStreamSynchronize(t->stream));
    return TURBOREG_OK;
}

int turboreg_mlp_get_state(turboreg_mlp* t, float* m, float* v, int32_t* step)
{
    if (!t || !m || !v || !step) return TURBOREG_ERR_INVALID_ARG;
    TM_CHECK(cudaSetDevice(t->device));
    TM_CHECK(cudaMemcpyAsync(m, t->mom, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost, t->stream));
    TM_CHECK(cudaMemcpyAsync(v, t->vel, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost, t->stream));
    TM_CHECK(cudaStreamSynchronize(t->stream));
    std::lock_guard<std::mutex> lk(t->host_mu);
    const int rc = report_skipped(t);
    *step = t->step;
    return rc;
}

int turboreg_mlp_set_state(turboreg_mlp* t, const float* m, const float* v, int32_t step)
{
    if (!t || !m || !v || step < 0) return TURBOREG_ERR_INVALID_ARG;
    TM_CHECK(cudaSetDevice(t->device));
    TM_CHECK(cudaMemcpyAsync(t->mom, m, sizeof(float) * kMlpParams, cudaMemcpyHostToDevice, t->stream));
    TM_CHECK(cudaMemcpyAsync(t->vel, v, sizeof(float) * kMlpParams, cudaMemcpyHostToDevice, t->stream));
    TM_CHECK(cudaStreamSynchronize(t->stream));
    std::lock_guard<std::mutex> lk(t->host_mu);
    *t->skipped = 0u;   // the steps are counted from here
    t->step = step;
    return TURBOREG_OK;
}

int turboreg_mlp_forward(turboreg_mlp* t, const float* feat, int32_t m, float* prob)
{
    if (!t || !feat || !prob || m < 1) return TURBOREG_ERR_INVALID_ARG;
    TM_CHECK(cudaSetDevice(t->device));
    TM_CHECK(cudaMemsetAsync(t->err, 0, sizeof(uint32_t), t->stream));
    launch_mlp_forward(feat, m, t->wbf, prob, t->err, t->stream);
    TM_CHECK(cudaGetLastError());
    uint32_t err = 0;
    TM_CHECK(cudaMemcpyAsync(&err, t->err, sizeof(uint32_t), cudaMemcpyDeviceToHost, t->stream));
    TM_CHECK(cudaStreamSynchronize(t->stream));
    std::lock_guard<std::mutex> lk(t->host_mu);
    const int rc = report_skipped(t);
    return err ? TURBOREG_ERR_TIMEOUT : rc;
}

int turboreg_mlp_grad(turboreg_mlp* t, const float* feat, const float* label, int32_t m, float* grad, float* loss)
{
    if (!t || !feat || !label || !grad || m < 1 || m > t->max_samples) return TURBOREG_ERR_INVALID_ARG;
    TM_CHECK(cudaSetDevice(t->device));
    int rc = backward(t, feat, label, m);
    if (rc != TURBOREG_OK) return rc;
    std::lock_guard<std::mutex> lk(t->host_mu);
    rc = fetch(t, t->grad, kMlpParams + 2);
    if (rc != TURBOREG_OK) return rc;
    std::memcpy(grad, t->host, sizeof(float) * kMlpParams);
    if (loss) *loss = t->host[kMlpParams];
    uint32_t err;
    std::memcpy(&err, t->host + kMlpParams + 1, sizeof(err));
    rc = report_skipped(t);
    return err ? TURBOREG_ERR_TIMEOUT : rc;
}

int turboreg_mlp_train_step(turboreg_mlp* t, const float* feat, const float* label, int32_t m, float lr,
                            float* loss)
{
    if (!t || !feat || !label || m < 1 || m > t->max_samples || !(lr > 0.f)) return TURBOREG_ERR_INVALID_ARG;
    TM_CHECK(cudaSetDevice(t->device));
    int rc = backward(t, feat, label, m);
    if (rc != TURBOREG_OK) return rc;
    t->step += 1;
    launch_mlp_adam(t->w, t->mom, t->vel, t->grad, t->wbf, t->step, lr, t->loss, loss ? t->step_loss : nullptr,
                    t->err, t->skipped, t->stream);
    TM_CHECK(cudaGetLastError());
    if (loss) {
        TM_CHECK(cudaStreamSynchronize(t->stream));
        std::lock_guard<std::mutex> lk(t->host_mu);
        *loss = *t->step_loss;
        return report_skipped(t);
    }
    return TURBOREG_OK;
}

}  // extern "C"
