// prop.cuh -- declarations shared by the proposal network's training and inference code.
#pragma once

#include <vector>

#include "hgm_internal.cuh"

namespace hgm {

constexpr int kPropHidden = 128;
constexpr uint32_t kPropMagic = 0x50524f50u;   // "PROP"

// Flat FP32 parameter vector: W1 [H x dp] (d_in used), b1, W2 [H x H], b2, w3, b3 (padded to 4).
struct PropLayout {
    int F = 0, d_in = 0, dp = 0;
    int64_t o_W1 = 0, o_b1 = 0, o_W2 = 0, o_b2 = 0, o_w3 = 0, o_b3 = 0, n = 0, n_logical = 0;
};

// Scratch of the training and forward passes, sized for batches of up to cap rows.
struct PropTrain {
    void *buf = nullptr;
    int cap = 0;
    float *part = nullptr;   // per CTA of a pass: its share of the gradient, L.n floats
    float *z3 = nullptr;     // logits of a forward pass whose output lies in its input
    float *loss = nullptr;   // mean loss of the last pass
    int *status = nullptr;   // 1 once a bounded tensor-core wait gave up
    cudaError_t ensure(const PropLayout &L, int B);
};

PropLayout prop_layout(int F);
void prop_pack(const PropLayout &L, const float *logical, std::vector<float> &flat);
void prop_unpack(const PropLayout &L, const float *flat, float *logical);
void prop_init(const PropLayout &L, uint64_t seed, std::vector<float> &logical);
// logits z3 [B] of X [B x d_in] (row stride ldx)
cudaError_t prop_forward(const PropLayout &L, const float *theta, PropTrain &w, const float *X, int ldx, int B,
                         float *logits, cudaStream_t st);
// gradient of the mean loss on (X, y) into grad (padded layout) and the loss into w.loss; with t > 0 also the t-th
// Adam step on theta (moments m, v)
cudaError_t prop_step(const PropLayout &L, float *theta, PropTrain &w, const float *X, int ldx, const float *y, int B,
                      float *grad, float *m, float *v, int64_t t, float lr, cudaStream_t st);

}  // namespace hgm

struct hgm_prop;
void prop_free(hgm_prop *p);   // device buffers of a proposal handle (prop_api.cu)

struct hgm_prop {
    uint32_t magic;
    hgm::PropLayout L;
    float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;   // device, L.n floats each
    int64_t step = 0;
    hgm::PropTrain train;
};
