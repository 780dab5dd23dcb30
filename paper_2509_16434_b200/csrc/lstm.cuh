// The recurrent cell, shared by the persistent time loop (lstm.cu) and the step-by-step kernels (encoder.cu).
#pragma once
#include "common.cuh"

constexpr int kLstmCounters = 256;  // rows of 32 words: counters of the persistent kernels

// One layer's sequence: T steps of Be envs, H units; arrays of T * Be rows (see ppo_model).
struct LstmSteps {
    int T, Be, H;
    const uint8_t *done;
    float *gates, *c, *cprev;
    bf16 *h, *hprev;
    unsigned int *counters;  // zero between launches
};

// The whole time loop of a layer in one launch; PPO_ERR_UNSUPPORTED (nothing launched) where it does not fit.
int lstm_fwd_steps(const LstmSteps &p, const bf16 *Wh, const float *xg, const float *bias, const float *h_init, const float *c_init,
                   int32_t *status, cudaStream_t st);
// A sequence of one step, W_x x included (X [Be][in]); hprev and cprev hold the state it starts from.
// ends: where the state after the step goes as well, fp32 and zero where done (null: nowhere; 16-byte aligned).  The last argument of the
// kernel: a step prepared once is launched again with others.
struct LstmStepEnds {
    float *h_out, *c_out;
    const uint8_t *done;
};
int lstm_one_step(const LstmSteps &p, const bf16 *X, int in, const bf16 *Wx, const bf16 *Wh, const float *bias, const LstmStepEnds &ends,
                  int32_t *status, cudaStream_t st);
// WhT: W_h^T [H][4H].  dhc: 4 * Be * H floats of scratch.
int lstm_bwd_steps(const LstmSteps &p, const bf16 *WhT, const float *dtop, bf16 *dg, float *dhc, int32_t *status, cudaStream_t st);

__device__ __forceinline__ float sigmoidf_(float x) { return 1.f / (1.f + __expf(-x)); }

// Gate pre-activations -> gate activations, cell state and output.
__device__ __forceinline__ void lstm_cell(float pi, float pf, float pg, float po, float c_prev, float &gi, float &gf, float &gg,
                                          float &go, float &c, float &h) {
    gi = sigmoidf_(pi);
    gf = sigmoidf_(pf);
    gg = tanhf(pg);
    go = sigmoidf_(po);
    c = gf * c_prev + gi * gg;
    h = go * tanhf(c);
}

// Gradient of the output (dh) and of the cell state (dc_in, from the next step) -> gradients of the gate pre-activations and
// of the state the step started from.
__device__ __forceinline__ void lstm_cell_back(float dh, float dc_in, float gi, float gf, float gg, float go, float c, float c_prev,
                                               float &di, float &df, float &dgg, float &dgo, float &dc_out) {
    const float tc = tanhf(c);
    const float dc = dc_in + dh * go * (1.f - tc * tc);
    di = dc * gg * gi * (1.f - gi);
    df = dc * c_prev * gf * (1.f - gf);
    dgg = dc * gi * (1.f - gg * gg);
    dgo = dh * tc * go * (1.f - go);
    dc_out = dc * gf;
}
