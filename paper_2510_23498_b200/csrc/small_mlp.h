// Row-local kernels for small dense velocities: see small_mlp.cu.
#pragma once
#include "common.cuh"
#include "rk_fused.h"

namespace mpode {

constexpr int SMALL_MAX_L = 4;

struct SmallMlp {
    int B, L, stages, act, time, bias, round_increment;
    int alone;                                         // every stage of the tableau depends on the one before it and no other
    int wr[SMALL_MAX_L + 1], wp[SMALL_MAX_L + 1];      // layer widths; rounded up to multiples of 8
    const float* theta; long long woff[SMALL_MAX_L], boff[SMALL_MAX_L];
    // weights in the order they are used (launch_small_pack): matrix instruction fragments, or rows in float32; forward: columns = outputs, reduction = inputs; backward: the other way round.  Biases and time column: low format, padded with zeros
    uint4 *wf[SMALL_MAX_L], *wb[SMALL_MAX_L];
    void *b16[SMALL_MAX_L], *wt16;
    const RkStepScalars* scal;                         // device, indexed by absolute step
    void* traj;                                        // low [(n + 1)][B][d]
    // forward
    int n_steps; const float* y0; float* yT;
    // backward: steps step_hi, step_hi - 1, ... (count of them); slot s of the slabs belongs to step step_hi - s
    int step_hi, count, recompute, vjp, commit;
    float* a; const float* cot;                        // fp32 [B][d]; [n][B][d] running-cost cotangents or null (commit only)
    int e; const int* e_dev;                           // log2 of the adjoint scale (on the device when e_dev is given)
    void* xs[SMALL_MAX_L];                             // layer inputs X_l (X_0 = Y_j): [slot][stages][B][wp_l]
    void* zs[SMALL_MAX_L + 1];                         // cotangents dZ_l, l = 1 .. L (dZ_L = kappa_j): [slot][stages][B][wp_l]
    void* psi[4];                                      // without commit: psi_j, low [B][wp_0]
    unsigned* flag;
    unsigned* err;                                     // a bounded wait that gave up
    unsigned long long wait_ns; int starve;            // limit of every wait; test of it: the backward kernel's weights stop coming
    int ring;                                          // buffers of the weight stream (set by the launch)
    // time-grid gradient (null: not wanted): [slot][blocks][3] shares; results of the last step [3]; t' [n + 1], updated per step
    float *tpart, *tvals, *tprime;
    // weight gradient: out = beta out + sum over the slots of coef[slot] (parameter gradient of the step)
    float* out; float beta; float coef[16];
};
constexpr int SMALL_MAX_CHUNK = 16;

// bytes of packed weights (both directions); whether the kernels take these widths
size_t small_pack_elems(mpode_dtype dt, int n, int k);      // of one layer and direction: n columns, reduction of k
size_t small_pack_bytes(mpode_dtype dt, int L, const int* wp);
bool small_mlp_supported(mpode_dtype dt, int B, int L, const int* wp);
bool small_backward_supported(mpode_dtype dt, int B);       // of a network that small_mlp_supported takes

void launch_small_pack(mpode_dtype dt, const SmallMlp& p, cudaStream_t st, long long* launches);
bool launch_small_forward(mpode_dtype dt, const SmallMlp& p, cudaStream_t st, long long* launches);
// Whether the backward kernels can be launched.  Asked before the first of them: a pass that has committed steps cannot change its path
// (a launch that the runtime refuses after that leaves its error for the driver)
bool small_backward_ready(mpode_dtype dt, const SmallMlp& p);
void launch_small_backward(mpode_dtype dt, const SmallMlp& p, cudaStream_t st, long long* launches);
int small_blocks(mpode_dtype dt, int B);                               // blocks of the forward and backward kernels
void launch_small_time(mpode_dtype dt, const SmallMlp& p, int blocks, cudaStream_t st, long long* launches);
bool small_wgrad_ready(mpode_dtype dt, const SmallMlp& p);
void launch_small_wgrad(mpode_dtype dt, const SmallMlp& p, cudaStream_t st, long long* launches);

}  // namespace mpode
