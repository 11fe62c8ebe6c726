// Row-local kernels whose weights stay in shared memory through the whole launch: see resident_mlp.cu.
#pragma once
#include "small_mlp.h"

namespace mpode {

// What a network and batch get from these kernels (fixed when the workspace is planned, for tableaux of up to four stages).
struct ResidentPlan {
    bool forward = false, backward = false;
    int mt_f = 1, mt_b = 1;             // row tiles of 8 per block
    int blocks_f = 0, blocks_b = 0;
    int sw[SMALL_MAX_L + 1] = {0};      // elements of a row of width wp[l] in shared memory
    int w_at[SMALL_MAX_L] = {0};        // element offset of layer l's weights in the image
    int b_at[SMALL_MAX_L] = {0}, t_at = 0;      // float offsets of the biases and the time column behind the weights
    int w_elems = 0, image_bytes = 0;
    int pieces = 0;                     // 16 x 8 pieces of the parameter gradient (bias columns included) that live in registers; 0: too many
    long long params = 0;
};

// Byte offsets of the rows' buffers in a block's shared memory (R rows of sw[l] elements each).  A parameter of the launch: indexed by layer
// in a kernel's own memory they would be trips to the L2, with nearly all of the L1 taken as shared memory.
struct ResidentBufs {
    int state = 0;                                      // bytes of a buffer of the state's width
    int z0 = 0, z[SMALL_MAX_L] = {0};                   // layer inputs or cotangents: two of the state's width, one of each hidden layer's
    int x00 = 0;                                        // backward: the stored state, two buffers,
    int keep = 0, keep_stage = 0, keep_at[SMALL_MAX_L] = {0};      // and every layer input of every stage
    int slots = 0;                                      // end of the buffers
};

struct ResidentMlp {
    SmallMlp s;
    ResidentPlan g;
    ResidentBufs b;                     // (set by the launch)
    unsigned char* image = nullptr;     // packed weights, biases and time column as they lie in shared memory
    float* partial = nullptr;           // parameter gradients of the blocks, or null: layer inputs and cotangents go to the slabs of `s`
};

ResidentPlan plan_resident(mpode_dtype dt, int B, int L, const int* wp, bool bias, bool time);
void launch_resident_pack(mpode_dtype dt, const ResidentMlp& p, cudaStream_t st, long long* launches);
bool launch_resident_forward(mpode_dtype dt, const ResidentMlp& p, cudaStream_t st, long long* launches);
bool resident_backward_ready(mpode_dtype dt, const ResidentMlp& p);      // as small_backward_ready
void launch_resident_backward(mpode_dtype dt, const ResidentMlp& p, cudaStream_t st, long long* launches);
void launch_resident_reduce(const ResidentMlp& p, cudaStream_t st, long long* launches);      // out = beta out + sum of the blocks' gradients

}  // namespace mpode
