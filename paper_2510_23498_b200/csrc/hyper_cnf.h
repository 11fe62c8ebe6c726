// Kernels of the hypernetwork flow with the exact trace (Sec. 6.1, the two-dimensional experiments): see hyper_cnf.cu.
#pragma once
#include "common.cuh"
#include "rk_fused.h"

namespace mpode {

constexpr int HYPER_MAX_D = 8;

size_t hyper_param_count(int h, int w, int d);       // A1, c1, A2, c2, A3, c3
size_t hyper_stage_floats(int h, int w, int d);      // h1, h2, the w weight sets and the products U_j . W_j of one stage time
size_t hyper_scratch_floats(int w, int d);           // the batch sums of the weight-set cotangents
bool hyper_shape_ok(int h, int w, int d);            // the weight sets of one stage time fit the kernels' shared memory

// k = [v; -tr] for one stage: `hyp` (hyper_stage_floats) receives the hypernetwork's rounded layers, A (low [w][B]) the units
void launch_hyper_forward(mpode_dtype dt, const float* theta, float tau16, int h, int w, int d, float* hyp, const void* Y, void* A, void* k,
                          void* k_l, int B, cudaStream_t st, long long* launches);
// psi and dg = (beta != 0 ? beta * dg : 0) + dtheta of one stage from its cotangent (kappa low [B, d], kappa_l low [B]).
// Sb: low [w][B] scratch for the unit cotangents; sums: hyper_scratch_floats; counter: a device word that is zero between calls;
// non-finite low-format values raise *flag (flag may be null)
void launch_hyper_vjp(mpode_dtype dt, const float* theta, float tau16, int h, int w, int d, const float* hyp, const void* Y, const void* A,
                      void* Sb, const void* kappa, const void* kappa_l, void* psi, float* sums, float* dg, float beta, int B, unsigned* flag,
                      unsigned* counter, cudaStream_t st, long long* launches);

// The whole solve (hyper_solve.cu).  launch_hyper_table evaluates the hypernetwork for every stage time of the solve into
// table[step][4] (hyper_stage_floats each); the forward kernel runs Alg. 1, the backward kernel (a cooperative launch) Alg. 2 with its
// scale decisions.
struct HyperSolve {
    int B, d, h, w, stages, n_steps, round_increment;
    const float* theta;
    const float* table; long long stage_floats;
    const RkStepScalars* scal;          // device [n_steps]
    void* traj;                         // low [(n_steps + 1)][B][d]
    // forward
    const float* y0; float* yT;         // fp32 [B][d], [B][d + 1]
    // backward
    const float* dLdyT; float* a; float* g; int accumulate;
    const float* cot;                   // fp32 [n_steps][B][d + 1] running-cost cotangents, or null
    int scaling, k_max, growth_rule, pbits, e0, e0_from_norm;
    float* part;                        // hyper_solve_part_floats: every block's sums of the weight-set cotangents over its samples
    float* tpart;                       // hyper_solve_tpart_floats: the weight sets' parts of the cotangent of h2
    float* dg;                          // [p] the attempt's parameter gradient
    float* a_new;                       // [B][d + 1] the adjoint the attempt would leave
    unsigned* words;                    // 16 device words, zero at launch
    unsigned long long wait_ns;         // limit of a grid barrier
    int starve;                         // test of that limit: the last block's last barrier waits for one arrival too many
    int *log_exp, *log_attempts, *log_doubled, *status;     // device [n_steps] each; status [4], zero at launch
};
bool hyper_solve_shape_ok(mpode_dtype dt, int h, int w, int d, int stages);
size_t hyper_solve_part_floats(mpode_dtype dt, int B, int h, int w, int d);
size_t hyper_solve_tpart_floats(int h, int w);
void launch_hyper_table(mpode_dtype dt, const float* theta, const RkStepScalars* scal, int n_steps, int stages, int h, int w, int d, float* table,
                        cudaStream_t st, long long* launches);
bool launch_hyper_solve_forward(mpode_dtype dt, const HyperSolve& p, cudaStream_t st, long long* launches);
bool launch_hyper_solve_backward(mpode_dtype dt, const HyperSolve& p, cudaStream_t st, long long* launches);

}  // namespace mpode
