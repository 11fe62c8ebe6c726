"""GPU parity at sizes where tiles, slices and padded rows end: just inside, on and just past their edges."""
import numpy as np
import pytest

from paper_2510_23498_b200 import inputs
from _harness import TOL, assert_parity, assert_same_log, rel_l2, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


# CUDA-core contractions: 64 x 64 tiles, reduction chunks of 32, clusters of 1, 2, 4 and 8 reduction slices, vector and scalar loads.
# Tolerance: the float32 mode's 1e-5 against the exact fp64 solution (sums of at most 1025 terms, 1025 * 2^-24 = 6e-5 at worst, 1e-6 typical).
@pytest.mark.parametrize("batch,d,hidden", [(1, 8, 16), (63, 8, 65), (64, 12, 64), (65, 5, 33), (300, 33, 130), (1025, 24, 64)])
def test_float32_mlp_at_tile_edges(batch, d, hidden):
    wl = inputs.mlp_block(batch=batch, n_steps=2, d=d, hidden=hidden, low="f32")
    gpu = run_gpu(wl, low="f32")
    assert_parity(gpu, run_oracle(wl, exact=True), TOL["f32"])
    assert gpu["stats"]["tc_contractions"] == 0 and gpu["stats"]["simt_contractions"] > 0


# 16-bit rows whose length is not a multiple of 8 elements are padded; hidden widths and state widths, each with its remainder, and
# batches that are and are not whole tiles of 64 sample pairs.  Tolerances: those of the formats (rounding-emulating oracle).
@pytest.mark.parametrize("batch,d,hidden,low", [(128, 63, 136, "bf16"), (64, 9, 71, "f16"), (130, 17, 65, "bf16"), (192, 64, 129, "f16")])
def test_flow_with_odd_widths_runs_on_the_tensor_cores(batch, d, hidden, low):
    wl = inputs.cnf_mlp(batch=batch, n_steps=2, d=d, hidden=hidden)
    scaling = "dynamic" if low == "f16" else "none"
    gpu = run_gpu(wl, low=low, scaling=scaling)
    assert_parity(gpu, run_oracle(wl, low=low, scaling=scaling), TOL[low])
    assert gpu["stats"]["simt_contractions"] == 0 and gpu["stats"]["tc_contractions"] > 0


# the same for MLPs (of these sizes on the row-local kernels; the padded fused program and layer-by-layer path are in test_gpu_fused_path.py)
@pytest.mark.parametrize("batch,d,hidden,low", [(200, 64, 137, "bf16"), (130, 33, 100, "bf16"), (257, 71, 65, "f16"), (128, 9, 72, "f16")])
def test_mlp_with_odd_widths_runs_on_the_tensor_cores(batch, d, hidden, low):
    wl = inputs.mlp_block(batch=batch, n_steps=2, d=d, hidden=hidden)
    scaling = "dynamic" if low == "f16" else "none"
    gpu = run_gpu(wl, low=low, scaling=scaling)
    assert_parity(gpu, run_oracle(wl, low=low, scaling=scaling), TOL[low])
    assert gpu["stats"]["simt_contractions"] == 0


# whole-solve kernels of the hypernetwork flow: one sample, a block's samples less and plus one, more sample groups than blocks, more
# weight sets than blocks, a hypernetwork as wide as a block's threads, and sets too large for shared memory (stage by stage)
@pytest.mark.parametrize("batch,d,hidden,w,n_steps", [(1, 2, 8, 16, 3), (7, 2, 32, 33, 2), (9, 3, 16, 200, 2), (2400, 2, 16, 32, 2), (40, 1, 128, 20, 2),
                                                      (30, 6, 8, 600, 2)])
def test_hypernetwork_flow_at_block_edges(batch, d, hidden, w, n_steps):
    wl = inputs.hyper_cnf(batch=batch, n_steps=n_steps, d=d, hidden=hidden, w=w)
    assert_parity(run_gpu(wl, "f32", "none"), run_oracle(wl, exact=True), TOL["f32"])
    gpu, orc = run_gpu(wl, "f16", "dynamic"), run_oracle(wl, "f16", "dynamic")
    assert_parity(gpu, orc, TOL["f16"])
    assert_same_log(gpu["log"], orc["log"])
    assert gpu["stats"]["whole_solve_launches"] == (0 if w == 600 else 2)


# whole-solve kernels of very small networks: every variant (state width 2 / 4 / 8, hidden width 32 / 64), one sample, a full block,
# one more than a block, a full cluster of 16 blocks
@pytest.mark.parametrize("batch,d,hidden", [(1, 2, 32), (64, 1, 5), (65, 4, 33), (513, 3, 32), (1024, 2, 64), (1000, 8, 30), (130, 7, 39)])
def test_tiny_network_variants(batch, d, hidden):
    wl = inputs.toy_mlp(batch=batch, n_steps=4, hidden=hidden)
    if d != 2:
        widths = [d, hidden, d]
        wl = inputs.mlp_block(batch=batch, n_steps=4, d=d, hidden=hidden, low="f16", scaling="dynamic")
        wl.vel["widths"], wl.theta = widths, inputs.mlp_theta(3, widths, True)
    gpu, orc = run_gpu(wl, "f16", "dynamic"), run_oracle(wl, "f16", "dynamic")
    assert_parity(gpu, orc, TOL["f16"])
    assert_same_log(gpu["log"], orc["log"])
    assert gpu["stats"]["whole_solve_launches"] == 2
    assert_parity(run_gpu(wl, "f32", "none"), run_oracle(wl, exact=True), TOL["f32"])


# row-local kernels of small dense networks, weights resident: one row, an odd row, two row tiles of 8 per block (2500: forward, and the other path
# backward), 1 to 4 layers, state widths that are not multiples of 8 or 16, several chunks of steps
@pytest.mark.parametrize("batch,widths,n_steps", [(1, [16, 24, 16], 3), (15, [40, 72, 40], 3), (17, [9, 33, 65, 9], 3), (300, [64, 64], 20),
                                                  (200, [72, 200, 200, 72], 2), (2500, [24, 40, 24], 2), (130, [16, 32, 48, 32, 16], 3)])
def test_small_networks_at_tile_edges(batch, widths, n_steps):
    wl = inputs.mlp_block(batch=batch, n_steps=n_steps, d=widths[0], hidden=widths[1])
    wl.vel["n_layers"], wl.vel["widths"], wl.theta = len(widths) - 1, widths, inputs.mlp_theta(3, widths, True)
    for low, scaling in (("bf16", "none"), ("f16", "dynamic"), ("f16", "none_safe")):
        gpu, orc = run_gpu(wl, low, scaling), run_oracle(wl, low, scaling)
        assert_parity(gpu, orc, TOL[low])
        assert gpu["stats"]["fused_launches"] > 0 and gpu["stats"]["simt_contractions"] == 0
        if scaling == "dynamic":
            assert_same_log(gpu["log"], orc["log"])


# tableaux with fewer than four stages: the buffers hold more of their steps (chunks of steps that end early, the longest chunk of 16), with
# the time terms of every step of a chunk
@pytest.mark.parametrize("solver,n_steps", [("euler", 37), ("midpoint", 21), ("kutta3", 9)])
@pytest.mark.parametrize("low", ["bf16", "f32"])
def test_small_networks_chunks_of_steps_per_tableau(solver, n_steps, low):
    wl = inputs.mlp_block(batch=300, n_steps=n_steps, d=40, hidden=72)
    wl.vel["n_layers"], wl.vel["widths"], wl.theta = 2, [40, 72, 40], inputs.mlp_theta(3, [40, 72, 40], True)
    wl.solver = solver
    gpu = run_gpu(wl, low, "none", want_dt=True)
    orc = run_oracle(wl, exact=True, want_dt=True) if low == "f32" else run_oracle(wl, low, "none", want_dt=True)
    assert_parity(gpu, orc, TOL[low])
    assert rel_l2(gpu["dL_dt"], orc["dL_dt"]) <= TOL[low]
    plain = run_gpu(wl, low, "none")
    assert np.array_equal(plain["a0"], gpu["a0"]) and plain["stats"]["fused_launches"] > 0
    assert rel_l2(plain["g"], gpu["g"]) <= 2.2e-6        # (steps may be grouped otherwise: float32 sums over at most 37 of them, 37 * 2^-24)


# the same in float32 (CUDA cores): one row, a block's 8 rows less and plus one, more row tiles than SMs, odd widths, 1 to 4 layers
@pytest.mark.parametrize("batch,widths,n_steps", [(1, [16, 24, 16], 3), (7, [16, 33, 65, 16], 3), (9, [64, 64], 20), (200, [72, 201, 200, 72], 2),
                                                  (1185, [24, 40, 24], 2), (130, [16, 32, 48, 32, 16], 3)])
def test_small_float32_networks_at_tile_edges(batch, widths, n_steps):
    wl = inputs.mlp_block(batch=batch, n_steps=n_steps, d=widths[0], hidden=widths[1], low="f32")
    wl.vel["n_layers"], wl.vel["widths"], wl.theta = len(widths) - 1, widths, inputs.mlp_theta(3, widths, True)
    gpu = run_gpu(wl, low="f32")
    assert_parity(gpu, run_oracle(wl, exact=True), TOL["f32"])
    assert gpu["stats"]["fused_launches"] > 0


# unscaled-safe passes of small dense networks: the step's parameter gradient alone leaves the format (its sums run over the batch; the
# cotangents and the adjoint stay finite), in one and in several gradient pieces, in one chunk of steps and across chunks, in all formats
@pytest.mark.parametrize("low,batch,widths,n_steps,size", [("f16", 1000, [64, 128, 64], 2, 100.0), ("f16", 1000, [64, 64], 20, 200.0), ("f16", 700, [72, 200, 200, 72], 2, 300.0),
                                                           ("bf16", 1000, [64, 128, 64], 2, 5e36), ("f32", 1000, [64, 128, 64], 2, 5e36)])
def test_small_networks_report_a_parameter_gradient_that_overflows(low, batch, widths, n_steps, size):
    from oracle import BY_NAME, Policy, make_velocity, odeint_backward, odeint_forward
    wl = inputs.mlp_block(batch=batch, n_steps=n_steps, d=widths[0], hidden=widths[1])
    wl.vel["n_layers"], wl.vel["widths"], wl.theta = len(widths) - 1, widths, inputs.mlp_theta(3, widths, True)
    dl = np.full((batch, widths[0]), size)
    gpu = run_gpu(wl, low, "none_safe", dLdyT=dl)
    assert gpu["stats"]["fused_launches"] > 0                                     # the row-local kernels
    assert gpu["status"] == 8 and np.all(np.isposinf(gpu["g"])) and np.all(np.isposinf(gpu["a0"]))
    vel, pol = make_velocity(wl.vel), Policy(low=low, scaling="none_safe")
    traj, _ = odeint_forward(vel, wl.theta, wl.y0, wl.tgrid, BY_NAME["rk4"], pol)
    _, _, log = odeint_backward(vel, wl.theta, traj, wl.tgrid, BY_NAME["rk4"], pol, dl)
    assert log.overflowed
    # the cotangents alone are finite: without the batch sum (one row) nothing overflows, on either side
    one = inputs.mlp_block(batch=1, n_steps=n_steps, d=widths[0], hidden=widths[1])
    one.vel, one.theta, one.y0 = wl.vel, wl.theta, wl.y0[:1]
    gpu = run_gpu(one, low, "none_safe", dLdyT=dl[:1])
    _, g, log = odeint_backward(vel, wl.theta, traj[:, :1], wl.tgrid, BY_NAME["rk4"], pol, dl[:1])
    assert gpu["status"] == 0 and not log.overflowed
    if low != "f32":
        assert rel_l2(gpu["g"], g) <= TOL[low]


# The row-local kernels wait for their weights with a limit (20 ms here).  The weights stop after the first stage: every block gives up, waits
# no more, runs to its end and leaves no copy in flight; the call reports it, and the same context then gives the usual result.
@pytest.mark.parametrize("low,scaling", [("bf16", "none"), ("f16", "dynamic"), ("f32", "none")])
def test_row_local_waits_that_run_out_are_reported(low, scaling):
    import time
    import torch
    from paper_2510_23498_b200 import binding
    wl = inputs.mlp_block(batch=300, n_steps=24, d=64, hidden=160)
    ref = run_gpu(wl, low, scaling)
    ctx = binding.Context(wl.vel, wl.batch, wl.n_steps, low=low, scaling=scaling)
    theta, y0 = torch.from_numpy(wl.theta).cuda(), torch.from_numpy(wl.y0).cuda()
    dl = torch.from_numpy(np.ascontiguousarray(ref["dLdyT"], dtype=np.float32)).cuda()
    ctx.forward(theta, y0, wl.tgrid, wl.solver)
    torch.cuda.synchronize()
    ctx.debug_waits(20_000_000, True)
    t0 = time.perf_counter()
    with pytest.raises(binding.MpodeError) as ei:
        ctx.backward(dl)
    assert ei.value.status == binding.ERR_CUDA and "wait timed out" in str(ei.value)
    assert time.perf_counter() - t0 < 2.0
    ctx.debug_waits(0, False)
    ctx.forward(theta, y0, wl.tgrid, wl.solver)
    a0, g, _, st = ctx.backward(dl)
    assert st == 0 and np.array_equal(a0.cpu().numpy(), ref["a0"]) and np.array_equal(g.cpu().numpy(), ref["g"])
    ctx.close()


# paired (value, tangent) tiles of 64 columns: one tile of 64 sample pairs, several, output columns that end inside a tile, on its edge and
# one vector past it, the smallest reduction length
@pytest.mark.parametrize("batch,d,hidden,low", [(64, 16, 72, "bf16"), (192, 24, 200, "f16"), (128, 72, 64, "bf16"), (512, 8, 256, "f16")])
def test_flow_with_narrow_paired_tiles(batch, d, hidden, low):
    wl = inputs.cnf_mlp(batch=batch, n_steps=2, d=d, hidden=hidden)
    scaling = "dynamic" if low == "f16" else "none"
    gpu = run_gpu(wl, low=low, scaling=scaling)
    assert_parity(gpu, run_oracle(wl, low=low, scaling=scaling), TOL[low])
    assert gpu["stats"]["simt_contractions"] == 0


# 64-channel convolutions whose second layer writes the next stage's input: solvers with such a stage everywhere (Heun, RK4, midpoint),
# nowhere (Euler) and in some stages only (the third-order and the 3/8 tableau); time steps that differ (non-uniform grid)
@pytest.mark.parametrize("solver", ["euler", "midpoint", "heun", "kutta3", "rk38", "rk4"])
def test_conv_block_next_stage_input_per_solver(solver):
    wl = inputs.conv_block(batch=3, n_steps=2, H=16, W=16, C=64, act="softplus", solver=solver)
    wl.tgrid = np.array([0.0, 0.375, 1.0], np.float32)
    for low, scaling in (("f16", "dynamic"), ("bf16", "none")):
        assert_parity(run_gpu(wl, low, scaling), run_oracle(wl, low, scaling), TOL[low])


# 64-channel convolutions: tiles in and out through shared memory.  Every image-row width, fewer tiles than SMs, and more than four per SM
# (the buffers of operand tiles wrap around)
@pytest.mark.parametrize("batch,H,W", [(1, 16, 8), (3, 8, 16), (2, 4, 32), (75, 32, 32)])
def test_conv_block_tile_buffers(batch, H, W):
    wl = inputs.conv_block(batch=batch, n_steps=1, H=H, W=W, C=64, act="softplus", solver="heun")
    assert_parity(run_gpu(wl, "bf16", "none"), run_oracle(wl, "bf16", "none"), TOL["bf16"])


# 64 channels, fewer pixels in all than one k-block of the tensor-core weight gradient
def test_conv_block_of_few_pixels():
    wl = inputs.conv_block(batch=1, n_steps=2, H=7, W=7, C=64, act="softplus")
    assert_parity(run_gpu(wl, "bf16", "none"), run_oracle(wl, "bf16", "none"), TOL["bf16"])


# column sums (bias and time-column gradients of the flow): batches of one row chunk, of chunks that end early, the largest that the
# cluster kernel takes and the next that it does not
@pytest.mark.parametrize("batch", [3, 130, 2048, 2112])
def test_flow_column_sums_at_chunk_edges(batch):
    wl = inputs.cnf_mlp(batch=batch, n_steps=1, d=16, hidden=72)
    assert_parity(run_gpu(wl, low="bf16"), run_oracle(wl, low="bf16"), TOL["bf16"])


def _network(batch, widths, n_steps, solver="rk4"):
    wl = inputs.mlp_block(batch=batch, n_steps=n_steps, d=widths[0], hidden=widths[1])
    wl.vel["n_layers"], wl.vel["widths"], wl.theta = len(widths) - 1, widths, inputs.mlp_theta(3, widths, True)
    wl.solver = solver
    return wl


# row-local kernels whose weights stay on the SM: one row, a block's 8 rows less and plus one, two and four row tiles a block; one layer (weights
# in registers: 2, 4, 6 and 8 reduction steps, parameter gradients in registers up to 64 pieces and in slabs above); widths of one and
# several tiles a warp, an odd number of reduction steps, and more than 16 of them.  Unscaled-safe passes in bfloat16: unscaled float16
# cotangents of a mean over 2369 x 128 entries, 2 / 303232 = 6.6e-6, are 110 units of the smallest subnormal, so that a value that rounds to its
# neighbour is 0.9 % off and the format's 2e-3 says nothing.
@pytest.mark.parametrize("batch,widths,n_steps", [(1, [24, 24], 3), (7, [64, 64], 5), (9, [72, 72], 3), (1185, [100, 100], 2), (2369, [128, 128], 2), (9, [40, 136, 40], 2),
                                                  (1190, [24, 130, 24], 2), (20, [16, 272, 16], 2), (9, [240, 64, 240], 2), (17, [33, 40, 33], 3), (300, [12, 20, 28, 12], 3)])
def test_resident_networks_at_tile_edges(batch, widths, n_steps):
    wl = _network(batch, widths, n_steps)
    for low, scaling in (("bf16", "none"), ("f16", "dynamic"), ("bf16", "none_safe")):
        gpu, orc = run_gpu(wl, low, scaling), run_oracle(wl, low, scaling)
        assert_parity(gpu, orc, TOL[low])
        assert gpu["stats"]["fused_launches"] > 0 and gpu["stats"]["simt_contractions"] == 0
        if scaling == "dynamic":
            assert_same_log(gpu["log"], orc["log"])


# tableaux whose stages depend on the one before alone (what the epilogues carry in registers) and on several, the time terms beside them
@pytest.mark.parametrize("solver", ["euler", "heun", "kutta3", "rk38"])
@pytest.mark.parametrize("widths", [[64, 64], [40, 72, 40]])
def test_resident_networks_per_tableau(solver, widths):
    wl = _network(100, widths, 5, solver)
    for low, scaling in (("bf16", "none"), ("f16", "dynamic")):
        gpu, orc = run_gpu(wl, low, scaling, want_dt=True), run_oracle(wl, low, scaling, want_dt=True)
        assert_parity(gpu, orc, TOL[low])
        assert rel_l2(gpu["dL_dt"], orc["dL_dt"]) <= TOL[low]
        plain = run_gpu(wl, low, scaling)
        assert np.array_equal(plain["a0"], gpu["a0"]) and np.array_equal(plain["yT"], gpu["yT"])


# weight gradients by clusters: fewer rows than two stages of the ring, pieces of 64 that end inside a tile, float32 with steps that meet one by one
@pytest.mark.parametrize("low,batch,widths,n_steps", [("f32", 3, [16, 72, 16], 5), ("f32", 513, [64, 200, 64], 3), ("f16", 2300, [64, 136, 64], 2), ("bf16", 31, [128, 160, 128], 9)])
def test_weight_gradient_clusters(low, batch, widths, n_steps):
    wl = _network(batch, widths, n_steps)
    scaling = "none" if low != "f16" else "dynamic"
    gpu = run_gpu(wl, low, scaling)
    assert_parity(gpu, run_oracle(wl, exact=True) if low == "f32" else run_oracle(wl, low, scaling), TOL[low])
    # a running gradient is added to, not overwritten: twice the same pass into one array
    import torch
    from paper_2510_23498_b200 import binding
    if scaling == "none":
        ctx = binding.Context(wl.vel, wl.batch, wl.n_steps, low=low)
        ctx.forward(torch.from_numpy(np.ascontiguousarray(wl.theta, dtype=np.float32)).cuda(), torch.from_numpy(np.ascontiguousarray(wl.y0, dtype=np.float32)).cuda(), wl.tgrid, wl.solver)
        dl = torch.from_numpy(np.ascontiguousarray(gpu["dLdyT"], dtype=np.float32)).cuda()
        _, g, _, _ = ctx.backward(dl)
        ctx.backward(dl, accumulate_into=g)
        assert rel_l2(g.cpu().numpy(), 2.0 * gpu["g"]) <= 1e-6      # (one more float32 rounding per entry and chunk of steps)
        ctx.close()


# Rows of a block that lie behind the batch must not reach a result: a velocity that leaves float16 along the trajectory from y = 0, but not
# along the samples'.  Several layers: every fourth hidden unit is 60000 at y = 0 and off (-60000) at the samples' y = -16, its outgoing weights 4;
# the other units see y + 16.  One layer: f = 0 at y = -15000 +- 8k, f(0) = 60000, slope 4.
def _overflows_at_zero(batch, widths, n_steps=2):
    wl = _network(batch, widths, n_steps)
    d, h = widths[0], widths[1]
    if len(widths) == 2:
        wl.theta = np.concatenate([np.concatenate([np.full((d, d), 4.0 / d), np.zeros((d, 1))], axis=1).ravel(), np.full(d, 60000.0)]).astype(np.float32)
        k = 8.0 * (np.arange(batch)[:, None] % 5 + np.arange(d // 2)[None, :] % 3)
        wl.y0 = (-15000.0 + np.concatenate([k, -k], axis=1)).astype(np.float32)
        return wl
    wl.y0 = (-16.0 + 0.25 * wl.y0).astype(np.float32)
    n0 = h * (d + 1)
    W0, b0, W1 = wl.theta[:n0].reshape(h, d + 1), wl.theta[n0:n0 + h], wl.theta[n0 + h:n0 + h + widths[2] * h].reshape(widths[2], h)
    b0[:] = 16.0 * W0[:, :d].sum(axis=1)
    W0[::4, :d], W0[::4, d], b0[::4], W1[:, ::4] = 7500.0 / d, 0.0, 60000.0, 4.0
    return wl


def _check_rows_behind_the_batch(wl, scalings):
    for scaling in scalings:
        gpu, orc = run_gpu(wl, "f16", scaling, k_max=40), run_oracle(wl, "f16", scaling, k_max=40)
        assert gpu["status"] == 0 and gpu["stats"]["fused_launches"] > 0
        assert_parity(gpu, orc, TOL["f16"])
        if scaling == "dynamic":
            assert_same_log(gpu["log"], orc["log"])
    gpu, orc = run_gpu(wl, "f16", "none", want_dt=True), run_oracle(wl, "f16", "none", want_dt=True)
    assert_parity(gpu, orc, TOL["f16"])
    assert rel_l2(gpu["dL_dt"], orc["dL_dt"]) <= TOL["f16"]


# (one and two row tiles a block, parameter gradients in registers and in slabs; one layer: its unscaled gradients leave the format)
@pytest.mark.parametrize("batch,widths", [(9, [16, 16]), (1203, [16, 16]), (9, [16, 24, 16]), (1203, [16, 24, 16]), (9, [64, 128, 64]), (1203, [64, 128, 64]), (3, [16, 32, 48, 16])])
def test_resident_networks_leave_rows_behind_the_batch_out(batch, widths):
    _check_rows_behind_the_batch(_overflows_at_zero(batch, widths), ("none", "dynamic") if len(widths) == 2 else ("none", "none_safe", "dynamic"))


# (the streaming kernels, 128 K weights: the extra rows' stage derivatives meet zero adjoints in the time terms)
def test_streaming_networks_leave_rows_behind_the_batch_out():
    _check_rows_behind_the_batch(_overflows_at_zero(17, [128, 256, 256, 128]), ("none", "none_safe", "dynamic"))


# weight gradients of the flow on both sides of the line between tiles of 64 columns and wider ones cut into slices: 16 and 17 k-blocks, outputs
# 256 columns and more wide and between 128 and 255
@pytest.mark.parametrize("batch,hidden", [(512, 264), (544, 264), (512, 136), (544, 136), (1024, 264)])
def test_flow_weight_gradient_tile_widths(batch, hidden):
    wl = inputs.cnf_mlp(batch=batch, n_steps=1, d=16, hidden=hidden)
    assert_parity(run_gpu(wl, low="bf16"), run_oracle(wl, low="bf16"), TOL["bf16"])


# The resident backward kernel with two row tiles of 8 a block (1185 to 2368 rows on 148 SMs): parameter gradients in registers (one layer and
# two) and in slabs, with the time terms beside them
@pytest.mark.parametrize("widths", [[64, 64], [40, 72, 40], [64, 128, 64]])
@pytest.mark.parametrize("want_dt", [False, True])
def test_resident_networks_with_two_row_tiles(widths, want_dt):
    wl = _network(1503, widths, 3)
    for low, scaling in (("bf16", "none"), ("f16", "dynamic")):
        gpu, orc = run_gpu(wl, low, scaling, want_dt=want_dt), run_oracle(wl, low, scaling, want_dt=want_dt)
        assert_parity(gpu, orc, TOL[low])
        assert gpu["stats"]["fused_launches"] > 0 and gpu["stats"]["simt_contractions"] == 0
        if want_dt:
            assert rel_l2(gpu["dL_dt"], orc["dL_dt"]) <= TOL[low]


# 16-bit networks whose weights stream (more than fit an SM, up to 160 K): one row, a block's 16 rows less and plus one, several blocks, two row
# tiles a block (forward; the other path backward); and a network whose forward pass is resident and whose backward pass streams.  Unscaled passes
# in bfloat16: unscaled float16 cotangents of a mean over 2401 x 128 entries, 2 / 307328 = 6.5e-6, are 109 units of the smallest subnormal, so
# that their rounding alone, half a unit, is up to 0.5 % of them (measured 0.6 % in dL/dy0), above the format's 2e-3.
@pytest.mark.parametrize("batch,widths,n_steps", [(1, [128, 256, 256, 128], 2), (15, [128, 256, 256, 128], 2), (17, [128, 256, 256, 128], 2), (200, [128, 256, 256, 128], 3), (2401, [128, 256, 256, 128], 1),
                                                  (200, [64, 256, 256, 64], 3), (33, [129, 250, 260, 129], 2)])
def test_streaming_networks_at_tile_edges(batch, widths, n_steps):
    wl = _network(batch, widths, n_steps)
    for low, scaling, want_dt in (("bf16", "none", False), ("f16", "dynamic", False), ("bf16", "none_safe", False), ("bf16", "none", True)):
        gpu, orc = run_gpu(wl, low, scaling, want_dt=want_dt), run_oracle(wl, low, scaling, want_dt=want_dt)
        assert_parity(gpu, orc, TOL[low])
        assert gpu["stats"]["fused_launches"] > 0 and gpu["stats"]["simt_contractions"] == 0
        if scaling == "dynamic":
            assert_same_log(gpu["log"], orc["log"])
        if want_dt:
            assert rel_l2(gpu["dL_dt"], orc["dL_dt"]) <= TOL[low]


# instance normalisation by the pixels of a plane: 4 and 16 of them a thread (up to 256 and 1024), read again and again above
@pytest.mark.parametrize("H,W", [(16, 16), (17, 16), (32, 32), (33, 32)])
@pytest.mark.parametrize("low", ["bf16", "f16"])
def test_parabolic_planes_at_register_edges(H, W, low):
    wl = inputs.parabolic_block(batch=2, n_steps=1, H=H, W=W, C=64, n_intervals=1, low=low, solver="euler")
    scaling = "dynamic" if low == "f16" else "none"
    assert_parity(run_gpu(wl, low, scaling), run_oracle(wl, low, scaling), TOL[low])


# weight gradients of unscaled-safe launches of one step, whose check goes with the addition to the output: clusters of one block and of several, and
# a step's gradient that alone leaves the format (a constant cotangent, summed over the batch: 1000 rows of 100 or 5e36)
@pytest.mark.parametrize("low,batch,widths,size", [("bf16", 9, [24, 40, 24], 5e36), ("bf16", 1000, [64, 128, 64], 5e36), ("f16", 1000, [72, 200, 200, 72], 300.0), ("f32", 1000, [16, 72, 16], 5e36)])
def test_weight_gradients_of_one_checked_step(low, batch, widths, size):
    wl = _network(batch, widths, 1)
    gpu = run_gpu(wl, low, "none_safe")
    if low != "f16":        # (unscaled float16 cotangents of a mean over 1000 x 72 entries are 466 units of the smallest subnormal: rounded to 0.1 % each)
        assert_parity(gpu, run_oracle(wl, exact=True) if low == "f32" else run_oracle(wl, low, "none_safe"), TOL[low])
    assert gpu["status"] == 0
    if batch > 9:
        gpu = run_gpu(wl, low, "none_safe", dLdyT=np.full((batch, widths[0]), size))
        assert gpu["status"] == 8 and np.all(np.isposinf(gpu["g"])) and np.all(np.isposinf(gpu["a0"]))
