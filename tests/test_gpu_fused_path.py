"""GPU parity of the fused Runge-Kutta program (rk_fused.cu) and of the layer-by-layer path for dense velocities, at networks above
the 160 K weights up to which the 16-bit formats take the row-local kernels: what the tests at smaller widths checked on these
paths before those kernels took their sizes.

Tolerances are those of the formats (rounding-emulating oracle) and of float32 mode (exact fp64 solution); scale logs identical.
"""
import numpy as np
import pytest

from paper_2510_23498_b200 import inputs
from _harness import TOL, assert_parity, assert_same_log, rel_l2, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


def _wide(batch, d, hidden, n_steps=2):
    assert 2 * d * hidden + hidden * hidden > 160 * 1024
    return inputs.mlp_block(batch=batch, n_steps=n_steps, d=d, hidden=hidden)


def _check(wl, low, scaling, path, **kw):
    orc, gpu = run_oracle(wl, low, scaling, **kw), run_gpu(wl, low, scaling, **kw)
    assert_parity(gpu, orc, TOL[low])
    if scaling == "dynamic":
        assert orc["log"].margin > 1e-4
        assert_same_log(gpu["log"], orc["log"])
    st = gpu["stats"]
    assert st["simt_contractions"] == 0 and st["whole_solve_launches"] == 0
    assert (st["fused_launches"] > 0, st["tc_contractions"] > 0) == ((True, False) if path == "fused" else (False, True))
    return gpu, orc


def test_networks_of_this_width_are_not_row_local():
    # the row-local kernels run a pass without finiteness decisions in one forward launch and one backward launch per chunk of steps, the
    # fused program recomputes and differentiates every step in launches of its own
    import torch
    from paper_2510_23498_b200 import binding
    for hidden, row_local in ((160, True), (520, False)):
        wl = inputs.mlp_block(batch=130, n_steps=4, d=72, hidden=hidden)
        ctx = binding.Context(wl.vel, wl.batch, wl.n_steps, low="bf16")
        ctx.set_profiling(True)
        _, yT = ctx.forward(torch.from_numpy(wl.theta).cuda(), torch.from_numpy(wl.y0).cuda(), wl.tgrid, wl.solver)
        ctx.backward(torch.ones_like(yT))
        assert ctx.collect_profile()["forward"]["launches"] == (1 if row_local else 1 + wl.n_steps)
        ctx.close()


@pytest.mark.parametrize("batch", [1, 127, 129, 300])
def test_fused_program_on_ragged_row_blocks_and_columns(batch):
    _check(_wide(batch, 72, 520), "bf16", "none", "fused")


# hidden widths that are not multiples of 8 are padded: one past, one short of a multiple, and odd widths that end inside a tile
@pytest.mark.parametrize("batch,d,hidden,low,scaling", [(200, 64, 513, "bf16", "none"), (130, 72, 519, "f16", "dynamic"), (257, 40, 1021, "bf16", "none_safe")])
def test_fused_program_with_padded_hidden_widths(batch, d, hidden, low, scaling):
    _check(_wide(batch, d, hidden), low, scaling, "fused")


# state widths that are not multiples of 8: padded rows on the layer-by-layer path (weight gradients on the tensor cores from 128 rows on)
@pytest.mark.parametrize("batch,d,hidden,low,scaling", [(130, 33, 400, "bf16", "none"), (257, 71, 521, "f16", "dynamic"), (128, 9, 460, "bf16", "none_safe")])
def test_layer_path_with_padded_state_rows(batch, d, hidden, low, scaling):
    _check(_wide(batch, d, hidden), low, scaling, "layers")


@pytest.mark.parametrize("d,path", [(64, "fused"), (61, "layers")])
def test_forced_overflow_is_retried_until_the_attempt_is_finite(d, path):
    # the finiteness flags come from the tensor-core epilogues, and the retries launch the same programs again
    wl = _wide(136, d, 520, n_steps=3)
    gpu, orc = _check(wl, "f16", "dynamic", path, k_max=60, init_scale_exp_override=40)
    assert max(gpu["log"]["attempts"]) > 1 and gpu["stats"]["retries"] == sum(k - 1 for k in gpu["log"]["attempts"])
    gpu = run_gpu(wl, "f16", "none_safe", init_scale_exp_override=40)
    assert gpu["status"] == 8 and np.all(np.isinf(gpu["g"])) and np.all(np.isinf(gpu["a0"]))
    gpu = run_gpu(wl, "f16", "dynamic", k_max=3, init_scale_exp_override=40)
    assert gpu["status"] == 7 and gpu["log"]["first_failed_step"] == 2 and gpu["log"]["attempts"][-1] == 3 and gpu["log"]["exp_used"][-1] == 40 - 3


@pytest.mark.parametrize("d", [64, 61])
def test_a_parameter_gradient_alone_that_overflows_is_reported(d):
    wl = _wide(1000, d, 520, n_steps=1)
    gpu = run_gpu(wl, "f16", "none_safe", dLdyT=np.full((1000, d), 100.0))
    assert gpu["status"] == 8 and np.all(np.isposinf(gpu["g"]))
    one = _wide(1, d, 520, n_steps=1)
    assert run_gpu(one, "f16", "none_safe", dLdyT=np.full((1, d), 100.0))["status"] == 0


@pytest.mark.parametrize("d,path", [(72, "fused"), (71, "layers")])
def test_dynamic_scaling_drains_the_stream_once_and_once_per_overflow(d, path):
    wl = _wide(130, d, 520, n_steps=4)
    gpu, _ = _check(wl, "f16", "dynamic", path, init_scale_exp_override=0)
    assert gpu["log"]["attempts"] == [1] * 4 and gpu["stats"]["host_syncs"] == 1 and gpu["stats"]["step_waits"] == 3
    gpu, _ = _check(wl, "f16", "dynamic", path, k_max=40, init_scale_exp_override=24)
    r = gpu["stats"]["retries"]
    assert r == sum(k - 1 for k in gpu["log"]["attempts"]) and r > 0 and gpu["stats"]["host_syncs"] == 1 + r


@pytest.mark.parametrize("solver", ["heun", "kutta3", "rk38"])
def test_other_tableaux_on_a_nonuniform_grid(solver):
    wl = _wide(48, 64, 520, n_steps=3)
    wl.solver = solver
    wl.tgrid = np.array([0.0, 0.1, 0.45, 1.0], dtype=np.float32)
    _check(wl, "bf16", "none", "fused")


@pytest.mark.parametrize("d,low,scaling", [(64, "f16", "dynamic"), (64, "bf16", "none"), (61, "f16", "dynamic"), (61, "bf16", "none"), (61, "f32", "none")])
def test_time_gradient_and_running_cost(d, low, scaling):
    wl = _wide(130, d, 520, n_steps=3)
    rc = (1.0 / (wl.batch * d) * np.random.default_rng(3).standard_normal((wl.n_steps, wl.batch, d))).astype(np.float32)
    orc = run_oracle(wl, exact=True, want_dt=True, running_cot=rc) if low == "f32" else run_oracle(wl, low, scaling, want_dt=True, running_cot=rc)
    gpu = run_gpu(wl, low, scaling, want_dt=True, running_cot=rc)
    assert_parity(gpu, orc, TOL[low])
    assert rel_l2(gpu["dL_dt"], orc["dL_dt"]) <= TOL[low]
    if scaling == "dynamic":
        assert_same_log(gpu["log"], orc["log"])


@pytest.mark.parametrize("d", [64, 61])
def test_repeats_are_bit_identical_and_gradients_accumulate(d):
    import torch
    from paper_2510_23498_b200 import binding
    wl = _wide(130, d, 520)
    r1, r2 = run_gpu(wl), run_gpu(wl)
    assert all(np.array_equal(r1[k], r2[k]) for k in ("yT", "traj", "a0", "g"))
    ctx = binding.Context(wl.vel, wl.batch, wl.n_steps, low=wl.low)
    ctx.forward(torch.from_numpy(wl.theta).cuda(), torch.from_numpy(wl.y0).cuda(), wl.tgrid, wl.solver)
    g = torch.full((ctx.p,), 3.0, device="cuda")
    ctx.backward(torch.from_numpy(r1["dLdyT"].astype(np.float32)).cuda(), accumulate_into=g)
    assert np.allclose(g.cpu().numpy(), r1["g"] + 3.0, rtol=1e-6, atol=1e-6)
    ctx.close()


@pytest.mark.parametrize("d", [64, 61])
def test_static_workspace_gives_the_same(d):
    import torch
    from paper_2510_23498_b200 import binding
    wl = _wide(200, d, 520)
    ref = run_gpu(wl)
    ctx = binding.Context(wl.vel, wl.batch, wl.n_steps, low=wl.low)
    assert ctx.workspace_bytes <= binding.STATIC_WORKSPACE_BYTES
    ctx.forward(torch.from_numpy(wl.theta).cuda(), torch.from_numpy(wl.y0).cuda(), wl.tgrid, wl.solver)
    dl = torch.from_numpy(ref["dLdyT"].astype(np.float32)).cuda()
    for _ in range(2):
        a0, g, st = ctx.backward_static_workspace(dl)
        torch.cuda.synchronize()
        assert st == 0 and rel_l2(a0.cpu().numpy(), ref["a0"]) <= TOL[wl.low] and rel_l2(g.cpu().numpy(), ref["g"]) <= TOL[wl.low]
    ctx.close()


def test_trajectory_aligned_to_16_bytes_only_goes_layer_by_layer():
    import torch
    from paper_2510_23498_b200 import binding
    wl = _wide(200, 64, 520)
    orc = run_oracle(wl)
    ctx = binding.Context(wl.vel, wl.batch, wl.n_steps, low=wl.low)
    n = (wl.n_steps + 1) * wl.batch * 64
    traj = torch.empty(n + 64, dtype=torch.bfloat16, device="cuda")[8:8 + n].view(wl.n_steps + 1, wl.batch, 64)
    assert traj.data_ptr() % 32 == 16
    _, yT = ctx.forward(torch.from_numpy(wl.theta).cuda(), torch.from_numpy(wl.y0).cuda(), wl.tgrid, wl.solver, traj=traj)
    _, dl = wl.loss(yT.cpu().numpy().astype(np.float64))
    a0, g, _, st = ctx.backward(torch.from_numpy(dl.astype(np.float32)).cuda())
    assert st == 0 and ctx.stats()["fused_launches"] == 0 and ctx.stats()["tc_contractions"] > 0
    assert_parity(dict(yT=yT.cpu().numpy(), traj=traj.float().cpu().numpy(), a0=a0.cpu().numpy(), g=g.cpu().numpy()), orc, TOL[wl.low])
    ctx.close()
