"""The C-ABI shared library builds without a GPU, loads, and exports every symbol include/mpode.h declares."""
import ctypes
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "mpode.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(mpode_[a-z0-9_]+)\s*\(", text)))


def test_library_builds_loads_and_exports_header_symbols():
    from paper_2510_23498_b200 import binding, build
    path = build.build()
    assert os.path.exists(path)
    lib = ctypes.CDLL(path)
    names = _declared_symbols()
    assert len(names) >= 15
    for n in names:
        assert hasattr(lib, n), "missing export %s" % n
    assert sorted(binding.EXPORTS) == names


def test_host_only_calls_work_without_a_device():
    from paper_2510_23498_b200 import binding
    lib = binding.load_library()
    assert lib.mpode_status_string(7).decode() == "dynamic adjoint scaling failed"
    rk4 = lib.mpode_tableau_rk4().contents
    assert rk4.stages == 4 and abs(sum(rk4.b[j] for j in range(4)) - 1.0) < 1e-15
    assert [rk4.c[j] for j in range(4)] == [0.0, 0.5, 0.5, 1.0]
    assert lib.mpode_tableau_euler().contents.stages == 1
    # context creation is host-side bookkeeping: sizes can be queried without a GPU
    import ctypes as C
    widths = (C.c_int * 4)(256, 1024, 1024, 256)
    desc = binding.VelocityDesc(0, 256, 3, C.cast(widths, C.POINTER(C.c_int)), 2, 1, 1, 0, 0, 0)
    pol = binding.Policy(1, 0, 0, 0, 0, binding.NO_OVERRIDE)
    h = C.c_void_p()
    assert lib.mpode_create(C.byref(h), C.byref(desc), 8192, 64, C.byref(pol)) == 0
    assert lib.mpode_param_count(h) == 1576192                       # 257*1024+1024 + 1024*1024+1024 + 1024*256+256
    assert lib.mpode_trajectory_bytes(h, 64) == 65 * 8192 * 256 * 2
    mixed = lib.mpode_workspace_bytes(h)
    lib.mpode_destroy(h)
    pol32 = binding.Policy(0, 0, 0, 0, 0, binding.NO_OVERRIDE)
    assert lib.mpode_create(C.byref(h), C.byref(desc), 8192, 64, C.byref(pol32)) == 0
    full = lib.mpode_workspace_bytes(h) + lib.mpode_trajectory_bytes(h, 64)
    lib.mpode_destroy(h)
    # every large buffer is in the low format: mixed mode needs about half of float32 mode
    assert (mixed + 65 * 8192 * 256 * 2) / full <= 0.55
    # The whole solve also holds the caller's float32 state, adjoint, terminal cotangent, parameters and gradient, the same in
    # both modes.  With them the ratio is 0.565: a KNOWN SHORTFALL against the 0.55 target (the fused backward's second cotangent
    # slots, two extra kappa slots and the slice partial sums of the weight gradient are what exceeds one half).  Asserted so that
    # it cannot grow unnoticed; the benchmark line reports the same figure as memory.ratio with memory.target.
    caller = 3 * 8192 * 256 * 4 + 2 * 1576192 * 4
    whole = (mixed + 65 * 8192 * 256 * 2 + caller) / (full + caller)
    assert 0.55 < whole <= 0.566, whole
    bad = binding.VelocityDesc(0, 256, 3, C.cast(widths, C.POINTER(C.c_int)), 2, 1, 1, 0, 0, 0)
    bad.d = 128
    assert lib.mpode_create(C.byref(h), C.byref(bad), 8, 4, C.byref(pol)) == 1


def test_convolutions_of_few_pixels_can_be_created():
    # fewer than 64 pixels in all, channels that the tensor-core weight gradient would take: its slice plan must not divide by zero
    import ctypes as C
    from paper_2510_23498_b200 import binding
    lib = binding.load_library()
    for kind, side, channels in (("conv", 7, 64), ("conv", 1, 64), ("parabolic", 3, 128)):
        desc = binding.VelocityDesc(binding.KINDS[kind], side * side * channels, 0, None, binding.ACTS["relu"], 1, 1, side, side, channels, 1, 1)
        pol = binding.Policy(binding.DTYPES["f16"], 0, 0, 0, 0, binding.NO_OVERRIDE)
        h = C.c_void_p()
        assert lib.mpode_create(C.byref(h), C.byref(desc), 1, 2, C.byref(pol)) == 0
        assert lib.mpode_workspace_bytes(h) > 0
        lib.mpode_destroy(h)


def test_policies_that_look_at_every_step_plan_no_gradients_of_blocks():
    # Small dense networks, MB: the buffers of a pass whose weight gradients come from slabs.  The parameter gradients of all blocks, which unscaled
    # passes add up instead, are up to 0.9 MB more.
    import ctypes as C
    from paper_2510_23498_b200 import binding
    lib = binding.load_library()
    for scaling, low, batch, ws, steps, mb in (("dynamic", "bf16", 836, [80, 80], 5, 2.49), ("none_safe", "bf16", 602, [23, 88, 23], 30, 1.12), ("dynamic", "f16", 350, [80, 80], 5, 1.11)):
        widths = (C.c_int * len(ws))(*ws)
        desc = binding.VelocityDesc(binding.KINDS["mlp"], ws[0], len(ws) - 1, C.cast(widths, C.POINTER(C.c_int)), binding.ACTS["tanh"], 1, 1, 0, 0, 0, 0, 1)
        h = C.c_void_p()
        assert lib.mpode_create(C.byref(h), C.byref(desc), batch, steps, C.byref(binding.Policy(binding.DTYPES[low], binding.SCALINGS[scaling], 10, 0, 0, binding.NO_OVERRIDE, 0))) == 0
        assert lib.mpode_workspace_bytes(h) <= mb * 1e6
        lib.mpode_destroy(h)


def test_a_refused_whole_solve_launch_fails_the_call_and_nothing_else_runs():
    # The hypernetwork flow plans its workspace for the whole-solve kernels alone: where the runtime refuses their launch (here every
    # launch, there is no device) the call fails with a status, and no kernel of another path is queued, for which no buffers exist.
    # Without a device no address is followed, so made-up ones do.
    import ctypes as C
    import pytest
    import torch
    from paper_2510_23498_b200 import binding
    if torch.cuda.is_available():
        pytest.skip("needs a machine whose launches are refused")
    lib = binding.load_library()
    widths = (C.c_int * 2)(16, 32)
    desc = binding.VelocityDesc(binding.KINDS["cnf_hyper"], 2, 1, C.cast(widths, C.POINTER(C.c_int)), 0, 0, 0, 0, 0, 0, 0, 0)
    pol = binding.Policy(1, 0, 0, 0, 0, binding.NO_OVERRIDE)
    h = C.c_void_p()
    assert lib.mpode_create(C.byref(h), C.byref(desc), 100, 2, C.byref(pol)) == 0
    t = (C.c_float * 3)(0.0, 0.5, 1.0)
    at = [(1 << 40) + (i << 30) for i in range(5)]
    assert lib.mpode_forward(h, None, at[0], at[1], t, 2, lib.mpode_tableau_rk4(), None, at[2], at[3], at[4], lib.mpode_workspace_bytes(h)) == binding.ERR_CUDA
    stats = binding.Stats()
    lib.mpode_get_stats(h, C.byref(stats))
    assert stats.kernel_launches <= 1 and stats.whole_solve_launches <= 1          # the table of weight sets at most
    lib.mpode_destroy(h)


def test_row_local_kernels_lie_over_the_buffers_of_the_other_path():
    # Small dense networks run row-local kernels in place of the fused or layer-by-layer path, never both in a call: their packed weights,
    # layer inputs and cotangents take no bytes of their own.  Bounds: what the other path alone needs (MB, rounded up), and for the
    # float32 network the layer inputs and cotangents of one RK4 step, 2 * 4 * 1024 * (64 + 256 + 256) * 4 = 18.9 MB, and its weights.
    import ctypes as C
    from paper_2510_23498_b200 import binding
    lib = binding.load_library()
    for widths, batch, steps, low, scaling, most in (([64, 64], 1024, 100, "bf16", "none", 2.5), ([24, 40, 24], 512, 64, "bf16", "none_safe", 0.8),
                                                     ([64, 128, 64], 1000, 64, "f16", "none", 4.1), ([72, 200, 200, 72], 1000, 16, "f16", "dynamic", 8.9),
                                                     ([64, 256, 256, 64], 2048, 64, "bf16", "none", 20.7), ([64, 256, 256, 64], 1024, 16, "f32", "none", 19.8)):
        arr = (C.c_int * len(widths))(*widths)
        linear = len(widths) == 2
        desc = binding.VelocityDesc(binding.KINDS["mlp"], widths[0], len(widths) - 1, C.cast(arr, C.POINTER(C.c_int)),
                                    binding.ACTS["none" if linear else "softplus"], 0 if linear else 1, 0 if linear else 1, 0, 0, 0, 0, 0)
        pol = binding.Policy(binding.DTYPES[low], binding.SCALINGS[scaling], 0, 0, 0, binding.NO_OVERRIDE)
        h = C.c_void_p()
        assert lib.mpode_create(C.byref(h), C.byref(desc), batch, steps, C.byref(pol)) == 0
        assert lib.mpode_workspace_bytes(h) <= most * 1e6, (widths, batch, low, lib.mpode_workspace_bytes(h))
        lib.mpode_destroy(h)


def test_hypernetwork_flow_plans_partial_sums_for_the_blocks_that_hold_samples():
    # Five samples are one block: one row of the 287 weight sets' sums (18 floats for each of four stages, 83 KB) and not one for each of the
    # 148 SMs (12 MB); 100 000 samples use every SM
    import ctypes as C
    from paper_2510_23498_b200 import binding
    lib = binding.load_library()

    def size(batch):
        widths = (C.c_int * 2)(15, 287)
        desc = binding.VelocityDesc(binding.KINDS["cnf_hyper"], 8, 1, C.cast(widths, C.POINTER(C.c_int)), 0, 0, 0, 0, 0, 0, 0, 0)
        pol = binding.Policy(1, 0, 0, 0, 0, binding.NO_OVERRIDE)
        h = C.c_void_p()
        assert lib.mpode_create(C.byref(h), C.byref(desc), batch, 5, C.byref(pol)) == 0
        out = lib.mpode_workspace_bytes(h)
        lib.mpode_destroy(h)
        return out

    assert size(5) < 2.4e6 and size(100000) > 12e6


def test_cnf_workspace_has_no_float32_cotangent_scratch_where_the_epilogue_takes_the_activation_step():
    # c5 (2048 x 784, 785 -> 2048 -> 2048 -> 784): with a batch that is a multiple of 64 and widths of at least 64 the backward
    # step through an activation runs in the tensor-core epilogue, so mixed mode plans no [2 B, 2048] float32 buffer (33.5 MB);
    # a ragged batch keeps the two-kernel form and its buffer
    import ctypes as C
    from paper_2510_23498_b200 import binding
    lib = binding.load_library()
    widths = (C.c_int * 4)(784, 2048, 2048, 784)

    def sizes(batch, low):
        desc = binding.VelocityDesc(binding.KINDS["cnf"], 784, 3, C.cast(widths, C.POINTER(C.c_int)), binding.ACTS["softplus"], 1, 1,
                                    0, 0, 0, 0, 0)
        pol = binding.Policy(low, 0, 0, 0, 0, binding.NO_OVERRIDE)
        h = C.c_void_p()
        assert lib.mpode_create(C.byref(h), C.byref(desc), batch, 8, C.byref(pol)) == 0
        out = lib.mpode_workspace_bytes(h), lib.mpode_trajectory_bytes(h, 8)
        lib.mpode_destroy(h)
        return out

    ws16, traj16 = sizes(2048, 1)
    ws32, traj32 = sizes(2048, 0)
    assert traj16 * 2 == traj32 == 9 * 2048 * 784 * 4
    assert (ws16 + traj16) / (ws32 + traj32) <= 0.52
    ragged, _ = sizes(2047, 1)
    assert ragged > ws16 + 30e6 * 2047 / 2048

