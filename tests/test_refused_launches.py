"""What the velocities do where the runtime refuses a launch.  Here it refuses every one (no device), so no address is followed and made-up
ones do; on a machine with a device these tests are skipped."""
import os
import subprocess

import pytest


def _run(tmp_path, body):
    """Compile `body` (the inside of main, with velocity.h) against the library and return what it prints."""
    import torch
    from paper_2510_23498_b200 import build
    if torch.cuda.is_available():
        pytest.skip("needs a machine whose launches are refused")
    lib = build.build()
    src = tmp_path / "t.cu"
    src.write_text('#include <stdio.h>\n#include "velocity.h"\nusing namespace mpode;\nint main() {\n%s\nreturn 0; }\n' % body)
    exe = str(tmp_path / "t")
    subprocess.run([build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", build.CSRC, str(src), lib,
                    "-Xlinker", "-rpath," + os.path.dirname(lib), "-o", exe], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout.split()


def test_the_row_local_backward_path_is_declined_before_its_first_step(tmp_path):
    # Whether the kernels can be launched is settled when the pass begins: later, chunks of steps would already have been committed
    out = _run(tmp_path, """
    int widths[4] = {64, 128, 128, 64};
    for (int low = 0; low < 3; ++low) {
        mpode_velocity_desc d{};
        d.kind = MPODE_VEL_MLP; d.d = 64; d.n_layers = 3; d.widths = widths; d.act = MPODE_ACT_TANH; d.append_time = d.has_bias = 1;
        Velocity* v = make_velocity(d, 100, (mpode_dtype)low, 4);
        Layout lay;
        v->plan(lay);
        FusedSolve fs;
        fs.n_steps = 4; fs.stages = 4; fs.traj = (void*)(1ull << 40); fs.scalars.resize(4);
        long long launches = 0;
        v->prepare(nullptr, (void*)(1ull << 41), (const float*)(1ull << 42), nullptr, &launches);
        printf("%d\\n", (int)v->fused_backward_begin(nullptr, (void*)(1ull << 41), fs, &launches));
    }""")
    assert out == ["0", "0", "0"]


def test_the_convolution_keeps_its_time_channel_where_the_64_channel_kernel_is_declined(tmp_path):
    # The 64-channel kernel adds tau times a slope to its bias table, which no other kernel reads.  Declined although the shape is its
    # own (16-pixel rows), the first convolution has to take the steps of a shape that is not (64-pixel rows): the table with the time
    # channel for the general tensor-core kernel, and where that is declined too the 65-channel form.
    out = _run(tmp_path, """
    for (int side : {16, 64}) {
        mpode_velocity_desc d{};
        d.kind = MPODE_VEL_CONV3X3_2; d.d = side * side * 64; d.H = d.W = side; d.C = 64; d.act = MPODE_ACT_RELU; d.append_time = 1;
        Velocity* v = make_velocity(d, 4, MPODE_BF16, 1);
        Layout lay;
        v->plan(lay);
        long long launches = 0;
        v->forward(nullptr, (void*)(1ull << 41), 0, (const void*)(1ull << 40), 0.5f, &launches);
        printf("%lld\\n", launches);
    }""")
    assert out == ["3", "3"]
