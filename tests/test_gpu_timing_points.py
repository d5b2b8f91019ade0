"""Kernel timing modes and launch count of the kernel sequence whose second filter writes the points: its
own steps, the row prefixes among them (the separate compaction's steps: test_gpu_timing.py)."""
import pytest

import scene

pytestmark = pytest.mark.gpu

STAGES = ((4, 5.0, 20.0), (2, 5.0, 20.0))
STEPS = {"prep_compose_clear", "project_zbuf", "pool3", "jbf_stage1", "bp_rows", "jbf_stage2"}


@pytest.mark.parametrize("timing,steps", [(0, set()), (1, STEPS), (2, {"jbf_stage2"})])
def test_steps_and_launches_of_a_1080p_frame(timing, steps):
    import torch
    from paper_2601_01210_gb300 import Densifier, build
    from paper_2601_01210_gb300.frames import FrameBuffers
    build.build()
    v = scene.make_view(21, res="1080p", scene_kind="room", n_scans=1, beams=64, az_steps=1024)
    with Densifier(dict(num_stages=2, stages=STAGES, launch_policy=1, timing=timing)) as d:
        b = FrameBuffers(v.camera, v.rgb, [(s.xyz, s.lidar_to_world) for s in v.scans])
        for _ in range(3):
            assert d.poll(d.submit(b.frame), -1) == 0
        torch.cuda.synchronize()
        times = d.kernel_times()
        assert d.kernel_launches() == 3 * len(STEPS)
        assert set(times) == steps and all(n == 3 and us > 0.0 for us, n in times.values())
