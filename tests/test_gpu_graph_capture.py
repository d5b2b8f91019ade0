"""Every graph of a context is captured by its first batch: no later batch pays for one, whichever kernel
sequence its size takes (points by the separate compaction or by the second filter)."""
import pytest

import scene

pytestmark = pytest.mark.gpu

STAGES = ((4, 5.0, 20.0), (2, 5.0, 20.0))


@pytest.mark.parametrize("sizes", [(1, 2), (2, 1)])   # frames of 960 x 540 in the batches: below and above 2^19 pixels
@pytest.mark.parametrize("slots", [1, 3])
@pytest.mark.parametrize("autotune", [0, 1])
def test_first_batch_captures_every_graph(sizes, slots, autotune):
    import torch
    from paper_2601_01210_gb300 import Densifier, build
    from paper_2601_01210_gb300.frames import FrameBuffers
    build.build()
    v = scene.make_view(21, res="540p", scene_kind="room", n_scans=1, beams=64, az_steps=512)
    bufs = [FrameBuffers(v.camera, v.rgb, [(s.xyz, s.lidar_to_world) for s in v.scans]) for _ in range(2)]
    with Densifier(dict(num_stages=2, stages=STAGES, launch_policy=1, batches_in_flight=slots, autotune=autotune)) as d:
        assert d.describe()["graphs"] == 0
        graphs, kernels = [], []
        for n in sizes:
            for t in [d.submit(b.frame) for b in bufs[:n]]:
                assert d.poll(t, -1) == 0
            torch.cuda.synchronize()
            graphs.append(d.describe()["graphs"])
            kernels.append(d.kernel_launches())
            d.reset_kernel_times()
        if d.describe()["stages"][1]["chosen"]["loop"] == "block":
            assert kernels[0] != kernels[1]   # the two sequences
        assert graphs[0] == graphs[1] > 0
