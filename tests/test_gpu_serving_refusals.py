"""The device's own refusal (DENSIFY_E_AGAIN) in the serving loop, under a load that forces it whatever the
speed of the GPU: more frames due at once than the context admits, with buffers to spare."""
import numpy as np
import pytest

import scene

pytestmark = pytest.mark.gpu

STAGES = ((4, 5.0, 20.0), (2, 5.0, 20.0))


@pytest.mark.parametrize("batches_in_flight", [1, 2])
def test_a_burst_beyond_the_limit_is_refused_and_served(batches_in_flight):
    import torch
    from paper_2601_01210_gb300 import Densifier, build
    from paper_2601_01210_gb300.frames import FrameBuffers
    from paper_2601_01210_gb300.serve import ServeLoop
    build.build()
    v = scene.make_view(21, res="qvga", scene_kind="room", n_scans=1, beams=32, az_steps=256)
    ring = [[FrameBuffers(v.camera, v.rgb, [(s.xyz, s.lidar_to_world) for s in v.scans]) for _ in range(3)]
            for _ in range(4)]
    with Densifier(dict(num_stages=2, stages=STAGES, max_inflight=2, batches_in_flight=batches_in_flight,
                        launch_policy=0)) as d:
        # three frames of four viewpoints due at once, two admitted: the first turn's third submit is refused
        arr = sorted((0.0, k) for k in range(4) for _ in range(3))
        st = ServeLoop(d, [[b.frame for b in r] for r in ring]).run(arr, 0.0, drain_s=10.0)
    torch.cuda.synchronize()
    assert st.completed == 12
    assert st.e_again > 0 and st.buffer_waits == 0
    first = ring[0][0].results()
    for r in ring:
        for b in r:
            assert np.array_equal(b.results()["depth"], first["depth"])
