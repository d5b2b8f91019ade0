"""A bounded wait that gives up inside densify_frame_noalloc reaches a caller that asks for the status
(the call itself has returned by then). Injected on the host; no wait on the GPU runs out."""
import pytest

import scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stages", [((4, 5.0, 20.0), (2, 5.0, 20.0)), ((4, 3.0, 20.0),)])
def test_wait_failure_is_reported_once(stages):
    import torch
    from paper_2601_01210_gb300 import build
    from paper_2601_01210_gb300 import densify as D
    from paper_2601_01210_gb300.frames import FrameBuffers
    build.build()
    v = scene.make_view(808, res="qvga", scene_kind="room", n_scans=2, beams=48, az_steps=512)
    b = FrameBuffers(v.camera, v.rgb, [(s.xyz, s.lidar_to_world) for s in v.scans], num_stages=len(stages))
    p = D.densify_default_params()
    p.num_stages = len(stages)
    for i, st in enumerate(stages):
        p.stage[i] = D.densify_stage(*st)
    stream = torch.cuda.Stream()

    def frame():
        assert D.densify_frame_noalloc(p, b.frame, stream.cuda_stream) == D.DENSIFY_OK

    def status():
        return D.densify_noalloc_status(stream.cuda_stream)
    frame()
    assert status() == D.DENSIFY_OK and b.n_points() > 0
    assert D.densify_inject_noalloc_wait_failure() == D.DENSIFY_OK
    frame()
    frame()   # a later frame does not hide the failure
    assert status() == D.DENSIFY_E_CUDA
    assert "bounded wait" in D.densify_last_error(None)
    assert status() == D.DENSIFY_OK   # reported once
    frame()
    assert status() == D.DENSIFY_OK
