"""A bounded wait that gives up while the sigma gradient runs (its pooling stages rows by bulk copies)
reaches the caller. The failure is injected on the host, into the status word whose address the
gradient's kernels get; no wait on the GPU runs out."""
import pytest

import scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stages", [((4, 5.0, 20.0), (2, 5.0, 20.0)), ((4, 3.0, 20.0),)])
def test_wait_failure_of_the_gradient_reaches_the_caller(stages):
    import torch
    from paper_2601_01210_gb300 import Densifier, build
    from paper_2601_01210_gb300 import densify as D
    from paper_2601_01210_gb300.frames import FrameBuffers
    build.build()
    v = scene.make_view(808, res="qvga", scene_kind="room", n_scans=2, beams=48, az_steps=512)
    gt = torch.full((240, 320), 3.0, device="cuda")
    with Densifier(dict(num_stages=len(stages), stages=stages)) as d:
        b = FrameBuffers(v.camera, v.rgb, [(s.xyz, s.lidar_to_world) for s in v.scans], num_stages=len(stages))
        first = d.sigma_grad(b.frame, gt)
        assert first[2] > 0 and d.sigma_grad(b.frame, gt) == first   # healthy, twice
        assert D.densify_inject_wait_failure(d.ctx) == D.DENSIFY_OK
        with pytest.raises(D.DensifyError) as e:
            d.sigma_grad(b.frame, gt)
        assert e.value.status == D.DENSIFY_E_CUDA and "bounded wait" in str(e.value)
        assert D.densify_submit(d.ctx, b.frame)[0] == D.DENSIFY_E_CUDA   # the context stays failed
        torch.cuda.synchronize()
        assert D.densify_destroy(d.ctx) == D.DENSIFY_OK
        d.ctx = None
