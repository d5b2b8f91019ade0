"""The no-allocation entry's single stage on either side of its rule between the list form and the plain
kernel (points per pixel; radius 2 by image size), against the context's list form: masks, z-buffer,
point count and colours exact, depth within 3e-5 (FP32 rounding)."""
import numpy as np
import pytest

from test_gpu_list_dense import _view

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [2, 4, 7])
@pytest.mark.parametrize("size,density,copies", [((320, 240), 0.05, 1), ((320, 240), 0.9, 1), ((320, 240), 0.9, 3),
                                                 ((1280, 820), 0.02, 1), ((1280, 820), 0.2, 1), ((1280, 820), 0.5, 3)])
def test_both_sides_of_the_rule_match_the_context(size, density, copies, radius):
    import torch
    from paper_2601_01210_gb300 import Densifier, build
    from paper_2601_01210_gb300 import densify as D
    from paper_2601_01210_gb300.frames import FrameBuffers
    build.build()
    v = _view(*size, density)

    def buffers():
        return FrameBuffers(v.camera, v.rgb, [(s.xyz, s.lidar_to_world) for s in v.scans] * copies, debug=True, num_stages=1)
    a, b = buffers(), buffers()
    stage = (radius, 4.0, 20.0)
    with Densifier(dict(num_stages=1, stages=(stage,), launch_policy=1)) as d:
        assert d.describe()["stages"][0]["chosen"]["loop"] == "list"
        assert d.poll(d.submit(a.frame), -1) == 0
    p = D.densify_default_params()
    p.num_stages, p.stage[0] = 1, D.densify_stage(*stage)
    assert D.densify_frame_noalloc(p, b.frame, None) == D.DENSIFY_OK, D.densify_last_error(None)
    torch.cuda.synchronize()
    x, y = a.results(), b.results()
    for k in ("zbuf", "valid", "rgba", "n"):
        assert np.array_equal(x[k], y[k]), k
    np.testing.assert_allclose(y["depth"], x["depth"], rtol=3e-5)
