"""After its first call, densify_frame_noalloc leaves the device's free memory unchanged whatever the
later frames are: other alignments of the colour rows (other kernels), stages, radii, poolings and
colour widths. In a process of its own, where the first call is the first use of the library."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CALLS = r"""
import numpy as np, torch
from paper_2601_01210_gb300 import densify as D
W, H = 192, 96
xyz = torch.rand(2000, 3, device="cuda") * 2 + torch.tensor([-1.0, -1.0, 2.0], device="cuda")
out = dict(out_depth=torch.zeros(H, W, device="cuda"), out_valid=torch.zeros(H, W, dtype=torch.uint8, device="cuda"),
           out_points=torch.zeros(H * W, 4, device="cuda"), out_points_n=torch.zeros(1, dtype=torch.int64, device="cuda"))
rgb = torch.zeros(H * 3 * (W + 1), dtype=torch.uint8, device="cuda")
def call(pitch, ns, r1, r2, sc=20.0, pool=3, **kw):
    f = D.make_frame(W, H, 150.0, 150.0, W / 2, H / 2, np.eye(4), rgb, [(xyz, np.eye(4))], rgb_pitch=pitch, **out)
    p = D.densify_default_params()
    p.num_stages, p.pool = ns, pool
    p.stage[0], p.stage[1] = D.densify_stage(r1, 5.0, sc), D.densify_stage(r2, 5.0, sc)
    for k, v in kw.items():
        setattr(p, k, v)
    assert D.densify_frame_noalloc(p, f, None) == 0, D.densify_last_error(None)
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]
aligned, unaligned = 3 * W, 3 * W + 3
free = call(unaligned, 2, 4, 2)
for pitch in (aligned, unaligned):
    for r in range(1, 8):
        for sc in (20.0, 5.0):
            assert call(pitch, 1, r, 0, sc) == free, (pitch, 1, r, sc)
            for r2 in (1, 2, 3):
                assert call(pitch, 2, r, r2, sc) == free, (pitch, 2, r, r2, sc)
    for kw in (dict(pool=2), dict(stage2_input=1), dict(emit_points=0), dict(kernel_variant=1), dict(kernel_variant=2)):
        assert call(pitch, 2, 4, 2, **kw) == free, (pitch, kw)
"""


def test_free_memory_stays_after_the_first_call():
    from paper_2601_01210_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", CALLS], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
