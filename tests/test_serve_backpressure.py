"""What the serving loop counts when admission pushes back, against the simulated device: the device's
refusals apart from the frames held for their viewpoint's own output buffer, the latter a frame each,
however fast the loop turns."""
import pytest

from paper_2601_01210_gb300.serve import ServeLoop
from test_serve_host import FakeClock, FakeDevice


class Clock(FakeClock):
    def __init__(self, tick):
        super().__init__()
        self.tick = tick

    def __call__(self):
        self.t += self.tick
        return self.t


def _frames(views, ring):
    return [[("view", v, s) for s in range(ring)] for v in range(views)]


@pytest.mark.parametrize("tick", [1e-5, 1e-6])
def test_own_buffers_count_once_a_frame(tick):
    clock = Clock(tick)
    dev = FakeDevice(clock, max_inflight=64, per_batch_s=5e-3)
    arr = [(1e-4 * k, 0) for k in range(5)] + [(5e-5, 1)]   # view 0: five frames within one batch's time, one buffer
    st = ServeLoop(dev, _frames(2, 1), clock=clock).run(sorted(arr), 0.001, drain_s=2.0)
    assert st.completed == 6
    assert (st.e_again, st.buffer_waits, st.refused_again) == (0, 4, 4)
    assert st.summary()["e_again_retries"] == 0 and st.summary()["buffer_waits"] == 4


def test_device_refusals_are_counted_apart():
    clock = Clock(1e-5)
    dev = FakeDevice(clock, max_inflight=2, per_batch_s=1e-3)
    arr = sorted((0.0, v) for v in range(4) for _ in range(3))
    st = ServeLoop(dev, _frames(4, 3), clock=clock).run(arr, 0.0, drain_s=2.0)   # at most 2 in flight: never out of buffers
    assert st.completed == 12
    assert st.e_again > 0 and st.buffer_waits == 0
    assert st.refused_again == st.e_again == st.summary()["e_again_retries"]
