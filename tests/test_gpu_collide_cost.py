"""The collision filter's time over its two kernels: a candidate has a lane in large sets (from 32768
candidates on) and a warp below.  The change must not make a set cost more than its size, whatever
the robot: chains whose bodies crowd one another leave many body pairs to the link spheres' tests."""
import numpy as np
import pytest
import torch

from paper_2510_07514_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu

EDGE = 32768


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    c = api.Context(0)
    yield c
    c.close()


def _time(f):
    """Median device time (us) of calls queued behind one another."""
    for _ in range(3):
        f()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(22)]
    for e in ev:
        f()
        e.record()
    torch.cuda.synchronize()
    return float(np.median([a.elapsed_time(b) for a, b in zip(ev, ev[1:])])) * 1e3


@pytest.mark.parametrize("obstacles", [0, 1, 20, 110])
@pytest.mark.parametrize("which", ["panda60", 0, 3, 5, 7])
def test_a_larger_set_costs_no_more_than_its_size(ctx, which, obstacles):
    rob = inputs.panda_with_spheres(np.random.default_rng(5)) if which == "panda60" else inputs.cfg3_chains()[which]
    rid = ctx.add_robot(rob)
    boxes = 10 if obstacles > 100 else 0
    sid = ctx.set_scene(inputs.random_scene(np.random.default_rng(3), obstacles - boxes, boxes)) if obstacles else -1
    th = torch.as_tensor(inputs.joint_samples(np.random.default_rng(4), rob, 4 * EDGE).T.copy(), dtype=torch.float32, device="cuda")

    def run(C):
        part = th[:, :C].contiguous()
        return _time(lambda: ctx.collide(rid, sid, part))

    # a warp per candidate takes a time linear in the candidates and a constant, so at most this; 15%
    # for the clock, and the 3 us of a launch
    warp = run(EDGE - 1)
    for C in (EDGE, 3 * EDGE // 2, 2 * EDGE, 4 * EDGE):
        assert run(C) <= 1.15 * warp * C / EDGE + 3, C
