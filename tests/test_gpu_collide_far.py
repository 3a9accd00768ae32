"""Collision verdicts of a scene far from the base against the extent of its obstacles: the cells that
large sets sort the obstacles into (a candidate per lane) must allow for the rounding of coordinates
that are large against a cell.  Against small sets of the same candidates (a warp per candidate, no
cells): the same verdict for every one."""
import numpy as np
import pytest
import torch

from paper_2510_07514_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu

BIG = 49500


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    c = api.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("per_body", [1, 8])
@pytest.mark.parametrize("far", [0.0, 1e3, 3e4, 4e5])
@pytest.mark.parametrize("boxes", [0, 6])
def test_verdicts_far_from_the_base(ctx, far, per_body, boxes):
    rng = np.random.default_rng(17)
    rob = inputs.panda_with_spheres(np.random.default_rng(5))
    first = np.concatenate([np.flatnonzero(rob.sph_body == b)[:per_body] for b in range(1, 9)])
    rob.sph_body, rob.sph_xyzr = rob.sph_body[first], rob.sph_xyzr[first]
    rob.a = np.array(rob.a, dtype=np.float64)
    rob.a[0] += far  # the arm stands this far from the origin
    rid = ctx.add_robot(rob)
    for trial in range(6):  # each a few obstacles within a small box
        at = np.array([far, 0.0, 0.0]) + rng.uniform([-0.5, -0.5, 0.1], [0.5, 0.5, 0.9])
        scene = inputs.random_scene(rng, 0, 0)
        scene.sph_xyzr = np.concatenate([at + rng.uniform(-0.05, 0.05, (4, 3)), rng.uniform(0.01, 0.04, (4, 1))], 1)
        if boxes:
            lo = at + rng.uniform(-0.06, 0.04, (boxes, 3))
            scene.box_lohi = np.concatenate([lo, lo + rng.uniform(0.0, 0.03, (boxes, 3))], 1)
        sid = ctx.set_scene(scene)
        th = torch.as_tensor(inputs.joint_samples(rng, rob, BIG).T.copy(), dtype=torch.float32, device="cuda")
        big = ctx.collide(rid, sid, th)
        small = torch.cat([ctx.collide(rid, sid, th[:, k:k + 16500].contiguous()) for k in range(0, BIG, 16500)])
        assert 0 < int(small.sum()) < BIG
        assert torch.equal(big, small), int((big != small).sum())
