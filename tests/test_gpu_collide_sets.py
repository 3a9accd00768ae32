"""Large candidate sets of the collision filter (a candidate per lane) against small ones (a warp
per candidate, themselves checked against the oracle): the same verdict for every candidate, for
scenes at the edges of the lane kernel's cells and words."""
import numpy as np
import pytest
import torch

from paper_2510_07514_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu

BIG = 33000  # more than the first size of the lane kernel


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    c = api.Context(0)
    yield c
    c.close()


def _scene(kind):
    rng = np.random.default_rng(7)
    s = inputs.random_scene(rng, 0, 0)
    if kind == "mixed":
        return inputs.random_scene(rng, 200, 20)
    if kind == "spheres":  # the last word of a mask full, and one more obstacle
        return inputs.random_scene(rng, 33, 0)
    if kind == "boxes":
        return inputs.random_scene(rng, 0, 33)
    if kind == "most":  # as many as the lane kernel takes
        return inputs.random_scene(rng, 448, 64, r_range=(0.01, 0.03))
    if kind == "one":
        s.sph_xyzr = np.array([[0.4, 0.1, 0.5, 0.05]])
    if kind == "flat":  # a point-like and a plane-like obstacle
        s.sph_xyzr = np.array([[0.5, 0.0, 0.4, 1e-6]])
        s.box_lohi = np.array([[-50.0, -50.0, 0.05, 50.0, 50.0, 0.05]])
    if kind == "far":
        s.sph_xyzr = np.array([[1e4, 1e4, 1e4, 0.5], [0.5, 0.2, 0.5, 0.1]])
    if kind == "unbounded":
        s.box_lohi = np.array([[-np.inf, -np.inf, -np.inf, np.inf, np.inf, 0.1], [0.3, 0.3, 0.3, 0.4, 0.4, 0.4]])
        s.sph_xyzr = np.array([[0.5, 0.2, 0.5, 0.1]])
    return s


def _robot(which):
    if which == "panda60":
        return inputs.panda_with_spheres(np.random.default_rng(5))
    if which == "base":  # spheres on the base, none on some bodies, few in all
        r = inputs.panda_with_spheres(np.random.default_rng(6))
        keep = (r.sph_body % 2 == 0)
        r.sph_body = np.concatenate([[0, 0], r.sph_body[keep]]).astype(np.int32)
        r.sph_xyzr = np.concatenate([[[0, 0, 0.05, 0.1], [0.4, 0, 0.4, 0.1]], r.sph_xyzr[keep]])
        r.ignore = (np.abs(np.subtract.outer(np.arange(9), np.arange(9))) <= 1).astype(np.uint8)
        return r
    return inputs.cfg3_chains()[int(which)]


@pytest.mark.parametrize("which", ["panda60", "base", "0", "5"])
@pytest.mark.parametrize("kind", ["none", "mixed", "spheres", "boxes", "most", "one", "flat", "far", "unbounded"])
def test_large_sets_give_the_verdicts_of_small_ones(ctx, which, kind):
    rob = _robot(which)
    rid = ctx.add_robot(rob)
    sid = -1 if kind == "none" else ctx.set_scene(_scene(kind))
    th = torch.as_tensor(inputs.joint_samples(np.random.default_rng(9), rob, BIG).T.copy(), dtype=torch.float32, device="cuda")
    th[1, 77] = float("nan")
    big = ctx.collide(rid, sid, th)
    for a, b in ((0, 11000), (11000, 22000), (22000, BIG)):
        assert torch.equal(ctx.collide(rid, sid, th[:, a:b].contiguous()), big[a:b])
    assert set(big.unique().tolist()) <= {0, 1}


@pytest.mark.parametrize("top_k,boxes", [(1, 20), (3, 0), (16, 20)])
def test_ranking_of_few_targets_equals_that_of_many(ctx, top_k, boxes):
    """The collision-aware ranking takes CTAs of twice the warps for few targets; a target's index
    keys its random streams, so the first ones of a long list are the same solves."""
    rng = np.random.default_rng(40 + top_k)
    rob = inputs.panda()
    scene = inputs.random_scene(rng, 200, boxes)
    rid, sid = ctx.add_robot(rob), ctx.set_scene(scene)
    tg = ctx.fk(rid, torch.as_tensor(inputs.joint_samples(rng, rob, 400).T.copy(), dtype=torch.float32, device="cuda"))
    many = ctx.solve(rid, sid, tg, 128, top_k, 3, rob.n)
    for T in (1, 2, 97):
        few = ctx.solve(rid, sid, tg[:T].contiguous(), 128, top_k, 3, rob.n)
        for x, y in zip(few, many):
            assert torch.equal(x.view(torch.int32), y[:T].view(torch.int32))
