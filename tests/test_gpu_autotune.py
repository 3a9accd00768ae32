"""The autotuner leaves alone the launch settings that its calibration batch does not use: small batches
run kernels of a fixed configuration, and long chains take fewer warps per CTA than asked for, so the
settings' times differ by noise only."""
import numpy as np
import pytest
import torch

from paper_2510_07514_gb300 import api, build, hjcd, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    c = api.Context(0)
    yield c
    c.close()


def _item(ctx, rob, T, seeds):
    rid = ctx.add_robot(rob)
    th = torch.as_tensor(inputs.joint_samples(np.random.default_rng(2), rob, T).T.copy(), dtype=torch.float32, device="cuda")
    return ctx.batch_item(rid, -1, ctx.fk(rid, th), seeds, 1, 3, rob.n)[0]


@pytest.mark.parametrize("T,seeds", [(1, 64), (4, 1000)])
def test_a_small_batch_leaves_the_launch_configuration(ctx, T, seeds):
    it = _item(ctx, inputs.panda(), T, seeds)
    try:
        for blk, wp in ((128, 4), (256, 2), (64, 8)):
            hjcd.hjcd_set_launch_config(ctx.h, blk, wp)
            _, rep = hjcd.hjcd_autotune(ctx.h, [it], None, 0.02, 1)
            assert (rep.ccd_block, rep.lm_warps) == (blk, wp)
    finally:
        hjcd.hjcd_set_launch_config(ctx.h, 64, 8)  # the defaults


def test_warps_that_come_to_the_same_launch_are_left(ctx):
    it = _item(ctx, inputs.dof_scaling_robot(24), 16, 1000)
    try:
        for wp in (8, 4, 2):
            hjcd.hjcd_set_launch_config(ctx.h, 64, wp)
            _, rep = hjcd.hjcd_autotune(ctx.h, [it], None, 0.02, 1)
            assert rep.lm_warps == wp and rep.ccd_block in (64, 128, 256)
    finally:
        hjcd.hjcd_set_launch_config(ctx.h, 64, 8)
