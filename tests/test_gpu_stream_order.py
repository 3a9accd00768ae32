"""A solve's launches in the order of its stream.

The kernels of small batches are set up while the one before still runs; none may touch memory
before it is complete.  Targets written by slow work queued just before a solve, and overwritten
by work queued just after it, must give the results of the solve alone, bit for bit, as must
solves queued back to back that share one workspace.
"""
import numpy as np
import pytest
import torch

from paper_2510_07514_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    c = api.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("T,seeds,scene", [(1, 16, False), (1, 1000, True), (16, 64, True), (8, 1000, False)])
def test_queued_writes_before_and_after_a_solve(ctx, T, seeds, scene):
    wl = inputs.cfg2(16, 64)
    n = wl.robot.n
    rid, sid = ctx.add_robot(wl.robot), ctx.set_scene(wl.scene) if scene else -1
    th = torch.as_tensor(inputs.joint_samples(np.random.default_rng(5), wl.robot, 4 * T), dtype=torch.float32)
    tg = ctx.fk(rid, th.t().contiguous().cuda()).view(4, T, 7)
    alone = [[x.clone() for x in ctx.solve(rid, sid, tg[k].contiguous(), seeds, 2, 11 + k, n)] for k in range(4)]
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        a = torch.randn(4096, 4096, device="cuda")
        buf, outs = torch.zeros(T, 7, device="cuda"), []
        for k in range(4):
            b = a @ a  # keeps the stream busy while the solve's launches are queued
            buf.copy_(tg[k] + 0.0 * b[0, 0].clamp(-1, 1).nan_to_num())
            outs.append(ctx.solve(rid, sid, buf, seeds, 2, 11 + k, n, stream=st))
            buf.zero_()
            outs[-1] = [x.clone() for x in outs[-1]]
    st.synchronize()
    for x, y in zip(alone, outs):
        for p, q in zip(x, y):
            assert torch.equal(p.view(torch.int32), q.view(torch.int32))
