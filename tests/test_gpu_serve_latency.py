"""The serving loop holds a small batch back for company only while others run: a client that waits for
each answer before it asks again, and requests that could not share a batch anyway, are launched as
soon as a stream is free."""
import time

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


def _request(ctx, seeds, caps, seed):
    rob = inputs.panda()
    rid = ctx.add_robot(rob)
    th = torch.as_tensor(inputs.joint_samples(np.random.default_rng(seed), rob, 1).T.copy(), dtype=torch.float32, device="cuda")
    return ctx.batch_item(rid, -1, ctx.fk(rid, th).cpu(), seeds, 1, seed, rob.n, device=torch.device("cpu"),
                          params=api.make_params(cd_max_iters=caps[0], lm_max_iters=caps[1]))


@pytest.mark.parametrize("inflight", [1, 3])
@pytest.mark.parametrize("caps", [(32, 20), (1, 1)])
def test_a_client_that_waits_for_each_answer_is_not_held_back(ctx, inflight, caps):
    it, out = _request(ctx, 64, caps, 3)
    hjcd.hjcd_server_start(ctx.h, max_inflight=inflight)
    try:
        queued = []
        for _ in range(200):
            info = hjcd.hjcd_wait(ctx.h, hjcd.hjcd_submit(ctx.h, it), 60.0)
            assert info.status == 0 and info.batch_requests == 1
            queued.append(info.queued_ms)
    finally:
        hjcd.hjcd_server_stop(ctx.h)
    # the scheduler's wake-up (about 10 us), not a share of the pace
    assert np.median(queued[20:]) < 0.05


def test_requests_that_cannot_share_a_batch_do_not_wait_for_one_another(ctx):
    items = [_request(ctx, 1000, (1, 1), 5 + k) for k in range(8)]
    alone = []
    for _ in range(30):
        t0 = time.perf_counter()
        ctx.solve_batch([items[0][0]])
        alone.append(time.perf_counter() - t0)
    hjcd.hjcd_server_start(ctx.h, max_inflight=3, max_batch_seeds=1000)
    try:
        spans = []
        for _ in range(30):
            t0 = time.perf_counter()
            ids = [hjcd.hjcd_submit(ctx.h, it) for it, _ in items]
            infos = [hjcd.hjcd_wait(ctx.h, i, 60.0) for i in ids]
            spans.append(time.perf_counter() - t0)
            assert all(inf.status == 0 and inf.batch_requests == 1 for inf in infos)
    finally:
        hjcd.hjcd_server_stop(ctx.h)
    # no longer than the requests one after another, with the serving loop's share of each
    assert np.median(spans[3:]) < len(items) * (np.median(alone[3:]) + 60e-6)
