"""The selection's time does not hang on the scores: keys that are all equal (the seeds of an invalid
target all score infinity), a few distinct ones, or squeezed together by others far away take about
as long as spread ones, in the top-K, the ranking and the collision-aware ranking."""
import numpy as np
import pytest
import torch

from paper_2510_07514_gb300 import api, build, hjcd, inputs

pytestmark = pytest.mark.gpu

T, M = 600, 8192  # enough targets for the device's time to show behind the calls' own
KINDS = ["equal", "inf", "few", "ulps", "two", "nan"]


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    c = api.Context(0)
    yield c
    c.close()


def _scores(kind, rng, inf=True):
    if kind == "equal":
        return np.full(M, 0.25, np.float32)
    if kind == "inf":
        return np.full(M, np.inf if inf else 3e38, np.float32)
    if kind == "few":
        return rng.choice(np.array([0.0, 1e-30, 0.5, 1.0, 3e38], np.float32), M)
    if kind == "ulps":
        return (np.float32(3.0).view(np.uint32) + rng.integers(0, 5, M).astype(np.uint32)).view(np.float32)
    if kind == "two":
        return rng.choice(np.array([0.1, 1e9], np.float32), M)
    s = (rng.chisquare(2, M) * 5).astype(np.float32)
    if kind == "nan":
        s[rng.random(M) < 0.2] = np.nan
    return s


def _dev(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _time(f):
    """Median time (us) of a call, from the events around it."""
    for _ in range(2):
        f()
    ms = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        ms.append(a.elapsed_time(b))
    return float(np.median(ms)) * 1e3


def test_topk_time_does_not_hang_on_the_scores(ctx):
    rob = inputs.panda()
    rid = ctx.add_robot(rob)
    th = torch.rand(7, T * M, device="cuda")
    off = _dev(np.arange(T + 1) * M, torch.int64)
    for ratio in (1, 4):
        K = max(1, M // ratio)
        B = K * (M // K)
        b_off, tb = _dev(np.arange(T + 1) * B, torch.int64), torch.empty(7, T * B, device="cuda")
        params = api.make_params(dup_ratio=ratio)

        def run(kind):
            score = _dev(np.tile(_scores(kind, np.random.default_rng(2)), T))
            return _time(lambda: hjcd.hjcd_topk_dup(ctx.h, rid, T, off, score, th, T * M, b_off, tb, T * B, None, 5, params))

        spread = run("spread")
        for kind in KINDS:
            assert run(kind) <= 2 * spread, (ratio, kind)


@pytest.mark.parametrize("top_k", [1, 64])
def test_rank_time_does_not_hang_on_the_scores(ctx, top_k):
    rob = inputs.panda()
    rid = ctx.add_robot(rob)
    th = torch.rand(7, T * M, device="cuda")
    off = _dev(np.arange(T + 1) * M, torch.int64)
    oe = torch.full((T * M,), 1e-3, device="cuda")
    q, e = torch.empty(T, top_k, 7, device="cuda"), torch.empty(T, top_k, 2, device="cuda")
    cnt = torch.empty(T, dtype=torch.int32, device="cuda")

    def run(kind, conv=1.0):
        rng = np.random.default_rng(2)
        score = _dev(np.tile(_scores(kind, rng, inf=False), T))
        pe = _dev(np.tile(np.where(rng.random(M) < conv, 5e-4, 2e-3), T))
        return _time(lambda: hjcd.hjcd_rank(ctx.h, rid, T, off, th, T * M, score, pe, oe, None, 1e-3, 1e-2, None, top_k, q, e, cnt))

    spread = run("spread")
    assert run("spread", 0.5) <= 2 * spread  # both classes
    for kind in KINDS:
        assert run(kind) <= 2 * spread, kind


def test_padding_rows_cost_no_more_than_poses(ctx):
    """A batch of a fixed size whose last rows are zero quaternions: invalid targets, no iterations."""
    rob = inputs.panda()
    rid = ctx.add_robot(rob)
    tg = ctx.fk(rid, _dev(inputs.joint_samples(np.random.default_rng(3), rob, 16).T.copy()))
    pad = tg.clone()
    pad[8:] = 0
    whole = _time(lambda: ctx.solve(rid, -1, tg, M, 1, 5, 7))
    assert _time(lambda: ctx.solve(rid, -1, pad, M, 1, 5, 7)) <= 1.1 * whole + 10
    q, e, c = ctx.solve(rid, -1, pad, M, 1, 5, 7)
    ref = ctx.solve(rid, -1, tg[:8].contiguous(), M, 1, 5, 7)
    torch.cuda.synchronize()
    assert int(c[8:].abs().sum()) == 0 and bool(q[8:].isnan().all()) and bool(e[8:].isnan().all())
    for x, y in zip((q, e, c), ref):
        assert torch.equal(x[:8].view(torch.int32), y.view(torch.int32))


@pytest.mark.parametrize("targets", [24, 500])
def test_collision_aware_ranking_of_equal_scores(ctx, targets):
    """Copies of one seed, unperturbed and unpolished, all score the same; the first ones by index are
    taken, as after the filter over all candidates."""
    rng = np.random.default_rng(8)
    rob = inputs.panda_with_spheres(np.random.default_rng(5))
    rid, sid = ctx.add_robot(rob), ctx.set_scene(inputs.random_scene(rng, 40, 4))
    tg = ctx.fk(rid, _dev(inputs.joint_samples(rng, rob, targets).T.copy()))
    params = api.make_params(dup_ratio=100000, dup_sigma=0.0, lm_max_iters=0)
    other = api.make_params(dup_ratio=100000, dup_sigma=0.05, lm_max_iters=0)
    lazy = ctx.solve(rid, sid, tg, M, 16, 3, 7, params=params)
    hjcd.hjcd_set_profiling(ctx.h, 1)
    try:
        def rank_ms(p):
            ms = []
            for _ in range(7):
                ctx.solve(rid, sid, tg, M, 16, 3, 7, params=p)
                ms.append(hjcd.hjcd_phase_times(ctx.h)[4])
            return float(np.median(ms))

        assert rank_ms(params) <= 2 * rank_ms(other)
    finally:
        hjcd.hjcd_set_profiling(ctx.h, 0)
    hjcd.hjcd_set_collision_mode(ctx.h, 0)
    try:
        whole = ctx.solve(rid, sid, tg, M, 16, 3, 7, params=params)
    finally:
        hjcd.hjcd_set_collision_mode(ctx.h, 1)
    torch.cuda.synchronize()
    assert int(lazy[2].max()) == 16  # (a colliding seed's copies all collide)
    for x, y in zip(lazy, whole):
        assert torch.equal(x.view(torch.int32), y.view(torch.int32))
