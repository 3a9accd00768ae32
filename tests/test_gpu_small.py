"""Small batches: the PO-CCD and PJ-IK kernels that spread a candidate's work over a CTA.

They run the one-thread-per-candidate kernels' operations in the same order, so a candidate's
results must be the same bits whether its batch is small (spread kernels) or large.  Sizes: one
candidate, the edges of a CTA's 16, more CTAs than fit at once; chains of one joint up to the
longest, joint tables with and without offsets.
"""
import numpy as np
import pytest
import torch

from paper_2510_07514_gb300 import api, build, hjcd, inputs

pytestmark = pytest.mark.gpu

BIG = 24000  # candidates: more than the spread kernels take (64 per SM)


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    c = api.Context(0)
    yield c
    c.close()


def _robot(which):
    if which == "offsets":  # joint offsets, limits past pi, a rotated flange
        r = inputs.panda()
        r.theta_off = np.linspace(-0.7, 0.9, 7)
        r.lo, r.hi = r.lo - 1.0, r.hi + 1.5
        c, s = np.cos(0.4), np.sin(0.4)
        r.flange = r.flange @ np.array([[c, 0, s, 0], [0, 1, 0, 0], [-s, 0, c, 0], [0, 0, 0, 1.0]])
        return r
    if which.startswith("planar"):
        return inputs.planar([0.3] * int(which[6:]))
    if which.startswith("random"):
        return inputs.cfg3_chains()[int(which[6:])]
    return inputs.dof_scaling_robot(int(which[5:]))


def _case(ctx, which, seed):
    rob = _robot(which)
    rid = ctx.add_robot(rob)
    rng = np.random.default_rng(seed)
    T = 24
    tg = ctx.fk(rid, torch.as_tensor(inputs.joint_samples(rng, rob, T).T.copy(), dtype=torch.float32, device="cuda"))
    tgt = torch.as_tensor(np.arange(BIG) * T // BIG, dtype=torch.int32, device="cuda")
    cand = torch.as_tensor(np.arange(BIG) % 1000, dtype=torch.int32, device="cuda")
    th = torch.as_tensor(inputs.joint_samples(rng, rob, BIG).T.copy(), dtype=torch.float32, device="cuda")
    return rob, rid, tg, tgt, cand, th


def _run(ctx, stage, rob, rid, tg, tgt, cand, th, params, sl):
    """The stage on candidates sl: theta, score, errors, iterations (rows of the slice)."""
    tgt, cand, th = tgt[sl].contiguous(), cand[sl].contiguous(), th[:, sl].clone(memory_format=torch.contiguous_format)
    C = tgt.numel()
    sc, pe, oe = (torch.empty(C, device="cuda") for _ in range(3))
    it = torch.empty(C, dtype=torch.int32, device="cuda")
    if stage == "ccd":
        hjcd.hjcd_po_ccd(ctx.h, rid, tg.shape[0], tg, 1e-3, 1e-2, 77, params, C, tgt, cand, th, th, C, 0, params.cd_max_iters,
                         sc, pe, oe, it)
    else:
        hjcd.hjcd_pjik(ctx.h, rid, tg.shape[0], tg, 1e-3, 1e-2, 77, params, C, tgt, cand, th, C, 0, params.lm_max_iters, sc, pe,
                       oe, it)
    torch.cuda.synchronize()
    return [x.cpu().numpy() for x in (th, sc, pe, oe, it)]


@pytest.mark.parametrize("stage", ["ccd", "lm"])
@pytest.mark.parametrize("which", ["planar1", "planar2", "planar3", "random0", "chain7", "offsets", "random5", "chain24"])
def test_small_batches_give_the_bits_of_large_ones(ctx, stage, which):
    case = _case(ctx, which, 11)
    for over in ({}, dict(lm_A=0, cd_max_iters=1, lm_max_iters=1), dict(lm_A=6, lm_lambda=1e-6, lm_trust_R=2.0)):
        params = api.make_params(**over)
        big = _run(ctx, stage, *case, params, slice(0, BIG))
        for a, b in ((0, 1), (5, 20), (16, 32), (40, 57), (100, 101 + 2432), (0, 9728)):
            small = _run(ctx, stage, *case, params, slice(a, b))
            for x, y in zip(small, big):
                np.testing.assert_array_equal(x.view(np.uint32), np.ascontiguousarray(y[..., a:b]).view(np.uint32))


@pytest.mark.parametrize("which,seeds,cap", [("random0", 997, 20), ("chain7", 1000, 20), ("chain12", 333, 20), ("random5", 500, 20),
                                             ("chain7", 256, 0), ("chain7", 256, 4), ("chain7", 256, 6), ("random0", 256, 7)])
def test_small_solves_give_the_rows_of_large_ones(ctx, which, seeds, cap):
    """Every size class of the polish (spread; spread, then the rest packed afresh; one lane per
    candidate, then few or many left) against one launch of one lane per candidate, also with caps
    around the iterations after which the candidates are packed afresh."""
    rob = _robot(which)
    rid = ctx.add_robot(rob)
    T = 36000 // seeds + 1
    params = api.make_params(lm_max_iters=cap)
    th = torch.as_tensor(inputs.joint_samples(np.random.default_rng(3), rob, T).T.copy(), dtype=torch.float32, device="cuda")
    tg = ctx.fk(rid, th)
    big = ctx.solve(rid, -1, tg, seeds, 64, 5, rob.n, params=params)
    for t in (1, 3, 6000 // seeds, 11500 // seeds, 14000 // seeds, 30000 // seeds):
        small = ctx.solve(rid, -1, tg[:t].contiguous(), seeds, 64, 5, rob.n, params=params)
        for x, y in zip(small, big):
            assert torch.equal(x.view(torch.int32), y[:t].view(torch.int32))


def test_a_small_mixed_batch_gives_each_request_its_bits(ctx):
    """Robots of different joint counts in one small batch (CTAs that straddle requests) against
    each request in a batch of its own robot too large for the spread kernels."""
    rng = np.random.default_rng(8)
    items, big = [], []
    for which in ("random0", "chain24", "chain7", "planar2"):
        rob = _robot(which)
        rid = ctx.add_robot(rob)
        th = torch.as_tensor(inputs.joint_samples(rng, rob, 40).T.copy(), dtype=torch.float32, device="cuda")
        tg = ctx.fk(rid, th)
        items.append(ctx.batch_item(rid, -1, tg[:3].contiguous(), 301, 8, 21, rob.n))
        big.append(ctx.solve(rid, -1, tg, 301, 8, 21, rob.n))
    ctx.solve_batch([it for it, _ in items])
    torch.cuda.synchronize()
    for (_, got), ref in zip(items, big):
        for x, y in zip(got, ref):
            assert torch.equal(x.view(torch.int32), y[:3].view(torch.int32))


def test_a_large_mixed_batch_gives_each_request_its_bits(ctx):
    """Eight robots of 6 to 20 joints with uneven seed counts in one batch (the packed PO-CCD column,
    rows in descending chain length) against each request alone."""
    rng = np.random.default_rng(12)
    items, alone = [], []
    for k in range(8):
        rob = _robot("random%d" % k)
        rid = ctx.add_robot(rob)
        th = torch.as_tensor(inputs.joint_samples(rng, rob, 20).T.copy(), dtype=torch.float32, device="cuda")
        tg = ctx.fk(rid, th)
        spt = rng.integers(30, 700, 20).astype(np.int32)
        items.append(ctx.batch_item(rid, -1, tg, int(spt.max()), 8, 21 + k, rob.n, samples_per_target=spt))
        alone.append(ctx.solve(rid, -1, tg, int(spt.max()), 8, 21 + k, rob.n, samples_per_target=spt))
    ctx.solve_batch([it for it, _ in items])
    torch.cuda.synchronize()
    for (_, got), ref in zip(items, alone):
        for x, y in zip(got, ref):
            assert torch.equal(x.view(torch.int32), y.view(torch.int32))


@pytest.mark.parametrize("which", ["planar1", "chain7", "random2", "offsets", "chain24"])
def test_fk_does_not_depend_on_the_batch(ctx, which):
    """Two candidates share a thread and a warp's 64 poses one store: every remainder, and an output
    buffer that does not start on 16 bytes, gives each candidate the pose it has alone."""
    rob = _robot(which)
    rid = ctx.add_robot(rob)
    rng = np.random.default_rng(4)
    th = torch.as_tensor(inputs.joint_samples(rng, rob, 1000).T.copy(), dtype=torch.float32, device="cuda")
    alone = torch.cat([ctx.fk(rid, th[:, c:c + 1].contiguous()) for c in range(200)])
    for C in (1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 200):
        assert torch.equal(ctx.fk(rid, th[:, :C].contiguous()), alone[:C])
        buf = torch.full((7 * C + 9,), -7.0, device="cuda")
        hjcd.hjcd_fk(ctx.h, rid, C, th, th.stride(0), buf[1:], None)  # a stride past C, 4-byte alignment
        torch.cuda.synchronize()
        assert torch.equal(buf[1:1 + 7 * C].view(C, 7), alone[:C])
        assert buf[0] == -7.0 and bool((buf[1 + 7 * C:] == -7.0).all())


@pytest.mark.parametrize("T,top_k", [(1, 1), (7, 3), (2000, 64)])
def test_results_do_not_depend_on_where_the_buffers_live(ctx, T, top_k):
    """Poses, references and outputs in device or host memory in any mix: small host results come
    through the library's pinned buffer, larger ones (2000 x 64 rows) by copies."""
    rob = _robot("chain7")
    rid = ctx.add_robot(rob)
    rng = np.random.default_rng(6)
    th = torch.as_tensor(inputs.joint_samples(rng, rob, T).T.copy(), dtype=torch.float32, device="cuda")
    tg = ctx.fk(rid, th)
    qc = torch.as_tensor(inputs.joint_samples(rng, rob, T), dtype=torch.float32, device="cuda")
    tg_h, qc_h = tg.cpu(), qc.cpu()
    shapes = ((T, top_k, 7), (T, top_k, 2), (T,))
    ref = None
    for mask in (0, 7, 1, 2, 4, 5):
        out = [torch.full(sh, -1, dtype=torch.int32 if k == 2 else torch.float32, device="cpu" if mask >> k & 1 else "cuda")
               for k, sh in enumerate(shapes)]
        src, cur = (tg_h, qc) if mask & 1 else (tg, qc_h)
        ctx.solve(rid, -1, src, 40, top_k, 9, 7, out=out, q_current=cur)
        torch.cuda.synchronize()
        got = [o.cpu().numpy().view(np.uint32) for o in out]
        if ref is None:
            ref = got
            assert (out[2] == min(top_k, 40)).all()
            assert torch.isnan(out[0][:, 40:]).all() and torch.isnan(out[1][:, 40:]).all()
        for a, b in zip(got, ref):
            np.testing.assert_array_equal(a, b)
