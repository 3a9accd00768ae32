"""Per-target selection (top-K and ranking) against a stable sort, for the score distributions and
sizes at the edges of its bucket pass: counts around the bin counts and the warp, ranges of a few
ulp and of the whole exponent, many equal scores, infinities and NaN."""
import numpy as np
import pytest
import torch

from paper_2510_07514_gb300 import api, build, hjcd, inputs

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 32, 33, 64, 127, 128, 129, 1000, 1024, 1025, 2048, 2049, 8191, 8192]


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    c = api.Context(0)
    yield c
    c.close()


def _scores(kind, M, rng):
    if kind == "wide":
        return np.exp(rng.uniform(-80, 80, M)).astype(np.float32)
    if kind == "ulps":
        return (np.float32(3.0).view(np.uint32) + rng.integers(0, 5, M).astype(np.uint32)).view(np.float32)
    if kind == "equal":
        return np.full(M, 0.25, np.float32)
    if kind == "few":
        return rng.choice(np.array([0.0, -0.0, 1e-30, 1.0, np.inf, 3e38], np.float32), M)
    s = (rng.chisquare(2, M) * 5).astype(np.float32)  # "nan": a usual spread with NaN and infinity in it
    s[rng.random(M) < 0.2] = np.nan
    s[rng.random(M) < 0.1] = np.inf
    return s


def _dev(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("kind", ["wide", "ulps", "equal", "few", "nan"])
@pytest.mark.parametrize("ratio", [1, 4, 3000])
def test_topk_order(ctx, kind, ratio):
    rng = np.random.default_rng(2)
    rob = inputs.panda()
    rid = ctx.add_robot(rob)
    for sizes in (SIZES, [1000]):  # several CTAs a target with one target alone
        m_off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        K = [max(1, m // ratio) for m in sizes]
        b_off = np.concatenate([[0], np.cumsum([k * (m // k) for k, m in zip(K, sizes)])]).astype(np.int64)
        score = np.concatenate([_scores(kind, m, rng) for m in sizes])
        th = inputs.joint_samples(rng, rob, len(score)).T.astype(np.float32)
        tb = torch.empty((7, int(b_off[-1])), device="cuda")
        src = torch.empty(int(b_off[-1]), dtype=torch.int32, device="cuda")
        hjcd.hjcd_topk_dup(ctx.h, rid, len(sizes), _dev(m_off, torch.int64), _dev(score), _dev(th), len(score),
                           _dev(b_off, torch.int64), tb, tb.shape[1], src, 5, api.make_params(dup_ratio=ratio, dup_sigma=0.0))
        torch.cuda.synchronize()
        src, tb = src.cpu().numpy(), tb.cpu().numpy()
        for t, m in enumerate(sizes):
            s = score[m_off[t]:m_off[t + 1]]
            want = np.tile(np.argsort(s + 0.0, kind="stable")[:K[t]], m // K[t])  # NaN sorts last
            np.testing.assert_array_equal(src[b_off[t]:b_off[t + 1]], want)
            np.testing.assert_array_equal(tb[:, b_off[t]:b_off[t + 1]], th[:, m_off[t] + want])


@pytest.mark.parametrize("kind", ["wide", "ulps", "equal", "few", "nan"])
@pytest.mark.parametrize("top_k", [1, 16, 64])
def test_rank_order(ctx, kind, top_k):
    rng = np.random.default_rng(3)
    rob = inputs.panda()
    rid = ctx.add_robot(rob)
    b_off = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    C, T = int(b_off[-1]), len(SIZES)
    score = np.concatenate([_scores(kind, m, rng) for m in SIZES])
    conv, hit = rng.random(C) < 0.5, rng.random(C) < 0.4
    perr, oerr = np.where(conv, 5e-4, 2e-3).astype(np.float32), rng.uniform(0, 0.01, C).astype(np.float32)
    th = inputs.joint_samples(rng, rob, C).T.astype(np.float32)
    q = torch.empty((T, top_k, 7), device="cuda")
    e = torch.empty((T, top_k, 2), device="cuda")
    cnt = torch.empty(T, dtype=torch.int32, device="cuda")
    hjcd.hjcd_rank(ctx.h, rid, T, _dev(b_off, torch.int64), _dev(th), C, _dev(score), _dev(perr), _dev(oerr),
                   _dev(hit, torch.uint8), 1e-3, 1e-2, None, top_k, q, e, cnt)
    torch.cuda.synchronize()
    q, e, cnt = q.cpu().numpy(), e.cpu().numpy(), cnt.cpu().numpy()
    for t in range(T):
        g = np.arange(b_off[t], b_off[t + 1])
        g = g[np.isfinite(score[g]) & ~hit[g]]
        want = g[np.lexsort((g, score[g] + 0.0, ~conv[g]))][:top_k]
        assert cnt[t] == len(want)
        np.testing.assert_array_equal(q[t, :len(want)], th[:, want].T)
        np.testing.assert_array_equal(e[t, :len(want)], np.stack([perr[want], oerr[want]], 1))
        assert np.isnan(q[t, len(want):]).all()
