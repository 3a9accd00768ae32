"""Small batches take kernels that spread a candidate over a CTA only where that is the shorter way: no
stage of a batch just below their largest size takes longer than of one just above it, whatever the
chain, down to a single joint."""
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


def _time(f):
    """Median device time (us) of a call among queued ones."""
    f()
    ms = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(8):
            f()
        b.record()
        torch.cuda.synchronize()
        ms.append(a.elapsed_time(b) / 8)
    return float(np.median(ms)) * 1e3


@pytest.mark.parametrize("stage", ["ccd", "lm"])
@pytest.mark.parametrize("which", ["planar1", "planar2", "planar3", "planar4", "planar5", "chain7", "chain24"])
def test_a_smaller_batch_takes_no_longer(ctx, stage, which):
    rob = inputs.planar([0.3] * int(which[6:])) if which.startswith("planar") else inputs.dof_scaling_robot(int(which[5:]))
    rid = ctx.add_robot(rob)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(1)
    T, most = 8, 64 * sms + 64
    tg = ctx.fk(rid, torch.as_tensor(inputs.joint_samples(rng, rob, T).T.copy(), dtype=torch.float32, device="cuda"))
    params = api.make_params()

    def run(C):
        th = torch.as_tensor(inputs.joint_samples(np.random.default_rng(2), rob, C).T.copy(), dtype=torch.float32, device="cuda")
        tgt = torch.as_tensor(np.arange(C) * T // C, dtype=torch.int32, device="cuda")
        cand = torch.as_tensor(np.arange(C) % 1000, dtype=torch.int32, device="cuda")
        out, sc, pe, oe = torch.empty_like(th), *(torch.empty(C, device="cuda") for _ in range(3))
        it = torch.empty(C, dtype=torch.int32, device="cuda")

        def call():
            if stage == "ccd":
                hjcd.hjcd_po_ccd(ctx.h, rid, T, tg, 1e-3, 1e-2, 7, params, C, tgt, cand, th, out, C, 0, 32, sc, pe, oe, it)
            else:
                out.copy_(th)
                hjcd.hjcd_pjik(ctx.h, rid, T, tg, 1e-3, 1e-2, 7, params, C, tgt, cand, out, C, 0, 20, sc, pe, oe, it)

        return _time(call)

    above = run(most)
    for per_sm in (32, 48, 64):
        assert run(per_sm * sms) <= 1.08 * above + 2, per_sm  # (the clock, and the candidates' own spread)


@pytest.mark.parametrize("ratio", [1, 4])
@pytest.mark.parametrize("which", ["random0", "random3", "chain7", "chain12"])
def test_a_smaller_polish_takes_no_longer(ctx, which, ratio):
    """The polish of a mid-size batch leaves its last candidates to a second launch; of a chain that often
    runs to the cap, or with every seed polished, that must not take longer than the one launch of a
    batch past those sizes (216 candidates per SM)."""
    rob = inputs.cfg3_chains()[int(which[6:])] if which.startswith("random") else inputs.dof_scaling_robot(int(which[5:]))
    rob.sph_body, rob.sph_xyzr = rob.sph_body[:0], rob.sph_xyzr[:0]
    rid = ctx.add_robot(rob)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    most = 216 * sms // 1000 + 2
    tg = ctx.fk(rid, torch.as_tensor(inputs.joint_samples(np.random.default_rng(16), rob, most).T.copy(), dtype=torch.float32,
                                     device="cuda"))
    params = api.make_params(dup_ratio=ratio)

    def polish_us(T):
        part = tg[:T].contiguous()
        ctx.solve(rid, -1, part, 1000, 1, 5, rob.n, params=params)
        us = []
        for _ in range(7):
            ctx.solve(rid, -1, part, 1000, 1, 5, rob.n, params=params)
            us.append(1e3 * hjcd.hjcd_phase_times(ctx.h)[2])
        return float(np.median(us))

    hjcd.hjcd_set_profiling(ctx.h, 1)
    try:
        above = polish_us(most)
        for T in (8, 12, 16, 20, 24, most - 2):
            assert polish_us(T) <= 1.08 * above + 5, T
    finally:
        hjcd.hjcd_set_profiling(ctx.h, 0)
