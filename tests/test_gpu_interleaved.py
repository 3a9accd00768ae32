"""Solves with device outputs, which return while they run, between solves with host outputs on other
streams, over one context: they share its workspace and its pinned buffer, which is released for the
next image after a solve's first launch and holds the error flag and the small host results."""
import numpy as np
import pytest
import torch

from paper_2510_07514_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scene", [False, True])
def test_device_and_host_outputs_in_turn(scene):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    rob = inputs.panda_with_spheres(np.random.default_rng(5))
    # sizes that grow the pinned buffer from solve to solve: results through it (up to 1 MB), then by copies
    sizes = [(1, 64, 1), (7, 100, 3), (60, 40, 8), (300, 40, 16), (900, 32, 24), (2000, 32, 24), (3, 1000, 2)]
    cases = []
    for k, (T, seeds, top_k) in enumerate(sizes):
        rng = np.random.default_rng(50 + k)
        cases.append((inputs.joint_samples(rng, rob, T), seeds, top_k, 70 + k))
    obstacles = inputs.random_scene(np.random.default_rng(1), 60, 5)

    def targets(ctx, rid, th):
        return ctx.fk(rid, torch.as_tensor(th.T.copy(), dtype=torch.float32, device="cuda"))

    ref = []
    with api.Context(0) as ctx:
        rid, sid = ctx.add_robot(rob), ctx.set_scene(obstacles) if scene else -1
        for th, seeds, top_k, seed in cases:
            out = ctx.solve(rid, sid, targets(ctx, rid, th), seeds, top_k, seed, 7)
            torch.cuda.synchronize()
            ref.append([x.cpu().view(torch.int32) for x in out])
    for turn in range(3):
        with api.Context(0) as ctx:  # a fresh context: its buffers grow from nothing
            rid, sid = ctx.add_robot(rob), ctx.set_scene(obstacles) if scene else -1
            tgs = [targets(ctx, rid, c[0]) for c in cases]
            hosts = [t.cpu() for t in tgs]
            torch.cuda.synchronize()
            a, b = torch.cuda.Stream(), torch.cuda.Stream()
            got = []
            for k, (th, seeds, top_k, seed) in enumerate(cases):
                big = cases[-2]  # in flight on the other stream while the host waits for its own
                got.append((len(cases) - 2, ctx.solve(rid, sid, tgs[-2], big[1], big[2], big[3], 7, stream=a)))
                got.append((k, ctx.solve(rid, sid, tgs[k], seeds, top_k, seed, 7, stream=a if turn == 1 else b)))
                got.append((k, ctx.solve(rid, sid, hosts[k], seeds, top_k, seed, 7, stream=b)))
            torch.cuda.synchronize()
            for k, out in got:
                for x, y in zip(out, ref[k]):
                    assert torch.equal(x.cpu().view(torch.int32), y)
