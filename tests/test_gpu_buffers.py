"""Device buffers of a solve, which its kernels read and write in place, at any byte address."""
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


def _at(offset, data):
    """The bytes of a 32-bit device tensor at an offset into a buffer of bytes (and the buffer)."""
    raw = data.contiguous().view(torch.uint8).flatten()
    buf = torch.full((raw.numel() + 16,), 171, dtype=torch.uint8, device="cuda")
    buf[offset:offset + raw.numel()] = raw
    return buf, buf[offset:offset + raw.numel()]


@pytest.mark.parametrize("T,top_k", [(1, 1), (5, 3)])
@pytest.mark.parametrize("offset", [1, 2, 3, 4])
def test_device_buffers_at_any_byte(ctx, T, top_k, offset):
    rob = inputs.panda()
    rid = ctx.add_robot(rob)
    rng = np.random.default_rng(6)
    tg = ctx.fk(rid, torch.as_tensor(inputs.joint_samples(rng, rob, T).T.copy(), dtype=torch.float32, device="cuda"))
    qc = torch.as_tensor(inputs.joint_samples(rng, rob, T), dtype=torch.float32, device="cuda")
    ref = ctx.solve(rid, -1, tg, 40, top_k, 9, 7, q_current=qc)
    shapes, types = ((T, top_k, 7), (T, top_k, 2), (T,)), (torch.float32, torch.float32, torch.int32)
    outs = [_at(offset, torch.zeros(s, dtype=d, device="cuda")) for s, d in zip(shapes, types)]
    tg_b, qc_b = _at(offset, tg), _at(offset, qc)
    o = ctx.opts(40, top_k, 9)
    hjcd.hjcd_solve_nearest(ctx.h, rid, -1, T, tg_b[1], qc_b[1], o, outs[0][1], outs[1][1], outs[2][1], None)
    torch.cuda.synchronize()
    for (buf, part), r in zip(outs, ref):
        assert torch.equal(part, r.contiguous().view(torch.uint8).flatten())
        assert bool((buf[:offset] == 171).all()) and bool((buf[offset + part.numel():] == 171).all())
