"""The memory of the fused path's volume: its slabs pad the disparities to 64 bytes per pixel; where
the device or a server's budget has no room for them, the volume is kept with its pixels padded
to four entries, and the maps are the same."""

import numpy as np
import pytest

from synth import make_pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_00476_gb300 import zncc as Z  # noqa: E402

W, H, ITERS = 900, 200, 2
CASES = [(17, Z.ZNCC_F32), (20, Z.ZNCC_F32), (20, Z.ZNCC_F16), (32, Z.ZNCC_F16)]


def volume_bytes(d, storage):
    return W * H * ((d + 3) // 4 * 4) * (4 if storage == Z.ZNCC_F32 else 2)


def pair(d):
    return make_pair(H, W, d, seed=d, disp="planes")


def run(ctx, p, storage):
    out = torch.full((H, W), -1, dtype=torch.int16, device="cuda")
    ctx.zncc_run(torch.from_numpy(p.left).cuda(), torch.from_numpy(p.right).cuda(), out, 20.0, 0.1, ITERS, storage)
    torch.cuda.synchronize()
    return out.cpu().numpy().view(np.uint16)


@pytest.mark.parametrize("d,storage", CASES)
def test_run_without_memory_for_slabs(d, storage, monkeypatch):
    p = pair(d)
    with Z.ZnccContext(W, H, d, 9) as ctx:
        want = run(ctx, p, storage)
    need = volume_bytes(d, storage)
    with Z.ZnccContext(W, H, d, 9) as ctx:
        monkeypatch.setenv("ZNCC_FAIL_DEVICE_ALLOC", f">{need - 1}")
        with pytest.raises(RuntimeError):
            run(ctx, p, storage)
        monkeypatch.setenv("ZNCC_FAIL_DEVICE_ALLOC", f">{need}")
        assert np.array_equal(run(ctx, p, storage), want)
        monkeypatch.delenv("ZNCC_FAIL_DEVICE_ALLOC")
        assert np.array_equal(run(ctx, p, storage), want)
        assert ctx.device_faults() == 0


@pytest.mark.parametrize("d,storage", CASES)
def test_server_admits_a_shape_whose_slabs_exceed_its_budget(d, storage):
    p = pair(d)
    with Z.ZnccContext(W, H, d, 9) as ctx:
        want = run(ctx, p, storage)
    budget = W * H * 44 + volume_bytes(d, storage)
    if storage == Z.ZNCC_F16:
        budget += W * H * 12 * (2 * ITERS - 1)
    disp = np.zeros((H, W), np.uint16)
    with Z.ZnccServer(budget, 2) as srv:
        t = srv.submit(p.left, p.right, d, 9, 20.0, 0.1, ITERS, storage)
        assert srv.poll(t, disp, 20_000_000) == Z.ZNCC_OK
    assert np.array_equal(disp, want)
