"""The slab-stored line passes (the fused path's default) against the general line passes
(cp.async staging, volume [H][W][D]): the same sums in the same association, so the maps are
equal, over line lengths on both sides of every change of block shape and scan group, columns and
rows that leave a block partly empty, and disparity counts that leave a slab or slice partly
empty."""

import numpy as np
import pytest

from synth import make_pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_00476_gb300 import zncc as Z  # noqa: E402

STORAGE = {"f32": Z.ZNCC_F32, "f16": Z.ZNCC_F16}


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def run(ctx, left, right, iters, storage, sigma_s=20.0):
    disp = torch.full(left.shape, -1, dtype=torch.int16, device="cuda")
    ctx.zncc_run(left, right, disp, sigma_s, 0.1, iters, STORAGE[storage])
    torch.cuda.synchronize()
    assert ctx.device_faults() == 0
    return disp


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("w,h,d,iters", [
    (1, 1, 1, 1), (16, 16, 4, 2), (17, 33, 5, 2), (31, 3, 16, 1), (64, 256, 17, 2), (65, 257, 31, 1), (321, 320, 33, 2),
    (385, 384, 48, 2), (449, 448, 20, 1), (513, 512, 24, 1), (641, 40, 32, 2), (769, 30, 64, 1), (833, 9, 8, 2),
    (1025, 17, 36, 2), (1409, 12, 40, 2), (1537, 10, 24, 1), (2049, 6, 12, 2), (2817, 5, 64, 1), (3072, 4, 20, 2),
    (9, 641, 20, 2), (7, 1025, 36, 1), (5, 1100, 256, 2), (4, 2047, 64, 1), (3, 2049, 12, 2), (3, 4096, 20, 2),
    (1242, 375, 100, 3)])
def test_slab_passes_equal_general_passes(w, h, d, iters, storage):
    p = make_pair(h, w, max(d, 2), seed=w + 3 * h + d, disp="planes")
    left, right = dev(p.left), dev(p.right)
    with Z.ZnccContext(w, h, d, 5) as ctx:
        new = run(ctx, left, right, iters, storage)
        again = run(ctx, left, right, iters, storage)
        ctx.set_tuning(Z.ZNCC_TUNE_LINE_LOADS, 1)
        ref = run(ctx, left, right, iters, storage)
    assert torch.equal(new, ref) and torch.equal(again, ref)


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("key,value", [(Z.ZNCC_TUNE_V_LPC, 1), (Z.ZNCC_TUNE_V_LPC, 2), (Z.ZNCC_TUNE_H_TQ, 2),
                                       (Z.ZNCC_TUNE_H_TQ, 8), (Z.ZNCC_TUNE_V_TQ, 4), (Z.ZNCC_TUNE_ROW_SPB, 1)])
def test_slab_passes_equal_general_passes_with_tuning(key, value, storage):
    p = make_pair(130, 400, 40, seed=5, disp="planes")
    left, right = dev(p.left), dev(p.right)
    with Z.ZnccContext(400, 130, 40, 7) as ctx:
        ctx.set_tuning(key, value)
        new = run(ctx, left, right, 2, storage)
        ctx.set_tuning(Z.ZNCC_TUNE_LINE_LOADS, 1)
        ref = run(ctx, left, right, 2, storage)
    assert torch.equal(new, ref)


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_slab_passes_in_a_batch(storage):
    """Pairs that share launches and pairs that do not, of uneven sizes and disparity counts."""
    shapes = [(200, 60, 20), (640, 192, 33), (200, 70, 64), (1100, 20, 16), (200, 64, 20), (33, 500, 24)]
    pairs = [make_pair(h, w, d, seed=i, disp="planes") for i, (w, h, d) in enumerate(shapes)]
    ims = [(dev(p.left), dev(p.right)) for p in pairs]
    ctxs = [Z.ZnccContext(w, h, d, 5) for w, h, d in shapes]
    out = [torch.full(l.shape, -1, dtype=torch.int16, device="cuda") for l, _ in ims]
    Z.zncc_run_batch(ctxs, [l for l, _ in ims], [r for _, r in ims], out, 20.0, 0.1, 2, STORAGE[storage])
    torch.cuda.synchronize()
    for c, (l, r), o in zip(ctxs, ims, out):
        c.set_tuning(Z.ZNCC_TUNE_LINE_LOADS, 1)
        assert torch.equal(o, run(c, l, r, 2, storage))
        c.close()


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("w,h,d,off", [(1, 1, 8, 0), (40, 384, 16, 0), (41, 385, 24, 0), (375, 130, 40, 0), (1280, 20, 32, 0),
                                       (1281, 9, 64, 0), (200, 193, 128, 0), (200, 193, 100, 0), (64, 50, 20, 0),
                                       (64, 50, 17, 0), (64, 50, 32, 1), (64, 50, 32, 4), (7, 450, 8, 0)])
def test_aggregation_of_a_callers_volume_equals_general_passes(w, h, d, off, storage):
    """dt_aggregate with and without the TMA-staged passes (by pixel alignment, start address and
    line length): the same sums in the same association, so the same values bit for bit."""
    rng = np.random.default_rng(w + h + d + off)
    tdt = torch.float32 if storage == "f32" else torch.float16
    guide = dev(rng.integers(0, 256, (h, w), dtype=np.uint8) // 16 * 3)
    v = torch.from_numpy(rng.uniform(-1, 1, (h, w, d)).astype(np.float32)).cuda()
    with Z.ZnccContext(w, h, d, 3) as ctx:
        got = []
        for loads in (0, 1):
            buf = torch.zeros(off + h * w * d, dtype=tdt, device="cuda")
            cost = buf[off:].view(h, w, d)
            cost.copy_(v)
            ctx.set_tuning(Z.ZNCC_TUNE_LINE_LOADS, loads)
            ctx.dt_aggregate(guide, cost, 20.0, 0.3, 2, STORAGE[storage])
            torch.cuda.synchronize()
            got.append(cost.clone())
        assert ctx.device_faults() == 0
    assert torch.equal(got[0], got[1])


def test_carries_through_long_rows_with_many_steps():
    """Rows of 14 warps and more with many steps per block: one chunk's lanes carry through the scan
    groups."""
    w, h, d = 1700, 80, 800
    p = make_pair(h, w, d, seed=11, disp="planes")
    left, right = dev(p.left), dev(p.right)
    with Z.ZnccContext(w, h, d, 3) as ctx:
        new = run(ctx, left, right, 2, "f32")
        ctx.set_tuning(Z.ZNCC_TUNE_LINE_LOADS, 1)
        ref = run(ctx, left, right, 2, "f32")
    assert torch.equal(new, ref)
