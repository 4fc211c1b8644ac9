"""Which line kernel a fused run took, in which block shape, and what it stored: every variant of
the slab passes (lanes per chunk, lines per block, two columns to a warp, the carry chain) leaves
the volume of the general passes bit for bit, and the runs of this file did take that variant."""

import numpy as np
import pytest

from synth import make_pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_00476_gb300 import zncc as Z  # noqa: E402

STORAGE = {"f32": (Z.ZNCC_F32, torch.float32, torch.int32), "f16": (Z.ZNCC_F16, torch.float16, torch.int16)}
SLAB, GENERAL = 2, 1


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def run(ctx, left, right, storage, loads, iters=2):
    """Map, stored volume (its bits) and line launches of a run."""
    flag, tdt, bits = STORAGE[storage]
    ctx.set_tuning(Z.ZNCC_TUNE_LINE_LOADS, loads)
    disp = torch.full(left.shape, -1, dtype=torch.int16, device="cuda")
    ctx.zncc_run(left, right, disp, 20.0, 0.1, iters, flag)
    vol = torch.empty((*left.shape, ctx.D), dtype=tdt, device="cuda")
    ctx.stored_volume(vol, flag)
    torch.cuda.synchronize()
    assert ctx.device_faults() == 0
    return disp, vol.view(bits), [ctx.launch_shape(k) for k in ("dt_hpair", "dt_vpair", "dt_vpair_wta")]


def shape_of(launch):
    return tuple(launch[k] for k in ("lanes", "lines", "columns", "chain"))


# (lanes, lines, columns to a warp, chain) of the row, column and column + WTA passes
@pytest.mark.parametrize("storage,w,h,d,rows,cols,wta", [
    ("f32", 64, 50, 20, (4, 1, 1, 0), (4, 4, 2, 0), (4, 4, 2, 0)),
    ("f32", 300, 700, 33, (4, 1, 1, 0), (4, 2, 2, 0), (4, 2, 2, 0)),
    ("f32", 900, 400, 256, (4, 1, 1, 0), (4, 4, 1, 0), (4, 4, 1, 0)),
    ("f32", 100, 513, 16, (4, 1, 1, 0), (4, 3, 1, 0), (4, 4, 1, 0)),
    ("f32", 1700, 80, 800, (4, 1, 1, 1), (4, 4, 2, 0), (4, 4, 2, 0)),
    ("f32", 2049, 20, 40, (2, 1, 1, 0), (4, 4, 2, 0), (4, 4, 2, 0)),
    ("f32", 12, 4096, 20, (4, 1, 1, 0), (2, 1, 1, 0), (2, 1, 1, 0)),
    ("f16", 64, 50, 20, (8, 1, 1, 0), (8, 4, 1, 0), (8, 4, 1, 0)),
    ("f16", 1242, 375, 33, (8, 1, 1, 0), (8, 3, 1, 0), (8, 3, 1, 0)),
    ("f16", 1000, 500, 128, (8, 1, 1, 0), (8, 2, 1, 0), (8, 2, 1, 0)),
    ("f16", 1000, 260, 800, (8, 1, 1, 0), (8, 4, 1, 0), (8, 4, 1, 0)),
    ("f16", 1700, 80, 800, (4, 1, 1, 0), (8, 4, 1, 0), (8, 4, 1, 0)),
    ("f16", 2049, 20, 40, (4, 1, 1, 0), (8, 4, 1, 0), (8, 4, 1, 0)),
    ("f16", 3072, 12, 20, (2, 1, 1, 0), (8, 4, 1, 0), (8, 4, 1, 0)),
    ("f16", 40, 2000, 24, (8, 1, 1, 0), (4, 1, 1, 0), (4, 1, 1, 0)),
    ("f16", 12, 4096, 20, (8, 1, 1, 0), (2, 1, 1, 0), (2, 1, 1, 0))])
def test_slab_passes_store_the_general_passes_volume(storage, w, h, d, rows, cols, wta):
    p = make_pair(h, w, max(d, 2), seed=w + h + d, disp="planes")
    left, right = dev(p.left), dev(p.right)
    with Z.ZnccContext(w, h, d, 5) as ctx:
        disp, vol, launches = run(ctx, left, right, storage, 0)
        assert [l["variant"] for l in launches] == [SLAB] * 3
        assert [shape_of(l) for l in launches] == [rows, cols, wta]
        ref_disp, ref_vol, ref_launches = run(ctx, left, right, storage, 1)
        assert [l["variant"] for l in ref_launches] == [GENERAL] * 3
    assert torch.equal(vol, ref_vol) and torch.equal(disp, ref_disp)


def test_carry_chain_in_a_batch():
    """Pairs that share the row launches, with enough steps a block for the carry chain."""
    w, h, d, n = 1700, 16, 600, 7
    pairs = [make_pair(h, w, d, seed=i, disp="planes") for i in range(n)]
    ims = [(dev(p.left), dev(p.right)) for p in pairs]
    ctxs = [Z.ZnccContext(w, h, d, 5) for _ in range(n)]
    out = [torch.full((h, w), -1, dtype=torch.int16, device="cuda") for _ in range(n)]
    Z.zncc_run_batch(ctxs, [l for l, _ in ims], [r for _, r in ims], out, 20.0, 0.1, 2, Z.ZNCC_F32)
    assert ctxs[0].launch_shape("dt_hpair")["variant"] == SLAB and ctxs[0].launch_shape("dt_hpair")["chain"] == 1
    vols = []
    for c in ctxs:
        vols.append(torch.empty((h, w, d), dtype=torch.float32, device="cuda"))
        c.stored_volume(vols[-1], Z.ZNCC_F32)
    torch.cuda.synchronize()
    for c, (l, r), o, v in zip(ctxs, ims, out, vols):
        disp, vol, _ = run(c, l, r, "f32", 1)
        assert torch.equal(v.view(torch.int32), vol) and torch.equal(o, disp)
        c.close()


def test_stored_volume_needs_a_run_of_that_type():
    p = make_pair(20, 40, 8, seed=1)
    left, right = dev(p.left), dev(p.right)
    disp = torch.empty((20, 40), dtype=torch.int16, device="cuda")
    vol = torch.empty((20, 40, 8), dtype=torch.float32, device="cuda")
    with Z.ZnccContext(40, 20, 8, 3) as ctx:
        for iters, storage, ok in ((0, Z.ZNCC_F32, False), (1, Z.ZNCC_F16, False), (1, Z.ZNCC_F32, True), (0, Z.ZNCC_F32, False)):
            ctx.zncc_run(left, right, disp, 20.0, 0.1, iters, storage)
            if ok:
                ctx.stored_volume(vol)
            else:
                with pytest.raises(Z.ZnccError):
                    ctx.stored_volume(vol)
        torch.cuda.synchronize()


def test_no_stored_volume_after_a_replayed_host_run():
    """A replayed run writes the volume in the layout of its capture, not of the last direct run."""
    w, h, d = 64, 32, 20
    p = make_pair(h, w, d, seed=3)
    left, right = dev(p.left), dev(p.right)
    host = [torch.from_numpy(np.ascontiguousarray(a)).pin_memory() for a in (p.left, p.right)]
    host.append(torch.zeros((h, w), dtype=torch.int16).pin_memory())
    args = [host[0].numpy(), host[1].numpy(), host[2].numpy().view(np.uint16)]
    disp = torch.empty((h, w), dtype=torch.int16, device="cuda")
    vol = torch.empty((h, w, d), dtype=torch.float16, device="cuda")
    with Z.ZnccContext(w, h, d, 5, stream=torch.cuda.Stream()) as ctx:
        torch.cuda.synchronize()
        ctx.zncc_run(left, right, disp, 20.0, 0.1, 2, Z.ZNCC_F16)
        ctx.stored_volume(vol, Z.ZNCC_F16)
        for _ in range(3):                  # issued, captured, replayed
            ctx.zncc_run_host(*args, 20.0, 0.1, 2, Z.ZNCC_F32)
        ctx.zncc_run(left, right, disp, 20.0, 0.1, 2, Z.ZNCC_F16)
        ctx.zncc_run_host(*args, 20.0, 0.1, 2, Z.ZNCC_F32)
        with pytest.raises(Z.ZnccError):
            ctx.stored_volume(vol, Z.ZNCC_F16)
