"""The cost volume's stores at every alignment: volumes whose pixels do not start on whole groups
of four entries (odd disparity counts, buffers off the alignment) hold the same values bit for bit
as the volume of the next multiple of four disparities (a cost does not depend on the range), and
nothing is written around them."""

import numpy as np
import pytest

from synth import make_pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_00476_gb300 import zncc as Z  # noqa: E402

DTYPES = {"f32": (torch.float32, Z.ZNCC_F32), "f16": (torch.float16, Z.ZNCC_F16)}
GUARD = 64                                              # entries kept on both sides of the volume


def volume(left, right, d, win, dtype, off, minb2):
    tdt, flag = DTYPES[dtype]
    h, w = left.shape
    buf = torch.full((GUARD + off + h * w * d + GUARD,), 7.0, dtype=tdt, device="cuda")
    cost = buf[GUARD + off:GUARD + off + h * w * d].view(h, w, d)
    with Z.ZnccContext(w, h, d, win) as ctx:
        ctx.set_tuning(Z.ZNCC_TUNE_ROW_MINB2, minb2)
        ctx.zncc_cost_volume(left, right, cost, flag)
        torch.cuda.synchronize()
        assert ctx.device_faults() == 0
    assert (buf[:GUARD + off] == 7.0).all() and (buf[GUARD + off + h * w * d:] == 7.0).all()
    return cost


# widths of eight, four and two lanes per 16-pixel chunk, whole and partial chunks; disparities
# that leave a group, a lane quad or a slice partly empty; entries from an aligned address
@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("w,h,d,win,off", [
    (1, 1, 1, 3, 0), (16, 2, 3, 3, 0), (17, 3, 2, 5, 1), (250, 4, 31, 9, 0), (640, 2, 33, 7, 2), (641, 2, 17, 9, 3),
    (1024, 2, 66, 11, 0), (1025, 2, 15, 9, 0), (1279, 3, 63, 9, 1), (1300, 2, 130, 13, 0), (2049, 2, 7, 9, 0),
    (2500, 2, 9, 9, 1), (2559, 2, 61, 5, 0), (3072, 1, 22, 15, 0), (64, 5, 32, 9, 1), (64, 5, 32, 9, 2),
    (1100, 2, 16, 9, 3), (2100, 2, 8, 9, 2)])
def test_stores_at_every_alignment(w, h, d, win, off, dtype):
    p = make_pair(h, w, max(d, 2), seed=w + 5 * h + d, disp="planes")
    left, right = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (p.left, p.right))
    want = volume(left, right, (d + 3) // 4 * 4, win, dtype, 0, 0)[:, :, :d]
    for minb2 in (0, 1):
        assert torch.equal(volume(left, right, d, win, dtype, off, minb2), want)


# volumes of more than half a million entries, whose lanes trade entries before the stores: blocks of
# eight, four and two lanes per chunk, one and two per SM
@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("w,h,d,win,off", [
    (1024, 512, 1, 3, 0), (1023, 257, 2, 3, 1), (70, 420, 18, 9, 0), (641, 50, 17, 9, 3), (250, 70, 31, 9, 0),
    (1025, 40, 15, 5, 0), (1300, 13, 33, 13, 1), (1999, 5, 54, 9, 0), (2049, 38, 7, 9, 0), (2500, 24, 9, 9, 1),
    (3072, 8, 22, 15, 0), (600, 30, 32, 7, 2)])
def test_stores_of_larger_volumes(w, h, d, win, off, dtype):
    assert w * h * d >= 1 << 19
    test_stores_at_every_alignment(w, h, d, win, off, dtype)
