"""The cost kernel's choice between one and two blocks per SM where shared memory decides it: wide
rows with the deepest disparity ranges, whose padded layout (two blocks) does not fit, run in the
other one, and the maps do not depend on the choice."""

import numpy as np
import pytest

from synth import make_pair
from test_gpu_limits import check_against_oracle, dev, gpu_run

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_00476_gb300 import zncc as Z  # noqa: E402


@pytest.mark.parametrize("value,blocks", [(1, 2), (2, 1), (3, 2), (100, 2)])
def test_every_tuning_value_is_accepted(value, blocks):
    p = make_pair(40, 200, 32, seed=3)
    left, right = dev(p.left), dev(p.right)
    disp = torch.empty((40, 200), dtype=torch.int16, device="cuda")
    with Z.ZnccContext(200, 40, 32, 9) as ctx:
        ctx.set_tuning(Z.ZNCC_TUNE_ROW_MINB2, value)
        ctx.zncc_run(left, right, disp, 20.0, 0.1, 1, Z.ZNCC_F32)
        torch.cuda.synchronize()
        assert ctx.launch_shape("zncc_cost_hpair")["variant"] == blocks
    check_against_oracle(p, disp.cpu().numpy().view(np.uint16), 32, 9, 1, Z.ZNCC_F32)


# whole rows where a split would compute as many slices a block (three of a row; two and slice 0 again)
@pytest.mark.parametrize("w,h,d,blocks", [(1900, 120, 33, 120), (1000, 100, 96, 100), (1900, 120, 16, 120)])
def test_i8_rows_are_not_split_for_nothing(w, h, d, blocks):
    p = make_pair(h, w, d, seed=w + d)
    left, right = dev(p.left), dev(p.right)
    disp = torch.full((h, w), -1, dtype=torch.int16, device="cuda")
    with Z.ZnccContext(w, h, d, 9) as ctx:
        ctx.zncc_run(left, right, disp, 20.0, 0.1, 1, Z.ZNCC_I8)
        torch.cuda.synchronize()
        assert ctx.launch_shape("zncc_cost_hpair")["blocks"] == blocks
    check_against_oracle(p, disp.cpu().numpy().view(np.uint16), d, 9, 1, Z.ZNCC_I8)


# (rows enough for four units per SM: the two-block layout is tried first)
@pytest.mark.parametrize("w,d,win", [(2560, 1024, 3), (2560, 1024, 9), (2560, 1024, 15), (2305, 1000, 9), (2400, 784, 9)])
def test_i8_rows_whose_padded_layout_does_not_fit(w, d, win):
    h = 7
    p = make_pair(h, w, d, seed=w + d + win)
    got = gpu_run(p, d, win, 1, Z.ZNCC_I8)
    check_against_oracle(p, got, d, win, 1, Z.ZNCC_I8)


@pytest.mark.parametrize("storage,iters", [(Z.ZNCC_F32, 0), (Z.ZNCC_F32, 1), (Z.ZNCC_F16, 1), (Z.ZNCC_I8, 1)])
@pytest.mark.parametrize("w,h,d", [(2560, 6, 1024), (2304, 20, 64), (1280, 30, 900), (160, 40, 64), (640, 100, 260)])
def test_maps_do_not_depend_on_the_blocks(w, h, d, storage, iters):
    p = make_pair(h, w, d, seed=w + h + d)
    left, right = dev(p.left), dev(p.right)
    maps = []
    for minb2 in (0, 1, 2):
        disp = torch.full((h, w), -1, dtype=torch.int16, device="cuda")
        with Z.ZnccContext(w, h, d, 9) as ctx:
            ctx.set_tuning(Z.ZNCC_TUNE_ROW_MINB2, minb2)
            ctx.zncc_run(left, right, disp, 20.0, 0.1, iters, storage)
            torch.cuda.synchronize()
            assert ctx.device_faults() == 0
        maps.append(disp.cpu().numpy())
    assert np.array_equal(maps[0], maps[1]) and np.array_equal(maps[0], maps[2])
