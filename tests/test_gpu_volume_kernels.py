"""Window statistics and WTA of a stored volume at the edges of their kernels' tiles, alignments
and loads: whole numbers, compared exactly (1/sigma to its float rounding)."""

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_00476_gb300 import zncc as Z  # noqa: E402


# (W, H, r, bytes from an aligned address to the first pixel, pitch - W): widths around the
# centres of a block (512 columns less the window), heights around its 8 rows, rows that do and
# do not start on 4 bytes
@pytest.mark.parametrize("w,h,r,off,pad", [
    (506, 8, 1, 0, 2), (507, 9, 1, 0, 1), (508, 7, 1, 4, 0), (1000, 17, 4, 0, 0), (1001, 16, 4, 1, 3),
    (499, 3, 5, 2, 1), (500, 24, 5, 0, 4), (494, 8, 7, 0, 2), (495, 1, 7, 0, 1), (3, 40, 7, 3, 2), (1, 1, 2, 0, 0)])
def test_window_stats_tiles_and_alignment(w, h, r, off, pad):
    rng = np.random.default_rng(w + 31 * h + r)
    pitch = w + pad
    buf = rng.integers(0, 256, off + pitch * h + 64, dtype=np.uint8)
    dev = torch.from_numpy(buf).cuda()
    img = dev[off:off + pitch * h].view(h, pitch)[:, :w]
    with Z.ZnccContext(w, h, 4, 2 * r + 1) as ctx:
        S, Q = (torch.empty((h, w), dtype=torch.int32, device="cuda") for _ in range(2))
        inv = torch.empty((h, w), dtype=torch.float32, device="cuda")
        ctx.zncc_window_stats(img, S, Q, inv)
        S2 = torch.zeros(h * w + 1, dtype=torch.int32, device="cuda")       # rows off 16 bytes
        assert Z.lib().zncc_window_stats(ctx._h, img.data_ptr(), pitch, S2[1:].data_ptr(), None, None) == Z.ZNCC_OK
        torch.cuda.synchronize()
    s, q = oracle.window_sums(np.ascontiguousarray(img.cpu().numpy()), r)
    assert np.array_equal(S.cpu().numpy(), s) and np.array_equal(Q.cpu().numpy(), q)
    assert np.array_equal(S2[1:].view(h, w).cpu().numpy(), s)
    var = (2 * r + 1) ** 2 * q.astype(np.int64) - s.astype(np.int64) ** 2
    ref = np.where(var > 0, 1.0 / np.sqrt(np.maximum(var, 1)), 0.0)
    assert np.allclose(inv.cpu().numpy(), ref, rtol=4e-7, atol=0)


# the same where the image is large enough for the kernel that walks down the rows (5 M pixel reads)
@pytest.mark.parametrize("w,h,r,off,pad", [
    (1667, 1000, 1, 0, 1), (1666, 1000, 1, 4, 2), (1012, 1009, 2, 0, 0), (499, 1121, 5, 2, 1), (500, 1024, 5, 0, 4),
    (494, 777, 7, 0, 2), (495, 775, 7, 1, 1), (1920, 1080, 5, 0, 0), (1001, 556, 4, 3, 7)])
def test_window_stats_of_large_images(w, h, r, off, pad):
    test_window_stats_tiles_and_alignment(w, h, r, off, pad)


# D around the lanes per pixel and loads per lane, volumes that start off 16 bytes
@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("d,off", [(1, 0), (2, 0), (3, 1), (8, 0), (8, 1), (31, 0), (32, 0), (33, 0), (36, 2),
                                   (64, 0), (66, 0), (128, 0), (132, 4), (256, 0), (260, 0), (1021, 0), (1024, 0)])
def test_wta_loads_ties_and_special_values(d, off, dtype):
    w, h = 37, 5
    rng = np.random.default_rng(7 * d + off)
    tdt, flag = (torch.float32, Z.ZNCC_F32) if dtype == "f32" else (torch.float16, Z.ZNCC_F16)
    v = rng.integers(-3, 4, (h, w, d)).astype(np.float32)            # many ties
    v[0, 0] = -np.inf                                                # nothing beats the start: 0
    v[0, 1] = np.nan
    v[1, :, d // 2:] = -np.inf
    v[2, :, ::2] = np.nan
    v[3] = np.where(v[3] == 0, -0.0, v[3])
    buf = torch.zeros(off + h * w * d, dtype=tdt, device="cuda")
    cost = buf[off:].view(h, w, d)
    cost.copy_(torch.from_numpy(v))
    disp = torch.empty((h, w), dtype=torch.int16, device="cuda")
    with Z.ZnccContext(w, h, d, 3) as ctx:
        ctx.wta_disparity(cost, disp, flag)
        torch.cuda.synchronize()
    n = np.where(np.isnan(v), -np.inf, v)
    ref = np.where(n.max(-1) == -np.inf, 0, n.argmax(-1))            # argmax: the smallest d of a tie
    assert np.array_equal(disp.cpu().numpy(), ref)


# pixels that start at every place of a 16-byte vector, around the lanes per pixel (24, 48 and 96
# vectors) and the short pixels; the volume's first and last pixels share vectors with what lies
# around it, which must not count
@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("d,off", [(5, 1), (9, 0), (12, 0), (14, 2), (15, 0), (16, 1), (17, 0), (20, 0), (28, 1), (34, 0), (93, 0), (95, 1), (97, 3),
                                   (155, 0), (186, 2), (190, 0), (193, 5), (255, 0), (379, 0), (385, 7), (765, 1), (1019, 3)])
def test_wta_of_pixels_off_16_bytes(d, off, dtype):
    w, h = 41, 3
    rng = np.random.default_rng(11 * d + off)
    tdt, flag = (torch.float32, Z.ZNCC_F32) if dtype == "f32" else (torch.float16, Z.ZNCC_F16)
    v = rng.integers(-40, 41, (h, w, d)).astype(np.float32)
    v[0, :, d - 1] = 50.0                                            # the best at either end of a pixel
    v[1, :, 0] = 50.0
    v[2, ::2] = -60.0
    buf = torch.full((16 + off + h * w * d + 16,), 99.0, dtype=tdt, device="cuda")
    cost = buf[16 + off:16 + off + h * w * d].view(h, w, d)
    cost.copy_(torch.from_numpy(v))
    disp = torch.empty((h, w), dtype=torch.int16, device="cuda")
    with Z.ZnccContext(w, h, d, 3) as ctx:
        ctx.wta_disparity(cost, disp, flag)
        torch.cuda.synchronize()
    assert np.array_equal(disp.cpu().numpy(), v.argmax(-1))


# radii 3 and 6, rows off 4 bytes on both sides of the sizes from which they walk down the rows too
@pytest.mark.parametrize("w,h,r,off,pad", [
    (1004, 801, 3, 0, 0), (700, 601, 6, 0, 0), (1202, 449, 6, 0, 0), (1201, 660, 6, 2, 2), (1199, 700, 6, 1, 2),
    (1241, 375, 7, 0, 0), (1003, 1111, 4, 3, 0), (1666, 1000, 1, 0, 0), (1001, 1500, 3, 0, 0)])
def test_window_stats_of_large_images_radii_and_rows_off_4_bytes(w, h, r, off, pad):
    test_window_stats_tiles_and_alignment(w, h, r, off, pad)


# the kernels that read packed statistics of left centres and of right centres down to 1 - D, at
# sizes where both statistics are computed down the rows (5 M reads, 4-byte rows): equal to the
# costs of the kernel that computes its own statistics
@pytest.mark.parametrize("w,h,d,r", [(1920, 600, 8, 2), (1920, 600, 9, 2), (1920, 600, 10, 2), (1920, 600, 11, 2), (1664, 450, 32, 4)])
def test_packed_statistics_of_large_images(w, h, d, r):
    rng = np.random.default_rng(w + d)
    left, right = (torch.from_numpy(rng.integers(0, 256, (h, w), dtype=np.uint8)).cuda() for _ in range(2))
    with Z.ZnccContext(w, h, d, 2 * r + 1) as ctx:
        want, scan = (torch.empty((h, w, d), dtype=torch.float32, device="cuda") for _ in range(2))
        ctx.zncc_cost_volume(left, right, want)
        ctx.zncc_cost_volume_scan(left, right, scan)
        assert torch.equal(scan, want)
        ctx.zncc_cost_volume_mma(left, right, scan)
        assert torch.equal(scan, want)


# volumes of more than a million entries: pixels of one to six rounds of loads at eight lanes
# (up to 192 vectors) and of 16 lanes
@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("d,off", [(189, 1), (379, 3), (385, 0), (511, 2), (523, 0), (765, 1), (769, 0), (999, 2), (1021, 5)])
def test_wta_of_large_volumes_off_16_bytes(d, off, dtype):
    w = 41
    h = (1 << 20) // (w * d) + 1
    rng = np.random.default_rng(d + off)
    tdt, flag = (torch.float32, Z.ZNCC_F32) if dtype == "f32" else (torch.float16, Z.ZNCC_F16)
    v = rng.integers(-40, 41, (h, w, d)).astype(np.float32)
    v[0, :, d - 1] = 50.0                                            # the best at either end of a pixel
    v[1, :, 0] = 50.0
    v[2, ::2] = -60.0
    buf = torch.full((16 + off + h * w * d + 16,), 99.0, dtype=tdt, device="cuda")
    cost = buf[16 + off:16 + off + h * w * d].view(h, w, d)
    cost.copy_(torch.from_numpy(v))
    disp = torch.empty((h, w), dtype=torch.int16, device="cuda")
    with Z.ZnccContext(w, h, d, 3) as ctx:
        ctx.wta_disparity(cost, disp, flag)
        torch.cuda.synchronize()
    assert np.array_equal(disp.cpu().numpy(), v.argmax(-1))
