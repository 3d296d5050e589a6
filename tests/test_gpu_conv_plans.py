"""The convolution and weight-gradient plans at the sizes where their tiles
end: x segments and row pairs, odd heights, one-voxel volumes, channel tiles
of every width, single and several K chunks, against the FP64 oracle.  The
operands are the same BF16 numbers on both sides, so only the FP32
accumulation differs: relative L2 1e-4 (its rounding, at most 27 * 256 sums of
2^-24 each, grows as their square root to about 5e-6), and every output
within 1e-3 of the largest (a voxel, tap or channel in the wrong place is off
by the outputs' own size)."""
import numpy as np
import pytest

from oracle import nn as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _need_gpu(libsoc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _bf(a):
    h = torch.from_numpy(np.asarray(a, np.float32)).to(torch.bfloat16)
    return h.cuda(), h.float().numpy().astype(np.float64)


def _close(got, ref):
    got = got.float().cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 1e-4 * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= 1e-3 * max(np.abs(ref).max(), 1.0)


# forward and input gradient: one and several K chunks of 16 or 32, one-plane
# volumes, the narrowest and widest rows of the slab kernel
@pytest.mark.parametrize("shape,cin,cout", [((7, 23, 16, 8), 16, 16), ((3, 52, 16, 16), 16, 48),
                                             ((160, 1, 16, 8), 16, 32), ((2, 20, 32, 64), 48, 16),
                                             ((1, 39, 16, 128), 32, 16), ((5, 8, 48, 32), 96, 32),
                                             ((4, 40, 16, 8), 64, 160), ((2, 5, 16, 64), 16, 256)])
def test_conv_slabs(libsoc, shape, cin, cout):
    rng = np.random.default_rng([cin, cout, shape[1]])
    x, x64 = _bf(rng.standard_normal(shape + (cin,)))
    w, w64 = _bf(rng.standard_normal((cout, 27, cin)) / np.sqrt(27 * cin))
    b = rng.standard_normal(cout).astype(np.float32)
    ref = O.conv3d(x64, w64, b.astype(np.float64))
    y = torch.full(shape + (cout,), 7.0, dtype=torch.float32, device="cuda")
    libsoc.conv3d(x, w, torch.from_numpy(b).cuda(), out_f32=y)
    _close(y, ref)
    y16 = torch.full(shape + (cout,), 7.0, dtype=torch.bfloat16, device="cuda")
    libsoc.conv3d(x, w, torch.from_numpy(b).cuda(), relu=True, out=y16)
    assert np.linalg.norm(y16.float().cpu().numpy() - np.maximum(ref, 0)) <= 1e-2 * np.linalg.norm(ref)
    gy, gy64 = _bf(rng.standard_normal(shape + (cout,)))
    gx = torch.full(shape + (cin,), 7.0, dtype=torch.float32, device="cuda")
    libsoc.conv3d_dgrad(gy, w, torch.empty(cout * 27 * cin, dtype=torch.bfloat16, device="cuda"), gx)
    _close(gx, O.conv3d_dgrad(gy64, w64))
    assert libsoc.nn_error_flag() == 0


# the plane-marching kernel: boxes that end in the middle of a row, of a group
# and of their planes, the narrowest and widest rows, fewer planes than a box
# may have, one to four K chunks of 16 or 32, channel tiles of 16, 48 and 80
@pytest.mark.parametrize("shape,cin,cout", [((2, 37, 40, 64), 16, 48), ((3, 50, 17, 16), 64, 32),
                                             ((1, 39, 24, 128), 48, 16), ((60, 5, 21, 8), 16, 96),
                                             ((4, 13, 70, 32), 32, 32), ((30, 3, 40, 32), 16, 16),
                                             ((90, 7, 16, 8), 32, 80)])
def test_conv_marches(libsoc, shape, cin, cout):
    test_conv_slabs(libsoc, shape, cin, cout)


# the per-tap kernel: two, three, four and many stages (as many producers, at
# most four), several boxes a block, one and several K chunks
@pytest.mark.parametrize("shape,cin,cout", [((2, 24, 24, 24), 64, 64), ((2, 24, 24, 24), 64, 128),
                                             ((1, 20, 12, 24), 64, 256), ((2, 13, 10, 27), 48, 32),
                                             ((3, 50, 21, 24), 16, 16), ((1, 2, 3, 5), 32, 16)])
def test_conv_taps(libsoc, shape, cin, cout):
    test_conv_slabs(libsoc, shape, cin, cout)


@pytest.mark.parametrize("shape,cin,cout", [((1, 1, 1, 1), 16, 16), ((2, 3, 5, 8), 16, 32), ((1, 4, 7, 9), 32, 16),
                                             ((1, 3, 9, 16), 64, 48), ((1, 2, 11, 17), 128, 16), ((2, 2, 3, 65), 16, 80),
                                             ((1, 3, 2, 130), 48, 32), ((3, 6, 6, 4), 256, 64), ((1, 20, 21, 33), 16, 16),
                                             ((1, 12, 40, 64), 48, 16)])
def test_weight_gradient_plans(libsoc, shape, cin, cout):
    rng = np.random.default_rng([cin, cout, shape[3]])
    x, x64 = _bf(rng.standard_normal(shape + (cin,)))
    gy, gy64 = _bf(rng.standard_normal(shape + (cout,)))
    gw = torch.ones((cout, 27, cin), dtype=torch.float32, device="cuda")       # accumulated into
    gb = torch.ones(cout, dtype=torch.float32, device="cuda")
    libsoc.conv3d_wgrad(gy, x, gw, gb)
    rw, rb = O.conv3d_wgrad(gy64, x64)
    _close(gw, rw + 1.0)
    _close(gb, rb + 1.0)
    again = torch.ones((cout, 27, cin), dtype=torch.float32, device="cuda")
    libsoc.conv3d_wgrad(gy, x, again, None)
    assert torch.equal(again, gw)                                              # fixed order of sums
    assert libsoc.nn_error_flag() == 0
