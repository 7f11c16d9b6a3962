"""The weight gradient of x and dy with values that are not finite: the sum over the output voxels of the
volume, with zero padding, whichever kernel takes the layer.  A voxel of x reaches the taps that meet
it inside the volume and no others; one of dy meets the padding too (0 x NaN = NaN).  All other sums
are of small integers, exact in FP32."""
import numpy as np
import pytest

from test_wgrad_halo import _plan

pytestmark = pytest.mark.gpu

# shape, channels, whether the kernel that stages x once takes it: one and several tiles along x, tiles
# that reach past the last row or plane, several chunk groups and slices, segments, and the other kernel
SHAPES = [((1, 1, 16), 16, 16, True), ((3, 5, 32), 48, 16, True), ((9, 9, 32), 96, 32, True), ((6, 7, 80), 32, 96, True),
          ((5, 13, 16), 112, 16, True), ((19, 11, 32), 80, 16, True), ((30, 33, 112), 16, 32, True),
          ((7, 10, 64), 64, 64, False), ((23, 16, 16), 64, 128, False), ((11, 6, 48), 192, 64, False),
          ((5, 13, 16), 64, 64, False)]          # its last stage reaches past the volume
BAD = (np.nan, np.inf, -np.inf)


def _direct(x, dy):
    D, H, W, cin = x.shape
    xp = np.pad(x, ((1, 1), (1, 1), (1, 1), (0, 0)))
    g = dy.reshape(-1, dy.shape[-1])
    with np.errstate(invalid="ignore"):
        return np.stack([np.einsum("pk,pc->kc", g, xp[t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H,
                                                      t % 3:t % 3 + W].reshape(-1, cin)) for t in range(27)], 1)


def _check(x, dy):
    import torch
    from paper_2211_03516_gb300 import unet as U
    dw = torch.zeros((dy.shape[-1], 27, x.shape[-1]), device="cuda:0")
    U.conv3d_wgrad(torch.from_numpy(x).to("cuda:0", torch.bfloat16), torch.from_numpy(dy).to("cuda:0", torch.bfloat16),
                   dw, 27)
    U.check_errors()
    np.testing.assert_array_equal(dw.cpu().numpy(), _direct(x, dy).astype(np.float32))


@pytest.mark.parametrize("shape,cin,cout,once", SHAPES)
def test_single_voxels(shape, cin, cout, once):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert (_plan(shape, cin, cout, sms) is not None) == once
    D, H, W = shape
    rng = np.random.default_rng(4)
    x, dy = rng.integers(-4, 5, shape + (cin,)).astype(np.float64), rng.integers(1, 5, shape + (cout,)) * 1.0
    # a channel each: corners, edges, faces, the inside, the last voxel of one tile and the first of the next
    where = [(0, 0, 0), (D - 1, H - 1, W - 1), (0, H - 1, 0), (D - 1, 0, W - 1), (D // 2, H // 2, 0), (D // 2, H // 2, W - 1),
             (D // 2, H - 1, W // 2), (D - 1, H // 2, W // 2), (0, H // 2, W // 2), (D // 2, 0, W // 2),
             (D // 2, H // 2, W // 2), (D // 3, H // 3, 15), (D // 3, H // 3, 16 % W)]
    some = x.copy()
    for k, (q, c) in enumerate(zip(where, rng.permutation(cin))):
        some[q + (c,)] = BAD[k % 3]
    _check(some, dy)
    some = dy.copy()
    for k, (p, c) in enumerate(zip(where, rng.permutation(cout))):
        some[p + (c,)] = BAD[k % 3]
    _check(x, some)


def test_whole_faces():
    """Every channel of a face, and of its opposite."""
    shape, cin, cout = (5, 13, 16), 112, 16
    rng = np.random.default_rng(5)
    dy = rng.integers(1, 5, shape + (cout,)) * 1.0
    for face in ((slice(None), slice(None), 0), (slice(None), slice(None), -1), (slice(None), -1), (-1,)):
        x = rng.integers(-4, 5, shape + (cin,)).astype(np.float64)
        x[face] = np.inf
        _check(x, dy)


def test_long_runs_of_positions():
    """One voxel on a face of the large volume: the sums that it leaves finite are summed again."""
    import torch
    from paper_2211_03516_gb300 import unet as U
    D, H, W, cin, cout = 184, 128, 128, 48, 16
    gen = torch.Generator(device="cuda:0").manual_seed(6)
    x = torch.randint(-2, 3, (D, H, W, cin), device="cuda:0", generator=gen).to(torch.bfloat16)
    dy = torch.randint(1, 3, (D, H, W, cout), device="cuda:0", generator=gen).to(torch.bfloat16)
    x[90, 64, 0, 7] = float("inf")
    dw = torch.zeros((cout, 27, cin), device="cuda:0")
    U.conv3d_wgrad(x, dy, dw, 27)
    U.check_errors()
    x[90, 64, 0, 7] = 0
    xp, g = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1)).double(), dy.reshape(-1, cout).double()
    for t in range(27):
        ref = g.T @ xp[t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H, t % 3:t % 3 + W].reshape(-1, cin)
        if t % 3 != 2:          # dx = 1 meets column 0 from outside only
            ref[:, 7] = float("inf")
        assert torch.equal(dw[:, t].double(), ref), t
