"""The weight gradient that stages each tile of x once for all 27 taps: its plan's limits and an
emulation of its staging, operands and epilogue on integers (CPU), and its results on a GPU."""
import ctypes

import numpy as np
import pytest

SHAPES = [((1, 1, 16), 16, 16), ((3, 5, 32), 48, 16), ((2, 3, 48), 16, 48), ((9, 9, 32), 96, 32), ((7, 10, 64), 64, 64),
          ((6, 7, 80), 32, 96), ((5, 13, 16), 112, 16), ((17, 7, 32), 16, 32), ((19, 11, 32), 80, 16)]
PLAN = "TZ TY XB cg ngroups Ct nslices nt kp slots slot_bytes x_bytes ncols nsplit nx ny ntiles seg run".split()


def _plan(shape, cin, cout, sms, taps=27):
    from paper_2211_03516_gb300 import build
    build.build()
    from paper_2211_03516_gb300 import vamrt
    f = vamrt.lib().vamrt_conv3d_wgrad_halo_plan
    f.argtypes = [ctypes.c_int32] * 7 + [ctypes.c_void_p]
    out = (ctypes.c_int32 * 20)()
    assert f(*shape, cin, cout, taps, sms, ctypes.addressof(out)) == 0
    return dict(zip(PLAN, list(out)[1:])) if out[0] else None


def _direct(x, dy):
    D, H, W, cin = x.shape
    xp = np.pad(x, ((1, 1), (1, 1), (1, 1), (0, 0)))
    g = dy.reshape(-1, dy.shape[-1])
    return np.stack([g.T @ xp[t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H, t % 3:t % 3 + W].reshape(-1, cin)
                     for t in range(27)], 1)


def _box(a, c0, x0, y0, z0, n, chunk_last):
    """What a TMA box of 16 channels, n = (x, y, z, chunks) writes: slots [.][16], zeros outside."""
    nx, ny, nz, nch = n
    D, H, W, C = a.shape
    out = np.zeros((nz, nch, ny, nx, 16), a.dtype)
    for z in range(max(z0, 0), min(z0 + nz, D)):
        for k in range(min(nch, (C - c0) // 16)):
            for y in range(max(y0, 0), min(y0 + ny, H)):
                lo, hi = max(x0, 0), min(x0 + nx, W)
                out[z - z0, k, y - y0, lo - x0:hi - x0] = a[z, y, lo:hi, c0 + 16 * k:c0 + 16 * k + 16]
    return (out.swapaxes(0, 1) if chunk_last else out).reshape(-1, 16)


BIG = (184, 128, 128), 48, 16        # sums of 30176 positions: runs of positions, tiles of one plane


@pytest.mark.parametrize("sms", [152, 7])
@pytest.mark.parametrize("shape,cin,cout", SHAPES + [((2, 13, 128), 48, 16)])
def test_emulated_on_integers(shape, cin, cout, sms):
    p = _plan(shape, cin, cout, sms)
    if shape == (2, 13, 128):            # the tile of the large volume, on a few of its rows
        p = _plan(*BIG, sms)
        if p is None:
            return
        assert p["TZ"] == 1 and p["run"] > 16384
        cuts = [b * p["run"] * p["ntiles"] // np.prod(BIG[0]) for b in range(p["nsplit"])] + [p["ntiles"]]
        assert cuts[0] == 0 and all(a < b for a, b in zip(cuts, cuts[1:])) and p["seg"] >= p["ntiles"]
        p["ny"], p["nsplit"] = -(-13 // p["TY"]), 1
        p["ntiles"] = 2 * p["nx"] * p["ny"]
    if p is None:           # left to the kernel that stages a copy of x per tap
        assert np.prod(shape) < 100 * sms or cin * cout > 64 * sms
        return
    TZ, TY, XB, cg, Ct, kp, nt = (p[k] for k in "TZ TY XB cg Ct kp nt".split())
    N = 3 * Ct
    RY, nc, nb, yblk = TY + 2, cin // 16, p["Ct"] // 16, TZ * TY * XB
    xs = (TZ + 2) * RY * cg * XB
    assert p["x_bytes"] == 32 * xs and p["slot_bytes"] == 32 * (xs + 3 * nb * yblk)
    assert 2 <= p["slots"] <= 4 and p["slots"] * p["slot_bytes"] <= 220 * 1024 and p["x_bytes"] % 256 == 0
    assert p["slot_bytes"] % 256 == 0 and XB % 16 == 0 and max(XB, TZ + 2, cg, nb) <= 256
    assert nt * kp * N <= p["ncols"] <= 512 and (TY * XB // 16) % kp == 0 and N <= 256 and N % 16 == 0 and 8 * nt >= (3 * cg - 1) * RY + 3
    assert p["ngroups"] * p["nslices"] * p["nsplit"] <= sms and 1 <= p["nsplit"] <= p["ntiles"] and p["seg"] >= 1
    assert (p["ngroups"] - 1) * cg < nc <= p["ngroups"] * cg and p["nslices"] * Ct == cout
    rng = np.random.default_rng(1)
    x, dy = rng.integers(-4, 5, shape + (cin,)), rng.integers(-4, 5, shape + (cout,))
    dw = np.zeros((cout, 27, cin), np.int64)
    r16 = np.arange(16)
    for group in range(p["ngroups"]):
        chunk0, ncg = group * cg, min(cg, nc - group * cg)
        for sl in range(p["nslices"]):
            acc = np.zeros((nt, 128, N), np.int64)
            for tile in range(p["ntiles"]):
                tx, r = tile % p["nx"], tile // p["nx"]
                ty, tz = r % p["ny"], r // p["ny"]
                slot = [_box(x, 16 * chunk0, tx * XB, ty * TY - 1, tz * TZ - 1, (XB, RY, TZ + 2, cg), False)]
                for dx in (-1, 0, 1):
                    slot.append(_box(dy, sl * Ct, tx * XB - dx, ty * TY, tz * TZ, (XB, TY, TZ, nb), True))
                slot = np.concatenate(slot)
                assert slot.shape[0] * 32 == p["slot_bytes"]
                for m in range(nt):
                    for oz in range(TZ):
                        for i in range(TY * XB // 16):
                            a0 = (8 * m + oz * RY * cg) * XB + 16 * i
                            b0 = xs + oz * TY * XB + 16 * i
                            A = slot[a0 + r16[:, None] + XB * np.arange(8)[None, :]].reshape(16, 128)
                            B = slot[b0 + r16[:, None] + yblk * np.arange(3 * nb)[None, :]].reshape(16, N)
                            acc[m] += A.T @ B
            for row in range(nt * 128):
                s = row // 16
                dyy, ch, dz = s % RY, s // RY % cg, s // RY // cg
                if dyy < 3 and dz < 3 and ch < ncg:
                    for n in range(N):
                        dw[sl * Ct + n % Ct, dz * 9 + dyy * 3 + n // Ct, 16 * (chunk0 + ch) + row % 16] += \
                            acc[row // 128, row % 128, n]
    np.testing.assert_array_equal(dw, _direct(x, dy))


@pytest.mark.gpu
@pytest.mark.parametrize("shape,cin,cout", SHAPES + [((40, 66, 128), 48, 16), ((30, 33, 112), 16, 32), ((23, 16, 16), 128, 128)])
def test_on_the_gpu(shape, cin, cout):
    """Integers of at most 4: every partial sum stays below 2^24, so FP32 sums are exact."""
    import torch
    from paper_2211_03516_gb300 import unet as U
    rng = np.random.default_rng(2)
    x, dy = rng.integers(-4, 5, shape + (cin,)), rng.integers(-4, 5, shape + (cout,))
    dw = torch.zeros((cout, 27, cin), device="cuda:0")
    U.conv3d_wgrad(torch.from_numpy(x).to("cuda:0", torch.bfloat16), torch.from_numpy(dy).to("cuda:0", torch.bfloat16),
                   dw, 27)
    U.check_errors()
    np.testing.assert_array_equal(dw.cpu().numpy(), _direct(x, dy).astype(np.float32))


@pytest.mark.gpu
def test_large_volume_on_the_gpu():
    """Runs of positions; sums of three million products of integers within 2, exact in FP32."""
    import torch
    from paper_2211_03516_gb300 import unet as U
    (D, H, W), cin, cout = BIG
    gen = torch.Generator(device="cuda:0").manual_seed(3)
    x = torch.randint(-2, 3, (D, H, W, cin), device="cuda:0", generator=gen).to(torch.bfloat16)
    dy = torch.randint(-2, 3, (D, H, W, cout), device="cuda:0", generator=gen).to(torch.bfloat16)
    dw = torch.zeros((cout, 27, cin), device="cuda:0")
    U.conv3d_wgrad(x, dy, dw, 27)
    U.check_errors()
    xp, g = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1)).double(), dy.reshape(-1, cout).double()
    for t in range(27):
        ref = g.T @ xp[t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H, t % 3:t % 3 + W].reshape(-1, cin)
        assert torch.equal(dw[:, t].double(), ref), t
