"""The convolution that walks along z: its plan's limits and an emulation of its stages, operands,
accumulator ring and epilogue on integers (CPU), and its results on a GPU."""
import ctypes

import numpy as np
import pytest

SHAPES = [((1, 1, 8), 16, 16), ((4, 5, 16), 32, 16), ((9, 3, 128), 16, 32), ((7, 6, 40), 16, 16), ((3, 17, 64), 16, 16),
          ((5, 4, 112), 32, 16), ((6, 2, 200), 16, 16), ((13, 9, 80), 16, 16), ((2, 9, 232), 16, 16),
          ((3, 5, 64), 48, 16), ((2, 3, 40), 80, 16)]
PLAN = "T TY mg adv ncols cps box_bytes stage_bytes ns nslice ry nblk".split()
RING = 5


def _plan(shape, cin, cout, sms, taps=27):
    from paper_2211_03516_gb300 import build
    build.build()
    from paper_2211_03516_gb300 import vamrt
    f = vamrt.lib().vamrt_conv3d_march_plan
    f.argtypes = [ctypes.c_int32] * 7 + [ctypes.c_void_p]
    out = (ctypes.c_int32 * 13)()
    assert f(*shape, cin, cout, taps, sms, ctypes.addressof(out)) == 0
    return dict(zip(PLAN, list(out)[1:])) if out[0] else None


def _direct(x, w):
    D, H, W, _ = x.shape
    xp = np.pad(x, ((1, 1), (1, 1), (1, 1), (0, 0)))
    return sum(xp[t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H, t % 3:t % 3 + W] @ w[:, t].T for t in range(27))


@pytest.mark.parametrize("sms", [152, 3])
@pytest.mark.parametrize("shape,cin,cout", SHAPES)
def test_emulated_on_integers(shape, cin, cout, sms):
    p = _plan(shape, cin, cout, sms)
    if p is None:
        return
    (D, H, W), nc = shape, cin // 16
    T, TY, mg, adv = p["T"], p["TY"], p["mg"], p["adv"]
    assert T * RING * 48 <= p["ncols"] <= 512 and p["nslice"] * p["nblk"] <= sms and p["nslice"] * 16 == cout
    sb = 32 * p["cps"]          # bytes of a slot: 16 channels of each of cps chunks
    assert (2 if p["cps"] > 1 else 3) <= p["ns"] <= 8 and nc * 27 * 512 + p["ns"] * p["stage_bytes"] <= 220 * 1024 and p["stage_bytes"] % 1024 == 0
    assert p["box_bytes"] == (TY + 2) * W * sb and TY + 2 <= 256 and adv % 8 == 0 and W % 8 == 0
    rng = np.random.default_rng(1)
    x, w = rng.integers(-4, 5, shape + (cin,)), rng.integers(-4, 5, (cout, 27, cin))
    y = np.zeros(shape + (cout,), np.int64)
    hits = np.zeros(shape + (p["nslice"],), int)
    tot = p["ry"] * D
    for block in range(p["nslice"] * p["nblk"]):
        sl, blk = block % p["nslice"], block // p["nslice"]
        l, l1, g = blk * tot // p["nblk"], (blk + 1) * tot // p["nblk"], 0
        acc = np.full((T, RING, 128, 48), 10 ** 9, np.int64)          # never read before it is overwritten
        while l < l1:
            col, z0 = l // D, l % D
            z1, y0 = min(D, z0 + l1 - l), col * TY
            for z in range(z0 - 1, z1 + 1):
                lo, hi = max(z - 1, z0), min(z + 1, z1 - 1)
                n, b0, s0, fresh = hi - lo + 1, lo - (z - 1), (g + lo - z0) % RING, z + 1 < z1
                for c in range(nc):
                    stage = np.full((p["stage_bytes"] // sb, 16), 777, np.int64)
                    box = np.zeros((TY + 2, W, 16), np.int64)
                    for r in range(TY + 2):
                        if 0 <= z < D and 0 <= y0 - 1 + r < H:
                            box[r] = x[z, y0 - 1 + r, :, 16 * c:16 * c + 16]
                    stage[8:8 + (TY + 2) * W] = box.reshape(-1, 16)
                    for dy in range(3):
                        B = np.stack([w[16 * sl + k % 16, (2 - k // 48) * 9 + dy * 3 + k // 16 % 3, 16 * c:16 * c + 16]
                                      for k in range(144)])
                        for t in range(T):
                            a0 = 8 + dy * W + adv * t - 8 * mg
                            assert a0 % 8 == 0 and 0 <= a0 and a0 + 128 <= stage.shape[0]
                            Dm = stage[a0:a0 + 128] @ B.T
                            apart = fresh and c == 0 and dy == 0
                            na = n - 1 if apart else n
                            n1 = min(n, RING - s0, na)
                            for k in range(na):
                                s = s0 + k if k < n1 else k - n1
                                acc[t, s] += Dm[:, 48 * (b0 + k):48 * (b0 + k) + 48]
                            if apart:
                                acc[t, (s0 + n - 1) % RING] = Dm[:, 48 * (b0 + n - 1):48 * (b0 + n)]
                if z - 1 >= z0:
                    for t in range(T):
                        A = acc[t, (g + z - 1 - z0) % RING]
                        for m in range(mg, mg + (adv if mg else 128)):
                            q = adv * t + m - 8 * mg
                            if q < 0 or q // W >= TY or y0 + q // W >= H:
                                continue
                            X = q % W
                            v = A[m, 16:32].copy()
                            if X > 0:
                                v += A[m - 1, :16]
                            if X < W - 1:
                                v += A[m + 1, 32:]
                            y[z - 1, y0 + q // W, X, 16 * sl:16 * sl + 16] = v
                            hits[z - 1, y0 + q // W, X, sl] += 1
            g += z1 - z0
            l += z1 - z0
    assert (hits == 1).all()
    np.testing.assert_array_equal(y, _direct(x, w))


@pytest.mark.gpu
@pytest.mark.parametrize("shape,cin,cout", SHAPES + [((40, 30, 128), 48, 16), ((33, 20, 64), 96, 32), ((30, 20, 96), 16, 48)])
def test_on_the_gpu(shape, cin, cout):
    """Integers of at most 4: every partial sum stays below 2^24, so FP32 results are exact."""
    import torch
    from paper_2211_03516_gb300 import unet as U
    rng = np.random.default_rng(2)
    x, w = rng.integers(-4, 5, shape + (cin,)), rng.integers(-4, 5, (cout, 27, cin))
    b = rng.integers(-9, 10, cout)
    dev = dict(device="cuda:0", dtype=torch.bfloat16)
    y = U.conv3d(torch.from_numpy(x).to(**dev), torch.from_numpy(w).to(**dev), torch.from_numpy(b).float().to("cuda:0"),
                 relu=True, out_dtype=torch.float32)
    U.check_errors()
    np.testing.assert_array_equal(y.cpu().numpy(), np.maximum(_direct(x, w) + b, 0).astype(np.float32))
