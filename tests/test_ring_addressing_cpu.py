"""CPU emulation of the grouped operators' windows (paper_2211_03516_gb300/csrc/ring.cuh).

For sampled pixel tiles the kernels' integer and FP32 steps of `bundle` and `corner` are
repeated on ray tables from the FP64 oracle's trace: the quarter turn, the rows, the window
that follows the bundle, the ring.  Checked for the kernels' alignments and
capacities at every group size: each sample's 8 corners lie in the rows and the window of its
stage, two stages fit the ring, and every cell lies inside the turned padded grid.  Needs no GPU.
"""
import math
import os
import re

import numpy as np
import pytest

from oracle import vam_oracle as O
from paper_2211_03516_gb300 import inputs as I

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2211_03516_gb300", "csrc")
SRC = "".join(open(os.path.join(CSRC, f)).read() for f in ("ring.cuh", "ring_project.cu", "ring_dose.cu"))
f32 = np.float32


def const(name):
    m = re.search(r"\b%s = ([0-9 *]+)[,;]" % name, SRC)
    assert m, name
    return int(eval(m.group(1)))


TU, TV = const("kProjTU"), const("kRingTV")
MAX_EX, MAX_EZ, MIN_EX, STEP_EZ, TAB = (const(n) for n in ("kMaxEX", "kMaxEZ", "kMinEX", "kStepEZ", "kRowTab"))
WORDS = [int(eval(x)) for x in re.search(r"kProjWords = S == 4 \? ([0-9 *]+) : ([0-9 *]+);", SRC).groups()]
DOSE_WORDS = const("kDoseWords")
# (alignment of z, granularity of EX, voxels of the ring, two buffers): projection of 4 and 2
# angles, dose of 4
FORMS = [(4 // S, 4 // S, WORDS[S != 4] // S, True) for S in (4, 2)] + [(4, 1, DOSE_WORDS // 4, False)]
assert const("kDoseTU") == TU and 3 * ((TAB - 3) // 2) + 1 < const("kDoseTab")


def q32(x):
    return np.rint(np.asarray(x) * 4294967296.0).astype(np.int64)


def table(w, pupil, u0, v0, a):
    """Entry points, directions, steps (voxels) and sample ranges of a tile's active rays."""
    out = []
    for u in range(u0, min(u0 + TU, w.nu)):
        for v in range(v0, min(v0 + TV, w.nv)):
            r = O.trace(w, pupil, u, v, a)
            if r["status"] != 2:
                continue
            K = int(r["k"])
            delta = r["ell"] / K
            j = np.arange(K)
            qz = (r["e"][2] + (j + 0.5) * delta * r["d2"][2]) / w.voxel_mm + 0.5 * (w.nz - 1)
            ins = np.nonzero((qz > -1.0) & (qz < w.nz))[0]
            if ins.size:
                out.append((*(np.asarray(r["e"]) / w.voxel_mm), *r["d2"], delta / w.voxel_mm, ins[0], ins[-1] + 1))
    return np.array(out, dtype=np.float64).reshape(-1, 9)


def place(w, T, theta):
    """Turned rays in padded Q32.32: turn, positions of sample jlo, steps, sample counts."""
    c, s = math.cos(theta), math.sin(theta)
    ex, ey, ez, bx, by, bz, dl = T[:, :7].T
    jlo, jhi = T[:, 7].astype(np.int64), T[:, 8].astype(np.int64)
    st = np.stack([(c * bx - s * by) * dl, (s * bx + c * by) * dl, bz * dl])
    q = q32(np.stack([c * ex - s * ey, s * ex + c * ey, 0.5 * (w.nz - 1) + 1.0 + ez]) + 0.5 * st)
    S = q32(st)
    top = (w.nz + 1) << 32
    for _ in range(4):
        z = q[2] + jlo * S[2]
        jlo = jlo + ((jlo < jhi) & ~((z >= 0) & (z < top)))
        z = q[2] + (jhi - 1) * S[2]
        jhi = jhi - ((jlo < jhi) & ~((z >= 0) & (z < top)))
    live = jlo < jhi
    q, S, jlo, jhi = q[:, live], S[:, live], jlo[live], jhi[live]
    dx, dy = int((S[0] >> 16).sum()), int((S[1] >> 16).sum())
    r = (0 if dy > 0 else 2) if abs(dy) >= abs(dx) else (1 if dx < 0 else 3)
    if r & 1:
        q[0], q[1] = q[1].copy(), -q[0]
        S[0], S[1] = S[1].copy(), -S[0]
    if r & 2:
        q[:2], S[:2] = -q[:2], -S[:2]
    nx, ny = (w.ny, w.nx) if r & 1 else (w.nx, w.ny)
    q[0] += q32(0.5 * (nx - 1) + 1.0)
    q[1] += q32(0.5 * (ny - 1) + 1.0)
    return r, (nx, ny), q + jlo * S, S, jhi - jlo


def window(q, S, n, align, exq, cap, split):
    """The kernels' Window, or None where the bundle is walked on global memory."""
    if (4 * S[1] < np.maximum(abs(S[0]), abs(S[2]))).any() or (S[1] <= 0).any():
        return None
    y0, y1 = int((q[1] >> 32).min()), int(((q[1] + (n - 1) * S[1]) >> 32).max()) + 1
    inv = f32(1.0) / S[1].astype(f32)
    ends = []
    for d in (0, 2):
        g = S[d].astype(f32) * inv
        for y in (y0, y1):
            t = ((y << 32) - q[1]).astype(f32) * f32(256.0 / 4294967296.0)
            a = (q[d] >> 24) + np.floor(t * g).astype(np.int64)
            ends.append((int(a.min()) - 4, int(a.max()) + 6))
    k, inv_n = f32(1.0 / 256.0), f32(1.0) / f32(y1 - y0)
    W = dict(y0=y0, y1=y1)
    width = []
    for name, (a, b) in (("x", ends[:2]), ("z", ends[2:])):
        W["l" + name] = f32(a[0]) * k
        W["ls" + name] = f32(b[0] - a[0]) * k * inv_n
        us = f32(b[1] - a[1]) * k * inv_n
        width.append(f32(max(a[1] - a[0], b[1] - b[0])) * k + abs(W["ls" + name]) + abs(us))
    if not (width[0] < MAX_EX and width[1] < MAX_EZ):
        return None
    W["EX"] = -(-max(int(math.floor(width[0] + f32(0.01))) + 3, MIN_EX) // exq) * exq
    W["EZ"] = -(-(int(math.floor(width[1] + f32(0.01))) + 3 + align - 1) // STEP_EZ) * STEP_EZ
    if W["EX"] > MAX_EX or W["EZ"] > MAX_EZ:
        return None
    rows = min(cap // (W["EX"] * W["EZ"]), TAB - 2)
    W["R"] = (rows >> 1) - 1 if split else (rows - 1) >> 1
    if W["R"] < 1:
        return None
    # two buffers of R + 1 rows, or a ring of 2 R + 1: a stage's rows and the next's
    assert (2 * W["R"] + (2 if split else 1)) * W["EX"] * W["EZ"] <= cap and 2 * W["R"] + 1 < TAB
    return W


def corner(W, y, align):
    t = (y - W["y0"]).astype(f32)

    def low(l, ls):
        m = (t.astype(np.float64) * np.float64(ls) + np.float64(l)).astype(f32)      # one rounding
        return np.floor(m - abs(ls)).astype(np.int64)

    return low(W["lx"], W["lsx"]), low(W["lz"], W["lsz"]) & ~(align - 1)


def check_block(w, T, theta):
    """(samples walked in the ring, all samples) of one tile, summed over the forms."""
    r, (nx, ny), q, S, n = place(w, T, theta)
    if n.size == 0:
        return 0, 0
    j = np.concatenate([np.arange(k) for k in n])
    ray = np.repeat(np.arange(n.size), n)
    cell = (q[:, ray] + j * S[:, ray]) >> 32
    for d, e in enumerate((nx, ny, w.nz)):
        assert cell[d].min() >= 0 and cell[d].max() + 1 <= e + 1        # turned padded grid
    boxed = 0
    for align, exq, cap, split in FORMS:
        W = window(q, S, n, align, exq, cap, split)
        if W is None:
            continue
        boxed += j.size
        assert cell[1].min() >= W["y0"] and cell[1].max() + 1 <= W["y1"]
        stage = (cell[1] - W["y0"]) // W["R"]
        assert (cell[1] + 1 <= W["y0"] + (stage + 1) * W["R"]).all()
        for dy in (0, 1):
            xo, zo = corner(W, cell[1] + dy, align)
            assert (cell[0] >= xo).all() and (cell[0] + 1 < xo + W["EX"]).all()
            assert (cell[2] >= zo).all() and (cell[2] + 1 < zo + W["EZ"]).all()
    return boxed, j.size * len(FORMS)


LARGE = I.WORKLOADS["large_768x768x1024_1000ang_4rays"]
RAGGED = I.TINY.scaled(nx=35, ny=34, nz=23, voxel_mm=0.4, nu=37, nv=23, pixel_u_mm=0.38, pixel_v_mm=0.41, n_angles=10,
                       f_number=3.5, pupil_pattern="sunflower", rays_per_pixel=4, pupil_mm=60.0)
# workload, tiles per workload, least fraction of samples walked in the ring
CASES = {
    "tiny": (I.TINY, 16, 1.0),
    "ragged": (RAGGED, 10, 0.9),
    "lens_train": (RAGGED.scaled(lens=I.telecentric_relay(), pupil_pattern="hex13", rays_per_pixel=13), 6, 0.9),
    "wide_stop": (RAGGED.scaled(jitter_per_pixel=True, f_number=1.2), 6, 0.0),
    "coarse_step": (RAGGED.scaled(step_vox=3.0), 6, 0.9),
    "fins18": (I.fins_workload(18), 6, 0.99),
    "mid_256cube_stratified_per_pixel": (I.MID, 6, 0.95),
    "tall_384x384x512": (I.WORKLOADS["tall_384x384x512_720ang_8rays"], 6, 0.99),
    "large_768x768x1024": (LARGE, 8, 0.99),
}


@pytest.mark.parametrize("name", list(CASES))
def test_ring_windows_hold_every_sample(name):
    w, n_tiles, least = CASES[name]
    rng = np.random.default_rng(7)
    pupil = I.workload_pupil(w)
    nut, nvt = -(-w.nu // TU), -(-w.nv // TV)
    tiles = [(0, 0), (nut - 1, nvt - 1), (nut // 2, nvt // 2), (nut // 4, 0)]
    tiles += [(int(rng.integers(nut)), int(rng.integers(nvt))) for _ in range(n_tiles - 4)]
    boxed = total = 0
    for tu, tv in tiles:
        T = table(w, pupil, tu * TU, tv * TV, int(rng.integers(w.rays_per_pixel)))
        if len(T):
            for theta in (0.0, math.pi / 4, float(rng.uniform(0, 2 * math.pi)), float(rng.uniform(0, 2 * math.pi))):
                b, n = check_block(w, T, theta)
                boxed, total = boxed + b, total + n
    assert total > 0 and boxed >= least * total, (boxed, total)
