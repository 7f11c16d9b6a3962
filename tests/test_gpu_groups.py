"""The grouped operators on scans of every group size against the FP64 oracle: quarter turns
(square grids), half turns, no partners, angle lists in any order, grids with nx != ny and odd
extents, bundles too wide for the shared-memory windows, volumes that are dense, or empty but
for a few voxels at the grid's corners and faces (stages that touch empty bricks only are
passed over).  Tolerance: 1e-5 relative L2, as for every FP32 operator."""
import numpy as np
import pytest
import torch

from oracle import vam_oracle as O
from paper_2211_03516_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = 1e-5
BASE = I.TINY.scaled(nx=35, ny=35, nz=41, voxel_mm=0.36, nu=37, nv=43, pixel_u_mm=0.38, pixel_v_mm=0.36, n_angles=144,
                     f_number=3.5, pupil_pattern="sunflower", rays_per_pixel=2, pupil_mm=60.0)
RNG = np.random.default_rng(5)
SHUFFLED = RNG.permutation(I.default_angles(148) + 0.1)
HALF = RNG.uniform(0.0, np.pi, 72)
PAIRED = np.concatenate([HALF, HALF + np.pi])
LOOSE = RNG.uniform(0.0, 2 * np.pi, 140)
# workload, angles (None: evenly spaced).  144 angles of 10 pixel tiles are enough for the grouped
# operators, the last four scans are not.
SCANS = {
    "quarter_turns": (BASE, None),
    "quarter_turns_shuffled": (BASE, SHUFFLED),
    "half_turns": (BASE.scaled(n_angles=142), None),
    "half_turns_listed": (BASE, PAIRED),
    "half_turns_oblong": (BASE.scaled(ny=38), None),
    "no_partners": (BASE.scaled(n_angles=141), None),
    "no_partners_listed_oblong": (BASE.scaled(nx=40), LOOSE),
    "coarse_steps": (BASE.scaled(step_vox=2.0), None),
    "wide_bundles": (BASE.scaled(f_number=1.1, pupil_mm=25.0, jitter_per_pixel=True), None),
    "wide_bundles_half_turns": (BASE.scaled(f_number=1.1, pupil_mm=25.0, jitter_per_pixel=True, ny=36), None),
    "few_quarter_turns": (BASE.scaled(n_angles=8), None),
    "few_no_partners": (BASE.scaled(n_angles=5, nx=40), None),
    "one_angle": (BASE.scaled(n_angles=1), None),
    "few_wide_bundles": (BASE.scaled(f_number=1.1, pupil_mm=25.0, jitter_per_pixel=True, n_angles=3), None),
}


def rel_l2(a, b):
    return float(np.linalg.norm(a.astype(np.float64) - b) / np.linalg.norm(b))


@pytest.fixture(scope="module")
def V():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2211_03516_gb300 import vamrt
    return vamrt


def volumes(w):
    dense = I.random_volume(w, seed=21) - 0.4
    few = np.zeros(w.vol_shape, np.float32)
    rng = np.random.default_rng(22)
    for z, y, x in ((0, w.ny // 2, w.nx // 2), (w.nz - 1, w.ny // 3, w.nx // 2), (w.nz // 2, w.ny // 2, 3),
                    (7, 4, w.nx // 2), (8, w.ny - 5, w.nx // 2), *rng.integers(6, 29, (4, 3))):
        few[z, y, x] = 1.0 + rng.random()
    return dense, few


@pytest.mark.parametrize("name", list(SCANS))
def test_projection_of_every_group_size(V, name):
    w, angles = SCANS[name]
    pupil = I.workload_pupil(w)
    P = V.Projector.from_workload(w, pupil, angles_rad=angles)
    for vol in volumes(w):
        y = P.adjoint(torch.from_numpy(vol).to("cuda:0")).cpu().numpy()
        assert rel_l2(y, O.adjoint(w, vol, pupil, angles=angles)) <= TOL
    assert float(P.adjoint(torch.zeros(w.vol_shape, device="cuda:0")).abs().max()) == 0.0


@pytest.mark.parametrize("name", list(SCANS))
def test_dose_of_every_group_size(V, name):
    """Projections of one sign and of both (two fixed-point conversions), dark angles, and a few
    lit pixels (angles of very different brightness within a group)."""
    w, angles = SCANS[name]
    pupil = I.workload_pupil(w)
    P = V.Projector.from_workload(w, pupil, angles_rad=angles)
    n = P.proj_shape[0]
    g = np.random.default_rng(23).random(P.proj_shape, dtype=np.float32)
    signed = g - 0.5
    signed[n // 2:, : w.nv // 2] = np.abs(signed[n // 2:, : w.nv // 2])
    few = np.zeros_like(g)
    few[np.arange(n), np.arange(n) * 5 % w.nv, np.arange(n) * 7 % w.nu] = 10.0 ** -(np.arange(n) % 5)
    few[0, w.nv // 2, 3:w.nu - 3] = 0.5
    for p in (g, signed, few):
        d = P.forward_dose(torch.from_numpy(p).to("cuda:0")).cpu().numpy()
        assert rel_l2(d, O.forward(w, p, pupil, angles=angles)) <= TOL
    assert float(P.forward_dose(torch.zeros(P.proj_shape, device="cuda:0")).abs().max()) == 0.0


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_dose_of_a_pixel_that_is_not_finite(V, bad):
    """Its rays' voxels are not finite, and only theirs; the rest of its block keeps its dose."""
    w = BASE
    pupil = I.workload_pupil(w)
    P = V.Projector.from_workload(w, pupil)
    g = torch.from_numpy(np.random.default_rng(24).random(P.proj_shape, dtype=np.float32)).to("cuda:0")
    one = torch.zeros_like(g)
    one[3, 20, 18] = 1.0
    touched = P.forward_dose(one) > 0
    # a corner of weight zero takes 0 x NaN = NaN: spare the touched voxels' neighbours
    away = torch.nn.functional.max_pool3d(touched[None].float(), 3, 1, 1)[0] == 0
    ref = P.forward_dose(g)
    g[3, 20, 18] = bad
    d = P.forward_dose(g)
    assert not torch.isfinite(d[touched]).any()
    assert torch.isfinite(d[away]).all()
    assert rel_l2(d[away].cpu().numpy(), ref[away].double().cpu().numpy()) <= TOL
