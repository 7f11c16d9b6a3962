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
BASE = I.TINY.scaled(nx=35, ny=35, nz=41, voxel_mm=0.36, nu=37, nv=43, pixel_u_mm=0.38, pixel_v_mm=0.36, n_angles=8,
                     f_number=3.5, pupil_pattern="sunflower", rays_per_pixel=3, pupil_mm=60.0)
SHUFFLED = np.random.default_rng(5).permutation(I.default_angles(12) + 0.1)
PAIRED = np.concatenate([[0.3, 1.1], np.array([0.3, 1.1]) + np.pi])
LOOSE = np.array([0.3, 1.1, 0.3 + np.pi / 2, 2.0])
# workload, angles (None: evenly spaced)
SCANS = {
    "quarter_turns": (BASE, None),
    "quarter_turns_shuffled": (BASE, SHUFFLED),
    "half_turns": (BASE.scaled(n_angles=6), None),
    "half_turns_listed": (BASE, PAIRED),
    "half_turns_oblong": (BASE.scaled(ny=38), None),
    "no_partners": (BASE.scaled(n_angles=5), None),
    "no_partners_listed_oblong": (BASE.scaled(nx=40), LOOSE),
    "one_angle": (BASE.scaled(n_angles=1), None),
    "coarse_steps": (BASE.scaled(step_vox=2.0), None),
    "wide_bundles": (BASE.scaled(f_number=1.1, pupil_mm=25.0, jitter_per_pixel=True), None),
    "wide_bundles_no_partners": (BASE.scaled(f_number=1.1, pupil_mm=25.0, jitter_per_pixel=True, n_angles=3), None),
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
