"""That the grouped operators run where they should: the path of every scan of test_gpu_groups.py, a
scan well above the limits against the oracle, accumulation in every storage type, and a voxel that
is not finite.  Tolerances: 1e-5 relative L2 for FP32 results; for 16-bit ones half a unit in the
last place of each value on top."""
import numpy as np
import pytest
import torch

from oracle import vam_oracle as O
from paper_2211_03516_gb300 import inputs as I
from test_gpu_groups import BASE, SCANS, rel_l2

pytestmark = pytest.mark.gpu

TOL = 1e-5
MANY = BASE.scaled(n_angles=288)
PATHS = {"quarter_turns": (4, 4), "quarter_turns_shuffled": (4, 4), "half_turns": (2, 1), "half_turns_listed": (2, 1),
         "half_turns_oblong": (2, 1), "no_partners": (1, 1), "no_partners_listed_oblong": (1, 1), "coarse_steps": (4, 4),
         "wide_bundles": (4, 4), "wide_bundles_half_turns": (2, 1), "few_quarter_turns": (1, 1),
         "few_no_partners": (1, 1), "one_angle": (1, 1), "few_wide_bundles": (1, 1)}


@pytest.fixture(scope="module")
def V():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2211_03516_gb300 import vamrt
    return vamrt


def test_every_scan_takes_its_path(V):
    assert set(PATHS) == set(SCANS)
    for name, (w, angles) in SCANS.items():
        assert V.Projector.from_workload(w, I.workload_pupil(w), angles_rad=angles).groups() == PATHS[name], name


@pytest.mark.parametrize("nu,n_angles,want", [(32, 720, (4, 4)), (16, 480, (1, 1)), (32, 722, (2, 1)), (16, 722, (1, 1))])
def test_small_pixel_arrays_over_a_large_grid(V, nu, n_angles, want):
    """About 22, 3.6, 22 and 5.5 samples per voxel: below 5 (groups of four) or 10 (of two) the copies of the
    volume cost more than groups save."""
    w = I.TINY.scaled(nx=256, ny=256, nz=256, voxel_mm=0.1, nu=nu, nv=nu, pixel_u_mm=0.4, pixel_v_mm=0.4, r_inner_mm=12.5,
                      n_angles=n_angles)
    P = V.Projector.from_workload(w, I.workload_pupil(w))
    assert P.groups() == want, P.sample_count() / 256 ** 3


def test_a_scan_above_the_limits(V):
    pupil = I.workload_pupil(MANY)
    P = V.Projector.from_workload(MANY, pupil)
    assert P.groups() == (4, 4)
    vol = I.random_volume(MANY, seed=51) - 0.4
    y = P.adjoint(torch.from_numpy(vol).to("cuda:0")).cpu().numpy()
    assert rel_l2(y, O.adjoint(MANY, vol, pupil)) <= TOL
    g = np.random.default_rng(52).random(P.proj_shape, dtype=np.float32) - 0.2
    d = P.forward_dose(torch.from_numpy(g).to("cuda:0")).cpu().numpy()
    assert rel_l2(d, O.forward(MANY, g, pupil)) <= TOL


@pytest.mark.parametrize("dtype,half_ulp", [(torch.float32, 2.0 ** -24), (torch.bfloat16, 2.0 ** -9), (torch.float16, 2.0 ** -12)])
def test_accumulation(V, dtype, half_ulp):
    """Added to what the output holds, rounded to its type once."""
    P = V.Projector.from_workload(MANY, I.workload_pupil(MANY))
    assert P.groups() == (4, 4)
    gen = torch.Generator(device="cuda:0").manual_seed(53)
    g = torch.rand(P.proj_shape, device="cuda:0", generator=gen) / 64
    f = torch.rand(P.vol_shape, device="cuda:0", generator=gen) / 64
    for op, x, shape in ((P.forward_dose, g, P.vol_shape), (P.adjoint, f, P.proj_shape)):
        start = torch.rand(shape, device="cuda:0", generator=gen).to(dtype)
        ref = start.double() + op(x).double()
        out = op(x, out=start.clone(), accumulate=True).double()
        assert float((out - ref).norm()) <= (2 * half_ulp + TOL) * float(ref.norm())
        assert bool(((out - ref).abs() <= 2 * half_ulp * ref.abs() + TOL * float(ref.max())).all())


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_projection_of_a_voxel_that_is_not_finite(V, bad):
    """The pixels whose rays see it are not finite, and only they."""
    P = V.Projector.from_workload(MANY, I.workload_pupil(MANY))
    assert P.groups() == (4, 4)
    f = torch.from_numpy(I.random_volume(MANY, seed=54)).to("cuda:0")
    one = torch.zeros_like(f)
    one[20, 17, 12] = 1.0
    seen = P.adjoint(one) > 0
    # a corner of weight zero takes 0 x NaN = NaN: spare the seeing pixels' neighbours
    away = torch.nn.functional.max_pool2d(seen[:, None].float(), 5, 1, 2)[:, 0] == 0
    ref = P.adjoint(f)
    f[20, 17, 12] = bad
    y = P.adjoint(f)
    assert not torch.isfinite(y[seen]).any()
    assert torch.equal(y[away], ref[away])
