"""Projections whose dark pixels hold -0.0, or negative values that vanish when they are weighted:
the dose is that of +0.0.  (Non-negative shares become fixed point by their bit pattern, in which
-0.0 is the lowest integer.)  Tolerance: 1e-5 relative L2, as for every FP32 operator."""
import numpy as np
import pytest
import torch

from paper_2211_03516_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = 1e-5
BASE = I.TINY.scaled(nx=35, ny=35, nz=41, voxel_mm=0.36, nu=37, nv=43, pixel_u_mm=0.38, pixel_v_mm=0.36, n_angles=288,
                     f_number=3.5, pupil_pattern="sunflower", rays_per_pixel=2, pupil_mm=60.0)
SCANS = {"quarter_turns": BASE, "no_partners": BASE.scaled(n_angles=287), "few_angles": BASE.scaled(n_angles=8),
         "wide_bundles": BASE.scaled(f_number=1.1, pupil_mm=25.0, jitter_per_pixel=True)}


@pytest.fixture(scope="module")
def V():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2211_03516_gb300 import vamrt
    return vamrt


@pytest.mark.parametrize("dtype,dark", [(torch.float32, -0.0), (torch.bfloat16, -0.0), (torch.float16, -0.0),
                                        (torch.float32, -1.5e-45)])
@pytest.mark.parametrize("name", list(SCANS))
def test_dose_of_dark_pixels_below_zero(V, name, dtype, dark):
    w = SCANS[name]
    P = V.Projector.from_workload(w, I.workload_pupil(w))
    gen = torch.Generator(device="cuda:0").manual_seed(31)
    g = torch.rand(P.proj_shape, device="cuda:0", generator=gen)
    # a third of the pixels dark, and every fifth angle whole: lit ones beside them in a group
    off = torch.rand(P.proj_shape, device="cuda:0", generator=gen) < 1 / 3
    off[::5] = True
    ref = P.forward_dose(g.masked_fill(off, 0.0).to(dtype)).double()
    d = P.forward_dose(g.masked_fill(off, dark).to(dtype)).double()
    assert float(ref.norm()) > 0
    assert float((d - ref).norm()) <= TOL * float(ref.norm())
