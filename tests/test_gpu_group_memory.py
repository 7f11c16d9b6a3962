"""A projector made while memory is short: the operators' four rotated copies of the volume are left
out and every call works one angle at a time.  Tolerance: 1e-5 relative L2 per FP32 operator."""
import pytest
import torch

from paper_2211_03516_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def V():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2211_03516_gb300 import vamrt
    return vamrt


def test_a_handle_made_while_memory_is_short(V):
    """It works one angle at a time, with the same results; one made with memory to spare groups."""
    w = I.TINY.scaled(nx=480, ny=480, nz=600, voxel_mm=0.05, nu=96, nv=96, pixel_u_mm=0.2, pixel_v_mm=0.27, r_inner_mm=11.8,
                      n_angles=180)
    pupil = I.workload_pupil(w)
    gen = torch.Generator(device="cuda:0").manual_seed(55)
    f = torch.rand(w.vol_shape, device="cuda:0", generator=gen)
    bytes_ = V.group_plan(V.GeometrySpec.from_workload(w, pupil), 152, 1 << 40, 1 << 40)[2]
    y = torch.empty((180, 96, 96), device="cuda:0")
    d = torch.empty(w.vol_shape, device="cuda:0")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    # one and a half times the copies stay free: enough for them, and for the rest of the handle
    spare = torch.cuda.mem_get_info()[0] - bytes_ * 3 // 2
    try:
        hold = torch.empty(spare, device="cuda:0", dtype=torch.uint8)
    except torch.OutOfMemoryError:
        pytest.skip("the device's free memory cannot be held in one piece")
    try:
        P = V.Projector.from_workload(w, pupil)
        assert P.groups() == (1, 1)
        P.adjoint(f, out=y)
        P.forward_dose(y, out=d)
        torch.cuda.synchronize()
    finally:
        del hold
        torch.cuda.empty_cache()
    Q = V.Projector.from_workload(w, pupil)
    assert Q.groups() == (4, 4)
    assert Q.info()["scratch_bytes"] - P.info()["scratch_bytes"] == bytes_
    y2 = Q.adjoint(f)
    assert float((y2 - y).double().norm()) <= TOL * float(y2.double().norm())
    d2 = Q.forward_dose(y2)
    assert float((d2 - d).double().norm()) <= 2 * TOL * float(d2.double().norm())
