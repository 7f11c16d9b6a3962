"""Which scans the operators take in groups of angles, by the host-only query (no GPU): partners,
sizes on both sides of the limits, samples for the volume's size, and the memory that the rotated
copies may take."""
import pytest

from paper_2211_03516_gb300 import inputs as I

PLENTY = 1 << 40
BASE = I.TINY.scaled(nx=35, ny=35, nz=41, voxel_mm=0.36, nu=37, nv=43, pixel_u_mm=0.38, pixel_v_mm=0.36, n_angles=144,
                     f_number=3.5, pupil_pattern="sunflower", rays_per_pixel=2, pupil_mm=60.0)     # 10 pixel tiles


def _plan(w, sms=152, free=PLENTY, angles=None, samples=PLENTY):
    from paper_2211_03516_gb300 import build
    build.build()
    from paper_2211_03516_gb300 import vamrt
    return vamrt.group_plan(vamrt.GeometrySpec.from_workload(w, I.workload_pupil(w), angles), sms, samples, free)


@pytest.mark.parametrize("kw,want", [
    (dict(), (4, 4)), (dict(n_angles=142), (2, 1)), (dict(n_angles=141), (1, 1)), (dict(ny=38), (2, 1)),
    (dict(n_angles=140), (4, 4)), (dict(n_angles=136), (4, 1)),      # 1400 and 1360 tiles: three waves are 1368
    (dict(n_angles=48), (4, 1)), (dict(n_angles=44), (1, 1)),        # 480 and 440 tiles: one wave is 456
    (dict(nz=8192), (4, 4)), (dict(nz=8193), (1, 1))])
def test_scans(kw, want):
    assert _plan(BASE.scaled(**kw))[:2] == want


def test_more_sms_need_larger_scans():
    assert _plan(BASE, sms=160)[:2] == (4, 1) and _plan(BASE, sms=480)[:2] == (1, 1)


def test_angle_lists():
    even = I.default_angles(144)
    assert _plan(BASE, angles=even[::-1] + 0.3)[:2] == (4, 4)
    assert _plan(BASE, angles=even ** 1.01)[:2] == (1, 1)


def test_few_samples_for_the_volume():
    voxels = 35 * 35 * 41
    assert _plan(BASE, samples=5 * voxels)[:2] == (1, 1) and _plan(BASE, samples=5 * voxels + 1)[:2] == (4, 4)
    half, voxels = BASE.scaled(ny=38), 35 * 38 * 41
    assert _plan(half, samples=10 * voxels)[:2] == (1, 1) and _plan(half, samples=10 * voxels + 1)[:2] == (2, 1)


def test_copies_leave_as_much_memory_free():
    bytes_ = _plan(BASE)[2]
    assert 16 * 37 * 37 * 44 < bytes_ < 16 * 37 * 37 * 44 + (1 << 20)
    assert _plan(BASE, free=2 * bytes_) == (4, 4, bytes_)
    assert _plan(BASE, free=2 * bytes_ - 1) == (1, 1, 0)
    assert _plan(BASE, free=0) == (1, 1, 0)


def test_bad_arguments():
    from paper_2211_03516_gb300 import vamrt
    with pytest.raises(vamrt.VamrtError, match="sms"):
        _plan(BASE, sms=0)
    with pytest.raises(vamrt.VamrtError, match="n_angles"):
        _plan(BASE.scaled(n_angles=65536))
