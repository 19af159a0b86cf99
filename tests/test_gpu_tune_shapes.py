"""The autotuner's last stage times each launch of the mixed flux once: on a mesh of four
waves of points or more shape 0 is the launch of shape 1, so one candidate is left
beside the handle's own, whichever that is; below, two."""
import pytest

from paper_1802_00704_gb300 import inputs as I
from tests.gpu_util import dev, needs_gpu, torch

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("shape", [0, 1, 2])
@pytest.mark.parametrize("large", [False, True])
def test_each_launch_is_timed_once(shape, large):
    from paper_1802_00704_gb300 import build, gks
    build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # 3 n^2 faces of two points on a periodic n x n mesh; four waves of 512 points per SM
    n = int((4 * 512 * sms / 6) ** 0.5) + (1 if large else -1)
    c = I.advection_case(n)
    assert (2 * c.mesh.n_face >= 4 * 512 * sms) == large
    m = gks.GksMesh(c.mesh, precision=gks.MIXED, basis_fp32=1, gmres_m=8, flux_shape=shape)
    r = m.autotune(dev(c.w0), trial_steps=1)
    # 54 solver candidates, no shorter restart
    assert r["n_failed"] == 0 and r["n_candidates"] == 54 + (1 if large else 2)
