"""Controller limits at the ends of their ranges in the kernel with several zones per
thread group, bit for bit against the group kernel (the comparison of test_gpu_slots)."""
import numpy as np
import pytest

from kn_inputs import Zones, custom_network
from test_gpu_slots import _both, env  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("frac", [1e-50, 1e-46, 1e-40, 0.0])
def test_smallest_step_fractions(env, frac):  # noqa: F811
    """dt_min_frac below the FP32 range at a late time: the limit frac t is still a step
    that FP32 holds, and an attempt rejected at or below it ends the zone at once.  One
    fast decay, k h = 2e-5 above eps_r, from t = 1e10 s with a step of 2e-42 s."""
    net = custom_network([1.0, 1.0], [((0,), (1,))], [np.log(1e37)], [0.0])
    n = 5
    z = Zones(Y0=np.full((n, 2), 0.5), T0=np.ones(n), rho0=np.ones(n), tau=np.zeros(n), t_start=np.full(n, 1e10),
              t_end=np.full(n, 2e10), dt_trial=np.full(n, 2e-42))
    r = _both(env, net, z, 32, eps_r=1e-6, eps_c=1.0, dt_min_frac=frac)
    if frac == 1e-50:
        assert (r["status"] == 2).all() and (r["rejects"] == 1).all()
