"""dH of FP32 trajectories with step coefficients that FP32 cannot hold (1/48,
1/12, 0.1932/8, beta / 6 = 5.9 / 6): rounded to FP32 they would scale every
kick or drift by up to 1 + 2^-24, and dH would be off by that part of what the
action gains over the trajectory, which is large from a hot start.

Allowed: 2^-27 of that gain, and 16 random roundings of the 32 V components
(2^-25 each) of forces near 1."""

import numpy as np
import pytest

from paper_0910_2950_gb300 import inputs

pytestmark = pytest.mark.gpu
DIMS = (8, 8, 8, 8)


@pytest.fixture(scope="module")
def fgmod():
    from paper_0910_2950_gb300 import build, fg
    build.build()
    fg.load()
    return fg


@pytest.mark.parametrize("link_reals", [18, 12])
@pytest.mark.parametrize("beta", [6.0, 5.9])
@pytest.mark.parametrize("integrator,steps", [("fg", 8), ("fg", 6), ("omelyan", 12), ("leapfrog", 24)])
def test_dh_against_fp64(fgmod, integrator, steps, beta, link_reals):
    u = inputs.hot_start(DIMS, 31)
    p = inputs.gaussian_momenta(DIMS, 32).astype(np.float32).astype(np.float64)
    got = {}
    with fgmod.Lattice(DIMS, beta, precision="fp32", link_reals=link_reals) as lat:
        lat.set_gauge(u)
        held = lat.get_gauge()
        lat.set_momenta(p)
        got["fp32"] = lat.trajectory(integrator, 1.0 / steps, 1.0, refresh=False, u_accept=0.0)
    with fgmod.Lattice(DIMS, beta, precision="fp64") as lat:
        lat.set_gauge(held)
        lat.set_momenta(p)
        got["fp64"] = lat.trajectory(integrator, 1.0 / steps, 1.0, refresh=False, u_accept=0.0)
    gain = abs(got["fp64"]["S_gauge1"] - got["fp64"]["S_gauge0"])
    bound = 2.0 ** -27 * gain + 16 * 2.0 ** -25 * np.sqrt(32 * np.prod(DIMS))
    assert abs(got["fp32"]["dH"] - got["fp64"]["dH"]) <= bound
