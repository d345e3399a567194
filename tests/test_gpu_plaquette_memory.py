"""The plaquette field of FP64 and double-float forces: memory that only handles
with forces to form hold, and that they can do without."""

import numpy as np
import pytest

from oracle import gauge
from paper_0910_2950_gb300 import inputs

pytestmark = pytest.mark.gpu
DIMS = (8, 6, 4, 10)
BETA = 6.0


@pytest.fixture(scope="module")
def fgmod():
    from paper_0910_2950_gb300 import build, fg
    build.build()
    fg.load()
    return fg


def test_only_forces_take_it(fgmod):
    plaquettes = 384 * int(np.prod(DIMS))
    with fgmod.Lattice(DIMS, BETA, kappa=0.12, precision="fp64") as lat:
        lat.set_gauge(inputs.hot_start(DIMS, 1))
        lat.cg_solve(inputs.gaussian_spinor_even(DIMS, 2))
        lat.plaquette()
        before = lat.device_bytes()
        lat.force()
        assert lat.device_bytes() >= before + plaquettes
    with fgmod.Lattice(DIMS, BETA, precision="df64") as lat:
        lat.set_gauge(inputs.hot_start(DIMS, 1))
        lat.action()
        before = lat.device_bytes()
        lat.set_momenta(inputs.gaussian_momenta(DIMS, 2))
        assert lat.device_bytes() >= before + plaquettes


@pytest.mark.parametrize("precision,tol", [("fp64", 64 * 2.0 ** -53), ("df64", 128 * 2.0 ** -47)])
def test_without_it(fgmod, monkeypatch, precision, tol):
    """Force bound as in test_gpu_plaquette_force; a batch and a single lattice
    agree; nothing is held for plaquettes."""
    monkeypatch.setenv("FG_PLAQUETTES", "0")
    u, p = inputs.hot_start(DIMS, 1), inputs.gaussian_momenta(DIMS, 2)
    with fgmod.Lattice(DIMS, BETA, precision=precision) as lat, \
            fgmod.Batch([DIMS, (4, 4, 4, 4)], [BETA, BETA], precision=precision) as bat:
        lat.set_gauge(u)
        lat.set_momenta(p)
        before = lat.device_bytes()
        lat.timing(True)
        assert np.max(np.abs(lat.force() - gauge.gauge_force(u, BETA))) <= 4.0 * BETA / 6.0 * 6.0 * 2.0 * tol
        assert lat.kernel_time("plaquette")[1] == 0 and lat.device_bytes() == before
        bat.set_gauge(0, u)
        bat.set_momenta(0, p)
        bat.trajectory("fg", 0.25, 0.5, refresh=False, always_accept=True)
        lat.trajectory("fg", 0.25, 0.5, refresh=False, u_accept=0.0)
        assert np.array_equal(bat.get_gauge(0), lat.get_gauge())
