"""FP64 and double-float fields on links that are unitary only to single
precision, as a program hands them over from an FP32 chain or a stored
configuration: the force is the derivative of the action at the links that
the handle holds, and dH follows.

Force: the bound of test_gpu_plaquette_force (64 roundings of the sums of
products that a component is made of; 128 in double-float, whose products
round at two steps).  dH: 64 roundings of H, which bounds what the forces of a
trajectory and the sums leave behind."""

import numpy as np
import pytest

from oracle import gauge
from oracle import integrators as it
from paper_0910_2950_gb300 import inputs

pytestmark = pytest.mark.gpu
BETA = 6.0
PRECISIONS = [("fp64", 2.0 ** -53, 64), ("df64", 2.0 ** -47, 128)]
DIMS = [(2, 2, 2, 2), (2, 6, 4, 16), (6, 4, 10, 2), (12, 10, 6, 8)]


@pytest.fixture(scope="module")
def fgmod():
    from paper_0910_2950_gb300 import build, fg
    build.build()
    fg.load()
    return fg


def single(u):
    """Links as single precision holds them."""
    return u.astype(np.complex64).astype(np.complex128)


@pytest.mark.parametrize("link_reals", [18, 12])
@pytest.mark.parametrize("precision,eps,n", PRECISIONS)
@pytest.mark.parametrize("dims", DIMS)
def test_force_is_the_derivative_at_the_links_held(fgmod, dims, precision, eps, n, link_reals):
    with fgmod.Lattice(dims, BETA, precision=precision, link_reals=link_reals) as lat:
        lat.set_gauge(single(inputs.hot_start(dims, 7)))
        want = gauge.gauge_force(lat.get_gauge(), BETA)
        assert np.max(np.abs(lat.force() - want)) <= 4.0 * BETA / 6.0 * 6.0 * 2.0 * n * eps


@pytest.mark.parametrize("integrator", ["fg", "omelyan"])
@pytest.mark.parametrize("precision,eps,n", PRECISIONS)
def test_dh_matches_oracle(fgmod, precision, eps, n, integrator):
    dims = (4, 4, 4, 4)
    u, p = single(inputs.hot_start(dims, 8)), inputs.gaussian_momenta(dims, 9)
    _, _, h0, h1 = it.trajectory(it.GaugeSystem(BETA), it.Integrator(integrator), u, p, 0.125)
    with fgmod.Batch([dims, dims], [BETA] * 2, precision=precision) as bat:
        for c in range(2):   # the other chain is unitary in 64 bits
            bat.set_gauge(c, u if c else inputs.hot_start(dims, 8))
            bat.set_momenta(c, p)
        batch = bat.trajectory(integrator, 0.125, 1.0, refresh=False, always_accept=True)[1]["dH"]
    with fgmod.Lattice(dims, BETA, precision=precision) as lat:
        lat.set_gauge(u)
        lat.set_momenta(p)
        alone = lat.trajectory(integrator, 0.125, 1.0, refresh=False, u_accept=0.0)["dH"]
    for got in (alone, batch):
        assert abs(got - (h1 - h0)) <= 64 * eps * h0


def test_form_follows_the_links(fgmod):
    """Staple sums until the links are projected, then plaquettes again."""
    dims = (4, 4, 4, 6)

    def plaquettes(lat):
        lat.timing_reset()
        lat.force()
        return lat.kernel_time("plaquette")[1]

    for precision in ("fp64", "df64"):
        with fgmod.Lattice(dims, BETA, precision=precision) as lat:
            lat.timing(True)
            assert plaquettes(lat) == 1           # cold start
            lat.set_gauge(single(inputs.hot_start(dims, 3)))
            assert plaquettes(lat) == 0
            lat.reunitarize()
            assert plaquettes(lat) == 1
            lat.set_gauge(single(inputs.hot_start(dims, 3)))
            lat.set_gauge(inputs.hot_start(dims, 3))
            assert plaquettes(lat) == 1


@pytest.mark.parametrize("precision", ["fp64", "df64"])
def test_mixed_batch_agrees_with_single_lattices(fgmod, precision):
    dims = [(4, 2, 2, 6), (12, 10, 6, 8), (2, 2, 2, 2), (2, 6, 4, 16)]
    starts = [inputs.hot_start(d, k) for k, d in enumerate(dims)]
    starts[1], starts[2] = single(starts[1]), single(starts[2])
    with fgmod.Batch(dims, [BETA] * len(dims), precision=precision) as bat:
        for turn in range(2):   # the second time other chains are off
            for k, d in enumerate(dims):
                bat.set_gauge(k, starts[k])
                bat.set_momenta(k, inputs.gaussian_momenta(d, k))
            for _ in range(2):
                bat.trajectory("fg", 0.25, 0.5, refresh=False, always_accept=True)
            for k, d in enumerate(dims):
                with fgmod.Lattice(d, BETA, precision=precision) as lat:
                    lat.set_gauge(starts[k])
                    lat.set_momenta(inputs.gaussian_momenta(d, k))
                    for _ in range(2):
                        lat.trajectory("fg", 0.25, 0.5, refresh=False, u_accept=0.0)
                    assert np.array_equal(bat.get_gauge(k), lat.get_gauge())
            starts = [inputs.hot_start(d, 10 + k) if 1 <= k <= 2 else single(starts[k]) for k, d in enumerate(dims)]


@pytest.mark.parametrize("precision", ["fp64", "df64"])
def test_compressed_links_stay_unitary(fgmod, precision):
    """12-real links over hundreds of trajectories: a rebuilt row must not feed
    its error back.  An FP64 handle that starts from the stored links goes on
    with the same bits (a double-float link can hold more than the 53 bits that
    the host's copy has)."""
    dims = (4, 4, 4, 4)
    with fgmod.Lattice(dims, BETA, precision=precision, link_reals=12, seed=5) as a, \
            fgmod.Lattice(dims, BETA, precision=precision, link_reals=12, seed=6) as b:
        a.set_gauge(inputs.hot_start(dims, 1))
        for _ in range(300):
            a.trajectory("fg", 0.125, 1.0, refresh=True, u_accept=0.0)
        u = a.get_gauge()
        defect = np.abs(np.einsum("...ij,...kj->...ik", u, u.conj()) - np.eye(3)).max()
        assert defect <= 64 * (2.0 ** -53 if precision == "fp64" else 2.0 ** -47)
        b.set_gauge(u)
        b.set_momenta(a.get_momenta())
        for lat in (a, b):
            lat.trajectory("fg", 0.125, 1.0, refresh=False, u_accept=0.0)
        assert precision == "df64" or np.array_equal(a.get_gauge(), b.get_gauge())
        a.timing(True)
        a.force()
        assert a.kernel_time("plaquette")[1] == 1
