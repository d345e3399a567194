"""The plaquette form of the gauge force (double-float and FP64 links) against
the oracle where its rows of 32 half-sites and its neighbour steps can go
wrong: extents of 2, rows that are not filled or straddle time slices, blocks
of one warp and of several.

A component is 4 beta / 6 times a sum of six entries of size below 2, each a
sum of products of four unitary matrices: some 40 roundings, 64 with the
scale's.  Twice that in double-float, whose products round at two steps."""

import numpy as np
import pytest

from oracle import gauge
from paper_0910_2950_gb300 import inputs

pytestmark = pytest.mark.gpu
BETA = 6.0
DIMS = [(2, 2, 2, 2), (4, 2, 2, 6), (2, 6, 4, 16), (6, 4, 10, 2), (12, 10, 6, 8), (16, 8, 8, 12)]


@pytest.fixture(scope="module")
def fgmod():
    from paper_0910_2950_gb300 import build, fg
    build.build()
    fg.load()
    return fg


@pytest.mark.parametrize("link_reals", [18, 12])
@pytest.mark.parametrize("precision,tol", [("fp64", 64 * 2.0 ** -53), ("df64", 128 * 2.0 ** -47)])
@pytest.mark.parametrize("dims", DIMS)
def test_force_matches_oracle(fgmod, dims, precision, tol, link_reals):
    u = inputs.hot_start(dims, 7)
    want = gauge.gauge_force(u, BETA)
    with fgmod.Lattice(dims, BETA, precision=precision, link_reals=link_reals) as lat:
        lat.set_gauge(u)
        assert np.max(np.abs(lat.force() - want)) <= 4.0 * BETA / 6.0 * 6.0 * 2.0 * tol


@pytest.mark.parametrize("precision", ["fp64", "df64"])
def test_batch_and_single_lattices_agree(fgmod, precision):
    dims = [(4, 2, 2, 6), (12, 10, 6, 8), (2, 2, 2, 2), (2, 6, 4, 16)]
    with fgmod.Batch(dims, [BETA] * len(dims), precision=precision) as bat:
        for k, d in enumerate(dims):
            bat.set_gauge(k, inputs.hot_start(d, k))
            bat.set_momenta(k, inputs.gaussian_momenta(d, k))
        bat.trajectory("omelyan", 0.25, 0.5, refresh=False, always_accept=True)
        for k, d in enumerate(dims):
            with fgmod.Lattice(d, BETA, precision=precision) as lat:
                lat.set_gauge(inputs.hot_start(d, k))
                lat.set_momenta(inputs.gaussian_momenta(d, k))
                lat.trajectory("omelyan", 0.25, 0.5, refresh=False, u_accept=0.0)
                assert np.array_equal(bat.get_gauge(k), lat.get_gauge())
