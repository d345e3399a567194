"""The link exponential over its range of exponents: at beta = 0 a QPQ step of
length dt is two drifts U <- exp(i (dt / 2) P) U, compared with the oracle's.

The series is summed for c1 = Tr A^2 / 2 < 1/4 and squared k times above
(2^k <= 3.5 |A|), so the error of an entry is a few roundings times
1 + |A|; 40 (1 + |A|) of them for each drift bound it, storage of P and U
included."""

import numpy as np
import pytest

from oracle import su3
from paper_0910_2950_gb300 import inputs

pytestmark = pytest.mark.gpu

DIMS = (4, 2, 2, 2)
# c1 = Tr A^2 / 2 of A = (dt / 2) P: zero, tiny, both sides of every change of the number of halvings, large
C1 = [0.0, 1e-20, 1e-8, 0.03, 0.249, 0.251, 0.99, 1.01, 3.99, 4.01, 60.0, 2500.0]


@pytest.fixture(scope="module")
def fgmod():
    from paper_0910_2950_gb300 import build, fg
    build.build()
    fg.load()
    return fg


@pytest.mark.parametrize("link_reals", [18, 12])
@pytest.mark.parametrize("reunitarize", [0, 1])
@pytest.mark.parametrize("precision,eps", [("fp32", 2.0 ** -24), ("df64", 2.0 ** -47), ("fp64", 2.0 ** -53)])
def test_drift_over_the_range_of_exponents(fgmod, precision, eps, reunitarize, link_reals):
    u = inputs.hot_start(DIMS, 3)
    p = inputs.gaussian_momenta(DIMS, 4)
    dt = 0.5
    # c1 = (dt / 2)^2 sum (p^a)^2 / 4; a single Gell-Mann direction (degenerate eigenvalues) on some links
    p[..., 3, :7] = 0.0
    p[..., 0, 0, 1:] = 0.0
    unit = p / np.sqrt(0.25 * dt * dt * np.sum(p * p, axis=-1, keepdims=True) / 4.0)
    with fgmod.Lattice(DIMS, beta=0.0, precision=precision, link_reals=link_reals, reunitarize=reunitarize) as lat:
        for c1 in C1:
            q = unit * np.sqrt(c1)
            lat.set_gauge(u)
            lat.set_momenta(q)
            lat.md_step("qpq", dt)
            want = su3.expi(su3.alg_to_mat(q), dt) @ u
            err = np.max(np.abs(lat.get_gauge() - want))
            size = np.sqrt(4.0 * c1 / 3.0)
            assert err <= 80.0 * eps * (1.0 + size), (c1, err)
