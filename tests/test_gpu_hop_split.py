"""The Dslash launches on both sides of the size where a block goes from one
direction a warp to eight hops a thread, and on lattices that fill neither's
blocks, against the oracle.

Mhat is two Dslash applications of 48 products an output component: random
roundings of some 4 ulp each, 16 ulp of the result's norm with margin (in the
storage format for half precision, in double-float and FP64 below FP64's
1e-12)."""

import numpy as np
import pytest

from oracle import fermion
from paper_0910_2950_gb300 import inputs

pytestmark = pytest.mark.gpu
KAPPA = 0.12
DIMS = [(2, 2, 2, 2), (6, 2, 4, 10), (16, 16, 12, 16), (16, 14, 16, 14)]


@pytest.fixture(scope="module")
def fgmod():
    from paper_0910_2950_gb300 import build, fg
    build.build()
    fg.load()
    return fg


@pytest.fixture(scope="module")
def case():
    made = {}

    def get(dims):
        if dims not in made:
            u = inputs.hot_start(dims, 5)
            x = inputs.gaussian_spinor_even(dims, 6)
            full = inputs.unpack_even(x, dims)
            made[dims] = (u, x, inputs.pack_even(fermion.mhat(u, KAPPA, full), dims),
                          inputs.pack_even(fermion.mhat_dag(u, KAPPA, full), dims))
        return made[dims]

    return get


@pytest.mark.parametrize("precision,eps", [("fp32", 2.0 ** -24), ("fp32_fp16cg", 2.0 ** -11), ("fp64", 1e-12 / 16)])
@pytest.mark.parametrize("dims", DIMS)
def test_operator_matches_oracle(fgmod, case, dims, precision, eps):
    u, x, want, want_dag = case(dims)
    with fgmod.Lattice(dims, kappa=KAPPA, precision=precision) as lat:
        lat.set_gauge(u)
        for dagger, w in ((False, want), (True, want_dag)):
            got = lat.apply_mhat_inner(x, dagger)
            assert np.linalg.norm(got - w) <= 16 * eps * np.linalg.norm(w)


@pytest.mark.parametrize("precision", ["fp32", "fp32_fp16cg", "fp64"])
@pytest.mark.parametrize("dims", DIMS)
def test_solve_meets_its_tolerance(fgmod, case, dims, precision):
    """The grand totals behind alpha, beta and the residual: the residual of
    the solution, by the oracle on the links as the handle holds them."""
    u, b, _, _ = case(dims)
    with fgmod.Lattice(dims, kappa=KAPPA, precision=precision, cg_tol=1e-10) as lat:
        lat.set_gauge(u)
        x, info = lat.cg_solve(b)
        held = lat.get_gauge()
    r = inputs.pack_even(fermion.mdagm(held, KAPPA, inputs.unpack_even(x, dims)), dims) - b
    assert info["true_residual"] <= 1e-10
    assert np.linalg.norm(r) <= 1.1e-10 * np.linalg.norm(b)
