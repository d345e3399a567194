"""Solves do not depend on the scale of the source: the 16-bit solvers keep
r / sigma, sigma following |r| down to 1e-10 |b|, which for the smallest
sources here lies among FP32's denormal numbers (some 13 bits of a residual's
double-float entry are left at 1e-41, two more than half precision holds)."""

import numpy as np
import pytest

from oracle import fermion
from paper_0910_2950_gb300 import inputs

pytestmark = pytest.mark.gpu
DIMS = (8, 8, 8, 8)
KAPPA = 0.12


@pytest.fixture(scope="module")
def fgmod():
    from paper_0910_2950_gb300 import build, fg
    build.build()
    fg.load()
    return fg


@pytest.mark.parametrize("exponent", [-103, -96, -60, 60, 100])
@pytest.mark.parametrize("precision", ["fp32_fp16cg", "fp32_bf16cg"])
def test_solve_of_a_scaled_source(fgmod, precision, exponent):
    u, b = inputs.hot_start(DIMS, 5), inputs.gaussian_spinor_even(DIMS, 6) * 2.0 ** exponent
    with fgmod.Lattice(DIMS, kappa=KAPPA, precision=precision, cg_tol=1e-10) as lat:
        lat.set_gauge(u)
        x, _ = lat.cg_solve(b)
        held = lat.get_gauge()
    r = inputs.pack_even(fermion.mdagm(held, KAPPA, inputs.unpack_even(x, DIMS)), DIMS) - b
    assert np.linalg.norm(r) <= 1.1e-10 * np.linalg.norm(b)
