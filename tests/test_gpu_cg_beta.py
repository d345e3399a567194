"""The six-launch CG iteration's beta, |r'|^2 / |r|^2 of the residuals as they
are stored: at small kappa Mhat is near the unit matrix, an iteration takes
|r|^2 down by up to 1e9, and a beta whose error is relative to |r|^2 instead
spoils the search directions or ends in NaN.

FP64 arithmetic sets the count; in FP32 a reliable update costs at most the
progress of one iteration, and two more are allowed for the rounding of the
last ones."""

import numpy as np
import pytest

from oracle import fermion
from paper_0910_2950_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fgmod():
    from paper_0910_2950_gb300 import build, fg
    build.build()
    fg.load()
    return fg


@pytest.mark.parametrize("kappa", [0.0005, 0.002, 0.01, 0.03, 0.12])
@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (16, 16, 12, 16)])
def test_solves_over_the_range_of_convergence(fgmod, monkeypatch, dims, kappa):
    monkeypatch.setenv("FG_CG_FOLD", "0")
    u, b = inputs.hot_start(dims, 5), inputs.gaussian_spinor_even(dims, 6)
    counts = {}
    for precision in ("fp64", "fp32", "fp32_fp16cg", "fp32_bf16cg"):
        with fgmod.Lattice(dims, kappa=kappa, precision=precision, cg_tol=1e-12) as lat:
            lat.set_gauge(u)
            x, counts[precision] = lat.cg_solve(b)
            held = lat.get_gauge()
        r = inputs.pack_even(fermion.mdagm(held, kappa, inputs.unpack_even(x, dims)), dims) - b
        assert np.linalg.norm(r) <= 1.1e-12 * np.linalg.norm(b)
    assert counts["fp32"]["iterations"] <= counts["fp64"]["iterations"] + counts["fp32"]["reliable_updates"] + 2
