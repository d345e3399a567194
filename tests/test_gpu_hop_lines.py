"""The Dslash of the inner solver on half-volumes around the sizes where FP64
goes from one direction a warp to eight hops a thread (131072 sites), and with
hundreds of blocks of 32 sites of which the last is not full; bounds as in
test_gpu_hop_split."""

import numpy as np
import pytest

from oracle import fermion
from paper_0910_2950_gb300 import inputs

pytestmark = pytest.mark.gpu
KAPPA = 0.12


@pytest.fixture(scope="module")
def fgmod():
    from paper_0910_2950_gb300 import build, fg
    build.build()
    fg.load()
    return fg


@pytest.mark.parametrize("dims,precisions", [((16, 16, 16, 64), ("fp64",)), ((16, 16, 16, 66), ("fp64",)),
                                             ((14, 14, 14, 14), ("fp64", "fp32", "fp32_fp16cg")),
                                             ((16, 16, 8, 10), ("fp32", "fp32_fp16cg"))])
def test_operator_matches_oracle(fgmod, dims, precisions):
    eps = {"fp64": 1e-12 / 16, "fp32": 2.0 ** -24, "fp32_fp16cg": 2.0 ** -11}
    u, x = inputs.hot_start(dims, 5), inputs.gaussian_spinor_even(dims, 6)
    full = inputs.unpack_even(x, dims)
    for dagger, op in ((False, fermion.mhat), (True, fermion.mhat_dag)):
        want = inputs.pack_even(op(u, KAPPA, full), dims)
        for precision in precisions:
            with fgmod.Lattice(dims, kappa=KAPPA, precision=precision) as lat:
                lat.set_gauge(u)
                got = lat.apply_mhat_inner(x, dagger)
            assert np.linalg.norm(got - want) <= 16 * eps[precision] * np.linalg.norm(want)
