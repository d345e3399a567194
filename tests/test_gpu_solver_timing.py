"""FP32 solves place their reliable updates by residuals that the host reads
while the GPU goes on: what it reads may not depend on how far the GPU has come.
Handles with the same inputs, run at the same time, give the same bits."""

import threading

import numpy as np
import pytest

from paper_0910_2950_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fgmod():
    from paper_0910_2950_gb300 import build, fg
    build.build()
    fg.load()
    return fg


@pytest.mark.parametrize("precision", ["fp32", "fp32_fp16cg"])
@pytest.mark.parametrize("dims", [(4, 4, 4, 8), (8, 8, 8, 16)])
def test_same_bits_at_any_pace(fgmod, dims, precision):
    u, chi = inputs.hot_start(dims, 31), inputs.gaussian_spinor_even(dims, 32)
    momenta = [inputs.gaussian_momenta(dims, 33 + k) for k in range(3)]
    got = {}

    def run(n):
        with fgmod.Lattice(dims, 5.6, precision=precision, kappa=0.12, seed=5) as lat:
            lat.set_gauge(u)
            lat.set_pseudofermion(chi)
            res = []
            for p in momenta:
                lat.set_momenta(p)
                res.append(lat.trajectory("fg", 0.25, 1.0, refresh=False, u_accept=0.0))
            got[n] = (res, lat.get_gauge())

    run(0)
    for _ in range(3):
        threads = [threading.Thread(target=run, args=(n,)) for n in range(1, 7)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for n in range(1, 7):
            assert got[n][0] == got[0][0]
            assert np.array_equal(got[n][1], got[0][1])
