"""Handles that share their GPU (fg_set_shared): the launches they take at sizes
where a handle alone takes others, against the oracle, and the two forms in
turn on one handle (captured batches of CG iterations hold the launches)."""

import numpy as np
import pytest

from oracle import fermion
from paper_0910_2950_gb300 import inputs, serve

KAPPA = 0.12
DIMS = [(2, 2, 2, 2), (6, 2, 4, 10), (8, 8, 8, 16), (16, 16, 12, 16)]


@pytest.fixture(scope="module")
def fgmod():
    from paper_0910_2950_gb300 import build, fg
    build.build()
    fg.load()
    return fg


@pytest.mark.gpu
@pytest.mark.parametrize("precision,eps", [("fp32", 2.0 ** -24), ("fp32_fp16cg", 2.0 ** -11)])
@pytest.mark.parametrize("dims", DIMS)
def test_operator_and_solve(fgmod, dims, precision, eps):
    """Bounds as in test_gpu_hop_split."""
    u, x = inputs.hot_start(dims, 5), inputs.gaussian_spinor_even(dims, 6)
    full = inputs.unpack_even(x, dims)
    want = inputs.pack_even(fermion.mhat(u, KAPPA, full), dims)
    with fgmod.Lattice(dims, kappa=KAPPA, precision=precision, cg_tol=1e-10) as lat:
        lat.set_shared()
        lat.set_gauge(u)
        assert np.linalg.norm(lat.apply_mhat_inner(x) - want) <= 16 * eps * np.linalg.norm(want)
        got, info = lat.cg_solve(x)
        held = lat.get_gauge()
    r = inputs.pack_even(fermion.mdagm(held, KAPPA, inputs.unpack_even(got, dims)), dims) - x
    assert info["true_residual"] <= 1e-10
    assert np.linalg.norm(r) <= 1.1e-10 * np.linalg.norm(x)


@pytest.mark.gpu
def test_changing_back_and_forth(fgmod):
    dims = (8, 8, 8, 16)
    u, b = inputs.hot_start(dims, 5), inputs.gaussian_spinor_even(dims, 6)
    got = {0: [], 1: []}
    with fgmod.Lattice(dims, kappa=KAPPA, precision="fp32") as lat:
        lat.set_gauge(u)
        for shared in (0, 1, 1, 0, 1, 0):
            lat.set_shared(shared)
            got[shared].append(lat.cg_solve(b)[0])
    for one in got.values():
        assert all(np.array_equal(x, one[0]) for x in one)
    with fgmod.Lattice(dims, kappa=KAPPA, precision="fp64") as lat:
        lat.set_gauge(u)
        alone = lat.cg_solve(b)[0]
        lat.set_shared()
        assert np.array_equal(alone, lat.cg_solve(b)[0])


@pytest.mark.parametrize("slots", [1, 2, 8])
def test_server_says_when_its_chains_run_together(monkeypatch, slots):
    made = []

    class Fake:
        def __init__(self, dims, beta, **kw):
            made.append(None)

        def set_shared(self, shared):
            made[-1] = bool(shared)

    monkeypatch.setattr(serve._fg, "Lattice", Fake)
    srv = serve.TrajectoryServer(slots=slots)
    srv.lattice_factory(serve.ChainSpec((4, 4, 4, 4), 5.9, 0.0, 1))
    srv.close()
    assert made == [slots > 1]
