"""GPU: the spatial order of a call, the reductions over splits and electrons,
at the sizes where their loops end (parts of the eight sorting CTAs, slices of
the partial sums, lanes of a walker), against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1011_4687_gb300 import build_lib, esp
from workloads import point_cells_environment, tiny_pd_environment

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    esp.load()


@pytest.mark.parametrize("n", [4096, 4097, 8191, 8200, 16393])
@pytest.mark.parametrize("spread", ["cells", "one cell", "outside"])
def test_order_of_ragged_calls(n, spread):
    """Every slot is filled once, whatever the cells: the call equals the
    oracle's sums position by position (a few distinct positions, repeated)."""
    wl = tiny_pd_environment(71, n_pairs=0, n_nuclei=40, n_pos=64, pos_radius=4.0)
    base = wl.positions.copy()
    if spread == "one cell":
        base = 0.1 + 1e-3 * base
    elif spread == "outside":
        base = base * 20.0
    ref = oracle.potential(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, base)
    pick = np.random.default_rng(n).integers(0, 64, size=n)
    with esp.Environment(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs) as env:
        V = env.eval(base[pick])
    # point charges of FP32C calls are summed to better than 1e-10 relative
    assert np.all(np.abs(V - ref[pick]) <= 1e-10 * np.maximum(np.abs(ref[pick]), 1.0))


@pytest.mark.parametrize("n", [17, 129, 511, 513])
@pytest.mark.parametrize("prec", ["fp64", "fp32c"])
def test_many_splits_of_few_positions(n, prec):
    """More than 64 partial sums per position (few blocks of positions, many tiles)."""
    wl = point_cells_environment(55, n_cells=20000, n_nuclei=36, n_positions=n)
    ref = oracle.potential(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, wl.positions)
    with esp.Environment(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, precision=prec) as env:
        V = env.eval(wl.positions)
        assert np.array_equal(V, env.eval(wl.positions))
    lim = 1e-10 * np.maximum(np.abs(ref), 1.0) if prec == "fp64" else 2e-6
    assert np.all(np.abs(V - ref) <= lim)


@pytest.mark.parametrize("n_walkers,n_elec", [(1, 1), (5, 31), (3, 32), (7, 33), (129, 2), (2, 200)])
def test_walker_sums(n_walkers, n_elec):
    wl = tiny_pd_environment(72, n_pairs=60, n_nuclei=6, n_pos=n_walkers * n_elec)
    with esp.Environment(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, precision="fp64") as env:
        V, E = env.eval_walkers(wl.positions, n_walkers, n_elec)
    exact = oracle.walker_energies(V, n_walkers, n_elec)
    # FP64 sums with compensation: two roundings of the result
    assert np.all(np.abs(E - exact) <= 2 * np.finfo(float).eps * np.maximum(np.abs(exact), np.abs(V).max()))
