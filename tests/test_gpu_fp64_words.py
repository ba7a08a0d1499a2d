"""GPU: FP64 evaluations whose far entries are summed in FP32 words, against the
oracle: every class, tile sizes, ragged numbers of positions (sorted and not),
positions between the charges and far outside, exponents that put the entries of
a tile on both sides of the far limit.  Bound 2e-13 of the sum of absolute terms:
the FP64 near terms and the oracle's own rounding (a few hundred units of 1e-16
after its recurrences); a lost word would show at 1e-8 or 1e-15 x 64."""
import numpy as np
import pytest

import oracle
from paper_1011_4687_gb300 import build_lib, esp
from workloads import PairList, realistic_environment, small_environment, tiny_pd_environment

pytestmark = pytest.mark.gpu
REL = 2e-13


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    esp.load()


def check(wl, pos, **kw):
    ref = oracle.potential(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, pos)
    kappa = oracle.abs_terms(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, pos)
    with esp.Environment(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, precision="fp64", screen_tol=0.0, **kw) as env:
        V = env.eval(pos)
        assert np.array_equal(V, env.eval(pos))
    assert np.all(np.abs(V - ref) <= REL * kappa), (np.abs(V - ref) / kappa).max()


@pytest.mark.parametrize("tile_size", [32, 64, 128, 256])
@pytest.mark.parametrize("n", [17, 127, 129, 600])
def test_every_class(tile_size, n):
    wl = realistic_environment(seed=2720, n_atoms=24, n_walkers=1, n_elec=600)
    check(wl, wl.positions[:n], tile_size=tile_size)


@pytest.mark.parametrize("exp_range", [(0.05, 0.5), (0.5, 5.0), (5.0, 5000.0)])
def test_inside_the_environment(exp_range):
    wl = tiny_pd_environment(82, n_pairs=900, n_nuclei=40, n_pos=700, exp_range=exp_range, spread=3.0, pos_radius=6.0)
    check(wl, np.concatenate([wl.positions, 40.0 * wl.positions[:50]]))


@pytest.mark.parametrize("n_walkers", [3, 50])
def test_s_charges_and_walkers(n_walkers):
    wl = small_environment(seed=93, n_nuclei=300, n_charges=1500, n_walkers=n_walkers, n_elec=33)
    check(wl, wl.positions)


def test_close_to_charges_and_centres():
    wl = small_environment(seed=94, n_nuclei=300, n_charges=900, n_walkers=1, n_elec=20)
    wl.pairs.alpha[:50] = wl.pairs.beta[:50] = 1e6  # sharp: far form right up to the centre
    wl.pairs.w[:50] = -(2e6 / np.pi) ** 1.5
    step = np.array([[1e-2, 0, 0], [1e-4, 1e-4, 0], [1e-7, 0, 0]])
    pos = np.concatenate([wl.nuclei_xyz[:3] + step, wl.pairs.A[:3] + step, wl.pairs.A[:1], wl.positions])
    check(wl, pos)


def test_point_charges_of_both_classes_and_scales():
    rng = np.random.default_rng(8)
    xyz, Z = rng.uniform(-9, 9, size=(700, 3)), rng.choice([0.1, -0.2, 3.0, 1e-40], size=700)
    pos = rng.uniform(-5, 5, size=(130, 3))
    for scale in (1.0, 1e-25, 1e25):
        ref = oracle.potential(xyz, Z * scale, PairList.empty(), pos)
        kappa = oracle.abs_terms(xyz, Z * scale, PairList.empty(), pos)
        with esp.Environment(xyz, Z * scale, PairList.empty(), precision="fp64") as env:
            assert np.all(np.abs(env.eval(pos) - ref) <= REL * kappa)
