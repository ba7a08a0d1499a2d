"""GPU: evaluations in words where far charges (a uniform field made of two)
coarsen the environment's coordinate grid: FP64 calls and few-position calls,
positions whose T = p |P - C|^2 lies on both sides of the far limit for sharp
exponents, and positions close to point charges, against the oracle.  Bound as
for FP64 evaluations in words elsewhere: 2e-13 of the sum of absolute terms."""
import numpy as np
import pytest

import oracle
from paper_1011_4687_gb300 import build_lib, esp
from workloads import PairList, tiny_pd_environment
from workloads.generate import s_charge_pairs

pytestmark = pytest.mark.gpu
REL = 2e-13


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    esp.load()


def with_field(xyz, Z, far):
    """Two charges at +-far on the x axis, 0.05 Ha each at the centre."""
    return (np.concatenate([xyz, [[far, 0.0, 0.0], [-far, 0.0, 0.0]]]),
            np.concatenate([Z, [0.05 * far, -0.05 * far]]))


def at_T(rng, C, p, n):
    """n positions with p |P - C|^2 log-uniform in 20..400 for entries of (C, p)."""
    k = rng.integers(0, C.shape[0], size=n)
    d = rng.normal(size=(n, 3))
    r = np.sqrt(np.exp(rng.uniform(np.log(20.0), np.log(400.0), size=n)) / p[k])
    return C[k] + d / np.linalg.norm(d, axis=1)[:, None] * r[:, None]


def check(xyz, Z, pairs, pos, prec):
    ref = oracle.potential(xyz, Z, pairs, pos)
    kappa = oracle.abs_terms(xyz, Z, pairs, pos)
    with esp.Environment(xyz, Z, pairs, precision=prec, screen_tol=0.0, point32_max_charge=0.0) as env:
        V = env.eval(pos)
    err = np.abs(V - ref) / kappa
    assert np.all(err <= REL), (err.max(), int(err.argmax()))


@pytest.mark.parametrize("far", [30.0, 1e3, 1e4, 3e4, 1e5, 1e7])
@pytest.mark.parametrize("n,prec", [(400, "fp64"), (16, "fp64"), (16, "fp32c")])
def test_sharp_charges(far, n, prec):
    rng = np.random.default_rng(31)
    C = rng.uniform(-6.0, 6.0, size=(7000, 3))
    p = np.exp(rng.uniform(np.log(1e2), np.log(1e6), size=7000))
    pairs = s_charge_pairs(C, p, rng.uniform(-1.0, 1.0, size=7000))
    xyz, Z = with_field(np.array([[7.0, 7.0, 7.0]]), np.array([3.0]), far)
    check(xyz, Z, pairs, at_T(rng, C, p, n), prec)


@pytest.mark.parametrize("far", [1e3, 1e4, 3e4])
def test_every_class(far):
    wl = tiny_pd_environment(83, n_pairs=900, n_nuclei=40, n_pos=10, exp_range=(500.0, 5e5), spread=3.0, pos_radius=6.0)
    rng = np.random.default_rng(32)
    p = wl.pairs.alpha + wl.pairs.beta
    C = (wl.pairs.alpha[:, None] * wl.pairs.A + wl.pairs.beta[:, None] * wl.pairs.B) / p[:, None]
    xyz, Z = with_field(wl.nuclei_xyz, wl.nuclei_Z, far)
    check(xyz, Z, wl.pairs, at_T(rng, C, p, 300), "fp64")


@pytest.mark.parametrize("far", [1e3, 1e4, 1e5])
@pytest.mark.parametrize("n", [16, 200])
def test_close_to_point_charges(far, n):
    rng = np.random.default_rng(33)
    xyz, Z = with_field(rng.uniform(-6.0, 6.0, size=(7000, 3)), rng.choice([1.0, 6.0, -7.0], size=7000), far)
    d = rng.normal(size=(n, 3))
    d *= (np.exp(rng.uniform(np.log(2e-4), 0.0, size=n)) / np.linalg.norm(d, axis=1))[:, None]
    check(xyz, Z, PairList.empty(), xyz[rng.integers(0, 7000, size=n)] + d, "fp64")


@pytest.mark.parametrize("far", [1e3, 3e4, 1e5, 5e5, 1e7])
def test_points_and_near_blocks_beside_fp32_sums(far):
    """FP32C: charges and near blocks (every tile: near_radius beyond the environment)
    keep 48 bits, 1e-11 of the absolute terms with three digits to spare."""
    rng = np.random.default_rng(34)
    C = rng.uniform(-6.0, 6.0, size=(700, 3))
    p = np.linspace(6.0, 80.0, 700)
    pairs = s_charge_pairs(C, p, np.full(700, -1.5))
    xyz, Z = with_field(rng.uniform(-6.0, 6.0, size=(70, 3)), rng.choice([1.0, 6.0, -7.0], size=70), far)
    d = rng.normal(size=(200, 3))
    d *= (np.exp(rng.uniform(np.log(2e-4), 0.0, size=200)) / np.linalg.norm(d, axis=1))[:, None]
    pos = np.concatenate([xyz[rng.integers(0, 70, size=200)] + d, at_T(rng, C, p, 100)])
    ref = oracle.potential(xyz, Z, pairs, pos)
    kappa = oracle.abs_terms(xyz, Z, pairs, pos)
    with esp.Environment(xyz, Z, pairs, near_radius=1e3) as env:
        assert np.all(np.abs(env.eval(pos) - ref) <= 1e-11 * kappa)
