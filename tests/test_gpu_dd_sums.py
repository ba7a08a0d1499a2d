"""GPU: the sums in pairs of FP32 numbers (point charges and near blocks of
FP32C calls) where they can go wrong: ragged tiles, positions on, very close to
and far outside the charges, values beyond FP32's range, every launch shape,
the batched kernel.  Bounds: the point-charge part keeps 48 bits per term, so
1e-11 of the sum of absolute terms holds with three digits to spare."""
import numpy as np
import pytest

import oracle
from paper_1011_4687_gb300 import build_lib, esp
from workloads import PairList, small_environment, tiny_pd_environment

pytestmark = pytest.mark.gpu
DD = 1e-11


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    esp.load()


# A faint s-charge: with it the point charges are part of an FP32C sum (alone
# they stay FP64); its FP32 terms err by less than 1e-14.
FAINT = PairList(np.array([[9.0, 9.0, 9.0]]), np.array([0.5]), np.zeros((1, 3), np.int32), np.array([[9.0, 9.0, 9.0]]),
                 np.array([0.5]), np.zeros((1, 3), np.int32), np.array([1e-8]))


def charges(seed, n, spread=10.0):
    rng = np.random.default_rng(seed)
    return rng.uniform(-spread, spread, size=(n, 3)), rng.choice([1.0, 6.0, 7.0, -8.0], size=n)


@pytest.mark.parametrize("n_charges", [1, 3, 4, 63, 64, 65, 130])
@pytest.mark.parametrize("kw", [dict(), dict(tile_size=32), dict(tile_size=256, pair_splits=2),
                                dict(threads_per_block=64, positions_per_thread=2),
                                dict(threads_per_block=256, positions_per_thread=1)])
def test_point_charges_ragged(n_charges, kw):
    xyz, Z = charges(n_charges, n_charges)
    pos = np.random.default_rng(1).uniform(-6.0, 6.0, size=(301, 3))
    ref = oracle.potential(xyz, Z, FAINT, pos)
    kappa = oracle.abs_terms(xyz, Z, FAINT, pos)
    with esp.Environment(xyz, Z, FAINT, **kw) as env:
        V = env.eval(pos)
    assert np.all(np.abs(V - ref) <= DD * kappa)


def test_point_charges_close_on_and_far():
    """On a charge: no finite value (the compensated sum of an infinite term);
    closer than the words resolve and outside their range (and non-finite
    positions): the FP64 code's values."""
    xyz, Z = charges(5, 70)
    step = np.array([1e-3, 0.0, 0.0])
    pos = np.concatenate([xyz[:1], xyz[1:2] + 1e-9 * step, xyz[2:3] + 1e-3 * step, xyz[3:4] + step,
                          [[1e3, 0, 0], [1e9, 1e9, 0], [np.nan, 0, 0]], np.zeros((40, 3))])
    ref = oracle.potential(xyz, Z, FAINT, pos[1:6])
    kappa = oracle.abs_terms(xyz, Z, FAINT, pos[1:6])
    with esp.Environment(xyz, Z, FAINT) as env:
        V = env.eval(pos)
    with esp.Environment(xyz, Z, FAINT, precision="fp64") as env:
        V64 = env.eval(pos)
    assert not np.isfinite(V[0]) and not np.isfinite(V64[0])
    assert np.all(np.abs(V[1:6] - ref) <= DD * kappa)
    assert np.isnan(V[6]) and np.isnan(V64[6])


@pytest.mark.parametrize("scale", [1e-30, 1e30, 1e60])
def test_charges_beyond_fp32_range(scale):
    xyz, Z = charges(6, 100)
    pos = np.random.default_rng(2).uniform(-6.0, 6.0, size=(40, 3))
    faint = FAINT.copy()
    faint.w *= min(scale, 1.0)
    ref = oracle.potential(xyz, Z * scale, faint, pos)
    kappa = oracle.abs_terms(xyz, Z * scale, faint, pos)
    with esp.Environment(xyz, Z * scale, faint, point32_max_charge=0.0, screen_tol=0.0) as env:
        assert np.all(np.abs(env.eval(pos) - ref) <= DD * kappa)


@pytest.mark.parametrize("n", [17, 129, 513, 4100])
def test_near_blocks_of_every_class(n):
    """near_radius beyond the environment: every block with a compact charge is
    near.  s and p/d products of sharp exponents (T on both sides of the Boys
    table's end), classes L = 0..4 (L <= 2 as dd sums, the rest FP64)."""
    wl = tiny_pd_environment(81, n_pairs=900, n_nuclei=10, n_pos=n, exp_range=(2.0, 40.0), spread=3.0,
                             pos_radius=4.0, same_center_frac=0.6)
    wl.pairs.w *= 2000.0  # compact charges: most tiles qualify
    ref = oracle.potential(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, wl.positions)
    kappa = oracle.abs_terms(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, wl.positions)
    with esp.Environment(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, near_radius=1e3, screen_tol=0.0) as env:
        assert env.info()["n_near_tiles"] >= 5
        V = env.eval(wl.positions)
    # (the tiles without a compact charge stay FP32)
    assert np.all(np.abs(V - ref) <= np.maximum(2e-6, 1.2e-7 * kappa))


def test_s_charges_all_near_reach_fp64_accuracy():
    wl = small_environment(seed=91, n_nuclei=50, n_charges=900, n_walkers=4, n_elec=33)
    # exponents above pi / |q|^2: every tile is near-capable
    wl.pairs.alpha[:] = wl.pairs.beta[:] = np.linspace(3.0, 40.0, len(wl.pairs))
    wl.pairs.w[:] = -1.5 * (2.0 * wl.pairs.alpha / np.pi) ** 1.5
    ref = oracle.potential(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, wl.positions)
    kappa = oracle.abs_terms(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, wl.positions)
    with esp.Environment(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, near_radius=1e3) as env:
        V = env.eval(wl.positions)
    assert np.all(np.abs(V - ref) <= DD * kappa)


def test_batch_sums_equal_single_calls():
    torch = pytest.importorskip("torch")
    wls = [small_environment(seed=92 + k, n_nuclei=30 + 40 * k, n_charges=300, n_walkers=3, n_elec=50 + k)
           for k in range(3)]
    envs = [esp.Environment(w.nuclei_xyz, w.nuclei_Z, w.pairs) for w in wls]
    pos = [torch.from_numpy(w.positions).cuda() for w in wls]
    with esp.Batch(envs) as b:
        out = b.eval(pos)
        torch.cuda.synchronize()
    for w, e, p, v in zip(wls, envs, pos, out):
        ref = oracle.potential(w.nuclei_xyz, w.nuclei_Z, w.pairs, w.positions)
        assert np.abs(v.cpu().numpy() - ref).max() <= 2e-6
        single = e.eval(p)
        e.synchronize()
        assert (v - single).abs().max().item() <= 1e-9
        e.close()
