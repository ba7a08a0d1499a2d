"""GPU: tiles dealt in parts (calls of few position blocks) against whole tiles
(one split) and the oracle: every tile size, ragged last parts, one or several
position blocks, environments of one class and of all.

FP32C, parts against whole tiles: every term and 4-term block is the same, only
the (sum, compensation) pairs are cut differently.  The compensation of N block
sums is about sqrt(N) 2^-25 of the absolute terms and takes sqrt(N) roundings of
2^-25 of itself: N 2^-50 of the absolute terms on either side.  FP64: 2e-13 of
the absolute terms (the near terms' recurrences and the oracle's own)."""
import numpy as np
import pytest

import oracle
from paper_1011_4687_gb300 import build_lib, esp
from workloads import realistic_environment, small_environment

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    esp.load()


WORKLOADS = {
    "classes": lambda: realistic_environment(seed=2721, n_atoms=24, n_walkers=1, n_elec=1100),
    "charges": lambda: small_environment(seed=95, n_nuclei=37, n_charges=1500, n_walkers=1, n_elec=1100),
}


@pytest.mark.parametrize("what", sorted(WORKLOADS))
@pytest.mark.parametrize("tile_size", [32, 64, 128, 256])
def test_parts(what, tile_size):
    wl = WORKLOADS[what]()
    ref = oracle.potential(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, wl.positions)
    kappa = oracle.abs_terms(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, wl.positions)
    args = (wl.nuclei_xyz, wl.nuclei_Z, wl.pairs)
    with esp.Environment(*args, precision="fp32c", tile_size=tile_size) as parts, \
            esp.Environment(*args, precision="fp32c", tile_size=tile_size, pair_splits=1) as whole, \
            esp.Environment(*args, precision="fp64", tile_size=tile_size, screen_tol=0.0) as f64:
        tol = 2 * (len(wl.pairs.alpha) / 4) * 2.0**-50
        for n in (17, 129, 512, 513, 1100):
            V, W = parts.eval(wl.positions[:n]), whole.eval(wl.positions[:n])
            assert np.all(np.abs(V - W) <= tol * kappa[:n]), (n, (np.abs(V - W) / kappa[:n]).max(), tol)
            assert np.array_equal(V, parts.eval(wl.positions[:n]))
            E = f64.eval(wl.positions[:n])
            assert np.all(np.abs(E - ref[:n]) <= 2e-13 * kappa[:n]), (n, (np.abs(E - ref[:n]) / kappa[:n]).max())
