"""GPU: few positions of distributions on both sides of the line between direct
FP64 entries (few entry-position pairs) and FP32 words, against the oracle: FP64
accuracy (2e-13 of the absolute terms, the terms' recurrences and the oracle's
own), with small point charges in FP32 2e-6 Ha."""
import numpy as np
import pytest

import oracle
from paper_1011_4687_gb300 import build_lib, esp
from workloads import realistic_environment

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    esp.load()


@pytest.mark.parametrize("n_atoms", [2, 24, 240])
@pytest.mark.parametrize("tile_size", [32, 64, 256])
def test_few_positions(n_atoms, tile_size):
    wl = realistic_environment(seed=2722, n_atoms=n_atoms, n_walkers=1, n_elec=16)
    args = (wl.nuclei_xyz, wl.nuclei_Z, wl.pairs)
    ref = oracle.potential(*args, wl.positions)
    kappa = oracle.abs_terms(*args, wl.positions)
    for precision, bound in (("fp64", 2e-13 * kappa), ("fp32c", np.maximum(2e-6, 2e-13 * kappa))):
        with esp.Environment(*args, precision=precision, tile_size=tile_size, screen_tol=0.0) as env:
            for n in (1, 2, 3, 7, 16):
                V = env.eval(wl.positions[:n])
                assert np.all(np.abs(V - ref[:n]) <= bound[:n]), (precision, n, np.abs(V - ref[:n]).max())
                assert np.array_equal(V, env.eval(wl.positions[:n]))
