"""GPU: few-position calls whose FP32 point charges stand beside distributions: in
FP64 and in words, fewer and more FP32 points than one wave of threads takes
(152 x 512 of one chunk), against the oracle.  Bound of an FP32C call: 2e-6 Ha."""
import numpy as np
import pytest

import oracle
from paper_1011_4687_gb300 import build_lib, esp
from workloads import point_cells_environment, realistic_environment

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cells", [300, 77_000, 90_000])
@pytest.mark.parametrize("n_atoms", [2, 40])
def test_cells_beside_distributions(n_cells, n_atoms):
    build_lib.build()
    cells = point_cells_environment(56, n_cells=n_cells, n_nuclei=36, n_positions=16)
    wl = realistic_environment(seed=2723, n_atoms=n_atoms, n_walkers=1, n_elec=16)
    xyz = np.concatenate([cells.nuclei_xyz, wl.nuclei_xyz])
    Z = np.concatenate([cells.nuclei_Z, wl.nuclei_Z])
    ref = oracle.potential(xyz, Z, wl.pairs, wl.positions)
    with esp.Environment(xyz, Z, wl.pairs) as env:
        for n in (1, 2, 4, 5, 16):
            V = env.eval(wl.positions[:n])
            assert np.abs(V - ref[:n]).max() <= 2e-6, n
            assert np.array_equal(V, env.eval(wl.positions[:n]))
