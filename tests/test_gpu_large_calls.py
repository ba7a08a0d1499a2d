"""GPU: calls of many position blocks, whose tile groups take at least eight splits
while the partial sums stay within 256 MB (to 2^22 positions), against one split.

Every term and 4-term block is the same and only the (sum, compensation) pairs are
cut differently: N 2^-50 of the absolute terms on either side for N block sums."""
import numpy as np
import pytest

import oracle
from paper_1011_4687_gb300 import build_lib, esp
from workloads import realistic_environment

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [233_473, 1_000_001, (1 << 22) + 513, (1 << 23) + 3])
def test_groups_of_large_calls(n):
    torch = pytest.importorskip("torch")
    build_lib.build()
    wl = realistic_environment(seed=2722, n_atoms=12, n_walkers=1, n_elec=500)
    pick = torch.from_numpy(np.random.default_rng(n).integers(0, 500, size=n)).cuda()
    pos = torch.from_numpy(wl.positions).cuda()[pick].contiguous()
    kappa = torch.from_numpy(oracle.abs_terms(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, wl.positions)).cuda()[pick]
    args = (wl.nuclei_xyz, wl.nuclei_Z, wl.pairs)
    with esp.Environment(*args) as env, esp.Environment(*args, pair_splits=1) as whole:
        V, W = env.eval(pos), whole.eval(pos)
        torch.cuda.synchronize()
    assert ((V - W).abs() / kappa).max().item() <= 2 * (len(wl.pairs.alpha) / 4) * 2.0**-50
