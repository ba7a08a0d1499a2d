"""GPU: the spatial order of a call's positions, at ragged ends of the eight sorting
CTAs' parts, in one cell and outside the grid: every slot is filled once, so the
call equals the oracle's sums position by position (64 distinct positions,
repeated; the oracle's values differ by far more than the bounds).

The environments keep their calls on the ordered paths: FP32C with a faint s-charge
beside the nuclei (nuclei alone are FP64), which adds less than 1e-14 of error to
the 48 bits of the nuclei's terms, 1e-11 with three digits to spare; FP64 with more
than 512 entries, 2e-13 of the sum of absolute terms as for all such calls."""
import numpy as np
import pytest

import oracle
from paper_1011_4687_gb300 import build_lib, esp
from workloads import PairList, tiny_pd_environment
from workloads.generate import s_charge_pairs

pytestmark = pytest.mark.gpu


def base_positions(spread):
    base = tiny_pd_environment(71, n_pairs=0, n_nuclei=40, n_pos=64, pos_radius=4.0).positions.copy()
    return 0.1 + 1e-3 * base if spread == "one cell" else 20.0 * base if spread == "outside" else base


@pytest.mark.parametrize("prec,n", [("fp32c", n) for n in (4096, 4097, 8191, 8200, 16393, 65537, 300001)] +
                         [("fp64", n) for n in (512, 513, 4097, 16393)])
@pytest.mark.parametrize("spread", ["cells", "one cell", "outside"])
def test_order(prec, n, spread):
    build_lib.build()
    rng = np.random.default_rng(9)
    xyz, Z = rng.uniform(-9.0, 9.0, size=(40 if prec == "fp32c" else 600, 3)), 3.0
    Z = np.full(xyz.shape[0], Z)
    pairs = s_charge_pairs(np.array([[9.0, 9.0, 9.0]]), np.array([1.0]), np.array([1e-8])) if prec == "fp32c" \
        else PairList.empty()
    base = base_positions(spread)
    ref = oracle.potential(xyz, Z, pairs, base)
    lim = (1e-11 if prec == "fp32c" else 2e-13) * oracle.abs_terms(xyz, Z, pairs, base)
    assert np.diff(np.sort(ref)).min() > 1e3 * lim.max()  # another position's value would show
    pick = np.random.default_rng(n).integers(0, 64, size=n)
    with esp.Environment(xyz, Z, pairs, precision=prec) as env:
        V = env.eval(base[pick])
    assert np.all(np.abs(V - ref[pick]) <= lim[pick])
