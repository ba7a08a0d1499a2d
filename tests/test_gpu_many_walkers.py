"""GPU: calls whose indices pass 32 bits: walker energies (one warp per walker: from
2^27 walkers on), position coordinates (from 2^31 / 3 positions on)."""
import numpy as np
import pytest

from paper_1011_4687_gb300 import build_lib, esp
from workloads import PairList
from workloads.generate import s_charge_pairs

pytestmark = pytest.mark.gpu


def test_walkers_beyond_2_27():
    torch = pytest.importorskip("torch")
    build_lib.build()
    n = (1 << 27) + 5
    with esp.Environment(np.array([[9.0, 0.0, 0.0]]), np.array([2.0]), PairList.empty(), precision="fp64") as env:
        pos = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
        pos[:, 0] = torch.arange(n, device="cuda") % 1000 * 1e-3
        E = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        V = torch.empty(n, dtype=torch.float64, device="cuda")
        env.eval_walkers(pos, n, 1, V_out=V, E_out=E)
        torch.cuda.synchronize()
        assert torch.equal(E, -V)
        assert (V * (9.0 - pos[:, 0]) - 2.0).abs().max().item() <= 1e-14


def test_coordinates_beyond_2_31():
    torch = pytest.importorskip("torch")
    build_lib.build()
    n = (1 << 31) // 3 + 1000
    faint = s_charge_pairs(np.array([[9.0, 9.0, 9.0]]), np.array([1.0]), np.array([1e-9]))
    with esp.Environment(np.array([[9.0, 0.0, 0.0]]), np.array([2.0]), faint) as env:
        pos = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
        pos[:, 0] = torch.arange(n, dtype=torch.int32, device="cuda") % 1000 * 1e-3
        V = env.eval(pos)
        torch.cuda.synchronize()
        # (the faint charge adds 1e-10)
        assert (V * (9.0 - pos[:, 0]) - 2.0).abs_().max().item() <= 1e-8
    del pos, V
    torch.cuda.empty_cache()
