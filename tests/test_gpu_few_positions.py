"""GPU: the few-position launch at the edges of its loops: one position up to
the largest call, part-filled chunks and pairs, tiles of every size, one entry,
nuclei beside FP32 cells (dd sums) and alone (FP64), repeated and interleaved
calls (the counters it leaves behind), against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1011_4687_gb300 import build_lib, esp
from workloads import PairList, point_cells_environment, realistic_environment

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    esp.load()


def check(V, ref, prec):
    lim = 1e-10 * np.maximum(np.abs(ref), 1.0) if prec == "fp64" else 2e-6
    assert np.all(np.abs(V - ref) <= lim), np.abs(V - ref).max()


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 31, 33, 48, 127, 128])
@pytest.mark.parametrize("prec", ["fp32c", "fp64"])
def test_cells(n, prec):
    wl = point_cells_environment(600 + n, n_cells=9001, n_nuclei=70, n_positions=n)
    ref = oracle.potential(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, wl.positions)
    with esp.Environment(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, precision=prec) as env:
        V = env.eval(wl.positions)
        check(V, ref, prec)
        assert np.array_equal(V, env.eval(wl.positions))


@pytest.mark.parametrize("tile_size", [32, 64, 128, 256])
@pytest.mark.parametrize("n", [1, 7, 16])
def test_distributions_and_nuclei_fp64(tile_size, n):
    wl = realistic_environment(seed=2719, n_atoms=30, n_walkers=1, n_elec=16)
    pos = wl.positions[:n]
    ref = oracle.potential(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, pos)
    for prec in ("fp64", "fp32c"):
        with esp.Environment(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, precision=prec, tile_size=tile_size,
                             point32_max_charge=0.0) as env:
            check(env.eval(pos), ref, "fp64")  # no FP32 entry: FP64 accuracy in both


@pytest.mark.parametrize("n_charges", [1, 2, 65])
def test_few_entries(n_charges):
    rng = np.random.default_rng(n_charges)
    xyz, Z = rng.uniform(-9, 9, size=(n_charges, 3)), rng.choice([0.1, -0.2, 3.0], size=n_charges)
    pos = np.concatenate([rng.uniform(-4, 4, size=(5, 3)), xyz[:1] + [[1e-4, 0, 0]]])
    ref = oracle.potential(xyz, Z, PairList.empty(), pos)
    with esp.Environment(xyz, Z, PairList.empty()) as env:
        V = env.eval(pos)
    kappa = oracle.abs_terms(xyz, Z, PairList.empty(), pos)
    # the last position sits on one charge: an FP32 term of it rounds |d|^2 three
    # times (half of that in its root), the root once, the product twice: four
    # FP32 units (2^-24 each) of the term
    assert np.all(np.abs(V - ref) <= np.maximum(2e-6, 4 * 2.0 ** -24 * kappa))


def test_calls_of_changing_size_and_graphs_interleave():
    torch = pytest.importorskip("torch")
    wl = point_cells_environment(77, n_cells=30000, n_nuclei=36, n_positions=128)
    ref = oracle.potential(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, wl.positions)
    pos = torch.from_numpy(wl.positions).cuda()
    with esp.Environment(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs,
                         stream=torch.cuda.current_stream().cuda_stream) as env:
        out = [torch.empty(n, dtype=torch.float64, device="cuda") for n in (1, 40)]
        with esp.Graph(env, pos[:1].clone(), out[0]) as g1, esp.Graph(env, pos[:40].clone(), out[1]) as g40:
            for n in (128, 1, 17, 500, 2, 128):
                p = pos[torch.arange(n, device="cuda") % 128]
                V = env.eval(p)
                g1.launch()
                g40.launch()
                torch.cuda.synchronize()
                check(V.cpu().numpy(), ref[np.arange(n) % 128], "fp32c")
                check(out[0].cpu().numpy(), ref[:1], "fp32c")
                check(out[1].cpu().numpy(), ref[:40], "fp32c")
