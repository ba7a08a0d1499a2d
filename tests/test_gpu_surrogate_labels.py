"""GPU: FP32C labels of a surrogate whose far tiles lie within near_radius of
label positions.  The FP32C kernel leaves such blocks to the dd kernel; a block in
neither sum shifts the labels by whole Coulomb terms (0.1 Ha each).  FP64 labels
have no such blocks, and FP32C ones are within 2e-6 Ha of them, so the errors of
the expansion against the labels differ by no more than that."""
import numpy as np
import pytest

from paper_1011_4687_gb300 import build_lib, esp
from workloads.generate import s_charge_pairs

pytestmark = pytest.mark.gpu
TOL = 2e-6


@pytest.fixture(scope="module", autouse=True)
def _lib():
    pytest.importorskip("torch")
    build_lib.build()
    esp.load()


def cluster_environment(seed, x, r, n):
    """Compact s-charges (exponent 40, potential above 2 Ha) in a ball of radius r about (x, 0, 0)."""
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(n, 3))
    C = d / np.linalg.norm(d, axis=1)[:, None] * rng.uniform(0.0, r, size=(n, 1)) + np.array([x, 0.0, 0.0])
    pairs = s_charge_pairs(C, np.full(n, 40.0), rng.uniform(-1.5, -0.5, size=n))
    return np.array([[20.0, 0.0, 0.0], [-20.0, 0.0, 0.0]]), np.array([8.0, 7.0]), pairs


# (ball, near_radius, charges, configuration): gaps to the 6 bohr QM sphere of 6 and 1 bohr
@pytest.mark.parametrize("ball,near_radius,n,cfg", [
    ((13.0, 1.0), 8.0, 40, dict()),
    ((13.0, 1.0), 1e3, 300, dict()),
    ((7.4, 0.4), -1.0, 40, dict(far_radius=6.2)),
])
def test_labels_include_near_blocks_of_far_tiles(ball, near_radius, n, cfg):
    xyz, Z, pairs = cluster_environment(4, *ball, n)
    info = {}
    for prec in (esp.FP64, esp.FP32C):
        with esp.Environment(xyz, Z, pairs, near_radius=near_radius, tile_size=32) as env, \
                esp.Surrogate(env, n_train=2048, n_valid=4096, epochs=0, label_precision=prec, **cfg) as sur:
            info[prec] = sur.info()
    assert info[esp.FP64]["n_far_entries"] >= n
    for key in ("baseline_max_err", "baseline_rms_err"):
        assert abs(info[esp.FP64][key] - info[esp.FP32C][key]) <= TOL, (key, info)
