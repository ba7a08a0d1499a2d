"""GPU: nuclei and merged monopoles alone keep FP64 in an FP32C batch and in a
surrogate, as in a single call.  One charge per system, so that no sum averages the
48 bits of a dd term (3e-15 in the root mean square, beyond the bound in most of
the positions).  Bound 9 x 2^-53 of the potential: offsets 1, their square sum
1.5, reciprocal square root 2, product 1, three additions of the sums."""
import numpy as np
import pytest

from paper_1011_4687_gb300 import build_lib, esp
from workloads import PairList, qm_positions

pytestmark = pytest.mark.gpu
REL = 9 * 2.0 ** -53


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    build_lib.build()
    return t


def exact(xyz, Z, pos):
    d = pos.astype(np.longdouble) - xyz.astype(np.longdouble)
    return np.longdouble(Z) / np.sqrt((d * d).sum(1))


@pytest.mark.parametrize("n", [40, 4200])
def test_batch(torch, n):
    rng = np.random.default_rng(n)
    xyz, Z = rng.uniform(-9.0, 9.0, size=(3, 3)), np.array([1.0, 8.0, -7.3])
    envs = [esp.Environment(xyz[k:k + 1], Z[k:k + 1], PairList.empty()) for k in range(3)]
    pos = [rng.uniform(-6.0, 6.0, size=(n + k, 3)) for k in range(3)]
    with esp.Batch(envs) as b:
        out = b.eval([torch.from_numpy(p).cuda() for p in pos])
        torch.cuda.synchronize()
    for k in range(3):
        ref = exact(xyz[k], Z[k], pos[k])
        assert np.abs((out[k].cpu().numpy() - ref) / ref).max() <= REL
        envs[k].close()


def test_surrogate(torch):
    xyz, Z = np.array([[3.1, -7.2, 1.7]]), np.array([7.3])
    pos = qm_positions(np.random.default_rng(3), 3000)
    with esp.Environment(xyz, Z, PairList.empty()) as env, esp.Surrogate(env, n_train=1024, n_valid=512, epochs=0) as sur:
        p = torch.from_numpy(pos).cuda()
        ref = exact(xyz[0], Z[0], pos)
        for V in (sur.predict(p), sur.eval(p)[0]):
            assert np.abs((V.cpu().numpy() - ref) / ref).max() <= REL
