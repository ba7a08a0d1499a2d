"""GPU: contexts of different tile sizes evaluated from several host threads at a
time: every launch succeeds (a kernel's shared-memory limit is common to them)
and every call returns what it returns alone."""
import threading

import numpy as np
import pytest

from paper_1011_4687_gb300 import build_lib, esp
from workloads import realistic_environment

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
def test_tile_sizes_side_by_side(precision):
    build_lib.build()
    wl = realistic_environment(seed=77, n_atoms=24, n_walkers=1, n_elec=40)
    pos = np.ascontiguousarray(wl.positions[:40])
    envs = [esp.Environment(wl.nuclei_xyz, wl.nuclei_Z, wl.pairs, precision=precision, tile_size=t)
            for t in (32, 256, 64, 256)]
    alone = [e.eval(pos) for e in envs]
    bad, gate = [], threading.Barrier(len(envs))

    def loop(env, ref):
        gate.wait()
        for _ in range(400):
            try:
                if not np.array_equal(env.eval(pos), ref):
                    bad.append("value")
            except Exception as ex:  # a refused launch
                bad.append(repr(ex))

    threads = [threading.Thread(target=loop, args=a) for a in zip(envs, alone)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for e in envs:
        e.close()
    assert not bad, (len(bad), bad[:3])
