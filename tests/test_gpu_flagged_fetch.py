"""A fetch after a step that raised a device flag returns that error, and the data too:
what is fetched stands as it is."""

import ctypes

import numpy as np
import pytest

from tests.gpu_util import make_sim, need_gpu

pytestmark = pytest.mark.gpu


def test_scalars_come_with_the_error():
    need_gpu()
    from paper_2003_03931_gb300 import _lib
    sim = make_sim(np=16, nc=8, a_init=0.1, a_final=0.5, n_steps=2)
    Q = np.full((3, sim.cfg.n), 3 * 256 + 32, np.int32)        # more than 2^32 units on a node
    sim.load_qp(Q, np.zeros((3, sim.cfg.n), np.float32), 0.1)
    sim.step(1)
    sc = _lib.Scalars()
    rc = sim.lib.pmpm_fetch(sim.h, _lib.SCALARS, ctypes.addressof(sc), ctypes.sizeof(sc))
    assert rc == _lib.PMPM_EOVERFLOW
    assert sc.step == 1 and sc.n == sim.cfg.n and 0.1 < sc.a < 0.5 and sc.sigma > 0.0
    assert sim.fetch_scalars()["step"] == 1                    # reported once
    sim.close()
