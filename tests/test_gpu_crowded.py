"""Boxes with many particles a cell, where each brick of cells has long loops: the
integer densities behind the coarse force, at the sizes where the bricks change."""

import numpy as np
import pytest

from oracle import force
from paper_2003_03931_gb300 import synth
from tests.gpu_util import make_sim, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc,pos_bytes", [(16, 1), (32, 1), (32, 2)])
def test_coarse_density_of_dense_boxes(nc, pos_bytes):
    # 64 particles a cell and more in clumps, in bricks of 4^3 cells (16^3) and 8 x 8 x 4
    need_gpu()
    bins = 256 if pos_bytes == 1 else 65536
    rng = np.random.default_rng(nc)
    sim = make_sim(np=4 * nc, nc=nc, a_init=0.02, a_final=1.0, n_steps=4, pos_bytes=pos_bytes)
    Q = synth.clustered_codes(rng, sim.cfg.n, nc, bins=bins)
    sim.load_qp(Q, synth.momenta(rng, sim.cfg.n), 0.3)
    want = force.ForceOperator(nc, pos_bytes).coarse_density(Q.T.astype(np.int64))
    np.testing.assert_array_equal(sim.fetch_coarse_density(), want.ravel())
    sim.close()
