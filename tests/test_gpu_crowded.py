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


@pytest.mark.parametrize("nc,nmesh,pos_bytes", [(16, 32, 1), (32, 128, 2), (64, 64, 1), (64, 256, 1)])
@pytest.mark.parametrize("in_cell", [1024, 1025, 32768])
def test_power_spectrum_of_a_crowded_cell(nc, nmesh, pos_bytes, in_cell):
    # both sides of the count from which the warps of a brick share its rows, and
    # everything in one cell, at the brick forms and node spacings
    need_gpu()
    from oracle import power
    bins = 256 if pos_bytes == 1 else 65536
    rng = np.random.default_rng(in_cell + nc)
    sim = make_sim(np=32, nc=nc, a_init=0.02, a_final=1.0, n_steps=4, pos_bytes=pos_bytes)
    Q = synth.uniform_codes(rng, sim.cfg.n, nc, bins=bins)
    here = np.all(Q // bins == np.array([[nc - 1], [0], [nc // 2]]), axis=0)   # none but these in that cell
    Q[:, here] = 0
    Q[:, :in_cell] = rng.integers(0, bins, size=(3, in_cell)) + bins * np.array([[nc - 1], [0], [nc // 2]])
    sim.load_qp(Q.astype(np.int32), synth.momenta(rng, sim.cfg.n), 0.3)
    k, pk, nm = sim.power_spectrum(nmesh, nmesh // 2)
    ko, po, no = power.power_spectrum(Q.T.astype(np.int64), nmesh, nmesh // 2, 4 * nc, pos_bytes=pos_bytes)
    np.testing.assert_array_equal(nm, no)
    # float32 transforms: the bar of the other forms
    np.testing.assert_allclose(pk, po, rtol=1e-4, atol=1e-6 * po.max())
    sim.close()
