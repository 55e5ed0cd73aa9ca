"""The column pass (short-range force by walking columns of tiles along z) at
the shapes where its parts change: the smallest box (its halo wraps onto
itself), ragged tiles of 4 and 5 cells, both position formats, and layers with
more particles than its tables, its first round of threads and its unchecked
deposit take.  Bar: the force of test_gpu_force.py, 1e-4 against the oracle."""

import numpy as np
import pytest

from oracle import force
from paper_2003_03931_gb300 import synth
from tests.gpu_util import make_sim, need_gpu, oracle_state, vector_rel_err

pytestmark = pytest.mark.gpu

TOL = 1e-4


def _check(sim):
    g = sim.fetch_force()
    ref = force.ForceOperator(sim.cfg.nc, sim.cfg.pos_bytes).particle_force(oracle_state(sim).codes()).T
    err = vector_rel_err(g, ref)
    assert err <= TOL, err


@pytest.mark.parametrize("np_,nc,tile_max,pos_bytes", [(16, 8, 5, 1), (16, 8, 4, 2), (16, 16, 5, 2), (32, 32, 5, 1),
                                                       (64, 32, 4, 2)])
def test_column_force_shapes(np_, nc, tile_max, pos_bytes):
    need_gpu()
    rng = np.random.default_rng(np_ + nc + tile_max)
    sim = make_sim(np=np_, nc=nc, a_init=0.02, a_final=1.0, n_steps=4, tile_max=tile_max, pos_bytes=pos_bytes)
    Q = synth.clustered_codes(rng, sim.cfg.n, nc, bins=256 if pos_bytes == 1 else 65536)
    sim.load_qp(Q, synth.momenta(rng, sim.cfg.n), 0.3)
    _check(sim)
    sim.close()


@pytest.mark.parametrize("in_cell", [250, 300, 5000])
def test_column_crowded_layer(in_cell):
    # all other particles uniform; `in_cell` share one coarse cell, one side of
    # the limit of 255 from which every node is checked, and past the 1024
    # particles whose cell comes from a table and the 256 of a first round
    need_gpu()
    nc = 16
    rng = np.random.default_rng(in_cell)
    sim = make_sim(np=32, nc=nc, a_init=0.02, a_final=1.0, n_steps=4)
    Q = synth.uniform_codes(rng, sim.cfg.n, nc)
    Q[:, :in_cell] = rng.integers(0, 256, size=(3, in_cell)) + 256 * np.array([[0], [7], [15]])
    sim.load_qp(Q.astype(np.int32), synth.momenta(rng, sim.cfg.n), 0.3)
    _check(sim)
    sim.close()


def test_column_flags_a_node_past_32_bits():
    # 4096 particles on one node: more than 2^32 of its 2^-21 units
    need_gpu()
    from paper_2003_03931_gb300._lib import PMPM_EOVERFLOW, PmpmError
    sim = make_sim(np=16, nc=8, a_init=0.1, a_final=0.5, n_steps=2)
    Q = np.full((3, sim.cfg.n), 3 * 256 + 32, np.int32)
    sim.load_qp(Q, np.zeros((3, sim.cfg.n), np.float32), 0.3)
    with pytest.raises(PmpmError) as e:
        sim.fetch_force()
    assert e.value.code == PMPM_EOVERFLOW
    sim.close()
