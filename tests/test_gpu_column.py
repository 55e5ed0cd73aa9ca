"""The column pass (short-range force by walking columns of tiles along z), which boxes
of 64^3 cells and more with over a particle a cell take: ragged tiles of 4 and 5
cells, both position formats, and layers with more particles than its tables, its first
round of threads and its unchecked deposit take.  Bar: the force of
test_gpu_force.py, 1e-4 against the oracle; and a step's momenta are the old ones
and the kick of that same force, bit for bit."""

import numpy as np
import pytest

from oracle import dynamics, force
from paper_2003_03931_gb300 import synth
from tests.gpu_util import make_sim, need_gpu, oracle_state, vector_rel_err

pytestmark = pytest.mark.gpu

NC = 64


def _check(sim, Q, P, a=0.3):
    sim.load_qp(Q.astype(np.int32), P, a)
    g = sim.fetch_force()
    st = oracle_state(sim)
    ref = force.ForceOperator(sim.cfg.nc, sim.cfg.pos_bytes).particle_force(st.codes()).T
    err = vector_rel_err(g, ref)
    assert err <= 1e-4, err
    kick, _ = dynamics.step_factors(sim.cfg.a_init, sim.cfg.a_final, sim.cfg.n_steps, 0, sim.cfg.n, 4 * sim.cfg.nc)
    sim.step(1)
    _, p = sim.fetch_step_qp()
    want = (st.momenta().T + (np.float32(kick) * g).astype(np.float32)).astype(np.float32)
    np.testing.assert_array_equal(p, want)


@pytest.mark.parametrize("tile_max,pos_bytes", [(5, 1), (5, 2), (4, 1), (4, 2)])
def test_shapes(tile_max, pos_bytes):
    need_gpu()
    rng = np.random.default_rng(tile_max + pos_bytes)
    sim = make_sim(np=128, nc=NC, a_init=0.02, a_final=1.0, n_steps=4, tile_max=tile_max, pos_bytes=pos_bytes)
    Q = synth.clustered_codes(rng, sim.cfg.n, NC, bins=256 if pos_bytes == 1 else 65536)
    _check(sim, Q, synth.momenta(rng, sim.cfg.n))
    sim.close()


@pytest.mark.parametrize("in_cell", [250, 300, 5000])
def test_crowded_layer(in_cell):
    # one side of the 255 particles a cell from which every node is checked, and past
    # the 1024 whose cell comes from a table and the 256 of a first round
    need_gpu()
    rng = np.random.default_rng(in_cell)
    sim = make_sim(np=128, nc=NC, a_init=0.02, a_final=1.0, n_steps=4)
    Q = synth.uniform_codes(rng, sim.cfg.n, NC)
    Q[:, :in_cell] = rng.integers(0, 256, size=(3, in_cell)) + 256 * np.array([[0], [7], [NC - 1]])
    _check(sim, Q, synth.momenta(rng, sim.cfg.n))
    sim.close()


def test_flags_a_node_past_32_bits():
    # 4096 particles on one node: more than 2^32 of its 2^-21 units
    need_gpu()
    from paper_2003_03931_gb300._lib import PMPM_EOVERFLOW, PmpmError
    rng = np.random.default_rng(1)
    sim = make_sim(np=128, nc=NC, a_init=0.1, a_final=0.5, n_steps=2)
    Q = synth.uniform_codes(rng, sim.cfg.n, NC)
    Q[:, :4096] = 3 * 256 + 32
    sim.load_qp(Q, np.zeros((3, sim.cfg.n), np.float32), 0.3)
    with pytest.raises(PmpmError) as e:
        sim.fetch_force()
    assert e.value.code == PMPM_EOVERFLOW
    sim.close()
