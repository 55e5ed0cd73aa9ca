"""Steps of boxes up to 32^3 cells, and of boxes with a particle a cell or fewer,
give the bits that they gave with 32^3-box tiles and the radix-2 (32^3 cells) or
two-step (larger meshes) coarse transforms pass by pass: a last bit of the force
moves the P(k) of such a box by up to 4e-4 within a schedule.  golden/step_bits.txt
holds, for each box, sigma and checksums of counts and v_c after its steps, from
the library before it had any other kernel for them."""

import os
import zlib

import numpy as np
import pytest

from paper_2003_03931_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "step_bits.txt")
ROWS = [line.split() for line in open(GOLDEN) if not line.startswith("#")]


def step_bits(np_, nc, pos_bytes, tile_max, lowmem, graphs, steps, seed):
    import torch
    stream = torch.cuda.Stream() if graphs else None
    from paper_2003_03931_gb300.sim import SimConfig, Simulation
    sim = Simulation(SimConfig(np=np_, nc=nc, a_init=0.02, a_final=1.0, n_steps=10, pos_bytes=pos_bytes,
                               tile_max=tile_max, lowmem=bool(lowmem)), device="cuda:0", stream=stream)
    if graphs:
        sim.graph_mode(True)
    sim.ic_zeldovich(seed, **synth.IC_SPECTRUM)
    sim.step(steps)
    got = (np.float32(sim.fetch_scalars()["sigma"]).view(np.uint32), zlib.crc32(sim.fetch_counts().tobytes()),
           zlib.crc32(sim.fetch_vc().tobytes()))
    sim.close()
    return " ".join("%08x" % v for v in got)


@pytest.mark.parametrize("row", ROWS, ids=["-".join(r[:8]) for r in ROWS])
def test_steps_keep_their_bits(row):
    need_gpu()
    assert step_bits(*map(int, row[:8])) == " ".join(row[8:])
