"""A step that fails on the host part-way (a CUDA call of the thread's that returned an
error is reported by the library's next check) leaves the sim where it was: the same
step can be taken again."""

import ctypes

import numpy as np
import pytest

from paper_2003_03931_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc,lowmem,graphs", [(16, False, False), (32, True, False), (64, False, False),
                                              (16, False, True)])
def test_the_same_step_again(nc, lowmem, graphs):
    need_gpu()
    import torch

    from paper_2003_03931_gb300._lib import PMPM_ECUDA, PmpmError
    from paper_2003_03931_gb300.sim import SimConfig, Simulation
    cfg = SimConfig(np=32, nc=nc, a_init=0.02, a_final=1.0, n_steps=3, lowmem=lowmem)
    cudart = ctypes.CDLL("libcudart.so.13")   # the library's: one per process
    states = []
    for fails in (False, True):
        sim = Simulation(cfg, device="cuda:0", stream=torch.cuda.Stream("cuda:0"))
        sim.graph_mode(graphs)
        sim.ic_zeldovich(5, **synth.IC_SPECTRUM)
        for _ in range(3):                    # the third's factors are the schedule's last
            if fails:
                sim.sync()
                cudart.cudaSetDevice(-1)      # returns an error and does nothing
                if not graphs or sim.fetch_scalars()["step"] < 2:
                    with pytest.raises(PmpmError) as e:
                        sim.step(1)
                    assert e.value.code == PMPM_ECUDA
                cudart.cudaGetLastError()
            sim.step(1)
        assert sim.fetch_scalars()["step"] == 3
        states.append((sim.fetch_counts(), sim.fetch_vc(), sim.fetch_scalars()["sigma"]))
        sim.close()
    for a, b in zip(*states):
        np.testing.assert_array_equal(a, b)
