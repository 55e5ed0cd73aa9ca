"""Mean |k| and mode counts of the power spectrum's shells, which follow from the mesh
alone, at every form of the mesh against exact sums."""

import math

import numpy as np
import pytest

from paper_2003_03931_gb300 import synth
from tests.gpu_util import make_sim, need_gpu

pytestmark = pytest.mark.gpu


def exact_shells(nmesh, box):
    """Mean |k| and modes of shell j = 1 .. nmesh/2: modes by |n|^2, roots summed by fsum."""
    s = np.arange(-nmesh // 2, nmesh // 2, dtype=np.int64) ** 2
    pairs = np.bincount(np.add.outer(s, s).reshape(-1))
    many = np.zeros(pairs.size + s.max(), np.int64)
    for v in s:
        many[v:v + pairs.size] += pairs
    k, modes = [], []
    for j in range(1, nmesh // 2 + 1):
        m = np.arange(j * j - j + 1, j * j + j + 1)
        modes.append(int(many[m].sum()))
        k.append(2 * math.pi / box * math.fsum(int(c) * math.sqrt(v) for c, v in zip(many[m], m.tolist())) / modes[-1])
    return np.array(k), np.array(modes)


@pytest.mark.parametrize("nc,nmesh", [(8, 8), (8, 16), (8, 32), (16, 64), (32, 128), (64, 256), (128, 512), (256, 1024)])
def test_mean_k_to_float64_rounding(nc, nmesh):
    # a root, a product and a place in a sum of 2 j terms, over 256 threads or fewer, and the
    # division: 16 roundings of 2^-53 in all
    need_gpu()
    sim = make_sim(np=16, nc=nc, a_init=0.02, a_final=1.0, n_steps=4, pk_mesh_max=nmesh)
    rng = np.random.default_rng(nmesh)
    sim.load_qp(synth.uniform_codes(rng, sim.cfg.n, nc), synth.momenta(rng, sim.cfg.n), 0.3)
    k, _, modes = sim.power_spectrum(nmesh, nmesh // 2)
    want, many = exact_shells(nmesh, 4.0 * nc)
    np.testing.assert_array_equal(modes, many)
    np.testing.assert_allclose(k, want, rtol=16 * 2.0 ** -53)
    sim.close()
