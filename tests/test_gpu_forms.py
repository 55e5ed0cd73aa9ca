"""The coarse chain, the scan and the short-range pass at the sizes where their forms
change; for the short-range pass also ragged tiles of 4 and 5 cells, both
position formats and crowded cells.  (The boxes here are small or sparse and take
32^3-box tiles; test_gpu_column.py has the same for the column pass.)  Bar: the
force of test_gpu_force.py, 1e-4 against the oracle."""

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


@pytest.mark.parametrize("np_,nc,tile_max,pos_bytes", [(16, 32, 5, 2), (32, 32, 5, 1), (64, 32, 4, 2), (32, 64, 5, 1)])
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
    nc = 32
    rng = np.random.default_rng(in_cell)
    sim = make_sim(np=32, nc=nc, a_init=0.02, a_final=1.0, n_steps=4)
    Q = synth.uniform_codes(rng, sim.cfg.n, nc)
    Q[:, :in_cell] = rng.integers(0, 256, size=(3, in_cell)) + 256 * np.array([[0], [7], [31]])
    sim.load_qp(Q.astype(np.int32), synth.momenta(rng, sim.cfg.n), 0.3)
    _check(sim)
    sim.close()


@pytest.mark.parametrize("nc", [8, 16, 32, 64])
def test_coarse_force_chain(nc):
    # the coarse chain's forms: one launch up to 16^3 cells, four at 32^3, and at 64^3 the
    # general transforms (a sparse box); far from everything the force is the coarse mesh's alone
    need_gpu()
    rng = np.random.default_rng(nc)
    sim = make_sim(np=8, nc=nc, a_init=0.02, a_final=1.0, n_steps=4)
    sim.load_qp(synth.uniform_codes(rng, sim.cfg.n, nc), synth.momenta(rng, sim.cfg.n), 0.3)
    _check(sim)
    sim.close()


@pytest.mark.parametrize("nc", [8, 32, 64, 128])
def test_scan_of_every_form(nc):
    # counts, offsets (through the decoded store), v_c and sigma of the one-, two-
    # and three-launch scans, sparse and with one crowded cell
    need_gpu()
    rng = np.random.default_rng(nc)
    sim = make_sim(np=32, nc=nc, a_init=0.02, a_final=1.0, n_steps=4)
    Q = synth.clustered_codes(rng, sim.cfg.n, nc)
    P = synth.momenta(rng, sim.cfg.n)
    sim.load_qp(Q, P, 0.3)
    st = oracle_state(sim)
    cell = (Q[0] >> 8) + nc * ((Q[1] >> 8) + nc * (Q[2] >> 8).astype(np.int64))
    np.testing.assert_array_equal(st.counts, np.bincount(cell, minlength=nc ** 3))
    S = np.stack([np.round(P[d].astype(np.float64) * 2 ** 24).astype(np.int64) for d in range(3)])
    sums = [np.zeros(nc ** 3, np.int64) for _ in range(3)]
    for d in range(3):
        np.add.at(sums[d], cell, S[d])
    live = np.flatnonzero(st.counts)
    U = 0
    for d in range(3):
        vc = (sums[d][live].astype(np.float32) * np.float32(2.0 ** -24)) / st.counts[live].astype(np.float32)
        np.testing.assert_array_equal(st.vc[live, d], vc)
        U += sum(int(s) ** 2 // int(c) for s, c in zip(sums[d][live], st.counts[live]))
    T = sum(int(s) ** 2 for s in S.reshape(-1))
    assert abs(float(st.sigma) / np.sqrt((T - U) * 2.0 ** -48 / (3 * sim.cfg.n)) - 1) < 1e-7
    m = np.sort(st.codes().T[0]), np.sort(Q[0])
    np.testing.assert_array_equal(*m)
    sim.close()


def _mean_k(nmesh, nbins, box):
    """Mean |k| of every shell, summed exactly over the distinct |n|^2."""
    import math
    s = np.arange(-nmesh // 2, nmesh // 2) ** 2
    two = np.add.outer(s, s).reshape(-1)
    pairs = np.bincount(two)
    many = np.zeros(pairs.size + s.max(), np.int64)
    for v in s:
        many[v:v + pairs.size] += pairs
    out = []
    for j in range(1, nbins + 1):
        m = np.arange(j * j - j + 1, j * j + j + 1)
        out.append(2 * math.pi / box * math.fsum(many[m] * np.sqrt(m)) / many[m].sum())
    return np.array(out)


@pytest.mark.parametrize("nc,nmesh,pos_bytes", [(8, 8, 1), (8, 32, 2), (16, 16, 1), (16, 32, 2), (32, 32, 1),
                                                (16, 64, 1), (32, 64, 2), (64, 64, 1), (32, 128, 1), (64, 128, 2),
                                                (64, 256, 1), (128, 512, 1)])
def test_power_spectrum_forms(nc, nmesh, pos_bytes):
    # every node spacing (1, 2 and 4 fine cells), position format and mesh form (one
    # CTA up to 16^3, three passes from 32^3) against the oracle; a tenth of the
    # particles in one cell
    need_gpu()
    from oracle import power
    bins = 256 if pos_bytes == 1 else 65536
    rng = np.random.default_rng(nmesh + nc)
    sim = make_sim(np=32, nc=nc, a_init=0.02, a_final=1.0, n_steps=4, pos_bytes=pos_bytes)
    Q = synth.clustered_codes(rng, sim.cfg.n, nc, bins=bins)
    Q[:, :3000] = rng.integers(0, bins, size=(3, 3000)) + bins * np.array([[nc - 1], [0], [nc // 2]])
    sim.load_qp(Q.astype(np.int32), synth.momenta(rng, sim.cfg.n), 0.3)
    nbins = nmesh // 2 - 1
    k, pk, nm = sim.power_spectrum(nmesh, nbins)
    ko, po, no = power.power_spectrum(Q.T.astype(np.int64), nmesh, nbins, 4 * nc, pos_bytes=pos_bytes)
    np.testing.assert_array_equal(nm, no)
    # (the oracle's k is a running sum of up to 4e5 roots, itself 1e-12 off)
    np.testing.assert_allclose(k, _mean_k(nmesh, nbins, 4.0 * nc), rtol=1e-12)
    # float32 transforms of a field whose strongest modes lead the weakest ones
    np.testing.assert_allclose(pk, po, rtol=1e-4, atol=1e-6 * po.max())
    sim.close()


@pytest.mark.parametrize("n,nc,nmesh", [(1000, 8, 32), (4097, 16, 64)])
def test_noalloc_any_number_of_particles(n, nc, nmesh):
    # the entry point on a caller's store takes any n, not only a sim's powers of two
    need_gpu()
    import ctypes

    import torch

    from oracle import power
    from paper_2003_03931_gb300 import _lib
    lib = _lib.load()
    rng = np.random.default_rng(n)
    Q = synth.uniform_codes(rng, n, nc)
    cell = (Q[0] >> 8) + nc * ((Q[1] >> 8) + nc * (Q[2] >> 8).astype(np.int64))
    Q = Q[:, np.argsort(cell, kind="stable")]
    m = [torch.from_numpy((Q[d] & 255).astype(np.uint8)).cuda() for d in range(3)]
    counts = torch.from_numpy(np.bincount(cell, minlength=nc ** 3).astype(np.int32)).cuda()
    nbins = nmesh // 2
    k, pk, nm = np.zeros(nbins), np.zeros(nbins), np.zeros(nbins, np.int64)
    rc = lib.pmpm_power_spectrum_noalloc(nc, n, m[0].data_ptr(), m[1].data_ptr(), m[2].data_ptr(), counts.data_ptr(),
                                         nmesh, nbins, k.ctypes.data, pk.ctypes.data, nm.ctypes.data,
                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, lib.pmpm_noalloc_last_error()
    ko, po, no = power.power_spectrum(Q.T.astype(np.int64), nmesh, nbins, 4 * nc)
    np.testing.assert_array_equal(nm, no)
    np.testing.assert_allclose(k, ko, rtol=1e-12)
    np.testing.assert_allclose(pk, po, rtol=1e-4, atol=1e-6 * po.max())


def test_column_flags_a_node_past_32_bits():
    # 4096 particles on one node: more than 2^32 of its 2^-21 units
    need_gpu()
    from paper_2003_03931_gb300._lib import PMPM_EOVERFLOW, PmpmError
    sim = make_sim(np=16, nc=32, a_init=0.1, a_final=0.5, n_steps=2)
    Q = np.full((3, sim.cfg.n), 3 * 256 + 32, np.int32)
    sim.load_qp(Q, np.zeros((3, sim.cfg.n), np.float32), 0.3)
    with pytest.raises(PmpmError) as e:
        sim.fetch_force()
    assert e.value.code == PMPM_EOVERFLOW
    sim.close()


@pytest.mark.parametrize("np_,nc,pos_bytes", [(4, 8, 1), (8, 8, 2), (16, 8, 1), (32, 8, 1), (64, 32, 2), (128, 32, 1)])
def test_initial_conditions_sizes(np_, nc, pos_bytes):
    # every split of the float64 passes up to 128 points, against the oracle's
    # transforms: the same cells and codes, momenta to float32 rounding
    need_gpu()
    from oracle import ic
    sim = make_sim(np=np_, nc=nc, a_init=0.02, a_final=1.0, n_steps=4, pos_bytes=pos_bytes)
    sim.ic_zeldovich(9, **synth.IC_SPECTRUM)
    got = oracle_state(sim)
    ref, _, _ = ic.zeldovich(9, np_, nc, 0.02, pos_bytes=pos_bytes, **synth.IC_SPECTRUM)
    np.testing.assert_array_equal(got.counts, ref.counts)
    for d in range(3):
        np.testing.assert_array_equal(np.sort(got.codes().T[d]), np.sort(ref.codes().T[d]))
    np.testing.assert_allclose(got.vc, ref.vc, rtol=1e-5, atol=1e-6 * np.abs(ref.vc).max())
    np.testing.assert_allclose(float(got.sigma), float(ref.sigma), rtol=1e-6)
    sim.close()
