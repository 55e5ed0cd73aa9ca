"""Forms of the passes that only large meshes take, each against float64 (or, for the
coarse force, whose boxes are too large for that, against the general transforms of
fft.cu): initial conditions of 256^3 to 1024^3 particles, power spectra of 1024^3 and
2048^3 points, the coarse force of up to 1024^3 cells, the scan of 512^3 cells."""

import math
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2003_03931_gb300 import synth
from tests.gpu_util import make_sim, need_gpu, oracle_state

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


# ---------------------------------------------------------------- initial conditions
def _noise(torch, seed, lo, hi):
    """White noise of lattice points lo .. hi - 1: SplitMix64 counters, Box-Muller."""
    def out(j):
        def shift(z, s):
            return (z >> s) & ((1 << (64 - s)) - 1)
        z = (j + 1) * -0x61C8864680B583EB + seed          # 0x9E37...7C15 as int64
        z = (z ^ shift(z, 30)) * -0x40A7B892E31B1A47      # 0xBF58...E5B9
        z = (z ^ shift(z, 27)) * -0x6B2FB644ECCEEE15      # 0x94D0...11EB
        return shift(z ^ shift(z, 31), 11).double()
    i = torch.arange(lo, hi, device="cuda")
    return torch.sqrt(-2 * torch.log((out(2 * i) + 1) * 2.0 ** -53)) * torch.cos(2 * math.pi * out(2 * i + 1) * 2.0 ** -53)


def _zeldovich(torch, seed, n, nc, a, slope, k_c, rms_disp):
    """Expected counts, integer coarse density (units 2^-27) and v_c in float64."""
    box, N = 4.0 * nc, n ** 3
    w = torch.empty(N, dtype=torch.float64, device="cuda")
    for lo in range(0, N, 1 << 24):
        w[lo:lo + (1 << 24)] = _noise(torch, seed, lo, min(N, lo + (1 << 24)))
    wk = torch.fft.rfftn(w.view(n, n, n))
    del w
    f = 2 * math.pi / box * torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")
    fr = 2 * math.pi / box * torch.arange(n // 2 + 1, dtype=torch.float64, device="cuda")
    kk = [fr[None, :], f[:, None], f]                          # x, y of a plane and all z
    psi = torch.empty((3, N), dtype=torch.float64, device="cuda")
    h = n // 2
    for d in range(3):
        t = torch.empty_like(wk)
        for z in range(n):                                     # a plane at a time
            k2 = kk[0] ** 2 + kk[1] ** 2 + kk[2][z] ** 2
            if z == 0:
                k2[0, 0] = 1.0
            c = torch.sqrt(k2 ** (slope / 2) * torch.exp(-k2 / (k_c * k_c))) / k2 * (kk[2][z] if d == 2 else kk[d])
            c[h, :] = 0.0
            c[:, h] = 0.0
            if z == 0:
                c[0, 0] = 0.0
            t[z] = 0.0 if z == h else 1j * c * wk[z]
        psi[d] = torch.fft.irfftn(t, s=(n, n, n)).reshape(-1)
        del t
    del wk
    scale = rms_disp / (a * math.sqrt(sum(float((psi[d] ** 2).sum()) for d in range(3)) / N))
    counts = torch.zeros(nc ** 3, dtype=torch.int64, device="cuda")
    rho = torch.zeros(nc ** 3, dtype=torch.int64, device="cuda")
    P = torch.zeros((3, nc ** 3), dtype=torch.float64, device="cuda")
    for lo in range(0, N, 1 << 24):
        i = torch.arange(lo, min(N, lo + (1 << 24)), device="cuda")
        lat = [i % n, i // n % n, i // (n * n)]
        Q = [torch.floor(((lat[d].double() + 0.5) * (box / n) + a * scale * psi[d, i]) * 64).long() % (256 * nc)
             for d in range(3)]
        key = Q[0] // 256 + nc * (Q[1] // 256 + nc * (Q[2] // 256))
        counts += torch.bincount(key, minlength=nc ** 3)
        for d in range(3):
            P[d] += torch.bincount(key, weights=a ** 1.5 * scale * psi[d, i], minlength=nc ** 3)
        s = [2 * q + 1 - 256 for q in Q]
        for c in range(8):
            o = (c & 1, c >> 1 & 1, c >> 2)
            node = [((s[d] >> 9) + o[d]) % nc for d in range(3)]
            wt = [(s[d] & 511) if o[d] else 512 - (s[d] & 511) for d in range(3)]
            rho.index_add_(0, node[0] + nc * (node[1] + nc * node[2]), wt[0] * wt[1] * wt[2])
    return counts, rho, P / counts.clamp(min=1)


@pytest.mark.parametrize("np_", [256, 512, 1024])
def test_initial_conditions(np_):
    # the same codes (every bit of them weighs in the coarse density), momenta to
    # float32 rounding
    need_gpu()
    import torch
    nc, a = 64, 0.02
    want = [t.cpu().numpy() for t in _zeldovich(torch, 9, np_, nc, a, **synth.IC_SPECTRUM)]
    torch.cuda.empty_cache()
    sim = make_sim(np=np_, nc=nc, a_init=a, a_final=1.0, n_steps=4)
    sim.ic_zeldovich(9, **synth.IC_SPECTRUM)
    np.testing.assert_array_equal(sim.fetch_counts(), want[0])
    np.testing.assert_array_equal(sim.fetch_coarse_density(), want[1])
    np.testing.assert_allclose(sim.fetch_vc(), want[2], rtol=1e-5, atol=1e-6 * np.abs(want[2]).max())
    sim.close()
    del sim
    torch.cuda.empty_cache()


# ---------------------------------------------------------------- power spectrum
def _spectrum(torch, Q, nmesh, nbins, box):
    """P(k) and modes of a few particles (codes Q [3, N]) by the direct sum over them."""
    U = int(256 * box / 4 / nmesh)                             # codes of a node spacing
    s = 2 * torch.from_numpy(Q.astype(np.int64)).cuda() + 1 - U
    i0, w = s // (2 * U), (s % (2 * U)).double() / (2 * U)
    k = torch.arange(nmesh, device="cuda")
    E = []
    for d in range(3):
        turn = torch.polar(torch.ones((), dtype=torch.float64, device="cuda"), -2 * math.pi / nmesh *
                           (k[:, None] * i0[d][None, :] % nmesh).double())
        step = torch.polar(torch.ones((), dtype=torch.float64, device="cuda"), -2 * math.pi / nmesh * k.double())[:, None]
        E.append(turn * ((1 - w[d])[None, :] + w[d][None, :] * step))
    n = torch.where(k < nmesh // 2, k, k - nmesh)
    xy = (n * n)[None, :] + (n * n)[:, None]
    P = torch.zeros(2 * nmesh, dtype=torch.float64, device="cuda")
    M = torch.zeros(2 * nmesh, dtype=torch.float64, device="cuda")
    for z in range(nmesh // 2 + 1):                            # a mode's mirror image counts with it
        G = E[1] @ (E[0] * E[2][z][None, :]).T                 # [ky, kx]
        j = torch.round(torch.sqrt((xy + z * z).double())).long().reshape(-1)
        mult = 1.0 if z in (0, nmesh // 2) else 2.0
        P += mult * torch.bincount(j, weights=(G.real ** 2 + G.imag ** 2).reshape(-1), minlength=2 * nmesh)
        M += mult * torch.bincount(j, minlength=2 * nmesh)
    P = P / M.clamp(min=1) * box ** 3 / Q.shape[1] ** 2
    return P[1:nbins + 1].cpu().numpy(), M[1:nbins + 1].long().cpu().numpy()


@pytest.mark.parametrize("nc,meshes", [(256, [1024, 512]), (512, [2048, 1024])])
def test_power_spectrum(nc, meshes):
    need_gpu()
    import torch
    rng = np.random.default_rng(nc)
    sim = make_sim(np=4, nc=nc, a_init=0.02, a_final=1.0, n_steps=4, pk_mesh_max=meshes[0])
    Q = synth.uniform_codes(rng, sim.cfg.n, nc)
    sim.load_qp(Q, synth.momenta(rng, sim.cfg.n), 0.3)
    for nmesh in meshes:
        k, pk, modes = sim.power_spectrum(nmesh, nmesh // 2)
        want, many = _spectrum(torch, Q, nmesh, nmesh // 2, 4.0 * nc)
        np.testing.assert_array_equal(modes, many)
        # float32 transforms: the bar of the other forms
        np.testing.assert_allclose(pk, want, rtol=1e-4)
        assert np.all(np.abs(k * 4.0 * nc / (2 * math.pi) - np.arange(1, nmesh // 2 + 1)) < 0.5)
    sim.close()
    del sim
    torch.cuda.empty_cache()


# ---------------------------------------------------------------- coarse force, scan
def test_coarse_passes(tmp_path):
    # two orders of float32 transforms of 3 log2 n stages each, forward and back: a few
    # times 2^-24 sqrt(60)
    need_gpu()
    from paper_2003_03931_gb300 import build
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe, lib = str(tmp_path / "coarse_check"), os.path.dirname(build.LIB)
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-o", exe, os.path.join(HERE, "gpu", "coarse_check.cu"),
                    build.LIB, "-lcudart", "-Xlinker", "-rpath=" + lib], check=True)
    import torch
    torch.cuda.empty_cache()
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300).stdout
    rms = dict((int(c), float(v)) for c, v in (line.split() for line in out.splitlines()))
    assert sorted(rms) == [64, 128, 256, 512, 1024]
    assert all(v < 2e-6 for v in rms.values()), rms


def test_scan_of_large_meshes():
    # eight cells a thread and three launches: counts, the store's order, v_c and sigma
    need_gpu()
    nc = 512
    rng = np.random.default_rng(nc)
    sim = make_sim(np=32, nc=nc, a_init=0.02, a_final=1.0, n_steps=4)
    Q = synth.clustered_codes(rng, sim.cfg.n, nc)
    Q[:, :300] = Q[:, :1]
    P = synth.momenta(rng, sim.cfg.n)
    sim.load_qp(Q, P, 0.3)
    st = oracle_state(sim)
    cell = (Q[0] >> 8) + nc * ((Q[1] >> 8) + nc * (Q[2] >> 8).astype(np.int64))
    live, at = np.unique(cell, return_inverse=True)
    many = np.bincount(at)
    assert st.counts.sum() == sim.cfg.n and np.count_nonzero(st.counts) == live.size
    np.testing.assert_array_equal(st.counts[live], many)
    np.testing.assert_array_equal(np.sort(st.codes().T[0]), np.sort(Q[0]))
    S = np.round(P.astype(np.float64) * 2 ** 24).astype(np.int64)
    U = 0
    for d in range(3):
        s = np.zeros(live.size, np.int64)
        np.add.at(s, at, S[d])
        np.testing.assert_array_equal(st.vc[live, d], (s.astype(np.float32) * np.float32(2.0 ** -24)) / many.astype(np.float32))
        U += sum(int(v) ** 2 // int(c) for v, c in zip(s, many))
    T = sum(int(v) ** 2 for v in S.reshape(-1))
    assert abs(float(st.sigma) / np.sqrt((T - U) * 2.0 ** -48 / (3 * sim.cfg.n)) - 1) < 1e-7
    sim.close()
