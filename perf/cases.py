"""The timed cases: what users of this framework have it do, through its public
entry points (paper_2003_03931_gb300.sim, .serve and the C ABI of
include/pmpm.h), over the range of boxes it takes.

Operations:
  force  the force at every particle of a resident box (PMPM_FORCE)
  kick   restart from a checkpoint, one step, the kicked momenta (PMPM_STEP_QP)
  run    a whole run: initial conditions or a checkpoint, some steps, P(k)
  ic     make a box: Zel'dovich initial conditions and their P(k)
  pk     the power spectrum of a resident box
  serve  a queue of whole-box requests on the batch engine

Results that the library hands over as doubles but computes in float32 (P(k)
from float32 transforms; sigma, a float32 value) are given back as float32.
A step's drifted codes and the store that it writes are roundings of its
momenta to whole codes, in an order within a cell that is not specified: the
momenta stand for one step, the spectrum (every particle's position) for a run.
"""

import ctypes
import math

import numpy as np
import torch

from paper_2003_03931_gb300 import _lib, serve
from paper_2003_03931_gb300.sim import SimConfig, Simulation

DEV = "cuda:0"
LCDM = dict(omega_m=0.258, omega_l=0.742)   # the paper's background
SLOPE, K_C = -1.5, math.pi / 2              # spectrum of the repository's workloads


def _case(op, np_, nc, **kw):
    c = dict(op=op, np=np_, nc=nc, pos_bytes=1, lowmem=False, lcdm=False, tile_max=5, graphs=False,
             rms=1.0, steps=1, n_steps=20, step0=8, from_ic=False, nmesh=np_, nbins=np_ // 2,
             noalloc=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest box of the workloads: one force evaluation (interactive
        # use, checks of a set-up); latency and launches count
        dict(_case("force", 32, 16), name="force_32"),
        # sparse box (one particle per coarse cell), 13 ragged tiles a side,
        # 2-byte positions: the precise format on a fine mesh
        dict(_case("force", 64, 64, pos_bytes=2, rms=2.0), name="force_64_sparse_pos2"),
        # an ordinary box, late and clustered
        dict(_case("force", 128, 64, rms=4.0), name="force_128_clustered"),
        # restart a small box and take one step (checkpoint, then analysis)
        dict(_case("kick", 64, 32, rms=1.5), name="kick_64"),
        # the 32^3 workload whole: initial conditions, 10 steps, P(k)
        dict(_case("run", 32, 16, from_ic=True, steps=10, n_steps=10, step0=0), name="run_32"),
        # the 128^3 workload up to the middle of its schedule, steps replayed as graphs
        dict(_case("run", 128, 64, from_ic=True, steps=10, step0=0, graphs=True), name="run_128_graphs"),
        # low-memory step on the LambdaCDM background, from a checkpoint
        dict(_case("run", 256, 128, lowmem=True, lcdm=True, steps=3, rms=2.0), name="run_256_lowmem"),
        # the benchmark's 512^3 box: two steps from a checkpoint, P(k)
        dict(_case("run", 512, 256, steps=2, rms=1.5), name="run_512"),
        # a new box: float64 initial conditions and their spectrum
        dict(_case("ic", 256, 128), name="ic_256"),
        # spectrum on a mesh finer than the lattice
        dict(_case("pk", 256, 128, nmesh=512, nbins=255, rms=3.0), name="pk_256_on_512"),
        # the smallest spectrum, by the entry point that allocates nothing
        dict(_case("pk", 32, 16, nmesh=32, nbins=16, noalloc=True), name="pk_32_noalloc"),
        # sixteen requests of the serving mix's sizes, all waiting at the start
        dict(_case("serve", 128, 64, steps=10, nmesh=0, nbins=0), name="serve_16"),
    ]


def draw(rng):
    op = rng.choice(["force", "force", "kick", "run", "run", "ic", "pk"])
    n = 2 ** rng.randint(5, 8)                                # 32 .. 256 per side
    nc = n // 2 if rng.random() < 0.7 else (n if n <= 128 else n // 4)
    lowmem = op in ("run", "pk") and rng.random() < 0.4
    nf = 4 * nc
    nmesh = min(max(nf >> rng.randint(0, 2), nf // 4), 512)
    if op == "run":
        nmesh = max(nmesh, nf // 2)                           # fine enough to tell the steps
    return _case(op, n, nc, pos_bytes=1 if lowmem else rng.choice([1, 1, 2]), lowmem=lowmem,
                 lcdm=op == "run" and rng.random() < 0.5, tile_max=rng.choice([5, 5, 4]),
                 graphs=op in ("run", "kick") and rng.random() < 0.4,
                 rms=round(0.3 * (5.0 / 0.3) ** rng.random(), 3), steps=rng.randint(1, 4),
                 n_steps=rng.randint(13, 40), step0=0 if op == "ic" else rng.randint(1, 8),
                 nmesh=nmesh, nbins=rng.randint(nmesh // 4, nmesh // 2))


# ---------------------------------------------------------------- inputs
def _schedule(case):
    return (0.01 if case["lcdm"] else 0.02), 1.0, case["n_steps"]


def _scale_factor(case, step):
    a0, a1, n = _schedule(case)
    return a0 * (a1 / a0) ** (step / n)


def _bins(case):
    return 256 if case["pos_bytes"] == 1 else 65536


def _field(n, box, seed, rms):
    """Displacements [3][n^3] (fine cells) of a Gaussian field with the
    workloads' spectrum, scaled to a 3-D rms: small ones are early boxes, a
    few cells are late ones with crossed shells and clusters."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    wk = torch.fft.rfftn(torch.randn((n, n, n), generator=g, device=DEV))
    k = 2 * math.pi / box * torch.fft.fftfreq(n, 1.0 / n, device=DEV)
    kr = 2 * math.pi / box * torch.fft.rfftfreq(n, 1.0 / n, device=DEV)
    kk = [kr[None, None, :], k[None, :, None], k[:, None, None]]       # x fastest
    k2 = kk[0] ** 2 + kk[1] ** 2 + kk[2] ** 2
    k2[0, 0, 0] = 1.0
    wk *= k2 ** (SLOPE / 4 - 1) * torch.exp(-k2 / (2 * K_C * K_C))
    wk[0, 0, 0] = 0
    psi = torch.stack([torch.fft.irfftn(1j * kk[d] * wk, s=(n, n, n)).reshape(-1) for d in range(3)])
    return psi * (rms / math.sqrt(float((psi.double() ** 2).sum()) / n ** 3))


def _tables():
    u = torch.arange(256, dtype=torch.float64, device=DEV)
    T = torch.tan(math.pi * ((u + 0.5) / 256 - 0.5)).float()
    E = torch.tan(math.pi * (u[1:] / 256 - 0.5)).float()
    return T, E


def _store(case, seed):
    """A box in the framework's storage format, on the GPU: position bins m
    and velocity bins u [3][N] ordered by cell, counts, v_c and sigma."""
    n, nc, B = case["np"], case["nc"], _bins(case)
    box, N = 4.0 * nc, n ** 3
    psi = _field(n, box, seed, case["rms"])
    i = torch.arange(N, device=DEV)
    q = [i % n, (i // n) % n, i // (n * n)]
    Q = torch.stack([torch.floor(((q[d].double() + 0.5) * (box / n) + psi[d].double()) * (B / 4)).long() % (nc * B)
                     for d in range(3)])
    a = _scale_factor(case, case["step0"])
    g = torch.Generator(device=DEV).manual_seed(seed + 1)
    p = math.sqrt(a) * (psi + 0.1 * case["rms"] * torch.randn(psi.shape, generator=g, device=DEV))
    del psi, q, i
    c = Q // B
    key, order = torch.sort(c[0] + nc * (c[1] + nc * c[2]), stable=True)
    Q, p = Q[:, order], p[:, order]
    counts = torch.bincount(key, minlength=nc ** 3)
    end = torch.cumsum(counts, 0)
    vc = torch.zeros((3, nc ** 3), device=DEV)
    dev2 = 0.0
    u = torch.empty((3, N), dtype=torch.uint8, device=DEV)
    for d in range(3):
        S = torch.cumsum(torch.round(p[d].double() * 2 ** 24).long(), 0)
        S = torch.cat([S.new_zeros(1), S])
        vc[d] = ((S[end] - S[end - counts]).double() * 2.0 ** -24 / counts.clamp(min=1)).float()
        dev2 += float(((p[d] - vc[d][key]).double() ** 2).sum())
    sigma = float(np.float32(math.sqrt(dev2 / (3 * N))))
    if sigma == 0.0:
        sigma = 2.0 ** -24
    _, E = _tables()
    for d in range(3):
        u[d] = torch.bucketize((p[d] - vc[d][key]) / sigma, E, right=True).to(torch.uint8)
    m = (Q % B).to(torch.uint8 if B == 256 else torch.int32)
    return dict(m=m, u=u, key=key, counts=counts.int(), vc=vc, sigma=sigma, a=a)


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h.numpy()


def _checkpoint(case, s):
    """The host state that load_state takes, in pinned memory."""
    m = s["m"] if case["pos_bytes"] == 1 else s["m"].to(torch.int16).view(torch.uint8)
    raw = torch.cat([m.reshape(-1), s["u"].reshape(-1)])
    return {"streams": _pinned(raw), "counts": _pinned(s["counts"]), "vc": _pinned(s["vc"]),
            "scalars": {"a": s["a"], "sigma": s["sigma"], "step": case["step0"]}}


def _sim(case):
    a0, a1, n = _schedule(case)
    cfg = SimConfig(np=case["np"], nc=case["nc"], a_init=a0, a_final=a1, n_steps=n,
                    tile_max=case["tile_max"], pos_bytes=case["pos_bytes"], lowmem=case["lowmem"],
                    pk_mesh_max=min(4 * case["nc"], 512), **(LCDM if case["lcdm"] else {}))
    sim = Simulation(cfg, device=DEV, stream=torch.cuda.Stream(DEV) if case["graphs"] else None)
    if case["graphs"]:
        sim.graph_mode(True)
    return sim


def _requests(case, seed):
    """16 requests of the serving mix without its 256^3 boxes, 5 to 10 steps;
    the seed gives every box its own initial conditions."""
    return serve.mixed_requests(16, seed=1, steps=(5, case["steps"]), sizes=(32, 64, 128),
                                weights=(0.4, 0.3, 0.3), seed_base=1000 * (seed + 1))


def prepare(case, seed):
    op = case["op"]
    if op == "serve":
        return dict(case=case, requests=_requests(case, seed), engine=serve.Engine(8 << 30, device=DEV))
    if op == "ic" or case["from_ic"]:
        return dict(case=case, sim=_sim(case), seed=seed)
    store = _store(case, seed)
    if case["noalloc"]:
        return dict(case=case, store=store, lib=_lib.load(), k=np.zeros(case["nbins"]),
                    pk=np.zeros(case["nbins"]), nm=np.zeros(case["nbins"], np.int64))
    st = dict(case=case, sim=_sim(case), host=_checkpoint(case, store))
    N = case["np"] ** 3
    if op in ("force", "pk"):
        st["sim"].load_state(st["host"])
        del st["host"]
    if op == "force":
        st["out"] = torch.empty((3, N), dtype=torch.float32, pin_memory=True)
    if op == "kick":
        st["out"] = torch.empty(24 * N, dtype=torch.uint8, pin_memory=True)
    return st


# ---------------------------------------------------------------- one pass
def _fetch(sim, what, out):
    _lib.check(sim.lib.pmpm_fetch(sim.h, what, ctypes.c_void_p(out.data_ptr()),
                                  out.numel() * out.element_size()), sim.h)


def _spectrum(k, pk, nm):
    return {"k": k, "pk": pk.astype(np.float32), "modes": nm}


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "serve":
        eng = state["engine"]
        ids = [eng.submit(r) for r in state["requests"]]
        eng.run()
        res = {r.id: r for r in eng.poll()}
        return [_spectrum(res[i].k, res[i].pk, res[i].nmodes) for i in ids]
    if op == "pk" and case["noalloc"]:
        s, m = state["store"], state["store"]["m"]
        rc = state["lib"].pmpm_power_spectrum_noalloc(
            case["nc"], m.shape[1], m[0].data_ptr(), m[1].data_ptr(), m[2].data_ptr(),
            s["counts"].data_ptr(), case["nmesh"], case["nbins"], state["k"].ctypes.data,
            state["pk"].ctypes.data, state["nm"].ctypes.data,
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        _lib.check(rc)
        return _spectrum(state["k"], state["pk"], state["nm"])
    sim = state["sim"]
    if op == "force":
        _fetch(sim, _lib.FORCE, state["out"])
        return state["out"]
    if op == "pk":
        return _spectrum(*sim.power_spectrum(case["nmesh"], case["nbins"]))
    if op == "kick":
        sim.load_state(state["host"])
        sim.step(1)
        _fetch(sim, _lib.STEP_QP, state["out"])
        return state["out"][12 * sim.cfg.n:].view(torch.float32).view(3, -1)
    if op == "ic" or case["from_ic"]:
        sim.ic_zeldovich(state["seed"], slope=SLOPE, k_c=K_C, rms_disp=0.3)
    else:
        sim.load_state(state["host"])
    if op == "ic":
        out = _spectrum(*sim.power_spectrum(case["nmesh"], case["nbins"]))
        return dict(out, counts=sim.fetch_counts(), vc=sim.fetch_vc(),
                    sigma=np.float32(sim.fetch_scalars()["sigma"]))
    sim.step(case["steps"])
    out = _spectrum(*sim.power_spectrum(case["nmesh"], case["nbins"]))
    return dict(out, sigma=np.float32(sim.fetch_scalars()["sigma"]))


# ---------------------------------------------------------------- the least work
def _box_work(op, np_, nc, nmesh, steps, pos_bytes, from_ic):
    """Bytes: stores and cell arrays read once and written once, results out.
    Flops: real transforms of 2.5 M log2 M (the whole fine and coarse meshes,
    one forward and three inverse, for a force), 8-node clouds."""
    N, C, F = np_ ** 3, nc ** 3, (4 * nc) ** 3
    store = (3 * pos_bytes + 3) * N + 16 * C

    def fft(m):
        return 2.5 * m * math.log2(m)
    force = 4 * fft(F) + 4 * fft(C) + 160 * N
    pk = fft(nmesh ** 3) + 40 * N + 10 * nmesh ** 3 if nmesh else 0
    if op == "force":
        return 3 * pos_bytes * N + 4 * C + 12 * N, force
    if op == "pk":
        return 3 * pos_bytes * N + 4 * C, pk
    if op == "kick":
        return 2 * store + 24 * N, force + 60 * N
    ic = 4 * fft(N) + 60 * N if from_ic else 0
    if op == "ic":
        return store + 16 * C, ic + pk
    return (2 * steps + 1) * store, ic + steps * (force + 60 * N) + pk


def work(case):
    if case["op"] == "serve":
        w = [_box_work("run", r.np, r.nc, r.mesh()[0], r.n_steps, 1, True) for r in _requests(case, 1)]
        return {"bytes": float(sum(x[0] for x in w)), "flops": float(sum(x[1] for x in w))}
    b, f = _box_work(case["op"], case["np"], case["nc"], case["nmesh"], case["steps"],
                     case["pos_bytes"], case["op"] == "ic" or case["from_ic"])
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------- 64-bit values
def _codes(case, s):
    nc, B = case["nc"], _bins(case)
    c = [s["key"] % nc, (s["key"] // nc) % nc, s["key"] // (nc * nc)]
    return torch.stack([c[d] * B + s["m"][d].long() for d in range(3)])


def _cloud(x, mesh):
    """Cloud-in-cell nodes and weights of positions x [3, N] in node spacings
    (nodes at i + 1/2): eight (flat node, weight) pairs."""
    t = x - 0.5
    i = torch.floor(t)
    w = t - i
    i = i.long()
    for k in range(8):
        o = (k & 1, (k >> 1) & 1, k >> 2)
        j = [(i[d] + o[d]) % mesh for d in range(3)]
        f = 1.0
        for d in range(3):
            f = f * (w[d] if o[d] else 1.0 - w[d])
        yield j[0] + mesh * (j[1] + mesh * j[2]), f


def _density(x, mesh):
    rho = torch.zeros(mesh ** 3, dtype=torch.float64, device=DEV)
    for j, w in _cloud(x, mesh):
        rho.index_add_(0, j, w)
    return rho.view(mesh, mesh, mesh)


def _ewald_real(x, box):
    """x component of the screened real-space part at x [M, 3] (nearest image
    first), alpha = 5 / box."""
    al = 5.0 / box
    f = torch.zeros(x.shape[0], dtype=torch.float64, device=DEV)
    x = x - box * torch.round(x / box)
    for n in range(27):
        r = x + box * torch.tensor([n % 3 - 1.0, n // 3 % 3 - 1.0, n // 9 - 1.0], dtype=torch.float64, device=DEV)
        r2 = (r * r).sum(1)
        ok = r2 > 0
        r1 = torch.sqrt(torch.where(ok, r2, torch.ones_like(r2)))
        s = torch.special.erfc(al * r1) + 2 / math.sqrt(math.pi) * al * r1 * torch.exp(-(al * r1) ** 2)
        f -= torch.where(ok, r[:, 0] * s / r1 ** 3, torch.zeros_like(s))
    return f


def _ewald_modes(box):
    h = torch.arange(-10, 11, dtype=torch.float64, device=DEV)
    h = torch.stack(torch.meshgrid(h, h, h, indexing="ij"), -1).reshape(-1, 3)
    h = h[(h * h).sum(1) > 0]
    k = 2 * math.pi / box * h
    k2 = (k * k).sum(1)
    return h, k, 4 * math.pi / box ** 3 * torch.exp(-k2 / (4 * (5.0 / box) ** 2)) / k2


def _kernels(nc):
    """x component of the coarse kernel [nc^3] (periodic pair force at coarse
    separations) and of the fine kernel at separations [-5, 5]^3 (the pair
    force less the coarse mesh's mean force between fine-cell centres)."""
    box = 4.0 * nc
    h, k, c = _ewald_modes(box)
    # sampling folds the Fourier part's modes onto the mesh's
    hm = h.long() % nc
    spec = torch.zeros(nc ** 3, dtype=torch.complex128, device=DEV)
    spec.index_add_(0, hm[:, 0] + nc * (hm[:, 1] + nc * hm[:, 2]), (1j * c * k[:, 0]))
    four = torch.fft.ifftn(spec.view(nc, nc, nc)).real * nc ** 3
    D = torch.arange(nc, dtype=torch.float64, device=DEV) * 4
    Dz, Dy, Dx = torch.meshgrid(D, D, D, indexing="ij")
    real = _ewald_real(torch.stack([Dx, Dy, Dz], -1).reshape(-1, 3), box).view(nc, nc, nc)
    K = four + real
    K[0, 0, 0] = 0.0
    K[:, :, nc // 2] = 0.0                                   # odd and periodic
    # the fine kernel
    d = torch.arange(-5, 6, dtype=torch.float64, device=DEV)
    dz, dy, dx = torch.meshgrid(d, d, d, indexing="ij")
    sep = torch.stack([dx, dy, dz], -1).reshape(-1, 3)
    per = _ewald_real(sep, box) - (torch.sin(sep @ k.T) * (c * k[:, 0])).sum(1)
    A = torch.zeros(sep.shape[0], dtype=torch.float64, device=DEV)
    s = torch.arange(64, device=DEV)
    src = torch.stack([s % 4, s // 4 % 4, s // 16]).double() + 0.5      # [3, 64]
    shift = 16                                                # keeps every node index positive
    for e in range(sep.shape[0]):
        tgt = src + sep[e][:, None]
        acc = torch.zeros((), dtype=torch.float64, device=DEV)
        nodes = []
        for p in (src, tgt):
            t = p / 4 - 0.5
            i = torch.floor(t)
            nodes.append((i.long(), t - i))
        (ia, wa), (ib, wb) = nodes
        W = [torch.stack([(1 - wa[q]) * (1 - wb[q]) + wa[q] * wb[q], (1 - wa[q]) * wb[q], wa[q] * (1 - wb[q])])
             for q in range(3)]                               # offset differences 0, +1, -1
        D0 = ib - ia
        for x, ox in enumerate((0, 1, -1)):
            for y, oy in enumerate((0, 1, -1)):
                for z, oz in enumerate((0, 1, -1)):
                    acc = acc + (W[0][x] * W[1][y] * W[2][z] *
                                 K[(D0[2] + oz) % nc, (D0[1] + oy) % nc, (D0[0] + ox) % nc]).sum()
        A[e] = acc / 64
    r2 = (sep * sep).sum(1)
    Ks = torch.where((r2 > 0) & (r2 < 36), per - A, torch.zeros_like(A))
    return K, Ks.view(11, 11, 11)


def _force64(case, Q):
    nc, cpf = case["nc"], _bins(case) // 4
    nf = 4 * nc
    x = (Q.double() + 0.5) / cpf
    K, Ks = _kernels(nc)
    wide = torch.zeros((nf, nf, nf), dtype=torch.float64, device=DEV)
    i = torch.arange(-5, 6, device=DEV) % nf
    wide[i[:, None, None], i[None, :, None], i[None, None, :]] = Ks
    out = torch.zeros(Q.shape, dtype=torch.float64, device=DEV)
    for kern, mesh, scale in ((wide, nf, 1.0), (K, nc, 4.0)):
        rho = torch.fft.rfftn(_density(x / scale, mesh) - Q.shape[1] / mesh ** 3)
        for d in range(3):
            kd = kern if d == 0 else kern.transpose(2, 2 - d).contiguous()
            F = torch.fft.irfftn(rho * torch.fft.rfftn(kd), s=(mesh, mesh, mesh)).reshape(-1)
            for j, w in _cloud(x / scale, mesh):
                out[d] += w * F[j]
    return out


def _spectrum64(case, x):
    """k and P(k) of positions x [3, N] (fine cells) on an nmesh^3 mesh."""
    m, box = case["nmesh"], 4.0 * case["nc"]
    rho = _density(x * (m / box), m)
    dk = torch.fft.rfftn(rho * (m ** 3 / x.shape[1]) - 1.0)
    f = torch.fft.fftfreq(m, 1.0 / m, dtype=torch.float64, device=DEV)
    fr = torch.arange(m // 2 + 1, dtype=torch.float64, device=DEV)
    r = torch.sqrt(f[:, None, None] ** 2 + f[None, :, None] ** 2 + fr[None, None, :] ** 2).reshape(-1)
    w = torch.full((m, m, m // 2 + 1), 2.0, dtype=torch.float64, device=DEV)
    w[:, :, 0] = w[:, :, -1] = 1.0                            # modes without a mirror image of their own
    w = w.reshape(-1)
    j = torch.round(r).long()
    nm = torch.bincount(j, weights=w)
    P = torch.bincount(j, weights=w * (dk.abs() ** 2).reshape(-1)) / nm * (box ** 3 / float(m) ** 6)
    k = torch.bincount(j, weights=w * r) / nm * (2 * math.pi / box)
    b = slice(1, case["nbins"] + 1)
    return {"k": k[b], "pk": P[b], "modes": None}


def _noise64(n, seed):
    """White noise of SplitMix64 counters 2i, 2i + 1 through Box-Muller."""
    out = np.empty(n)
    with np.errstate(over="ignore"):
        for a in range(0, n, 1 << 22):
            j = np.arange(2 * a, 2 * min(n, a + (1 << 22)), dtype=np.uint64)
            z = np.uint64(seed) + (j + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z = (z ^ (z >> np.uint64(31))) >> np.uint64(11)
            u1 = (z[0::2].astype(np.float64) + 1) * 2.0 ** -53
            u2 = z[1::2].astype(np.float64) * 2.0 ** -53
            out[a:a + u1.size] = np.sqrt(-2 * np.log(u1)) * np.cos(2 * np.pi * u2)
    return out


def _ic64(case, seed):
    n, nc, cpf = case["np"], case["nc"], _bins(case) // 4
    box, a = 4.0 * nc, _schedule(case)[0]
    wk = torch.fft.fftn(torch.from_numpy(_noise64(n ** 3, seed)).to(DEV).view(n, n, n))
    f = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=DEV)
    kk = [2 * math.pi / box * f.view([-1 if e == 2 - d else 1 for e in range(3)]) for d in range(3)]
    k2 = kk[0] ** 2 + kk[1] ** 2 + kk[2] ** 2
    k2[0, 0, 0] = 1.0
    amp = torch.sqrt(k2 ** (SLOPE / 2) * torch.exp(-k2 / (K_C * K_C))) / k2
    amp[0, 0, 0] = 0.0
    h = n // 2
    amp[h, :, :] = 0.0
    amp[:, h, :] = 0.0
    amp[:, :, h] = 0.0
    psi = torch.stack([torch.fft.ifftn(1j * kk[d] * amp * wk).real.reshape(-1) for d in range(3)])
    psi *= 0.3 / (a * torch.sqrt((psi ** 2).sum() / n ** 3))
    i = torch.arange(n ** 3, device=DEV)
    q = torch.stack([i % n, i // n % n, i // (n * n)]).double()
    x = (q + 0.5) * (box / n) + a * psi
    Q = torch.floor(x * cpf).long() % (nc * _bins(case))
    p = a ** 1.5 * psi
    c = Q // _bins(case)
    key = c[0] + nc * (c[1] + nc * c[2])
    cnt = torch.bincount(key, minlength=nc ** 3)
    vc = torch.stack([torch.bincount(key, weights=p[d], minlength=nc ** 3) / cnt.clamp(min=1) for d in range(3)])
    sigma = torch.sqrt(((p - vc[:, key]) ** 2).sum() / (3 * n ** 3))
    return dict(_spectrum64(case, (Q.double() + 0.5) / cpf), counts=None, vc=vc, sigma=sigma)


def exact(case, seed):
    """run()'s values in 64 bits from the same inputs.  A run of several steps
    has none: its roundings to whole codes are part of the method."""
    op = case["op"]
    if op in ("serve", "run"):
        return None
    if op == "ic":
        return _ic64(case, seed)
    s = _store(case, seed)
    Q = _codes(case, s)
    if op == "pk":
        return _spectrum64(case, (Q.double() + 0.5) / (_bins(case) // 4))
    g = _force64(case, Q)
    if op == "force":
        return g
    # one kick of the Einstein-de Sitter leapfrog in a (half steps at the
    # geometric means)
    n0 = case["step0"]
    a = [_scale_factor(case, n0 + e) for e in (-1, 0, 1)]
    rho = case["np"] ** 3 / (4.0 * case["nc"]) ** 3
    kick = 3 / (8 * math.pi * rho) * 2 * ((a[1] * a[2]) ** 0.25 - (a[0] * a[1]) ** 0.25)
    u = s["u"].long()
    T = torch.tan(math.pi * ((torch.arange(256, dtype=torch.float64, device=DEV) + 0.5) / 256 - 0.5))
    return s["vc"].double()[:, s["key"]] + s["sigma"] * T[u] + kick * g
