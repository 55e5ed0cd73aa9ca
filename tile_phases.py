"""Per-phase clock breakdown of the column pass (the short-range pass of a
step): a measurement tool beside bench.py (the library itself is not built
with it).

Builds a second copy of the library with -DPMPM_PHASE_CLOCKS, in which every
warp adds up clock64() between the marks of a layer, runs a box, and prints
the mean cycles per layer and warp of the chosen steps:

    python tile_phases.py [--workload c3_512] [--steps 1 10 20]
"""

import argparse
import ctypes
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)
PKG = os.path.join(ROOT, "paper_2003_03931_gb300")
PROF_LIB = os.path.join(PKG, "_build_phases", "libpmpm_phases.so")

# the intervals that the marks of k_column close, in a layer's order
PHASES = ["forward, tables | gather", "  wait", "z sum", "  wait", "inverse y", "inverse x", "  (deposit loads)",
          "deposit", "own loads", "  wait"]
N_MARKS, WARPS = 12, 8


def main(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--workload", default="c3_512")
    ap.add_argument("--steps", type=int, nargs="+", default=[1, 10, 20])
    args = ap.parse_args(argv)
    from paper_2003_03931_gb300 import build
    build.build(defines=("PMPM_PHASE_CLOCKS",), lib=PROF_LIB,
                build_dir=os.path.join(PKG, "_build_phases"))
    from paper_2003_03931_gb300 import _lib
    _lib.LIB_PATH = PROF_LIB
    from paper_2003_03931_gb300 import synth
    from paper_2003_03931_gb300.sim import SimConfig, Simulation
    w = dict(synth.WORKLOADS[args.workload])
    w["n_steps"] = max(w["n_steps"], max(args.steps) + 1)
    sim = Simulation(SimConfig(**w))
    sim.ic_zeldovich(1, **synth.IC_SPECTRUM)
    sim.lib.pmpm_debug_phases.argtypes = [ctypes.c_void_p, ctypes.c_int]
    buf = np.zeros(WARPS * N_MARKS, np.uint64)
    for step in sorted(args.steps):
        while sim.fetch_scalars()["step"] < step:
            sim.step(1)
        sim.sync()
        sim.lib.pmpm_debug_phases(buf.ctypes.data, buf.size)   # clears
        sim.step(1)
        sim.sync()
        sim.lib.pmpm_debug_phases(buf.ctypes.data, buf.size)
        b = buf.reshape(WARPS, N_MARKS).astype(np.float64)
        layers = b[:, 10:11].max()
        b = b[:, :len(PHASES)] / layers
        print(f"step {step}: {int(layers)} layers walked, {b.sum(axis=1).mean():.0f} cycles a layer")
        print("  %-30s" % "warp" + "".join(f"{i:7d}" for i in range(WARPS)))
        for i, name in enumerate(PHASES):
            print("  %-30s" % name + "".join(f"{v:7.0f}" for v in b[:, i]))
    sim.close()


if __name__ == "__main__":
    sys.exit(main())
