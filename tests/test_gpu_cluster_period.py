"""A field period of small lysosomes as one cluster launch (the autotuner's option
up to 512 NPs) against the per-step kernel at the same warps with all records in
one tile: bit for bit, over runs with discarded and recorded periods, at the edges
of its groups of 32 targets and of the cluster sizes, for one lysosome and for
batches whose lysosomes need fewer blocks than the largest, at T = 0, and for NPs at
one point. The step's own parity with the oracle is the existing tests'; one debug
step is checked here too.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import os, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import oracle
from paper_1407_2737_gb300 import inputs, kmc

def outputs(lyss, pinned, S):
    ctx = kmc.kmc_create(lyss, kmc.KMC_FP32_MIXED, center=np.zeros(3))
    if pinned:
        kmc.kmc_tuning(ctx, 8, 256, 0)
    H = np.linspace(0.015, 0.04, len(lyss))
    out = []
    for seed in (3, 4):  # moments and steps carry over
        kmc.kmc_run(ctx, H, 1e5, S, 3, 1, seed)
        try:
            kmc.kmc_sync(ctx)
        except kmc.KmcError as e:
            out.append(np.array([e.status]))
        for q in range(len(lyss)):
            for what in (kmc.KMC_READ_MOMENTS, kmc.KMC_READ_COUNTERS):
                out.append(kmc.kmc_read(ctx, what, q))
            if len(out[0]) > 1:
                for what in (kmc.KMC_READ_LOOP_M, kmc.KMC_READ_NP_ENERGY, kmc.KMC_READ_DHDIP):
                    out.append(kmc.kmc_read(ctx, what, q))
    kmc.kmc_destroy(ctx)
    return out

def sample(n, T=300.0):
    ly = inputs.lattice_nodes_lysosome(n, 14e-9, 0.1, Keff=2e4, T=T, seed=n)
    rng = np.random.default_rng(n)
    ly.pos = inputs.snap_to_float32(ly.pos + 1e-9 * rng.normal(size=ly.pos.shape), 14e-9)
    return ly

cases = [[sample(n)] for n in (1, 2, 31, 32, 33, 100, 255, 256, 257, 511, 512)]
cases += [[sample(5), sample(100), sample(64, T=0.0)], [sample(40 + 7 * q) for q in range(20)]]
twice = sample(70)
twice.pos[3] = twice.pos[60]
cases.append([twice])
for lyss in cases:
    for S in (1, 2, 25):
        got = outputs(lyss, False, S)
        want = outputs(lyss, True, S)
        assert len(got) == len(want)
        assert all(np.array_equal(g, w, equal_nan=True) for g, w in zip(got, want)), (
            [l.n for l in lyss], S)
ly = cases[5][0]
m = (oracle.initial_moments(ly.axis)).astype(np.float32).astype(np.float64)
ctx = kmc.kmc_create([ly], kmc.KMC_FP32_MIXED, center=np.zeros(3))
g = kmc.kmc_debug_step(ctx, [0.012], 5e-8, 5, 7, m)
o = oracle.step(ly, 0, m, 0.012, 5e-8, 5, 7)
rms = np.sqrt(np.mean(np.sum(o["B_dip"] ** 2, axis=1)))
assert np.max(np.linalg.norm(g["B_dip"] - o["B_dip"], axis=1)) <= 1e-5 * rms
assert np.array_equal(g["u"], o["u"])
print("cluster ok")
'''


def test_bits_of_the_per_step_kernel():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1407_2737_gb300 import build as kbuild
    lib = kbuild.build()
    env = dict(os.environ, KMC_LIB_PATH=lib, KMC_TUNE_CLUSTER="1")
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], env=env, capture_output=True,
                       text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0 and "cluster ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
