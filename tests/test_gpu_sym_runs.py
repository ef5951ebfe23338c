"""Whole runs of the symmetric plans that the autotuner may take, set by
kmc_launch_shape: FP64 parts against the oracle's runs, and every lysosome of a
batch against itself alone; balanced FP32 plans against the same steps launched one
by one. A run alone exercises the chains' offsets into items, updates and slots, and
the slots' reuse from step to step under programmatic launches.

Tolerances: those of an FP64 run (moments and loop 1e-9, the same jumps; a run with a
draw within 1e-9 of its probability is left out); the others are bit for bit.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1407_2737_gb300 import build as kbuild
    kbuild.build()


def _shape(**kw):
    s = dict.fromkeys(kmc.SHAPE_KEYS, 0)
    s.update(warps=4, tile=32, tpl=1, rpl=1)
    s.update(kw)
    return s


def _outputs(ctx, q):
    return [kmc.kmc_read(ctx, w, q) for w in (kmc.KMC_READ_MOMENTS, kmc.KMC_READ_LOOP_M,
                                              kmc.KMC_READ_NP_ENERGY, kmc.KMC_READ_COUNTERS)]


def _fp64_runs(parts):
    lyss = [inputs.make_lysosome(n, 12e-9, 0.05 if n > 3 else 0.01, Keff=1e4, seed=70 + n)
            for n in (300, 129, 65, 64, 33, 32, 31, 2, 1)]
    lyss[2].vol = lyss[2].vol * np.linspace(0.6, 1.4, lyss[2].n)
    lyss[4].T = 0.0
    ctx = kmc.kmc_create(lyss, kmc.KMC_FP64_PLAIN, center=np.zeros(3))
    kmc.kmc_launch_shape(ctx, _shape(fp64_parts=parts))
    kmc.kmc_run(ctx, 0.02, 1e5, 30, 2, 1, 5)
    got = [_outputs(ctx, q) for q in range(len(lyss))]
    assert kmc.kmc_launch_shape(ctx)["fp64_parts"] == parts
    kmc.kmc_destroy(ctx)
    compared = 0
    for q, ly in enumerate(lyss):
        o = oracle.run(ly, q, 0.02, 1e5, 30, 2, 1, 5, nthreads=4)
        if o["counters"]["near"]:
            continue
        compared += ly.n
        m, loop, _, cnt = got[q]
        assert cnt[kmc.CNT_JUMPS] == o["counters"]["flips"], (ly.n, parts)
        assert np.max(np.abs(m - o["m"])) <= 1e-9
        np.testing.assert_allclose(loop, o["loop_M"], rtol=0, atol=1e-9)
    assert compared > 300
    alone = kmc.kmc_create(lyss[:1], kmc.KMC_FP64_PLAIN, center=np.zeros(3))
    kmc.kmc_launch_shape(alone, _shape(fp64_parts=parts))
    kmc.kmc_run(alone, 0.02, 1e5, 30, 2, 1, 5)
    assert all(np.array_equal(a, b) for a, b in zip(_outputs(alone, 0), got[0]))
    assert got[0][3][kmc.CNT_JUMPS] > 0
    kmc.kmc_destroy(alone)


@pytest.mark.parametrize("parts", [1, 2, 4, 8, 16])
def test_fp64_parts_follow_the_oracle(parts):
    _fp64_runs(parts)


@pytest.mark.parametrize("sizes", [[1], [65], [700], [130, 700, 64, 1500, 1]])
@pytest.mark.parametrize("warps,cells", [(2, 2), (4, 1), (4, 2), (8, 1)])
def test_balanced_runs_are_their_steps(sizes, warps, cells):
    lyss = [inputs.lattice_nodes_lysosome(n, 14e-9, 0.1, Keff=1e4, seed=n) for n in sizes]
    vol = [l.vol / l.vol.sum() for l in lyss]
    off = np.concatenate([[0], np.cumsum(sizes)])
    for bal, supd in ((1, 0), (8, 1), (64, 0)):
        sh = _shape(warps=warps, tpl=2 * cells, sym_cells=cells, balanced=bal, sym_update=supd)
        run = kmc.kmc_create(lyss, kmc.KMC_FP32_MIXED, center=np.zeros(3))
        kmc.kmc_launch_shape(run, sh)
        kmc.kmc_run(run, 0.02, 1e5, 2, 4, 0, 5)  # the field is 20 and -20 mT: no rounding
        got = [_outputs(run, q) for q in range(len(lyss))]
        kmc.kmc_destroy(run)
        one = kmc.kmc_create(lyss, kmc.KMC_FP32_MIXED, center=np.zeros(3))
        kmc.kmc_launch_shape(one, sh)
        m = np.concatenate([kmc.kmc_read(one, kmc.KMC_READ_MOMENTS, q) for q in range(len(lyss))])
        loop, jumps = [], 0
        for k in range(8):
            g = kmc.kmc_debug_step(one, np.full(len(lyss), 0.02 * (1 - 2 * (k & 1))), 5e-6, 5, k, m)
            m = g["m_out"]
            jumps += g["flipped"].sum()
            loop.append([v @ m[a:b, 2] for v, a, b in zip(vol, off, off[1:])])
        kmc.kmc_destroy(one)
        assert np.array_equal(np.concatenate([g[0] for g in got]), m), (bal, supd)
        assert sum(g[3][kmc.CNT_JUMPS] for g in got) == jumps
        np.testing.assert_allclose([g[1] for g in got], np.transpose(loop), rtol=0, atol=1e-12)


def test_runs_of_the_debug_build():
    # bounds checks on every item, chain by chain
    from paper_1407_2737_gb300 import build as kbuild
    code = ("import sys; sys.path[:0] = [%r, %r]; import test_gpu_sym_runs as t; "
            "t._fp64_runs(4); t.test_balanced_runs_are_their_steps([130, 700, 1], 4, 2); "
            "print('debug ok')" % (ROOT, os.path.join(ROOT, "tests")))
    env = dict(os.environ, KMC_LIB_PATH=kbuild.build(debug=True))
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True,
                       timeout=600, cwd=ROOT)
    assert r.returncode == 0 and "debug ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
