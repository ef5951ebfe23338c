"""Balanced plans of the symmetric pair form (items of about equal work that may
start and end inside a cell of 64 NPs), which the autotuner times beside the
whole-cell ones: the field of every NP against the oracle's, at sizes with one
cell, one row group, ragged last cells and several chains, with few and with many
items, in the debug build too. A pair left out, taken twice or gathered from the
wrong slot moves some NP's field by far more than the FP32 tolerance (1e-5 of the
rms field, the step's). Only these plans are timed here (an environment variable);
the two update kernels add the slots in different orders, and both run.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import oracle
from paper_1407_2737_gb300 import inputs, kmc

for sizes in ([1], [65], [600], [2000], [130, 700, 64, 1500, 1]):
    lyss = [inputs.lattice_nodes_lysosome(n, 14e-9, 0.1, seed=n) for n in sizes]
    rng = np.random.default_rng(1)
    m = np.concatenate([oracle.initial_moments(l.axis) + 0.3 * rng.normal(size=(l.n, 3))
                        for l in lyss])
    m /= np.linalg.norm(m, axis=1, keepdims=True)
    m = m.astype(np.float32).astype(np.float64)
    for tpl in (2, 4):
        for upd in (1, 2):
            ctx = kmc.kmc_create(lyss, kmc.KMC_FP32_MIXED, center=np.zeros(3))
            kmc.kmc_pair_form(ctx, kmc.FORM_SYMMETRIC)
            kmc.kmc_targets_per_lane(ctx, tpl)
            kmc.kmc_sym_update(ctx, upd)
            g = kmc.kmc_debug_step(ctx, np.full(len(sizes), 0.01), 5e-8, 1, 2, m)
            off = 0
            for l in lyss:
                B = oracle.dipolar_field(l.pos, l.vol, l.Ms, m[off:off + l.n])
                rms = np.sqrt(np.mean(np.sum(B ** 2, axis=1))) or 1.0
                e = np.max(np.linalg.norm(g["B_dip"][off:off + l.n] - B, axis=1))
                assert e <= 1e-5 * rms, (sizes, tpl, upd, l.n, e / rms)
                off += l.n
            kmc.kmc_run(ctx, 0.02, 1e5, 10, 2, 1, 5)
            kmc.kmc_sync(ctx)
            kmc.kmc_destroy(ctx)
print("balanced ok")
'''


@pytest.mark.parametrize("bal,debug", [(1, False), (2, False), (8, False), (1, True)])
def test_balanced_plans(bal, debug):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1407_2737_gb300 import build as kbuild
    lib = kbuild.build(debug=debug)
    env = dict(os.environ, KMC_LIB_PATH=lib, KMC_TUNE_BAL=str(bal))
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], env=env, capture_output=True,
                       text=True, timeout=900, cwd=ROOT)
    assert r.returncode == 0 and "balanced ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
