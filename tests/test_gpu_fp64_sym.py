"""The symmetric pair form of FP64 contexts, which the autotuner times beside the
ordered kernels, at the edges of its cells of 32 NPs, its parts and its chains.

Tolerances: the FP64 step's (field within 1e-12 of sum_j |term_ij|, moments
1e-12). Which form the autotuner takes is a matter of timing, so the parts are
forced through the environment variable that names the candidates to time.
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

def batch():
    lyss = [inputs.make_lysosome(n, 12e-9, 0.05 if n > 3 else 0.01, seed=70 + n)
            for n in (1, 2, 31, 32, 33, 64, 65, 129, 300)]
    lyss[4].vol = lyss[4].vol * np.linspace(0.6, 1.4, lyss[4].n)
    lyss[5].T = 0.0
    return lyss

def moments(lyss):
    rng = np.random.default_rng(5)
    m = np.concatenate([oracle.initial_moments(l.axis) + 0.3 * rng.normal(size=(l.n, 3))
                        for l in lyss])
    return m / np.linalg.norm(m, axis=1, keepdims=True)

def terms(ly):
    d = ly.pos[None] - ly.pos[:, None]
    r = np.linalg.norm(d, axis=2)
    np.fill_diagonal(r, np.inf)
    w = 4e-7 * np.pi * ly.Ms * ly.vol / (4 * np.pi)
    return 4.0 * (w[None] / r ** 3).sum(axis=1)

lyss = batch()
m = moments(lyss)
ctx = kmc.kmc_create(lyss, kmc.KMC_FP64_PLAIN, center=np.zeros(3))
g = kmc.kmc_debug_step(ctx, np.full(len(lyss), 0.015), 5e-8, 3, 21, m)
assert kmc.kmc_pair_form(ctx) == kmc.FORM_SYMMETRIC
off = 0
for q, ly in enumerate(lyss):
    sl = slice(off, off + ly.n)
    off += ly.n
    o = oracle.step(ly, q, m[sl], 0.015, 5e-8, 3, 21)
    assert np.all(np.abs(g["B_dip"][sl] - o["B_dip"]) <= 1e-12 * terms(ly)[:, None] + 1e-300)
    assert np.array_equal(g["u"][sl], o["u"]) and np.array_equal(g["n_min"][sl], o["n_min"])
    ok = o["near"] == 0
    assert np.max(np.abs(g["m_out"][sl][ok] - o["m_out"][ok]), initial=0.0) <= 1e-12
# a run in chains; each lysosome alone gets the same bits
kmc.kmc_run(ctx, 0.02, 1e5, 30, 2, 1, 5)
kmc.kmc_sync(ctx)
got = [kmc.kmc_read(ctx, kmc.KMC_READ_MOMENTS, q) for q in range(len(lyss))]
kmc.kmc_destroy(ctx)
alone = kmc.kmc_create([lyss[0]], kmc.KMC_FP64_PLAIN, center=np.zeros(3))
kmc.kmc_debug_step(alone, [0.015], 5e-8, 3, 21, m[:1])
kmc.kmc_run(alone, 0.02, 1e5, 30, 2, 1, 5)
assert np.array_equal(kmc.kmc_read(alone, kmc.KMC_READ_MOMENTS, 0), got[0])
kmc.kmc_destroy(alone)
# two NPs at one point are skipped, as in the ordered kernel; pinning the
# ordered form leaves the symmetric one
two = inputs.make_lysosome(40, 12e-9, 0.05, seed=9)
two.pos[7] = two.pos[33]
m2 = moments([two])
B = []
for form in (0, kmc.FORM_ORDERED):
    ctx = kmc.kmc_create([two], kmc.KMC_FP64_PLAIN, center=np.zeros(3))
    if form:
        kmc.kmc_pair_form(ctx, form)
    B.append(kmc.kmc_debug_step(ctx, 0.01, 5e-8, 3, 2, m2)["B_dip"])
    assert kmc.kmc_pair_form(ctx) == (form or kmc.FORM_SYMMETRIC)
    kmc.kmc_destroy(ctx)
assert np.all(np.abs(B[0] - B[1]) <= 1e-12 * np.abs(B[1]).max())
# the failure-detection hook runs the ordered kernel and leaves the form as it was
ctx = kmc.kmc_create([two], kmc.KMC_FP64_PLAIN, center=np.zeros(3))
try:
    kmc.kmc_debug_stall(ctx)
except kmc.KmcError as e:
    assert e.status == kmc.KMC_ETIMEOUT
kmc.kmc_run(ctx, 0.02, 1e5, 10, 1, 0, 5)
kmc.kmc_sync(ctx)
assert kmc.kmc_pair_form(ctx) == kmc.FORM_SYMMETRIC
print("sym64 ok")
'''


@pytest.mark.parametrize("parts,debug", [(1, False), (4, False), (16, False), (2, True)])
def test_symmetric_form(parts, debug):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1407_2737_gb300 import build as kbuild
    lib = kbuild.build(debug=debug)
    env = dict(os.environ, KMC_LIB_PATH=lib, KMC_TUNE_F64=str(parts))
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], env=env, capture_output=True,
                       text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0 and "sym64 ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
