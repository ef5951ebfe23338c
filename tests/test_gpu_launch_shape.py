"""Launch shapes as a whole (kmc_launch_shape): what the autotuner took in one
process is read there and set in another one, which continues its checkpoint bit
for bit, for each kind of shape; and what no kernel of a context runs, or a pin
forbids, is refused and leaves the shape as it was.
"""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
F64, F32 = kmc.KMC_FP64_PLAIN, kmc.KMC_FP32_MIXED


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1407_2737_gb300 import build as kbuild
    kbuild.build()


CHILD = r'''
import json, os, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
from paper_1407_2737_gb300 import inputs, kmc
prec, sizes, out = int(sys.argv[2]), json.loads(sys.argv[3]), sys.argv[4]
lyss = [inputs.make_lysosome(n, 12e-9, 0.05, seed=n) for n in sizes]
ctx = kmc.kmc_create(lyss, prec, center=np.zeros(3))
if "KMC_TUNE_BAL" in os.environ:  # (of the symmetric form; the ordered one may be faster)
    kmc.kmc_pair_form(ctx, kmc.FORM_SYMMETRIC)
kmc.kmc_run(ctx, 0.02, 1e5, 30, 1, 0, 5)
kmc.kmc_save(ctx, out + ".state")
kmc.kmc_run(ctx, 0.02, 1e5, 30, 1, 0, 6)
np.savez(out, *[kmc.kmc_read(ctx, w, q) for q in range(len(sizes))
                for w in (kmc.KMC_READ_MOMENTS, kmc.KMC_READ_LOOP_M, kmc.KMC_READ_NP_ENERGY)])
print(json.dumps(kmc.kmc_launch_shape(ctx)))
'''


@pytest.mark.parametrize("prec,sizes,env,field,value", [
    (F64, [300, 129, 40], "KMC_TUNE_F64", "fp64_parts", 1),
    (F64, [300, 129, 40], "KMC_TUNE_F64", "fp64_parts", 16),
    (F32, [700, 130], "KMC_TUNE_BAL", "balanced", 4),
    (F32, [100, 45], "KMC_TUNE_CLUSTER", "cluster_period", 1),
    (F32, [300, 200], None, None, None)])
def test_a_shape_moves_to_another_process(prec, sizes, env, field, value, tmp_path):
    out = str(tmp_path / "run.npz")
    e = dict(os.environ)
    if env:
        e[env] = str(value)
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT, str(prec), json.dumps(sizes), out],
                       env=e, capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-3000:]
    shape = json.loads(r.stdout.strip().splitlines()[-1])
    assert field is None or shape[field] == value
    lyss = [inputs.make_lysosome(n, 12e-9, 0.05, seed=n) for n in sizes]
    ctx = kmc.kmc_create(lyss, prec, center=np.zeros(3))
    assert set(kmc.kmc_launch_shape(ctx).values()) == {0}
    assert kmc.kmc_launch_shape(ctx, shape) == shape
    kmc.kmc_load(ctx, out + ".state")
    kmc.kmc_run(ctx, 0.02, 1e5, 30, 1, 0, 6)
    got = [kmc.kmc_read(ctx, w, q) for q in range(len(sizes))
           for w in (kmc.KMC_READ_MOMENTS, kmc.KMC_READ_LOOP_M, kmc.KMC_READ_NP_ENERGY)]
    assert kmc.kmc_launch_shape(ctx) == shape
    kmc.kmc_destroy(ctx)
    with np.load(out) as want:
        assert all(np.array_equal(want[k], g) for k, g in zip(want.files, got))


def _shape(**kw):
    s = dict.fromkeys(kmc.SHAPE_KEYS, 0)
    s.update(warps=4, tile=64, tpl=1, rpl=1)
    s.update(kw)
    return s


SYM = dict(tile=32, tpl=2, sym_cells=1)
CLU = dict(warps=8, cluster_period=1)


@pytest.mark.parametrize("prec,n,kw", [
    (F32, 40, dict(warps=7, rpl=7)), (F32, 40, dict(rpl=2, warps=2)), (F32, 40, dict(tpl=0)),
    (F32, 40, dict(tpl=5)), (F32, 40, dict(chunk=100)), (F32, 40, dict(tile=48)),
    (F32, 40, dict(fp64_parts=1, tile=32)), (F32, 40, dict(SYM, fp64_parts=1)),
    (F32, 40, dict(SYM, balanced=-1)), (F32, 40, dict(SYM, balanced=65)),
    (F32, 40, dict(SYM, balanced=1, chunk=64)), (F32, 40, dict(SYM, cluster=2)),
    (F32, 40, dict(balanced=1)), (F32, 40, dict(sym_update=1)), (F32, 40, dict(cluster=1)),
    (F32, 40, dict(CLU, persistent=1)), (F32, 40, dict(CLU, tile=32)), (F32, 513, CLU),
    (F64, 40, CLU), (F64, 40, SYM), (F64, 40, dict(persistent=1)),
    (F64, 40, dict(tile=32, fp64_parts=3)), (F64, 40, dict(tile=32, fp64_parts=32)),
    (F64, 20000, dict(tile=32, fp64_parts=4))])
def test_refused_shapes(prec, n, kw):
    ly = inputs.lattice_nodes_lysosome(n, 14e-9, 0.1, seed=1)
    ctx = kmc.kmc_create([ly], prec, center=np.zeros(3))
    before = kmc.kmc_launch_shape(ctx, _shape(warps=8))
    with pytest.raises(kmc.KmcError) as e:
        kmc.kmc_launch_shape(ctx, _shape(**kw))
    assert e.value.status == kmc.KMC_EINVAL
    assert kmc.kmc_launch_shape(ctx) == before
    assert set(kmc.kmc_launch_shape(ctx, _shape(warps=0)).values()) == {0}
    kmc.kmc_destroy(ctx)


def test_shapes_keep_to_the_pins():
    ly = inputs.make_lysosome(200, 12e-9, 0.05, seed=3)
    for pin, mode, bad, good in (
            (kmc.kmc_persistent, 1, CLU, {}), (kmc.kmc_persistent, 2, {}, dict(persistent=1)),
            (kmc.kmc_pair_form, 1, SYM, CLU), (kmc.kmc_pair_form, 2, {}, SYM),
            (kmc.kmc_targets_per_lane, 2, {}, SYM), (kmc.kmc_sym_update, 2, SYM, {}),
            (kmc.kmc_cluster_split, 2, {}, dict(cluster=2, chunk=128))):
        ctx = kmc.kmc_create([ly], F32, center=np.zeros(3))
        pin(ctx, mode)
        with pytest.raises(kmc.KmcError) as e:
            kmc.kmc_launch_shape(ctx, _shape(**bad))
        assert e.value.status == kmc.KMC_EINVAL
        kmc.kmc_launch_shape(ctx, _shape(**good))
        kmc.kmc_destroy(ctx)


@pytest.mark.parametrize("mode", [1, 2])
def test_a_pinned_period_drops_the_clusters(mode):
    # in either order: pinned before tuning, the mode keeps the cluster period out
    ly = inputs.make_lysosome(90, 12e-9, 0.05, seed=3)
    ctx = kmc.kmc_create([ly], F32, center=np.zeros(3))
    kmc.kmc_launch_shape(ctx, _shape(**CLU))
    kmc.kmc_persistent(ctx, mode)
    kmc.kmc_run(ctx, 0.02, 1e5, 10, 1, 0, 5)
    s = kmc.kmc_launch_shape(ctx)
    assert s["cluster_period"] == 0 and (s["persistent"] == 0 or mode == 2)
    kmc.kmc_destroy(ctx)
