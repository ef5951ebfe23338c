"""The benchmark names the kernel that ran and counts its launches: shapes that share
warps, tile and chunk are told apart."""
import importlib.util
import os

import numpy as np
import pytest

from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BASE = dict(dict.fromkeys(kmc.SHAPE_KEYS, 0), warps=8, tile=64, tpl=1, rpl=1)
SYM = dict(BASE, warps=4, tile=32, tpl=2, sym_cells=1)


@pytest.mark.parametrize("shape,kernel,launches", [
    (BASE, "kmc_step_f32<8>", 20), (dict(BASE, cluster_period=1), "kmc_cluster_f32<8>", 1),
    (dict(BASE, persistent=1), "kmc_persist_f32<8>", 1),
    (SYM, "kmc_field_sym<4, 1> + kmc_update_sym<4>", 40),
    (dict(SYM, balanced=2, sym_update=1), "kmc_field_sym<4, 1> + kmc_update_sym_block<4>", 40)])
def test_launch_info(shape, kernel, launches):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    spec = importlib.util.spec_from_file_location("bench_mod", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    ly = inputs.make_lysosome(100, 12e-9, 0.05, seed=1)
    ctx = kmc.kmc_create([ly], kmc.KMC_FP32_MIXED, center=np.zeros(3))
    kmc.kmc_launch_shape(ctx, shape)
    kmc.kmc_run(ctx, 0.02, 1e5, 20, 1, 0, 1)
    info = bench.launch_info(kmc, ctx, [ly])
    kmc.kmc_destroy(ctx)
    assert info["kernel"] == kernel and info["launches_per_period"](20) == launches
    assert info["launch"].get("balanced", 0) == shape["balanced"]
