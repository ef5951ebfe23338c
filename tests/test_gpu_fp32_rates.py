"""FP32-mixed steps at step lengths that put a rate, both or their sum beyond FP32's
range: P, against the oracle's, within the FP32 step's bound (2e-3, fields of 1e-5),
and whole runs that hold no NP back."""
import numpy as np
import pytest

import oracle
from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [dict(warps=8, tile=64), dict(warps=4, tile=32, tpl=2, sym_cells=1)])
@pytest.mark.parametrize("ratio", [1e37, 3e38, 1e39, 1e45, 1e200, 1e-45, 1e-200])
def test_step_lengths_beyond_fp32(ratio, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    tau0 = 1e-10
    ly = inputs.make_lysosome(200, 5e-9, 0.02, Ms=1e6, Keff=1.6e5, T=300.0, tau0=tau0, seed=4)
    ctx = kmc.kmc_create([ly], kmc.KMC_FP32_MIXED, center=np.zeros(3))
    kmc.kmc_launch_shape(ctx, dict(dict.fromkeys(kmc.SHAPE_KEYS, 0), tpl=1, rpl=1) | shape)
    m = oracle.initial_moments(ly.axis).astype(np.float32).astype(np.float64)
    P = []
    for k in range(8):
        H = 0.15 * np.cos(2 * np.pi * k / 8)
        g = kmc.kmc_debug_step(ctx, [H], ratio * tau0, 11, k, m)
        o = oracle.step(ly, 0, m, H, ratio * tau0, 11, k)
        assert np.max(np.abs(g["P"] - o["P"])) < 2e-3
        P.append(o["P"])
        m = g["m_out"]
    assert (np.ptp(P) > 0.9) == (ratio > 1)
    kmc.kmc_run(ctx, 0.15, 1.0 / (8 * ratio * tau0), 8, 2, 0, 11)
    kmc.kmc_sync(ctx)
    cnt = kmc.kmc_read(ctx, kmc.KMC_READ_COUNTERS, 0)
    assert cnt[kmc.CNT_NONFINITE] == 0 and (cnt[kmc.CNT_JUMPS] > 500) == (ratio > 1)
    kmc.kmc_destroy(ctx)
