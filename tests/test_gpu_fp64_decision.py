"""Steps v-vii of an FP64 run where its FP32 shortcuts end: rates beyond FP32's
range in the draw u < P. Only kmc_run takes the shortcut (kmc_debug_step returns P
itself), so whole runs are compared with the oracle's.

Tolerance: the FP64 run's (moments 1e-9 after some dozens of steps, the draws
equal, which a single other decision breaks by far).
"""
import numpy as np
import pytest

import oracle
from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1407_2737_gb300 import build as kbuild
    kbuild.build()


@pytest.mark.parametrize("ratio", [1e37, 3e38, 1e39, 1e45, 1e-37, 1e-45])
def test_step_lengths_beyond_fp32(ratio):
    # barriers of 0 to 6 kT: nu0 t_step of 1e39 puts one rate, both or their sum
    # above FP32's largest number, and 1e-45 puts both below its smallest
    S, periods, tau0 = 20, 2, 1e-10
    ly = inputs.make_lysosome(200, 5e-9, 0.02, Ms=1e6, Keff=1.6e5, T=300.0, tau0=tau0, seed=4)
    f = 1.0 / (S * ratio * tau0)
    o = oracle.run(ly, 0, 0.15, f, S, periods, 0, 11, nthreads=4)
    ctx = kmc.kmc_create([ly], kmc.KMC_FP64_PLAIN, center=np.zeros(3))
    kmc.kmc_run(ctx, 0.15, f, S, periods, 0, 11)
    jumps, near = kmc.kmc_read(ctx, kmc.KMC_READ_COUNTERS, 0)[:2]
    m = kmc.kmc_read(ctx, kmc.KMC_READ_MOMENTS, 0)
    loop = kmc.kmc_read(ctx, kmc.KMC_READ_LOOP_M, 0)
    kmc.kmc_destroy(ctx)
    assert near == 0 and jumps == o["counters"]["flips"]
    assert jumps > 500 if ratio > 1 else jumps == 0
    assert np.max(np.abs(m - o["m"])) <= 1e-9
    np.testing.assert_allclose(loop, o["loop_M"], rtol=0, atol=1e-9)
